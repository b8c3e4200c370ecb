"""The fast sweep kernels against the staged sweep at the sizes where a tiling can go wrong:
one window, a window's edge, one row or column beyond it, remainders along z, many blocks."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -24


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_01701_gb300 import build as B
    B.build()
    import paper_2305_01701_gb300 as P
    return P


def _fields(P, nd, n, seed, h=None):
    """A history near yield: pure shear with noise, noisy velocities, shear zero on the walls.
    h: the edge of the cells (default: a box of edges near 1)."""
    rng = np.random.default_rng(seed)
    rates = [1.0, -1.0] if nd == 2 else [1.0, 0.0, -1.0]
    f = {}
    shape = {k: P.field_shape(nd, tuple(n) + (1,), k) for k in
             ["vx", "vy", "txx", "tyy", "txy", "p"] + (["vz", "tzz", "txz", "tyz"] if nd == 3 else [])}
    for d in range(nd):
        ax = nd - 1 - d
        x = np.arange(n[d] + 1) / n[d] - 0.5
        v = rates[d] * x.reshape([-1 if q == ax else 1 for q in range(nd)]) * np.ones(shape["v" + "xyz"[d]])
        f["v" + "xyz"[d]] = (v + 0.02 * rng.standard_normal(v.shape) if h is None else
                             v * n[d] * h + h * rng.standard_normal(v.shape))
        c = shape["t" + "xyz"[d] * 2]
        f["t" + "xyz"[d] * 2] = (1.2e-3 if nd == 2 else 1.7e-3) * rates[d] + 1e-4 * rng.standard_normal(c)
    for k, walls in (("txy", (0, 1)), ("txz", (0, 2)), ("tyz", (1, 2))):
        if k in shape:
            t = 1e-4 * rng.standard_normal(shape[k])
            for d in walls:
                ax = nd - 1 - d
                t[tuple(slice(None) if q != ax else [0, -1] for q in range(nd))] = 0.0
            f[k] = t
    f["p"] = 1e-4 * rng.standard_normal(shape["p"])
    return f


def _solve(P, nd, n, precision, kernel, iters, f, shape=-1, **opts):
    opts = dict(opts)
    force = opts.pop("force", 0.0)
    cohesion = 1.5e-3 * (1e3 if opts.pop("elastic", False) else 1.0)
    pending = opts.pop("pending", 0)   # commit after so many chunks, the solve undecided
    g = P.Grid(nd, n, L=opts.pop("L", (1.0, 0.8, 1.3)[:nd]), precision=precision)
    rng = np.random.default_rng(1)
    g.set_material(2.0, 1.0, opts.pop("mu_s", math.inf), 30.0, 0.0, cohesion * (1 + 0.01 * rng.standard_normal(int(np.prod(n)))))
    if "cell_g" in opts:
        g.set_shear_modulus(1.0 + 0.2 * opts.pop("cell_g") * rng.random(int(np.prod(n))))
    g.set_solver(tol=0.0, max_iter=iters, n_chk=opts.pop("chunk", iters // 2), **opts)
    g.set_kernel(kernel, shape)
    for k, a in f.items():
        g.set(k, a)
    bf = force * rng.standard_normal(sum(f["v" + c].size for c in "xyz"[:nd])) if force else None
    g.apply_increment(1.0, 1e-4, P.LOAD_XY if nd == 2 else P.LOAD_XZ, bf)
    info = g.solve_chunks(pending) if pending else g.solve_increment(raise_on_fail=False)
    g.commit_increment()
    out = {k: g.get(k) for k in list(f) + ["epl", "scale"]}
    g.close()
    return info, out


def _compare(f, out, ref, info, iref, iters, eps):
    """Both sweeps round every state value once or twice per iteration in another order: over
    `iters` iterations the difference stays below 4 iters ulp of the field group's scale (each
    rounding decays with the relaxation; the sum of all of them bounds it)."""
    bound = 4 * iters * eps
    groups = [[k for k in f if k[0] == "v"], [k for k in f if k[0] != "v"]]
    for names in groups:
        scale = max(np.abs(ref[k]).max() for k in names)
        for k in names:
            err = np.abs(out[k] - ref[k]).max() / scale
            assert err <= bound, (k, err, bound)
    plastic = ref["scale"] < 1.0
    assert plastic.any() and not plastic.all()
    assert np.abs(out["scale"] - ref["scale"]).max() <= bound * 10
    for k in ("max_sigma", "eps_rel"):
        assert abs(info[k] - iref[k]) <= 100 * bound * abs(iref[k]), (k, info[k], iref[k])


@pytest.mark.parametrize("n,kz", [((27, 19, 5), 0), ((28, 20, 6), 0), ((29, 21, 7), 3), ((31, 3, 9), 0), ((1, 45, 4), 0),
                                  ((84, 61, 2), 1), ((63, 47, 33), 0), ((90, 64, 21), 8), ((35, 130, 1), 0)])
def test_register_sweep_matches_the_staged_sweep_at_tile_edges_fp32(P, n, kz):
    iters = 20
    f = _fields(P, 3, n, 7)
    iref, ref = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_STAGED, iters, f)
    info, out = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_FUSED_REG, iters, f, shape=kz)
    _compare(f, out, ref, info, iref, iters, EPS32)


@pytest.mark.parametrize("n", [(27, 11, 5), (28, 12, 6), (29, 13, 7), (57, 25, 12), (90, 64, 21)])
@pytest.mark.parametrize("mu_s", [math.inf, 1e-3])
def test_register_sweep_with_a_per_cell_modulus_matches_the_staged_sweep_fp32(P, n, mu_s):
    iters = 20
    f = _fields(P, 3, n, 8)
    iref, ref = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_STAGED, iters, f, cell_g=1.0, mu_s=mu_s)
    info, out = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_AUTO, iters, f, cell_g=1.0, mu_s=mu_s)
    _compare(f, out, ref, info, iref, iters, EPS32)


@pytest.mark.parametrize("n,rows", [((30, 4), 0), ((31, 5), 0), ((32, 33), 3), ((62, 64), 4), ((63, 7), 0), ((2, 9), 3),
                                    ((300, 180), 3)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("opts", [{}, {"mu_s": 1e-3, "jaumann": False}, {"incompressible": True}])
def test_sweep_2d_matches_the_fused_sweep_at_strip_edges(P, n, rows, precision, opts):
    iters = 20
    f = _fields(P, 2, n, 5)
    pr = P.FP64 if precision == "fp64" else P.FP32_MIXED
    iref, ref = _solve(P, 2, n, pr, P.KERNEL_FUSED, iters, f, shape=rows, **opts)
    info, out = _solve(P, 2, n, pr, P.KERNEL_AUTO, iters, f, **opts)
    _compare(f, out, ref, info, iref, iters, 2.0 ** -53 if precision == "fp64" else EPS32)


@pytest.mark.parametrize("n", [(31, 7, 3), (32, 8, 2), (33, 9, 4), (64, 17, 5), (20, 70, 12)])
@pytest.mark.parametrize("opts", [{}, {"mu_s": 1e-3, "jaumann": False}, {"incompressible": True}])
def test_fp64_sweep_3d_matches_the_register_sweep_at_warp_edges(P, n, opts):
    iters = 20
    f = _fields(P, 3, n, 6)
    iref, ref = _solve(P, 3, n, P.FP64, P.KERNEL_FUSED_REG, iters, f, shape=0, **opts)
    info, out = _solve(P, 3, n, P.FP64, P.KERNEL_STAGED, iters, f, **opts)
    _compare(f, out, ref, info, iref, iters, 2.0 ** -53)


@pytest.mark.parametrize("n", [(58, 31), (59, 32), (60, 33), (61, 63), (119, 64), (120, 65), (121, 3)])
@pytest.mark.parametrize("tile", [3, 4])
@pytest.mark.parametrize("opts", [{}, {"mu_s": 1e-3, "jaumann": False}, {"freeze_iter": 5}])
def test_batched_strips_of_column_pairs_match_the_staged_sweep_fp32(P, n, tile, opts):
    iters = 20
    f = _fields(P, 2, n, 9)
    iref, ref = _solve(P, 2, n, P.FP32_MIXED, P.KERNEL_STAGED, iters, f, **opts)
    info, out = _solve(P, 2, n, P.FP32_MIXED, P.KERNEL_FUSED, iters, f, shape=tile, **opts)
    _compare(f, out, ref, info, iref, iters, EPS32)


@pytest.mark.parametrize("nd,n", [(2, (31, 300)), (2, (64, 7)), (3, (33, 5, 260)), (3, (28, 20, 6))])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_commit_history_copies_and_line_integrals(P, nd, n, precision):
    """The commit's trial near the yielding centres against the trial of every point (formed
    while the warm-start targets are recorded), the copies of a restore, the column integrals."""
    f = _fields(P, nd, n, 10)
    g = P.Grid(nd, n, L=(1.0, 0.8, 1.3)[:nd], precision=P.FP64 if precision == "fp64" else P.FP32_MIXED)
    g.set_material(2.0, 1.0, math.inf, 30.0, 0.0, np.full(int(np.prod(n)), 1.5e-3))
    g.set_solver(tol=2e-2, max_iter=50000, n_chk=10)
    for k, a in f.items():
        g.set(k, a)
    g.snapshot()
    names = list(f) + ["epl", "ux", "exx", "exy"]
    start = {k: g.get(k) for k in names}
    outs = []
    for on in (0, 1):
        g.warm_record(on)
        g.apply_increment(1.0, 1e-4, P.LOAD_XY if nd == 2 else P.LOAD_XZ)
        info = g.solve_increment()
        outs.append(({k: g.get(k) for k in names + ["scale"]}, (info["sxx_int_centre"], info["sxx_int_right"])))
        g.restore()
        for k in names:
            np.testing.assert_array_equal(g.get(k), start[k])
    (a, la), (b, lb) = outs
    assert (a["scale"] < 1.0).any() and (a["epl"] > 0.0).any() and (a["epl"] == 0.0).any()
    for k in a:
        np.testing.assert_array_equal(a[k], b[k])
    assert la == lb
    sxx = a["txx"] - a["p"]
    cols = (sxx[:, n[0] // 2], sxx[:, -1]) if nd == 2 else (sxx[:, n[1] // 2, n[0] // 2], sxx[:, n[1] // 2, -1])
    h = 0.8 / n[1] if nd == 2 else 1.3 / n[2]
    for got, c in zip(la, cols):
        assert abs(got - math.fsum(c * h)) <= len(c) * 2.0 ** -52 * np.abs(c * h).sum()
    g.close()


@pytest.mark.parametrize("n", [(11, 3), (12, 4), (13, 5), (24, 25), (64, 64), (27, 90), (171, 140), (300, 180), (383, 191)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("opts", [{}, {"mu_s": 1e-3, "jaumann": False, "incompressible": True}, {"freeze_iter": 5},
                                  {"force": 1e-3}])
def test_resident_2d_iterations_equal_the_two_launch_sweep(P, n, precision, opts):
    """One launch per chunk against two per iteration: the same operations, equal bits, at the
    edges of every lattice, over several chunks; the largest grids take two launches again."""
    iters = 24
    f = _fields(P, 2, n, 11)
    pr = P.FP64 if precision == "fp64" else P.FP32_MIXED
    iref, ref = _solve(P, 2, n, pr, P.KERNEL_STAGED, iters, f, chunk=6, **opts)
    info, out = _solve(P, 2, n, pr, P.KERNEL_AUTO, iters, f, chunk=6, **opts)
    for k in out:
        np.testing.assert_array_equal(out[k], ref[k])
    for k in ("iters", "max_sigma", "eps_rel", "eps_res"):
        assert info[k] == iref[k]


@pytest.mark.parametrize("n", [(3, 2, 2), (15, 15, 1), (27, 19, 5), (31, 9, 33), (90, 40, 24), (70, 30, 40)])
@pytest.mark.parametrize("opts", [{}, {"mu_s": 1e-3, "jaumann": False, "incompressible": True}, {"freeze_iter": 6}])
def test_resident_3d_iterations_match_the_staged_sweep_fp32(P, n, opts):
    """One launch per chunk: blocks of one point and of many, remainders in each direction."""
    iters = 24
    f = _fields(P, 3, n, 12)
    iref, ref = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_STAGED, iters, f, chunk=6, **opts)
    info, out = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_AUTO, iters, f, chunk=6, **opts)
    _compare(f, out, ref, info, iref, iters, EPS32)


@pytest.mark.parametrize("nd,n,precision", [(2, (24, 25), "fp64"), (2, (64, 64), "fp64"), (2, (300, 180), "fp32"),
                                            (3, (27, 19, 5), "fp32"), (3, (90, 40, 24), "fp32")])
@pytest.mark.parametrize("chunk", [2, 4, 10])
def test_commit_of_an_undecided_solve_takes_the_newest_iterate(P, nd, n, precision, chunk):
    """Whole chunks, then a commit while the stopping test has not decided: the resident kernels
    leave the state where the launch-per-iteration sweeps do."""
    iters = 20
    f = _fields(P, nd, n, 13)
    pr = P.FP64 if precision == "fp64" else P.FP32_MIXED
    (iref, ref), (info, out) = (_solve(P, nd, n, pr, k, 1000, f, chunk=chunk, pending=iters // chunk)
                                for k in (P.KERNEL_STAGED, P.KERNEL_AUTO))
    assert info["status"] == iref["status"] == P.PENDING
    if nd == 2:
        for k in out:
            np.testing.assert_array_equal(out[k], ref[k])
    else:
        _compare(f, out, ref, info, iref, iters, EPS32)


@pytest.mark.parametrize("n", [(27, 11, 5), (40, 33, 14)])
def test_commit_of_an_undecided_solve_with_a_per_cell_modulus(P, n):
    """The register sweep stores its return scales at checks; with a per-cell modulus also in the
    last iteration of a chunk, where the staged sweep has them: the commit of the undecided solve
    adds plastic strain to the same cells."""
    iters = 20
    f = _fields(P, 3, n, 14)
    kw = dict(chunk=10, pending=2, cell_g=1.0)
    iref, ref = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_STAGED, 1000, f, **kw)
    info, out = _solve(P, 3, n, P.FP32_MIXED, P.KERNEL_AUTO, 1000, f, **kw)
    assert info["status"] == iref["status"] == P.PENDING
    _compare(f, out, ref, info, iref, iters, EPS32)
    # a cell within rounding of yield may return on one side only
    differ = np.count_nonzero((out["epl"] > 0.0) != (ref["epl"] > 0.0))
    assert differ <= max(1, out["epl"].size // 1000), differ


@pytest.mark.parametrize("n", [(61, 33), (130, 90), (300, 180)])
def test_elastic_iterations_without_rotation_round_alike_in_every_fp32_2d_kernel(P, n):
    """The deviatoric rate is formed first and scaled once, in one order: strips, the launches per
    iteration and the resident iterations give the same bits where neither the return nor the
    rotation's means (whose sums each kernel shares in its own way) take part.  (In FP64 the
    compiler contracts the strips' products and sums, which are not packed there.)"""
    f = _fields(P, 2, n, 15)
    opts = dict(chunk=6, jaumann=False, elastic=True)
    _, ref = _solve(P, 2, n, P.FP32_MIXED, P.KERNEL_FUSED, 24, f, shape=4, **opts)
    for kernel in (P.KERNEL_STAGED, P.KERNEL_AUTO):
        _, out = _solve(P, 2, n, P.FP32_MIXED, kernel, 24, f, **opts)
        for k in out:
            np.testing.assert_array_equal(out[k], ref[k])


@pytest.mark.parametrize("nd,n,precision,kernel", [
    (3, (60, 33, 14), "fp32", "KERNEL_FUSED_REG"), (3, (60, 33, 14), "fp64", "KERNEL_FUSED_REG"),
    (3, (40, 33, 14), "fp32", "KERNEL_AUTO"),      # its check runs the register sweep
    (2, (64, 50), "fp64", "KERNEL_AUTO"), (2, (64, 50), "fp32", "KERNEL_AUTO"), (2, (300, 180), "fp32", "KERNEL_AUTO")])
def test_waits_that_run_out_end_the_solve_with_timeout(P, nd, n, precision, kernel):
    """A bound of 8 cycles, far below the latency of a plane's copy or of an exchanged word, ends
    the solve with EP_ERR_TIMEOUT; with the default bound back the grid solves as an untouched
    one.  Bounds around those latencies may end it or not, and leave the grid as usable."""
    f = _fields(P, nd, n, 16)
    rng = np.random.default_rng(1)
    coh = 1.5e-3 * (1 + 0.01 * rng.standard_normal(int(np.prod(n))))
    grids = []
    for _ in range(2):
        g = P.Grid(nd, n, L=(1.0, 0.8, 1.3)[:nd], precision=P.FP64 if precision == "fp64" else P.FP32_MIXED)
        g.set_material(2.0, 1.0, math.inf, 30.0, 0.0, coh)
        g.set_kernel(getattr(P, kernel), -1)
        for k, a in f.items():
            g.set(k, a)
        g.snapshot()
        grids.append(g)
    g, ref = grids

    def solve(x, wait):
        x.restore()
        x.set_solver(tol=0.0, max_iter=40, n_chk=10, wait_cycles=wait)
        x.apply_increment(1.0, 1e-4, P.LOAD_XY if nd == 2 else P.LOAD_XZ)
        return x.solve_increment(raise_on_fail=False)["status"]

    timeout, not_converged = 7, 5
    assert solve(ref, 0) == not_converged
    ref.commit_increment()
    want = {k: ref.get(k) for k in list(f) + ["epl", "scale"]}
    assert (want["scale"] < 1.0).any()
    for wait in (8, 300, 600, 1200, 2400, 4800, 9600):
        status = solve(g, wait)
        assert status in ((timeout,) if wait == 8 else (timeout, not_converged)), (wait, status)
        assert solve(g, 0) == not_converged
        g.commit_increment()
        for k, a in want.items():
            np.testing.assert_array_equal(g.get(k), a)
    g.close()
    ref.close()


@pytest.mark.parametrize("kernel,shape", [("KERNEL_AUTO", -1), ("KERNEL_STAGED", -1), ("KERNEL_FUSED", 0),
                                          ("KERNEL_FUSED", 3), ("KERNEL_FUSED", 4)])
@pytest.mark.parametrize("seed", [17, 18, 19])
def test_fp32_stopping_measures_of_2d_sweeps_are_formed_in_fp64(P, kernel, shape, seed):
    """max|tau - tau_chk| and max|p - p_chk| of FP32 states, against the same differences of the
    two checks' states on the host: equal to rounding in 64 bits."""
    n, chk = (70, 45), 2
    f = _fields(P, 2, n, seed)
    runs = [_solve(P, 2, n, P.FP32_MIXED, getattr(P, kernel), m, f, shape=shape, chunk=chk) for m in (2 * chk, 3 * chk)]
    (_, a), (info, b) = runs
    assert info["iters"] == 3 * chk
    # Eqs. PT1-PT24qq with the defaults of the grid and _solve's material and step
    dt, G, K, L, h = 1e-4, 1.0, 2.0, (1.0, 0.8), [w / m for w, m in zip((1.0, 0.8), n)]
    eta, Vp = G * dt, 0.9 / math.sqrt(2.0) * min(h)
    rho = 3.0 * math.sqrt(10.0) * math.pi / 2.0 * eta / (Vp * max(L))
    Gt = rho * Vp ** 2 / (0.5 + 4.0 / 3.0)
    bt = (1.0 / (2.0 * Gt)) / (1.0 / (2.0 * Gt) + 1.0 / (2.0 * eta))
    bp = (1.0 / (0.5 * Gt)) / (1.0 / (0.5 * Gt) + 1.0 / (K * dt))
    for keys, beta, got in ((("txx", "tyy", "txy"), bt, info["eps_tau"]), (("p",), bp, info["eps_p"])):
        gap = max(np.abs(b[k] - a[k]).max() for k in keys)
        want = gap / (chk * (1.0 - beta)) / info["max_sigma"]
        assert abs(got - want) <= 1e-11 * want, (keys, got, want)


@pytest.mark.parametrize("nd,n,precision,kernel,opts", [
    (3, (2, 2, 70000), "fp64", ("KERNEL_FUSED_REG", 0), {}),          # planes
    (3, (2, 530000, 1), "fp64", ("KERNEL_AUTO", -1), {}),             # row blocks
    (2, (2, 530000), "fp64", ("KERNEL_FUSED", 0), {}),                # the rotation's means
    (2, (2, 2100000), "fp32", ("KERNEL_FUSED", 0), {}),               # strips of rows
    (3, (2, 790000, 1), "fp32", ("KERNEL_STAGED", -1), {"cell_g": 1.0}),
])
def test_grids_longer_than_one_launch(P, nd, n, precision, kernel, opts):
    """More planes, row blocks or strips than a launch's 65,535 along y or z.  The FP64 grid that
    no fused sweep holds along y is compared with a per-cell modulus of the same value
    everywhere, which takes the general stage kernels."""
    iters = 8
    f = _fields(P, nd, n, 20, h=0.02)
    opts = dict(opts, L=tuple(0.02 * m for m in n))
    pr = P.FP64 if precision == "fp64" else P.FP32_MIXED
    general = {"cell_g": 0.0} if kernel[0] == "KERNEL_AUTO" else {}
    iref, ref = _solve(P, nd, n, pr, getattr(P, kernel[0]), iters, f, shape=kernel[1], **opts, **general)
    info, out = _solve(P, nd, n, pr, P.KERNEL_AUTO, iters, f, **opts)
    _compare(f, out, ref, info, iref, iters, 2.0 ** -53 if precision == "fp64" else EPS32)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_resident_chunks_after_other_chunks_of_the_same_solve(P, precision):
    """The kernel changed between the chunks of one solve, twice over: the resident sweep starts its
    exchange anew, and every chunk gives the staged sweep's bits."""
    n = (64, 50)
    f = _fields(P, 2, n, 21)
    outs = []
    for mixed in (False, True):
        g = P.Grid(2, n, L=(1.0, 0.8), precision=P.FP64 if precision == "fp64" else P.FP32_MIXED)
        g.set_material(2.0, 1.0, math.inf, 30.0, 0.0, np.full(n[0] * n[1], 1.5e-3))
        g.set_solver(tol=0.0, max_iter=1000, n_chk=10)
        for k, a in f.items():
            g.set(k, a)
        for _ in range(2):
            g.apply_increment(1.0, 1e-4)
            for chunk in range(6):
                g.set_kernel(P.KERNEL_AUTO if mixed and chunk % 3 else P.KERNEL_STAGED)
                assert g.solve_chunks(1)["status"] == P.PENDING
            g.commit_increment()
        outs.append({k: g.get(k) for k in list(f) + ["epl", "scale"]})
        g.close()
    for k, a in outs[0].items():
        np.testing.assert_array_equal(outs[1][k], a)


@pytest.mark.parametrize("grids", [[(2, (64, 64), "fp64"), (2, (64, 50), "fp64"), (2, (128, 128), "fp64")],
                                   [(2, (300, 180), "fp32"), (2, (383, 191), "fp32")],
                                   [(3, (90, 40, 24), "fp32"), (3, (40, 33, 14), "fp32"), (2, (300, 180), "fp32")]])
def test_resident_grids_solved_at_once_equal_one_after_the_other(P, grids):
    """Cooperative launches of several grids on their own streams, from a host thread each: the
    launches take turns where they do not fit the chip together, and the results are the same."""
    import threading

    def make(nd, n, precision):
        g = P.Grid(nd, n, L=(1.0, 0.8, 1.3)[:nd], precision=P.FP64 if precision == "fp64" else P.FP32_MIXED)
        g.set_material(2.0, 1.0, math.inf, 30.0, 0.0, np.full(int(np.prod(n)), 1.5e-3))
        g.set_solver(tol=0.0, max_iter=400, n_chk=20)
        for k, a in _fields(P, nd, n, 22).items():
            g.set(k, a)
        g.snapshot()
        return g

    def solve(g, out, q):
        for _ in range(5):
            g.apply_increment(1.0, 1e-4, P.LOAD_XY if g.ndim == 2 else P.LOAD_XZ)
            out[q] = g.solve_increment(raise_on_fail=False)["status"]
            g.commit_increment()

    gs = [make(*a) for a in grids]
    names = ["vx", "vy", "txx", "tyy", "txy", "p", "epl", "scale"]
    status = [None] * len(gs)
    for q, g in enumerate(gs):
        solve(g, status, q)
    want = [{k: g.get(k) for k in names} for g in gs]
    assert status == [5] * len(gs)
    for g in gs:
        g.restore()
    status = [None] * len(gs)
    threads = [threading.Thread(target=solve, args=(g, status, q)) for q, g in enumerate(gs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert status == [5] * len(gs)
    for g, w in zip(gs, want):
        for k in names:
            np.testing.assert_array_equal(g.get(k), w[k])
        g.close()
