// ep_words.cuh -- values exchanged between the blocks of one cooperative launch: they
// travel in words that also carry the number of the iteration that wrote them, so that
// the reader polls the value itself: one trip through L2 where a counter behind a fence
// takes four.  Three FP32 values share a 16-byte word (.b128, written and read as a
// whole; a word of 8 bytes per value: 383 x 191 2.7 us an iteration against 2.0); an
// FP64 value is two words of 8 bytes, each with the number (a .b128 word per value: 64^2
// 4.2 us against 4.0).
#pragma once

#include <cuda_runtime.h>

#include "ep_internal.cuh"

namespace ep {

struct alignas(16) Word {
  unsigned long long lo, hi;   // upper half of hi (FP64: of both): iteration number
};
__device__ __forceinline__ Word ld_relaxed(const Word *p) {
  Word v;
  asm volatile("{ .reg .b128 q; ld.relaxed.gpu.global.b128 q, [%2]; mov.b128 {%0, %1}, q; }"
               : "=l"(v.lo), "=l"(v.hi) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(Word *p, Word v) {
  asm volatile("{ .reg .b128 q; mov.b128 q, {%1, %2}; st.relaxed.gpu.global.b128 [%0], q; }"
               ::"l"(p), "l"(v.lo), "l"(v.hi) : "memory");
}

// three values of a point: one word in FP32, three in FP64
template <typename T>
constexpr int words_of() { return sizeof(T) == 4 ? 1 : 3; }

__device__ __forceinline__ void send(Word *w, long long, float a, float b, float c, unsigned tag) {
  st_relaxed(w, {(unsigned long long)__float_as_uint(b) << 32 | __float_as_uint(a),
                 (unsigned long long)tag << 32 | __float_as_uint(c)});
}
__device__ __forceinline__ void send(Word *w, double v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&w->lo), "l"(t | (b & 0xffffffffu)) : "memory");
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&w->hi), "l"(t | (b >> 32)) : "memory");
}
__device__ __forceinline__ void send(Word *w, long long stride, double a, double b, double c, unsigned tag) {
  send(w, a, tag);
  send(w + stride, b, tag);
  send(w + 2 * stride, c, tag);
}
// third: whether c is wanted
__device__ __forceinline__ bool receive(const Word *w, long long, unsigned tag, float *a, float *b, float *c, bool third) {
  const Word v = ld_relaxed(w);
  *a = __uint_as_float((unsigned)v.lo);
  *b = __uint_as_float((unsigned)(v.lo >> 32));
  if (third) *c = __uint_as_float((unsigned)v.hi);
  return (unsigned)(v.hi >> 32) == tag;
}
__device__ __forceinline__ bool receive(const Word *w, unsigned tag, double *v) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(&w->lo) : "memory");
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(b) : "l"(&w->hi) : "memory");
  *v = __longlong_as_double((long long)(b << 32 | (a & 0xffffffffu)));
  return (unsigned)(a >> 32) == tag && (unsigned)(b >> 32) == tag;
}
__device__ __forceinline__ bool receive(const Word *w, long long stride, unsigned tag, double *a, double *b, double *c,
                                        bool third) {
  bool ok = receive(w, tag, a);
  ok = receive(w + stride, tag, b) && ok;
  if (third) ok = receive(w + 2 * stride, tag, c) && ok;
  return ok;
}

// one reader's wait for its words: it gives up after the grid's bound (ep_solver_opts.
// wait_cycles), or when another reader has (looked up every 64 tries)
struct Wait {
  long long since;
  unsigned tries;
};
__device__ __forceinline__ Wait wait_begin() { return {clock64(), 0u}; }
// after a try that found a word missing
__device__ __forceinline__ bool wait_over(Wait &w, long long limit, DevInfo *di) {
  if (clock64() - w.since <= limit && ((++w.tries & 63) != 0 || *(volatile const int *)&di->done == 0)) return false;
  atomicCAS(&di->done, 0, 4);
  return true;
}

}  // namespace ep
