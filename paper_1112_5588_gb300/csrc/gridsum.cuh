// fp64 sums over a warp, a CTA and all CTAs of a cooperative launch (cg.cu, mlp.cu)
// or over the partial sums of a launch (krylov.cu). Over a grid every CTA gives its
// threads' values and every thread gets the total, with no return to the host and
// no second launch.
//
// A dependent fp64 add takes 70 cycles here and a warp's fp64 add holds the
// SM's fp64 pipe for 16, so that a shuffle tree of fp64 adds over 1024 threads
// costs 5000 cycles (2.5 us). The sums are therefore taken in integers: each
// level finds the largest exponent, shifts its values to it as fixed point,
// rounded to nearest, and adds them as integers, which is exact. A warp's values
// are each rounded at 2^-57 of the largest one or less, 160 CTAs' at 2^-60, and the
// sum at 2^-57 of itself: a warp's sum and the CTAs' are off by less than 2^-51 of
// the largest value and 2^-56 of the sum, trees of fp64 adds by up to 5 2^-53 and 8
// 2^-53 of the sum of the magnitudes.
//
// Between CTAs: a CTA writes its sum into a slot of its own as two words, each
// with the number of the sum (its epoch); one warp of every CTA reads all slots
// until each word shows the epoch, and adds them. A word carries its own epoch,
// so no ordering between words and no atomic counter is needed: one store and
// one load of L2 latency. Every slot has a 128-byte line of its own (with eight
// slots to a line the two dies' L2 partitions pass the line back and forth at
// every store: 4.0 us a sum with 152 CTAs of 256 threads, against 2.5). Two
// sets of slots are used in turn: a CTA writes epoch e + 2 only after it has
// seen every CTA's e + 1, which were written after their CTAs had read all of
// epoch e. The total does not depend on the order of the values.
//
// Waits are bounded: a CTA that gives up sets the error word and leaves, and
// every other wait looks at that word and leaves too.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pjds {
namespace kry {

constexpr int GS_MAX_CTAS = 320;        // slots of a set
constexpr int GS_CHUNK = 5;             // slots a lane reads at once: 160, one CTA on each SM
constexpr uint32_t GS_SPIN = 1u << 23;  // polls (several seconds) before a wait gives up

struct __align__(128) GridSlot {
  ulonglong2 w;
  unsigned long long pad[14];
};

// In caller memory; zero before the launch.
struct GridSlots {
  GridSlot slot[2][GS_MAX_CTAS];
  unsigned long long error;  // 1: a wait ran out
  unsigned long long pad[15];
  uint32_t arrived;          // CTAs at GridBarrier
  uint32_t pad2[31];
};

// A sum in fixed point: f 2^(e - 1079), |f| at most 2^57, e from 1 on; e = 0x7ff: f
// holds the bits of an infinity or a NaN.
struct Fixed {
  long long f;
  uint32_t e;
};

__device__ __forceinline__ Fixed fixed_of(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  Fixed a;
  a.e = (uint32_t)(b >> 52) & 0x7ffu;
  if (a.e == 0x7ffu) {
    a.f = (long long)b;
  } else {
    const unsigned long long m = ((b & 0xfffffffffffffull) | (a.e ? 0x10000000000000ull : 0ull)) << 4;
    a.f = (long long)b < 0 ? -(long long)m : (long long)m;
    a.e = a.e ? a.e : 1u;
  }
  return a;
}

// of a finite float, without the fp64 pipe
__device__ __forceinline__ Fixed fixed_of(float v) {
  const uint32_t b = __float_as_uint(v), k = (b >> 23) & 0xffu, m = (b & 0x7fffffu) | (k ? 0x800000u : 0u);
  Fixed a;
  a.f = (long long)m << 33;
  if ((int32_t)b < 0) a.f = -a.f;
  a.e = m ? max(k, 1u) + 896u : 1u;
  return a;
}

__device__ __forceinline__ double double_of(const Fixed &a) {
  if (a.e == 0x7ffu) return __longlong_as_double(a.f);
  if (a.f == 0) return 0.0;
  const bool neg = a.f < 0;
  unsigned long long m = neg ? 0ull - (unsigned long long)a.f : (unsigned long long)a.f;
  const int lz = __clzll((long long)m);
  const int e = (int)a.e + 7 - lz;  // biased exponent of the result (m has bit 63 - lz as its highest)
  if (e < 1 || e > 2045) return ldexp((double)a.f, (int)a.e - 1079);
  m <<= lz;
  // 53 bits, to nearest even; a carry runs into the exponent as it should
  const unsigned long long keep = m >> 11, low = m & 0x7ffull;
  const unsigned long long up = (low > 0x400ull || (low == 0x400ull && (keep & 1))) ? 1ull : 0ull;
  const unsigned long long b = (((unsigned long long)e - 1) << 52) + keep + up;
  return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

// Sum over the warp of N values a lane, in every lane.
template <int N>
__device__ __forceinline__ Fixed warp_sum(const Fixed (&a)[N]) {
  static_assert(N <= 7, "a lane's sum beyond 63 bits");
  constexpr int G = N > 1 ? 3 : 0;  // bits kept below a value's: N 2^(57 + G) is below 2^63
  uint32_t em = a[0].e;
#pragma unroll
  for (int q = 1; q < N; ++q) em = max(em, a[q].e);
  em = __reduce_max_sync(0xffffffffu, em);
  Fixed s;
  if (em == 0x7ffu) {  // an infinity or a NaN: finite values do not matter beside it
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (a[q].e == 0x7ffu) v += __longlong_as_double(a[q].f);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    s.e = 0x7ffu;
    s.f = __double_as_longlong(v);
    return s;
  }
  long long f = 0;
#pragma unroll
  for (int q = 0; q < N; ++q)  // (G + 1 bits more, and the last one rounded)
    f += (((long long)((unsigned long long)a[q].f << (G + 1)) >> min(em - a[q].e, 63u)) + 1) >> 1;
  // in three parts, whose sums over 32 lanes fit 32 bits
  const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)f & 0x3ffffffu);
  const uint32_t s1 = __reduce_add_sync(0xffffffffu, (uint32_t)(f >> 26) & 0x3ffffffu);
  const int32_t s2 = __reduce_add_sync(0xffffffffu, (int32_t)(f >> 52));
  int e = (int)em - G;
  if constexpr (N == 1) {  // below 2^62
    f = (long long)s0 + ((long long)s1 << 26) + ((long long)s2 << 52);
  } else {  // hi 2^26 + low, hi below 2^42
    const long long hi = ((long long)s2 << 26) + s1 + (s0 >> 26);
    const uint32_t low = s0 & 0x3ffffffu;
    const bool far = hi < -(1ll << 36) || hi >= (1ll << 36);
    f = far ? (hi << 20) + ((low + 32u) >> 6) : (hi << 26) + low;
    e += far ? 6 : 0;
  }
  // to 57 bits, from where the next sum's shifts drop nothing that a double holds, and e from 1 on
  const unsigned long long m = f < 0 ? 0ull - (unsigned long long)f : (unsigned long long)f;
  const int sh = max(m ? 7 - __clzll((long long)m) : 0, 1 - e);  // > 0: too large by sh bits
  s.f = sh > 0 ? (f + ((1u << sh) >> 1)) >> sh : (long long)((unsigned long long)f << -sh);
  s.e = (uint32_t)(e + sh);
  if (f == 0) s.e = 1u;
  if (s.e >= 0x7ffu) {  // the sum overflows
    s.e = 0x7ffu;
    s.f = f < 0 ? (long long)0xfff0000000000000ull : 0x7ff0000000000000ll;
  }
  return s;
}

__device__ __forceinline__ ulonglong2 gs_peek(const ulonglong2 *p) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}

// Words of a slot: the halves of f, beside the exponent and 20 bits of the epoch.
__device__ __forceinline__ ulonglong2 gs_pack(const Fixed &a, uint32_t epoch) {
  const unsigned long long f = (unsigned long long)a.f, tag = epoch & 0xfffffu;
  return make_ulonglong2((f & 0xffffffff00000000ull) | ((unsigned long long)a.e << 20) | tag, (f << 32) | tag);
}

struct GridSum {
  GridSlots *g;
  uint32_t epoch;  // of the last sum

  // Sum of `v` over all threads of all CTAs and then(total), evaluated once per
  // CTA (an fp64 division by every thread would hold the fp64 pipe for a
  // microsecond), in every thread. PUBLISH: global
  // writes made by any thread of the grid before the call are visible to every
  // thread after it (to ordinary loads, not to the read-only path). False: a
  // wait ran out; the kernel has to return.
  template <bool PUBLISH, typename F>
  __device__ __forceinline__ bool operator()(double v, double &total, double &result, F then) {
    __shared__ Fixed sh[33];
    __shared__ double sh_total, sh_result;
    __shared__ int sh_ok;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    const uint32_t tag = ++epoch & 0xfffffu;
    {
      const Fixed a[1] = {fixed_of(v)};
      const Fixed s = warp_sum<1>(a);
      if (l == 0) sh[w] = s;
    }
    __syncthreads();
    if (w == 0) {
      Fixed a[1] = {Fixed{0, 1}};
      if (l < nw) a[0] = sh[l];
      const Fixed s = warp_sum<1>(a);
      GridSlot *set = g->slot[epoch & 1];
      if (l == 0) {
        if (PUBLISH) __threadfence();
        const ulonglong2 p = gs_pack(s, epoch);
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(&set[blockIdx.x].w), "l"(p.x), "l"(p.y)
                     : "memory");
      }
      Fixed sum{0, 1};
      bool ok = true;
      // GS_CHUNK slots of a lane at a time, their loads in flight together
      for (uint32_t k0 = l; k0 < gridDim.x + l; k0 += 32 * GS_CHUNK) {
        ulonglong2 p[GS_CHUNK];
        bool all;
        uint32_t it = 0;
        do {
          all = true;
#pragma unroll
          for (int q = 0; q < GS_CHUNK; ++q)
            if (k0 + 32 * q < gridDim.x) p[q] = gs_peek(&set[k0 + 32 * q].w);
#pragma unroll
          for (int q = 0; q < GS_CHUNK; ++q)
            if (k0 + 32 * q < gridDim.x)
              all = all && ((uint32_t)p[q].x & 0xfffffu) == tag && ((uint32_t)p[q].y & 0xfffffu) == tag;
          if (!all && (++it >= GS_SPIN || ((it & 1023u) == 0 && *(volatile unsigned long long *)&g->error))) ok = false;
        } while (!all && ok);
        __syncwarp();
        Fixed b[GS_CHUNK];
#pragma unroll
        for (int q = 0; q < GS_CHUNK; ++q)
          b[q] = k0 + 32 * q < gridDim.x ? Fixed{(long long)((p[q].x & 0xffffffff00000000ull) | (p[q].y >> 32)),
                                                 (uint32_t)(p[q].x >> 20) & 0x7ffu}
                                         : Fixed{0, 1};
        const Fixed t = warp_sum<GS_CHUNK>(b);
        if (k0 == (uint32_t)l) {
          sum = t;
        } else {
          const Fixed two[1] = {l == 0 ? sum : l == 1 ? t : Fixed{0, 1}};
          sum = warp_sum<1>(two);
        }
      }
      if (PUBLISH) __threadfence();
      ok = __all_sync(0xffffffffu, ok);
      if (l == 0) {
        if (!ok) atomicExch(&g->error, 1ull);
        const double t = double_of(sum);
        sh_total = t;
        sh_result = then(t);
        sh_ok = ok;
      }
    }
    __syncthreads();
    total = sh_total;
    result = sh_result;
    return sh_ok != 0;
  }

  template <bool PUBLISH>
  __device__ __forceinline__ bool operator()(double v, double &total) {
    double none;
    return operator()<PUBLISH>(v, total, none, [](double t) { return t; });
  }
};

// A barrier of all CTAs that publishes global writes like GridSum<true>, without
// a value: one counter (1.2 us with 152 CTAs against 2.8 for a sum).
struct GridBarrier {
  GridSlots *g;
  uint32_t target;  // arrivals when all are here

  __device__ __forceinline__ bool operator()() {
    __shared__ int sh_ok;
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&g->arrived) : "memory");
      uint32_t v;
      int ok = 1;
      for (uint32_t it = 1;; ++it) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&g->arrived) : "memory");
        if ((int32_t)(v - target) >= 0) break;
        if (it >= GS_SPIN || ((it & 1023u) == 0 && *(volatile unsigned long long *)&g->error)) {
          ok = 0;
          atomicExch(&g->error, 1ull);
          break;
        }
      }
      sh_ok = ok;
    }
    __syncthreads();
    return sh_ok != 0;
  }
};

}  // namespace kry
}  // namespace pjds
