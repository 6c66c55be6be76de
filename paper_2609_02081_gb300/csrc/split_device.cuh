// split_device.cuh — device helpers shared by the split mode's kernels.
#pragma once
#include <cuda_runtime.h>

#include "split.hpp"

namespace hmat {

// Programmatic dependent launch.  allow_next_kernel: the next kernel of the stream
// may be scheduled from here on, not only when this one ends (it still waits for
// this one's results); wait_for_previous_kernel: returns when the previous kernel
// has finished and its writes are visible.  Every kernel launched this way waits,
// so a kernel's finish implies that all earlier ones have finished.  Such a kernel
// is resident while memory that it will read is still being written, so its
// parameters are not __restrict__ and nothing goes through __ldg: either would tell
// the compiler that the memory does not change while the kernel runs, and let it move
// a load above the wait or take it from the read-only cache.  Only the
// exponents allow the next one early: the encoder doing so let residue-GEMM CTAs
// settle while its last blocks ran, and a 512-product batch took 22.7 ms against
// 21.3 (n = 4096: 20.9 against 19.9); from the GEMM it makes no difference, since
// no CRT block fits beside it.
__device__ __forceinline__ void allow_next_kernel() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Scaled integer round(x * 2^s) of a double given as bits; |result| <= 2^b by construction.
// Zeros and subnormals give 0 (split mode flushes subnormal inputs).
__device__ __forceinline__ long long scaled_int(unsigned long long u, int s) {
  const int ef = (int)((u >> 52) & 0x7FF);
  if (ef == 0 || ef == 0x7FF) return 0;
  const unsigned long long mant = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = 1075 - ef - s;      // value * 2^s = mant * 2^-sh
  long long X;
  if (sh <= 0) X = (long long)(mant << (-sh));     // not reached for b <= 52
  else if (sh >= 60) X = 0;
  else X = (long long)((mant + (1ull << (sh - 1))) >> sh);
  return (u >> 63) ? -X : X;
}

// The job holding unit u of a stage: the last job whose prefix count of that
// stage (`which`: 0 exponents, 1 encoder A, 2 encoder B, 3 GEMM items, 4 CRT
// blocks, 5 and 6 the matrix form's encoder and CRT blocks) is at most u: a job
// without units in the stage is never found.  Every lane of a full warp calls it with the same u (each
// kernel's block index); the warp probes 32 jobs per round and narrows by a
// ballot, so a call of 1024 jobs takes two dependent rounds of loads instead
// of ten.
__device__ __forceinline__ int find_split_job(const SplitJob* jobs, int njobs, int64_t u, int which) {
  const int lane = threadIdx.x & 31;
  auto begin = [&](int g) -> int64_t {
    switch (which) {
      case 0: return jobs[g].exp_begin;
      case 1: return jobs[g].encA_begin;
      case 2: return jobs[g].encB_begin;
      case 3: return jobs[g].item_begin;
      case 4: return jobs[g].crt_begin;
      case 5: return jobs[g].enc2_begin;
      default: return jobs[g].crt2_begin;
    }
  };
  int lo = 0, hi = njobs - 1;               // the answer lies in [lo, hi]; begin(lo) <= u
  while (lo < hi) {
    const int step = (hi - lo + 32) / 32;   // lane l probes lo + l step
    const int g = lo + lane * step;
    const unsigned le = __ballot_sync(0xffffffffu, g <= hi && begin(g) <= u);
    lo += (31 - __clz(le)) * step;          // lane 0 (begin(lo) <= u) is always set
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// A load before wait_for_previous_kernel() of data that an earlier kernel than the
// previous one wrote (which the previous one has waited for): performed at the GPU's
// point of coherence, since this SM's L1 may still hold a line from before that write.
__device__ __forceinline__ unsigned long long load_coherent(const double* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// p itself, as a value that exists only from here on: loads through it, of whatever
// kind, cannot move above an earlier wait_for_previous_kernel().
template <class T>
__device__ __forceinline__ T* known_from_here(T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

// The job of unit u of a stage: the one in the arguments, or the table's.
template <bool kOne>
__device__ __forceinline__ const SplitJob& unit_job(const JobParam<kOne>& one, const SplitJob* jobs,
                                                    int njobs, int64_t u, int which) {
  if constexpr (kOne) return one.job;
  else return jobs[find_split_job(jobs, njobs, u, which)];
}

template <int L>
__device__ __forceinline__ double limbs_to_double(const uint32_t* xin, int neg, int scale_exp) {
  // whole-limb shifts bring the top nonzero limb (index h) to position L - 1;
  // selects only, so the limbs stay in registers
  uint32_t x[L];
#pragma unroll
  for (int q = 0; q < L; ++q) x[q] = xin[q];
  int h = L - 1;
#pragma unroll
  for (int s = 0; s < L - 1; ++s) {
    const bool z = x[L - 1] == 0;
#pragma unroll
    for (int q = L - 1; q > 0; --q) x[q] = z ? x[q - 1] : x[q];
    x[0] = z ? 0u : x[0];
    h -= z ? 1 : 0;
  }
  const uint32_t l2 = x[L - 1], l1 = x[L - 2], l0 = x[L - 3];
  if (l2 == 0) return neg ? -0.0 : 0.0;
  uint32_t sticky = 0;
#pragma unroll
  for (int q = 0; q < L - 3; ++q) sticky |= x[q];
  const int lz = __clz(l2);                       // normalise the 96-bit window [l2 l1 l0]
  unsigned long long hi = ((unsigned long long)l2 << 32) | l1;
  unsigned long long lo = (unsigned long long)l0 << 32;
  if (lz) {
    hi = (hi << lz) | (lo >> (64 - lz));
    lo <<= lz;
  }
  if (lo != 0 || sticky != 0) hi |= 1ull;         // sticky bit: one correct rounding below
  // value = W 2^(32(h-2)) with W ~ hi 2^(32 - lz): hi 2^E, hi in [2^63, 2^64)
  const int E = 32 * (h - 1) - lz + scale_exp;
  const int bexp = E + 1086;                      // IEEE biased exponent of hi 2^E
  if (bexp >= 1 && bexp <= 2046) {
    // normal result: round hi to 53 bits (nearest, ties to even) and assemble
    // the bits with integer operations; a mantissa carry bumps the exponent
    const unsigned long long mant = hi >> 11;
    const uint32_t rem = (uint32_t)hi & 0x7FFu;
    const unsigned long long up = (rem > 0x400u || (rem == 0x400u && (mant & 1ull))) ? 1ull : 0ull;
    const unsigned long long bits = ((unsigned long long)(bexp - 1) << 52) + mant + up;
    return __longlong_as_double((long long)(bits | ((unsigned long long)neg << 63)));
  }
  const double v = __ull2double_rn(hi);           // subnormal or overflowing result
  const double r = scalbn(v, E);
  return neg ? -r : r;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait2() { asm volatile("cp.async.wait_group 2;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait6() { asm volatile("cp.async.wait_group 6;\n" ::: "memory"); }

// |X| = [x3 x2 x1 x0] (below 2^127) times 2^scale_exp as a double, rounded
// to nearest even: the top 64 significant bits from the two 64-bit halves and
// one leading-zero count, the bits below as a sticky bit.
__device__ __forceinline__ double limbs4_to_double(const uint32_t* x, int neg, int scale_exp) {
  unsigned long long hi = ((unsigned long long)x[3] << 32) | x[2];
  unsigned long long lo = ((unsigned long long)x[1] << 32) | x[0];
  const bool hz = hi == 0ull;
  int e0 = hz ? scale_exp : 64 + scale_exp;       // weight 2^e0 of hi's bit 0
  hi = hz ? lo : hi;
  lo = hz ? 0ull : lo;
  if (hi == 0ull) return neg ? -0.0 : 0.0;
  const int lz = __clzll((long long)hi);
  unsigned long long top = (hi << lz) | ((lo >> 1) >> (63 - lz));   // bit 63 set
  if ((lo << lz) != 0ull) top |= 1ull;            // sticky bit: one correct rounding below
  const int E = e0 - lz;                          // value = top 2^E
  const int bexp = E + 1086;                      // IEEE biased exponent of top 2^E
  if (bexp >= 1 && bexp <= 2046) {
    const unsigned long long mant = top >> 11;
    const uint32_t rem = (uint32_t)top & 0x7FFu;
    const unsigned long long up = (rem > 0x400u || (rem == 0x400u && (mant & 1ull))) ? 1ull : 0ull;
    const unsigned long long bits = ((unsigned long long)(bexp - 1) << 52) + mant + up;
    return __longlong_as_double((long long)(bits | ((unsigned long long)neg << 63)));
  }
  const double v = __ull2double_rn(top);          // subnormal or overflowing result
  const double r = scalbn(v, E);
  return neg ? -r : r;
}

// S_e - q P for one output: acc holds S_e in L signed 64-bit limb sums (limb q
// weighs 2^(32 q)), S_e = X_e (mod P), 0 < S_e, |X_e| < 2^-1.25 P.  q is the
// nearest integer to a float estimate of S_e / P from the leading limbs (pb: the
// limb below P's top one, pinv = fl(2^(32 pb) / P)); returns X_e 2^scale_exp.
template <int L>
__device__ __forceinline__ double crt_value(const long long (&acc)[L], const uint32_t* P, int pb, float pinv,
                                            int scale_exp) {
  uint32_t x[L];
  long long t = acc[0];
  x[0] = (uint32_t)t;
#pragma unroll
  for (int q = 1; q < L; ++q) {            // signed carries; t ends as S >> 32 (L - 1), below 2^35
    t = acc[q] + (t >> 32);
    x[q] = (uint32_t)t;
  }
  float sf = fmaf((float)(int)(t >> 32), 4294967296.f, (float)x[L - 1]);
#pragma unroll
  for (int q = L - 2; q >= 0; --q)
    if (q >= pb) sf = fmaf(sf, 4294967296.f, (float)x[q]);
  const uint32_t qq = __float2uint_rn(sf * pinv);
  long long borrow = 0;
  unsigned long long mulc = 0;
#pragma unroll
  for (int q = 0; q < L; ++q) {            // x = S - qq P modulo 2^(32 L): X in two's complement
    const unsigned long long prod = (unsigned long long)P[q] * qq + mulc;
    mulc = prod >> 32;
    const long long diff = (long long)x[q] - (long long)(uint32_t)prod + borrow;
    x[q] = (uint32_t)diff;
    borrow = diff >> 32;
  }
  const uint32_t neg = x[L - 1] >> 31;     // |X| = (x ^ -neg) + neg, without a branch
  const uint32_t flip = 0u - neg;
  unsigned long long c = neg;
#pragma unroll
  for (int q = 0; q < L; ++q) {
    const unsigned long long tq = (unsigned long long)(x[q] ^ flip) + c;
    x[q] = (uint32_t)tq;
    c = tq >> 32;
  }
  if constexpr (L == 4) return limbs4_to_double(x, (int)neg, scale_exp);
  else return limbs_to_double<L>(x, (int)neg, scale_exp);
}

// Calls f(JobParam, table) with the version of the job argument that `jobs` holds.
template <class F>
cudaError_t with_jobs(const SplitJobs& jobs, F&& f) {
  if (jobs.table) return f(JobParam<false>{});
  JobParam<true> one;
  one.job = *jobs.one;
  return f(one);
}

}  // namespace hmat
