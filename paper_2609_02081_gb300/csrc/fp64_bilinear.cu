// fp64_bilinear.cu — plain FP64 bilinear biquaternion product, one fused kernel.
//
// C <- alpha op(A) op(B) + beta C with the paper's bilinear scheme
// (Sec. III B, Eq. bilinearH + Gauss, Eq. cmplx-3-real-mult), every real
// product accumulated in FP64.  Per output tile the kernel
//   prologue : stages the present components of op(A), op(B) (op = index
//              transpose + sign, Sec. III) and forms the plan's left/right
//              factors (the Hadamard sums and Gauss Re+Im sums) in shared
//              memory — nothing of them is written to global memory;
//   main loop: accumulates all (up to 24) real products in registers;
//   epilogue : recombines them into the eight output components with the
//              plan's weights (2, -1/4, ... exact dyadic scalings), applies the
//              complex alpha / beta update (Sec. III scaling and addition) and
//              stores C.
//
// GB300 note: FP64 FMA throughput is 2 per clock per SM (1.06 to 1.2 TFLOP/s
// measured), so a warp-wide DFMA occupies an SM sub-partition's FP64 pipe for 64
// clocks; the kernel is bound by that pipe alone.  24 accumulators per output point
// cap the tile at 32x32 per SM (24 x 1024 doubles = 192 KB of registers).  What is
// left to gain is the count of FP64 instructions that are not product FMAs, and a
// pipe that never waits:
//  - signs (of op and of the +-1 sums) are flips of the sign bit on the integer pipe;
//    a select between x + y and x - y costs both.  With the Hadamard sums as a
//    butterfly a point of a side takes 24 FP64 additions (80 before): 6 % of the
//    FP64 instructions at 32x32 tiles instead of 17 %;
//  - the factors of the next k-block are formed while this one's products run, one
//    barrier a block, the two warps of a sub-partition at different times;
//  - components are copied four k-blocks ahead: plans of few products spend less time
//    on a block than one copy takes (1 product, n = 1024: 5.99 ms with two blocks
//    ahead, 3.05 with four).
// n = 2048: 434 -> 365 ms; the products alone take 328 at 2 per clock and 2070 MHz.
#include <cuda_runtime.h>

#include "common.cuh"

namespace hmat {

constexpr int F_BM = 32, F_BN = 32, F_BK = 4, F_THREADS = 256;
constexpr int F_RING = 4;           // k-blocks of staged components: the copies run this far ahead
constexpr int F_KALIGN = 8;         // slices of a split inner dimension are multiples of this
static_assert(F_BM == 32 && F_BN == 32 && F_THREADS == 2 * F_BK * 32, "one factor point of one side per thread");
// products per pass: 24 accumulators per output point fill the register file;
// plans with more products run as several passes (host side)
constexpr int F_MAXP = 24;

struct Fp64Smem {
  double araw[F_RING][8][F_BK][F_BM];   // staged op(A) components
  double braw[F_RING][8][F_BK][F_BN];   // staged op(B) components
  double xs[2][kMaxFactors][F_BK][F_BM];   // left factors (double buffer)
  double ys[2][kMaxFactors][F_BK][F_BN];   // right factors
  double wd[8][F_MAXP];                 // recombination weights w4 / 4 of the loaded plan
  KPlan plan;
  JobDesc job;                          // the only job of a call (kOne)
  int plan_id;
};

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, bool valid) {
  const uint32_t s = smem_u32(smem);
  const int src_bytes = valid ? 8 : 0;   // 0: zero-fill, nothing read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Stage the k-block at k0 of the present components of op(A) (BM x BK, warps 0-3) and
// op(B) (BK x BN, warps 4-7); inner indices at or beyond kend read as zero.
__device__ __forceinline__ void stage_raw(Fp64Smem& s, int buf, const JobDesc& jb, int i0, int j0, int k0, int kend) {
  const bool left = threadIdx.x < F_THREADS / 2;
  const int t = threadIdx.x & (F_THREADS / 2 - 1);
  // reads run along the operand's stored rows: along k for op(A) and transposed op(B)
  const bool along_k = left ? !jb.transA : jb.transB;
  const int r = along_k ? t / F_BK : t % 32, kk = along_k ? t % F_BK : t / 32;
  const int at = (left ? i0 : j0) + r, kg = k0 + kk;
  const bool valid = at < (left ? jb.m : jb.n) && kg < kend;
  const int64_t ld = left ? jb.lda : jb.ldb;
  const int64_t off = !valid ? 0 : along_k ? (int64_t)at * ld + kg : (int64_t)kg * ld + at;
  const double* src = (left ? jb.A : jb.B) + off;
  const int64_t stride = left ? jb.sA : jb.sB;
  const uint32_t present = left ? jb.fa : jb.fb;
  double* dst = left ? &s.araw[buf][0][kk][r] : &s.braw[buf][0][kk][r];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    if (!((present >> c) & 1u)) continue;
    cp_async8(dst + c * F_BK * 32, src + (int64_t)c * stride, valid);
  }
}

// x with its sign bit flipped when bit 31 of mask is set: sign changes on the integer
// pipe, none of them an FP64 instruction
__device__ __forceinline__ double flip(double x, uint32_t mask) {
  return __hiloint2double(__double2hiint(x) ^ (int)(mask & 0x80000000u), __double2loint(x));
}

// The components of staged point (kk, r) with their op signs (bit c of neg), zeros
// where a component is absent.
__device__ __forceinline__ void load_point(const double (*raw)[F_BK][F_BM], int kk, int r, uint32_t present,
                                           uint32_t neg, double v[8]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = ((present >> c) & 1u) ? flip(raw[c][kk][r], neg << (31 - c)) : 0.0;
}

// Signed +-1 sum of v[0..3] with the four coefficients of a group (0, 1 or -1), in order.
__device__ __forceinline__ double signed_sum(const int8_t* coef, const double* v) {
  const uint32_t w = *reinterpret_cast<const uint32_t*>(coef);
  bool any = false;
  double acc = 0.0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (!(w >> (8 * e) & 0xFFu)) continue;
    const double x = flip(v[e], w << (24 - 8 * e));
    acc = any ? acc + x : x;
    any = true;
  }
  return acc;
}

// One side's factors of staged point v into f[slot][kk][r].  The eight groups of the
// full plan are the four components and their Hadamard sums, formed as a butterfly
// (8 additions for the four sums instead of 12); other plans sum term by term.
__device__ __forceinline__ void form_point(const double v[8], double (*f)[F_BK][F_BM], int kk, int r, int ngroups,
                                           bool hadamard, const int8_t (*cre)[4], const int8_t (*cim)[4],
                                           const int8_t (*slot)[3]) {
  auto emit = [&](int g, double re, double im) {
    const int sr = slot[g][0], si = slot[g][1], ss = slot[g][2];
    if (sr >= 0) f[sr][kk][r] = re;
    if (si >= 0) f[si][kk][r] = im;
    if (ss >= 0) f[ss][kk][r] = re + im;
  };
  if (hadamard) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      int e = 0;                        // the group's component
#pragma unroll
      for (int i = 1; i < 4; ++i) e = cre[g][i] ? i : e;
      const double re = e == 0 ? v[0] : e == 1 ? v[1] : e == 2 ? v[2] : v[3];
      const double im = e == 0 ? v[4] : e == 1 ? v[5] : e == 2 ? v[6] : v[7];
      emit(g, re, im);
    }
    const double p01 = v[0] + v[1], m01 = v[0] - v[1], p23 = v[2] + v[3], m23 = v[2] - v[3];
    const double q01 = v[4] + v[5], n01 = v[4] - v[5], q23 = v[6] + v[7], n23 = v[6] - v[7];
    emit(4, p01 + p23, q01 + q23);
    emit(5, p01 - p23, q01 - q23);
    emit(6, m01 + m23, n01 + n23);
    emit(7, m01 - m23, n01 - n23);
    return;
  }
  for (int g = 0; g < ngroups; ++g) {
    const double re = signed_sum(cre[g], v), im = signed_sum(cim[g], v + 4);
    emit(g, re, im);
  }
}

// Prologue: the left factors of the k-block staged in raw (warps 0-3, one point a
// thread) or its right factors (warps 4-7) into factor buffer fbuf.
__device__ __forceinline__ void form_factors(Fp64Smem& s, int rbuf, int fbuf, const JobDesc& jb, uint32_t negA,
                                             uint32_t negB) {
  const KPlan& p = s.plan;
  const int kk = (threadIdx.x >> 5) & (F_BK - 1), r = threadIdx.x & 31;
  double v[8];
  if (threadIdx.x < F_THREADS / 2) {
    load_point(s.araw[rbuf], kk, r, jb.fa, negA, v);
    form_point(v, s.xs[fbuf], kk, r, p.nlg, p.bilinear_left != 0, p.lre, p.lim, p.lslot);
  } else {
    load_point(s.braw[rbuf], kk, r, jb.fb, negB, v);
    form_point(v, s.ys[fbuf], kk, r, p.nrg, p.bilinear_right != 0, p.rre, p.rim, p.rslot);
  }
}

// Recombination of point pt's 24 products of the paper's full plan (T1, T2, T3 of
// P1, ..., P8): Gauss's differences, then the sums of P5..P8 as a butterfly; 56 FP64
// instructions where the weights' table takes 100.
__device__ __forceinline__ void recombine_full(const double acc[F_MAXP][4], int pt, double q[8]) {
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    double P[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const double t1 = acc[3 * r][pt], t2 = acc[3 * r + 1][pt];
      P[r] = part ? acc[3 * r + 2][pt] - t1 - t2 : t1 - t2;
    }
    const double s56 = P[4] + P[5], d56 = P[4] - P[5], s78 = P[6] + P[7], d78 = P[6] - P[7];
    q[4 * part] = fma(-0.25, s56 + s78, 2.0 * P[0]);
    q[4 * part + 1] = fma(0.25, s56 - s78, -2.0 * P[1]);
    q[4 * part + 2] = fma(0.25, d56 + d78, -2.0 * P[2]);
    q[4 * part + 3] = fma(0.25, d56 - d78, -2.0 * P[3]);
  }
}

// C[i][jj] <- alpha q + beta C[i][jj]
__device__ __forceinline__ void store_point(const JobDesc& jb, int i, int jj, const double q[8]) {
  double* cbase = jb.C + (int64_t)i * jb.ldc + jj;
  if (jb.alpha_re == 1.0 && jb.alpha_im == 0.0 && jb.beta_re == 0.0 && jb.beta_im == 0.0) {
#pragma unroll
    for (int e = 0; e < 8; ++e) cbase[(int64_t)e * jb.sC] = q[e];
    return;
  }
  const bool use_beta = (jb.beta_re != 0.0 || jb.beta_im != 0.0);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    double re = jb.alpha_re * q[e] - jb.alpha_im * q[e + 4];
    double im = jb.alpha_re * q[e + 4] + jb.alpha_im * q[e];
    if (use_beta) {
      const double cre = cbase[(int64_t)e * jb.sC];
      const double cim = cbase[(int64_t)(e + 4) * jb.sC];
      re += jb.beta_re * cre - jb.beta_im * cim;
      im += jb.beta_re * cim + jb.beta_im * cre;
    }
    cbase[(int64_t)e * jb.sC] = re;
    cbase[(int64_t)(e + 4) * jb.sC] = im;
  }
}

template <bool kOne>
struct Fp64One {
  JobDesc job;
};
template <>
struct Fp64One<false> {};

// kRanges: the call's tiles, laid end to end in k-blocks (each job's tiles
// ranges.per_tile of them apart), are cut into one range of ranges.width k-blocks per
// CTA, whatever tiles it crosses.  Each piece of a tile goes to slot (CTA + tile) of
// the partial outputs: along the ranges either number increases, so no two pieces
// share one.
// kOne: the call's only job, in the arguments: nothing to copy to the device first, and
// the launch need not wait for the 2.05 us grid on which dependent launches start
// (64 x 64 x 64: 74 -> 59 us, n = 256: 776 -> 756).
// kFull: every job runs the paper's full plan, whose product q multiplies left and right
// factor q: no plan look-ups between the products (n = 1024: 47.8 -> 47.4 ms).
template <bool kRanges, bool kOne, bool kFull>
__global__ void __launch_bounds__(F_THREADS, 1)
fp64_bilinear_kernel(const __grid_constant__ Fp64One<kOne> one, const JobDesc* jobs, int njobs, const KPlan* plans,
                     int64_t total_tiles, Fp64Ranges ranges) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Fp64Smem& s = *reinterpret_cast<Fp64Smem*>(smem_raw);
  const int t = threadIdx.x;
  const int ty = t / 16, tx = t % 16;   // output rows 2ty, 2ty+1; cols 2tx, 2tx+1
  // (a copy in shared memory: with the fields in constant memory the compiler spends
  // the registers that the products' operands are prefetched in)
  if constexpr (kOne) {
    static_assert(sizeof(JobDesc) % 8 == 0 && sizeof(JobDesc) / 8 <= F_THREADS, "copied in 8-byte words");
    if (t < (int)(sizeof(JobDesc) / 8))
      reinterpret_cast<uint64_t*>(&s.job)[t] = reinterpret_cast<const uint64_t*>(&one.job)[t];
  }
  if (t == 0) s.plan_id = -1;
  __syncthreads();

  // pos: an output tile (or tile-slice) of the call, or a k-block of this CTA's range
  const int64_t end = kRanges ? min(total_tiles, (int64_t)(blockIdx.x + 1) * ranges.width) : total_tiles;
  int64_t pos = kRanges ? (int64_t)blockIdx.x * ranges.width : blockIdx.x;
  while (pos < end) {
    const JobDesc& jb = kOne ? s.job : jobs[find_job(jobs, njobs, pos)];
    int64_t local;
    int kbeg, kend;
    double* part = nullptr;             // this piece's partial result, or null: C itself
    if constexpr (kRanges) {
      const int64_t within = pos - jb.tile_begin;
      local = within / jb.per_tile;
      const int64_t tile_end = jb.tile_begin + (local + 1) * jb.per_tile;
      const int kb = (int)(within - local * jb.per_tile);
      const int blocks = (int)(min(end, tile_end) - pos);
      kbeg = kb * F_BK;
      kend = min(jb.k, kbeg + blocks * F_BK);
      pos = min(end, tile_end);
      if (kbeg >= jb.k) continue;       // the padding behind the tile's last k-block
      part = ranges.part + (blockIdx.x + jb.tile0 + local) * (8 * F_BM * F_BN);
    } else {
      const int64_t ntile = (int64_t)jb.tiles_m * jb.tiles_n;
      local = (pos - jb.tile_begin) % ntile;
      const int64_t slice = (pos - jb.tile_begin) / ntile;   // 0 unless the inner dimension is split
      kbeg = (int)slice * jb.kchunk;
      kend = min(jb.k, kbeg + jb.kchunk);
      pos += gridDim.x;
      if (jb.kslices > 1) part = jb.part + (slice * ntile + local) * (8 * F_BM * F_BN);
    }
    const int i0 = (int)(local / jb.tiles_n) * F_BM;
    const int j0 = (int)(local % jb.tiles_n) * F_BN;
    if (s.plan_id != jb.plan) {
      __syncthreads();
      static_assert(sizeof(KPlan) % 8 == 0, "copied in 8-byte words");
      for (int w = t; w < (int)(sizeof(KPlan) / 8); w += F_THREADS)
        reinterpret_cast<uint64_t*>(&s.plan)[w] = reinterpret_cast<const uint64_t*>(plans + jb.plan)[w];
      if (t == 0) s.plan_id = jb.plan;
      __syncthreads();
      for (int w = t; w < 8 * F_MAXP; w += F_THREADS)
        s.wd[w / F_MAXP][w % F_MAXP] = 0.25 * (double)s.plan.w4[w / F_MAXP][w % F_MAXP];
      __syncthreads();
    }
    const int np = kFull ? F_MAXP : s.plan.np;

    double acc[F_MAXP][4];
#pragma unroll
    for (int q = 0; q < F_MAXP; ++q) acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.0;

    // One barrier per k-block.  While the products of block kb run, block kb + 1's
    // factors are formed from its staged components and block kb + F_RING's components
    // are copied; the left side's warps form before their products and the right side's
    // after, so that one of a sub-partition's two warps feeds the FP64 pipe throughout.
    uint32_t negA = 0, negB = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      negA |= jb.signA[c] < 0 ? 1u << c : 0u;
      negB |= jb.signB[c] < 0 ? 1u << c : 0u;
    }
    const int nkb = (kend - kbeg + F_BK - 1) / F_BK;
    if (nkb > 0) {
#pragma unroll
      for (int i = 0; i < F_RING; ++i) {
        if (i < nkb) stage_raw(s, i, jb, i0, j0, kbeg + i * F_BK, kend);
        cp_async_commit();
      }
      cp_async_wait<F_RING - 1>();
      __syncthreads();                // block 0 staged; the previous tile's products finished
      form_factors(s, 0, 0, jb, negA, negB);
    }
    for (int kb = 0; kb < nkb; ++kb) {
      cp_async_wait<F_RING - 2>();
      __syncthreads();                // block kb's factors and block kb + 1's components visible
      const int cur = kb & 1, ahead = kb + F_RING;
      // into the buffer whose factors are formed
      if (ahead < nkb) stage_raw(s, ahead % F_RING, jb, i0, j0, kbeg + ahead * F_BK, kend);
      cp_async_commit();
      const bool more = kb + 1 < nkb;
      if (more && t < F_THREADS / 2) form_factors(s, (kb + 1) % F_RING, cur ^ 1, jb, negA, negB);
#pragma unroll 2
      for (int kk = 0; kk < F_BK; ++kk) {
#pragma unroll
        for (int q = 0; q < F_MAXP; ++q) {
          if (q >= np) break;
          {
            const int fl = kFull ? q : s.plan.pl[q], fr = kFull ? q : s.plan.pr[q];
            const double2 x = *reinterpret_cast<const double2*>(&s.xs[cur][fl][kk][2 * ty]);
            const double2 y = *reinterpret_cast<const double2*>(&s.ys[cur][fr][kk][2 * tx]);
            acc[q][0] = fma(x.x, y.x, acc[q][0]);
            acc[q][1] = fma(x.x, y.y, acc[q][1]);
            acc[q][2] = fma(x.y, y.x, acc[q][2]);
            acc[q][3] = fma(x.y, y.y, acc[q][3]);
          }
        }
      }
      if (more && t >= F_THREADS / 2) form_factors(s, (kb + 1) % F_RING, cur ^ 1, jb, negA, negB);
    }
    cp_async_wait<0>();

    // Epilogue: recombination (weights w4/4, exact), then alpha / beta.
#pragma unroll
    for (int pt = 0; pt < 4; ++pt) {
      const int ti = 2 * ty + (pt >> 1), tj = 2 * tx + (pt & 1);
      double q[8];
      if (kFull || s.plan.bilinear_full) {
        recombine_full(acc, pt, q);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          double o = 0.0;
#pragma unroll
          for (int pp = 0; pp < F_MAXP; ++pp) {
            if (pp < np) {
              if (s.plan.w4[e][pp] != 0) o = fma(acc[pp][pt], s.wd[e][pp], o);
            }
          }
          q[e] = o;
        }
      }
      if (part) {                      // reduced later
        double* dst = part + ti * F_BN + tj;
#pragma unroll
        for (int e = 0; e < 8; ++e) dst[(int64_t)e * (F_BM * F_BN)] = q[e];
      } else if (i0 + ti < jb.m && j0 + tj < jb.n) {
        store_point(jb, i0 + ti, j0 + tj, q);
      }
    }
  }
}

// Split-k reduction of one job: C <- alpha (sum over the slices, in slice
// order) + beta C, one thread per output element.
__global__ void __launch_bounds__(256) fp64_splitk_reduce_kernel(JobDesc jb) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)jb.m * jb.n) return;
  const int i = (int)(idx / jb.n), jj = (int)(idx % jb.n);
  const int64_t ntile = (int64_t)jb.tiles_m * jb.tiles_n;
  const int64_t tile = (int64_t)(i / F_BM) * jb.tiles_n + jj / F_BN;
  const int within = (i % F_BM) * F_BN + jj % F_BN;
  double q[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) q[e] = 0.0;
  for (int sl = 0; sl < jb.kslices; ++sl) {
    const double* src = jb.part + ((int64_t)sl * ntile + tile) * 8 * (F_BM * F_BN) + within;
#pragma unroll
    for (int e = 0; e < 8; ++e) q[e] += src[(int64_t)e * (F_BM * F_BN)];
  }
  store_point(jb, i, jj, q);
}

// Reduction behind the ranges: C <- alpha (sum of the tile's pieces, in k order) +
// beta C, four blocks a tile, one thread per output element.
template <bool kOne>
__global__ void __launch_bounds__(256)
fp64_ranges_reduce_kernel(const __grid_constant__ Fp64One<kOne> one, const JobDesc* jobs, int njobs,
                          Fp64Ranges ranges) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t tile = blockIdx.x >> 2;
  int lo = 0, hi = kOne ? 0 : njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].tile0 <= tile) lo = mid;
    else hi = mid - 1;
  }
  const JobDesc& jb = [&]() -> const JobDesc& {
    if constexpr (kOne) return one.job;
    else return jobs[lo];
  }();
  const int64_t local = tile - jb.tile0;
  const int within = (int)(blockIdx.x & 3) * 256 + threadIdx.x;
  const int i = (int)(local / jb.tiles_n) * F_BM + within / F_BN;
  const int jj = (int)(local % jb.tiles_n) * F_BN + within % F_BN;
  if (i >= jb.m || jj >= jb.n) return;
  double q[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) q[e] = 0.0;
  const int64_t begin = jb.tile_begin + local * jb.per_tile;
  const int64_t last = begin + (jb.k + F_BK - 1) / F_BK - 1;   // before begin: k = 0, no pieces
  if (last >= begin) {
    const int64_t c0 = begin / ranges.width;
    const int pieces = (int)(last / ranges.width - c0) + 1;
    const double* src = ranges.part + (c0 + tile) * (8 * F_BM * F_BN) + within;
    // four pieces' loads in flight (a tile that every SM shares has a hundred or more)
#pragma unroll 4
    for (int c = 0; c < pieces; ++c, src += 8 * F_BM * F_BN) {
#pragma unroll
      for (int e = 0; e < 8; ++e) q[e] += src[(int64_t)e * (F_BM * F_BN)];
    }
  }
  store_point(jb, i, jj, q);
}

cudaError_t launch_fp64_ranges_reduce(const JobDesc* one, const JobDesc* d_jobs, int njobs, const Fp64Ranges& ranges,
                                      cudaStream_t stream) {
  const dim3 grid((unsigned)(4 * ranges.tiles));
  if (one)
    return launch_dependent(fp64_ranges_reduce_kernel<true>, grid, dim3(256), 0, stream, Fp64One<true>{*one}, d_jobs,
                            njobs, ranges);
  return launch_dependent(fp64_ranges_reduce_kernel<false>, grid, dim3(256), 0, stream, Fp64One<false>{}, d_jobs,
                          njobs, ranges);
}

cudaError_t launch_fp64_splitk_reduce(const JobDesc& jb, cudaStream_t stream) {
  const int64_t elems = (int64_t)jb.m * jb.n;
  if (elems <= 0) return cudaSuccess;
  fp64_splitk_reduce_kernel<<<(unsigned)((elems + 255) / 256), 256, 0, stream>>>(jb);
  return cudaGetLastError();
}

// Bytes of the split-k partial outputs of one product with kslices slices.
int64_t fp64_splitk_bytes(int64_t m, int64_t n, int kslices) {
  const int64_t tiles = ((m + F_BM - 1) / F_BM) * ((n + F_BN - 1) / F_BN);
  return kslices > 1 ? (int64_t)kslices * tiles * 8 * F_BM * F_BN * (int64_t)sizeof(double) : 0;
}

size_t fp64_smem_bytes() { return sizeof(Fp64Smem); }

cudaError_t fp64_configure() {
  cudaError_t e = cudaSuccess;
  auto set = [&e](auto kernel) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Fp64Smem));
  };
  set(fp64_bilinear_kernel<false, false, false>);
  set(fp64_bilinear_kernel<false, false, true>);
  set(fp64_bilinear_kernel<true, false, false>);
  set(fp64_bilinear_kernel<true, true, false>);
  set(fp64_bilinear_kernel<true, true, true>);
  return e;
}

// True when product q of the plan multiplies factors q and its products recombine as the
// paper's full plan (kFull).
bool fp64_full_plan(const KPlan& p) {
  for (int q = 0; q < F_MAXP; ++q)
    if (p.pl[q] != q || p.pr[q] != q) return false;
  return p.bilinear_full != 0 && p.np == F_MAXP && !p.four_m;
}

// d_jobs: njobs of them; one: the only job of a call cut into ranges, or null; full:
// every plan is fp64_full_plan
cudaError_t launch_fp64_bilinear(const JobDesc* one, const JobDesc* d_jobs, int njobs, const KPlan* d_plans,
                                 int64_t total_tiles, int grid, const Fp64Ranges& ranges, bool full,
                                 cudaStream_t stream) {
  auto go = [&](auto kernel, const auto& job) {
    return launch_dependent(kernel, dim3((unsigned)grid), dim3(F_THREADS), sizeof(Fp64Smem), stream, job, d_jobs,
                            njobs, d_plans, total_tiles, ranges);
  };
  if (one)
    return full ? go(fp64_bilinear_kernel<true, true, true>, Fp64One<true>{*one})
                : go(fp64_bilinear_kernel<true, true, false>, Fp64One<true>{*one});
  if (ranges.width > 0) return go(fp64_bilinear_kernel<true, false, false>, Fp64One<false>{});
  return full ? go(fp64_bilinear_kernel<false, false, true>, Fp64One<false>{})
              : go(fp64_bilinear_kernel<false, false, false>, Fp64One<false>{});
}

int64_t fp64_ranges_bytes(const Fp64Ranges& r) {
  return (r.ctas + r.tiles) * (int64_t)(8 * F_BM * F_BN * sizeof(double));
}

int fp64_block_k() { return F_BK; }
int fp64_tile_m() { return F_BM; }
int fp64_max_products() { return F_MAXP; }
int fp64_tile_n() { return F_BN; }
int fp64_tile_k() { return F_KALIGN; }

}  // namespace hmat
