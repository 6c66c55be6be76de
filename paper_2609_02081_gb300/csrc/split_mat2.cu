// split_mat2.cu — the matrix form of the split mode's full biquaternion products:
// encoder and CRT (the residue GEMM between them is split_gemm.cu's).
//
// Modulo an odd p all of whose prime factors are 1 modulo 4 there is an s with
// s^2 = -1, so i -> s and i -> -s map the complex integers onto two copies of
// Z_p, and through
//     q1 + q2 i + q3 j + q4 k  ->  [[q1 + I q2, q3 + I q4], [-q3 + I q4, q1 - I q2]]
// (I the imaginary unit of the coefficients) the biquaternions map onto two
// copies of the 2 x 2 matrices over Z_p.  A product is then two independent 2 x 2
// products, each with Strassen's seven multiplications in Winograd's variant
// (S. Winograd, "On multiplication of 2 x 2 matrices", 1971):
//     S1 = x21 + x22, S2 = S1 - x11, S3 = x11 - x21, S4 = x12 - S2,
//     T1 = y12 - y11, T2 = y22 - T1, T3 = y22 - y12, T4 = T2 - y21,
//     P1 = x11 y11, P2 = x12 y21, P3 = S4 y22, P4 = x22 T4, P5 = S1 T1, P6 = S2 T2, P7 = S3 T3,
//     c11 = P1 + P2, c12 = P1 + P6 + P5 + P3, c21 = P1 + P6 + P7 - P4, c22 = P1 + P6 + P7 + P5.
// That is 14 residue GEMMs per modulus where the paper's bilinear scheme has 24;
// the moduli are smaller (15 of 111 bits where the plans' 14 have 109), so a
// product at tol 1e-12 takes 210 GEMMs instead of 336.  Every residue is exact,
// and the integers recovered are those of the plans' forms.
//
// Factor plane f of a side and product plane f: P_{f+1} of the copy i -> s for
// f < 7, P_{f-6} of the copy i -> -s for f >= 7.
#include <cuda_runtime.h>

#include <cmath>

#include "split_device.cuh"

namespace hmat {

namespace {

constexpr int kPlanes = kMat2Planes;

// Per modulus: the digit weights w[d] = 2^(16 d) and s 2^(16 d), centred.
struct Mat2Mod {
  float npf, inv;       // -p, fl(1/p)
  float w[4], sw[4];
};
__constant__ Mat2Mod c_m2[kMaxModuli];
// [nmod][0]: CRT elements carrying 1/4, [nmod][1]: 1/(4 s); signed 32-bit digits
// (five padded to eight, for vector loads)
__constant__ int4 c_m2crt[kMaxModuli + 1][2][kMaxModuli][2];
__constant__ uint32_t c_m2P[kMaxModuli + 1][kLimbs];
__constant__ uint32_t c_m2off[kMaxModuli + 1][kLimbs];   // N P with N = nmod * kMat2WeightSum * kMat2HalfMax
__constant__ float c_m2Pinv[kMaxModuli + 1];
__constant__ int c_m2Pbase[kMaxModuli + 1];

// v - p round(v / p) on two lanes; v / p is off by at most |v| 2^-25 / p before
// the rounding, so |result| <= p / 2 + |v| 2^-25 + ... < 122 for |v| < 2^24
__device__ __forceinline__ float2 fmod2(float2 v, float2 npf, float2 inv) {
  const float2 q = __fadd2_rn(__ffma2_rn(v, inv, f2(12582912.0f)), f2(-12582912.0f));
  return __ffma2_rn(q, npf, v);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.0f), a); }

constexpr int kRows = 16, kK = 32, kThreads = 128, kPitch = kK + 2;

// ND balanced 16-bit digits of two neighbouring integers as floats: X = sum_d
// x_d 2^(16 d), the low ones in [-2^15, 2^15).  Adding 2^15 to every low digit
// makes them unsigned halves of the words, which a byte permute places under the
// exponent of 2^23.
template <int ND>
__device__ __forceinline__ void digits2(longlong2 X, float2 (&d)[ND]) {
  constexpr long long bias = ND == 3 ? 0x80008000ll : 0x800080008000ll;
  const unsigned long long a = (unsigned long long)(X.x + bias), b = (unsigned long long)(X.y + bias);
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  auto half = [](uint32_t word, uint32_t sel) {
    return __uint_as_float(__byte_perm(word, 0x4B000000u, sel)) - 8421376.0f;   // 2^23 + 2^15
  };
  d[0] = make_float2(half(al, 0x7610), half(bl, 0x7610));
  d[1] = make_float2(half(al, 0x7632), half(bl, 0x7632));
  if constexpr (ND == 3) {
    d[2] = make_float2((float)(int)ah, (float)(int)bh);
  } else {
    d[2] = make_float2(half(ah, 0x7610), half(bh, 0x7610));
    d[3] = make_float2((float)((int)ah >> 16), (float)((int)bh >> 16));
  }
}

// One thread's pair of k positions of one row: for every modulus the four matrix
// entries of both copies and the seven factors of each, 4-byte stores.
template <int ND, int SIDE>
__device__ __forceinline__ void encode_pair(const longlong2 (&E)[8], int nmod, unsigned char* out,
                                            uint32_t plane_bytes) {
  float2 d[8][ND];
#pragma unroll
  for (int e = 0; e < 8; ++e) digits2<ND>(E[e], d[e]);
  for (int l = 0; l < nmod; ++l) {
    const Mat2Mod& mc = c_m2[l];
    const float2 npf = f2(mc.npf), inv = f2(mc.inv);
    // entries 11, 12, 21, 22 of the copies i -> s (u) and i -> -s (v): |sum of
    // weighted digits| < 2^24 (checked when the root s is chosen)
    float2 u[4], v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float2 re = d[2 * e][0], im = __fmul2_rn(d[2 * e + 1][0], f2(mc.sw[0]));
#pragma unroll
      for (int q = 1; q < ND; ++q) {
        re = __ffma2_rn(d[2 * e][q], f2(mc.w[q]), re);
        im = __ffma2_rn(d[2 * e + 1][q], f2(mc.sw[q]), im);
      }
      u[e] = fmod2(__fadd2_rn(re, im), npf, inv);
      v[e] = fmod2(sub2(re, im), npf, inv);
    }
    // |residue| <= 121 is exact in BF16, whose bits are the upper half of the float's
    auto put = [&](float2 x) {
      *reinterpret_cast<uint32_t*>(out) = __byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x7632);
      out += plane_bytes;
    };
    auto factors = [&](const float2 (&x)[4]) {
      if (SIDE == 0) {
        const float2 s1 = __fadd2_rn(x[2], x[3]);
        const float2 s2 = sub2(s1, x[0]);
        const float2 s4 = sub2(x[1], s2);
        put(x[0]);
        put(x[1]);
        put(fmod2(s4, npf, inv));
        put(x[3]);
        put(fmod2(s1, npf, inv));
        put(fmod2(s2, npf, inv));
        put(fmod2(sub2(x[0], x[2]), npf, inv));
      } else {
        const float2 t3 = sub2(x[3], x[1]);
        const float2 t2 = __fadd2_rn(t3, x[0]);
        put(x[0]);
        put(x[2]);
        put(x[3]);
        put(fmod2(sub2(t2, x[2]), npf, inv));
        put(fmod2(sub2(x[1], x[0]), npf, inv));
        put(fmod2(t2, npf, inv));
        put(fmod2(t3, npf, inv));
      }
    };
    factors(u);
    factors(v);
  }
}

// One block per tile of 16 rows x 32 k of one side (op(A) rows or op(B)
// columns), every modulus.
//   phase 1: the present components of the tile are read (coalesced along
//            whichever index is contiguous in memory, all loads of a thread in
//            flight at once), scaled to integers, combined to the real and
//            imaginary parts of the four matrix entries and staged in shared memory;
//   phase 2: a thread takes two neighbouring k of one row, splits its eight
//            integers into float digits once, holds them in registers over the
//            moduli and stores one bfloat162 per factor plane: 16 lanes fill one
//            aligned half of a swizzled 128-byte row.
// Bound by its writes (28 bytes per modulus and element).
template <int ND>
__global__ void __launch_bounds__(kThreads, 4) mat2_encode_kernel(const SplitJob* __restrict__ jobs, int njobs,
                                                                  unsigned char* __restrict__ ws, int64_t first) {
  __shared__ __align__(16) long long ent[8][kRows][kPitch];
  __shared__ int s_row[kRows];
  const int64_t blk = first + blockIdx.x;
  const SplitJob& sj = jobs[find_split_job(jobs, njobs, blk, 5)];
  const JobDesc& d = sj.d;
  const int ktiles = sj.nkb * (kTileK / kK);
  const int64_t a_blocks = (int64_t)((d.m + kRows - 1) / kRows) * ktiles;
  int64_t local = blk - sj.enc2_begin;
  const int side = local >= a_blocks ? 1 : 0;
  if (side) local -= a_blocks;
  const int tile_rows = side ? sj.bn : kTileM;
  const int rows_pad = (side ? sj.tiles_n : sj.tiles_m) * tile_rows;
  const int r0 = (int)(local / ktiles) * kRows;
  const int k0 = (int)(local % ktiles) * kK;
  const int nout = side ? d.n : d.m;
  const uint32_t flags = side ? d.fb : d.fa;
  const double* base = side ? d.B : d.A;
  const int64_t ld = side ? d.ldb : d.lda, cs = side ? d.sB : d.sA;
  const int8_t* sign = side ? d.signB : d.signA;
  const bool contiguous = side ? (d.transB != 0) : (d.transA == 0);
  const int t = threadIdx.x;
  if (t < kRows) {
    const int r = r0 + t;
    s_row[t] = (r < nout) ? reinterpret_cast<const int32_t*>(ws + (side ? sj.off_texp : sj.off_sexp))[r] : 0;
  }
  constexpr int kPos = kRows * kK / kThreads;    // positions per thread
  unsigned long long raw[kPos][8];
#pragma unroll
  for (int u = 0; u < kPos; ++u) {
    const int idx = t + u * kThreads;
    const int rr = contiguous ? idx / kK : idx % kRows, kk = contiguous ? idx % kK : idx / kRows;
    const int r = r0 + rr, kg = k0 + kk;
    const bool in = r < nout && kg < d.k;
    const double* src = base + (contiguous ? (int64_t)r * ld + kg : (int64_t)kg * ld + r);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      raw[u][c] = 0ull;
      if (in && ((flags >> c) & 1u))
        raw[u][c] = (unsigned long long)__double_as_longlong(__ldcs(src + (int64_t)c * cs));
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kPos; ++u) {
    const int idx = t + u * kThreads;
    const int rr = contiguous ? idx / kK : idx % kRows, kk = contiguous ? idx % kK : idx / kRows;
    const int s = s_row[rr];
    long long X[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      X[c] = scaled_int(raw[u][c], s);
      if (sign[c] < 0) X[c] = -X[c];
    }
    // a_e = X[e], b_e = X[e + 4]: Re and Im of entries 11, 12, 21, 22
    ent[0][rr][kk] = X[0] - X[5];
    ent[1][rr][kk] = X[4] + X[1];
    ent[2][rr][kk] = X[2] - X[7];
    ent[3][rr][kk] = X[6] + X[3];
    ent[4][rr][kk] = -X[2] - X[7];
    ent[5][rr][kk] = X[3] - X[6];
    ent[6][rr][kk] = X[0] + X[5];
    ent[7][rr][kk] = X[4] - X[1];
  }
  __syncthreads();

  const int64_t tile_bytes = (int64_t)tile_rows * kTileK * 2;
  const uint32_t plane_bytes = (uint32_t)(side ? sj.encB_plane : sj.encA_plane);   // below 2^32 (checked on the host)
  unsigned char* enc = ws + (side ? sj.off_encB : sj.off_encA);
  const int nmod = sj.nmod;
#pragma unroll 1
  for (int pass = 0; pass < kRows * kK / 2 / kThreads; ++pass) {
    const int pos = t + pass * kThreads;
    const int rr = pos / (kK / 2), kp = 2 * (pos % (kK / 2));
    const int r = r0 + rr;
    if (r >= rows_pad) return;
    const int kg = k0 + kp;
    const int kb = kg / kTileK, c16 = (kg % kTileK) / 8, in16 = (kg % 8) * 2;
    const int rt = r / tile_rows, rin = r % tile_rows;
    unsigned char* out = enc + ((int64_t)rt * sj.nkb + kb) * tile_bytes + (int64_t)(rin >> 3) * 1024 +
                         (rin & 7) * 128 + ((c16 ^ (rin & 7)) << 4) + in16;
    longlong2 E[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) E[e] = *reinterpret_cast<const longlong2*>(&ent[e][rr][kp]);
    if (side) encode_pair<ND, 1>(E, nmod, out, plane_bytes);
    else encode_pair<ND, 0>(E, nmod, out, plane_bytes);
  }
}

// ------------------------------------------------------------------ CRT
// One block per output row segment of 128 elements (one row of 128 columns, or
// four rows of 32 for narrow products) and two threads per element: the first
// half works on the sums u + v of the two copies' residues, the other on u - v.
// The 14 planes of four moduli at a time are copied into a three-slot ring with
// cp.async, two groups ahead, one barrier per group.  With t = u +- v:
//   half 0: M1 = (c11 + c22)/4, M6 = (c22 - c11)/4, M3 = (c12 - c21)/4, M8 = -(c12 + c21)/4
//   half 1: M5 = (c11 + c22)/4s, M2 = (c11 - c22)/4s, M7 = (c12 - c21)/4s, M4 = (c12 + c21)/4s
// (M8 imaginary part of q4, ...): slot e of half h is component (4 h + e), moved
// to the other half's part for odd e.  The sums of c11, c12, c21, c22 times the
// CRT elements (which carry 1/4 or 1/(4s)) accumulate in signed 64-bit limb sums;
// the outputs are their sums and differences plus N P.
constexpr int kGroup = 4, kSlots = 3;

template <int L, bool kWide>
__global__ void __launch_bounds__(2 * kCrtCols, L <= 4 ? 4 : 3) mat2_crt_kernel(const SplitJob* __restrict__ jobs,
                                                                                int njobs,
                                                                                unsigned char* __restrict__ ws) {
  __shared__ __align__(16) uint8_t ring[kSlots][kGroup][kPlanes][kCrtCols];
  __shared__ double xch[8][kCrtCols];
  const int64_t blk = blockIdx.x;
  const SplitJob& sj = jobs[find_split_job(jobs, njobs, blk, 6)];
  const JobDesc& d = sj.d;
  const int nm = sj.nmod;
  const int tid = threadIdx.x;
  const int col = tid % kCrtCols, half = tid / kCrtCols;
  const int w = kWide ? kCrtCols : sj.crt_w;
  const int64_t local = blk - sj.crt2_begin;
  const int colblocks = (d.n + w - 1) / w;
  const int i0 = (int)(local / colblocks) * (kCrtCols / w);
  const int j0 = (int)(local % colblocks) * w;
  const int64_t ncols = (int64_t)sj.tiles_n * sj.bn;
  const int64_t plane = sj.res_plane;
  // threads below 2 * 14 * 8 copy two 16-byte chunks per group: chunk cc of plane
  // pc of moduli ml and ml + 2
  constexpr int kChunks = kCrtCols / 16;
  const int ml = tid / (kPlanes * kChunks), pc = tid % (kPlanes * kChunks) / kChunks, cc = tid % kChunks;
  const int cw = w / 16, crow = cc / cw, ccol = (cc % cw) * 16;
  const bool has = ml < 2 && i0 + crow < d.m && (int64_t)j0 + ccol < ncols;
  const unsigned char* src = ws + sj.off_res + ((int64_t)ml * kPlanes + pc) * plane + (int64_t)(i0 + crow) * ncols +
                             j0 + ccol;
  const int64_t mod2 = 2 * kPlanes * plane;     // bytes between moduli l and l + 2
  uint8_t* const dst = &ring[0][0][0][0] + (ml * kPlanes + pc) * kCrtCols + cc * 16;
  auto issue = [&](int g, int slot) {
    const int l = g * kGroup + ml;
    uint8_t* to = dst + slot * (kGroup * kPlanes * kCrtCols);
    if (has && l < nm) cp_async16(to, src + (int64_t)(2 * g) * mod2);
    if (has && l + 2 < nm) cp_async16(to + 2 * kPlanes * kCrtCols, src + (int64_t)(2 * g + 1) * mod2);
    cp_async_commit();
  };
  const int groups = (nm + kGroup - 1) / kGroup;
  issue(0, 0);
  issue(1, 1);
  long long acc[4][L];                          // c11, c12, c21, c22
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int q = 0; q < L; ++q) acc[e][q] = 0;
  const int sg = half ? -1 : 1;
  const int4* crt = c_m2crt[nm][half][0];
  int slot = 0;
#pragma unroll 1
  for (int g = 0; g < groups; ++g) {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");   // group g has landed
    __syncthreads();
    // the slot refilled here was read in group g - 1, which every thread has
    // finished at this barrier
    issue(g + 2, slot == 0 ? 2 : slot - 1);
#pragma unroll
    for (int m = 0; m < kGroup; ++m) {
      const int l = g * kGroup + m;
      if (l < nm) {
        const uint8_t(*pl)[kCrtCols] = ring[slot][m];
        int tt[7];
#pragma unroll
        for (int r = 0; r < 7; ++r) tt[r] = (int)(int8_t)pl[r][col] + sg * (int)(int8_t)pl[r + 7][col];
        const int u1 = tt[0] + tt[5], u2 = u1 + tt[6];
        const int c[4] = {tt[0] + tt[1], u1 + tt[4] + tt[2], u2 - tt[3], u2 + tt[4]};
        const int4 lo = crt[2 * l];
        int dg[L];
        dg[0] = lo.x;
        dg[1] = lo.y;
        dg[2] = lo.z;
        dg[3] = lo.w;
        if constexpr (L > 4) dg[4] = crt[2 * l + 1].x;
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int q = 0; q < L; ++q) acc[e][q] += (long long)c[e] * dg[q];
      }
    }
    slot = slot == kSlots - 1 ? 0 : slot + 1;
  }

  // outputs
  const int i = i0 + (kWide ? 0 : col / w), j = j0 + (kWide ? col : col % w);
  const bool valid = i < d.m && j < d.n;
  double q4v[4] = {0.0, 0.0, 0.0, 0.0};
  if (valid) {
    const int sc = -(reinterpret_cast<const int32_t*>(ws + sj.off_sexp)[i] +
                     reinterpret_cast<const int32_t*>(ws + sj.off_texp)[j]);
    const int pb = c_m2Pbase[nm];
    const float pinv = c_m2Pinv[nm];
    const uint32_t* P = c_m2P[nm];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      long long s[L];
#pragma unroll
      for (int q = 0; q < L; ++q) {
        const long long x = e < 2 ? acc[0][q] : acc[1][q], y = e < 2 ? acc[3][q] : acc[2][q];
        // e = 0: c11 + c22; 1: +-(c22 - c11); 2: c12 - c21; 3: -+(c12 + c21)
        const long long z = e == 0 ? x + y : e == 1 ? y - x : e == 2 ? x - y : -(x + y);
        s[q] = (long long)c_m2off[nm][q] + ((e & 1) && half ? -z : z);
      }
      q4v[e] = crt_value<L>(s, P, pb, pinv, sc);
    }
  }
  // slot e holds component own(e), whose partner under multiplication by i is own(e) ^ 4
  auto own = [&](int e) { return (4 * half + e) ^ ((e & 1) << 2); };
  double* cbase = d.C + (int64_t)i * d.ldc + j;
  const bool plain = (d.alpha_re == 1.0 && d.alpha_im == 0.0 && d.beta_re == 0.0 && d.beta_im == 0.0);
  if (plain) {                                  // block-uniform
    if (valid) {
#pragma unroll
      for (int e = 0; e < 4; ++e) cbase[(int64_t)own(e) * d.sC] = q4v[e];
    }
    return;
  }
  // both C values of a pair are read before the exchange barrier, written after it
  const bool use_beta = (d.beta_re != 0.0 || d.beta_im != 0.0);
  double cown[4] = {0.0, 0.0, 0.0, 0.0}, coth[4] = {0.0, 0.0, 0.0, 0.0};
  if (valid && use_beta) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      cown[e] = cbase[(int64_t)own(e) * d.sC];
      coth[e] = cbase[(int64_t)(own(e) ^ 4) * d.sC];
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) xch[own(e)][col] = q4v[e];
  __syncthreads();
  if (!valid) return;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    // real components: a_r Q - a_i Q' + b_r C - b_i C'; imaginary ones: plus signs
    const double sgn = own(e) < 4 ? -1.0 : 1.0;
    const double qo = xch[own(e) ^ 4][col];
    double v = d.alpha_re * q4v[e] + sgn * d.alpha_im * qo;
    if (use_beta) v += d.beta_re * cown[e] + sgn * d.beta_im * coth[e];
    cbase[(int64_t)own(e) * d.sC] = v;
  }
}

}  // namespace

cudaError_t mat2_configure(const int* moduli, const int* root, int n, const int32_t* crt_d, const uint32_t* crt_P,
                           const uint32_t* crt_off) {
  Mat2Mod mc[kMaxModuli];
  if (n != kMaxModuli) return cudaErrorInvalidValue;
  for (int l = 0; l < n; ++l) {
    const long long p = moduli[l];
    if (p > 2 * kMat2HalfMax + 1) return cudaErrorInvalidValue;
    auto centred = [p](long long v) {
      const long long r = ((v % p) + p) % p;
      return (float)(r > (p - 1) / 2 ? r - p : r);
    };
    mc[l].npf = -(float)p;
    mc[l].inv = 1.0f / (float)p;
    for (int q = 0; q < 4; ++q) {
      const long long wq = (1ll << (16 * q)) % p;
      mc[l].w[q] = centred(wq);
      mc[l].sw[q] = centred(wq * root[l]);
    }
  }
  cudaError_t e = cudaMemcpyToSymbol(c_m2, mc, sizeof(mc));
  if (e != cudaSuccess) return e;
  static int4 crt[kMaxModuli + 1][2][kMaxModuli][2];
  for (int m = 0; m <= kMaxModuli; ++m)
    for (int h = 0; h < 2; ++h)
      for (int l = 0; l < kMaxModuli; ++l) {
        const int32_t* x = crt_d + (((int64_t)m * 2 + h) * kMaxModuli + l) * kLimbs;
        crt[m][h][l][0] = make_int4(x[0], x[1], x[2], x[3]);
        crt[m][h][l][1] = make_int4(x[4], 0, 0, 0);
      }
  e = cudaMemcpyToSymbol(c_m2crt, crt, sizeof(crt));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2P, crt_P, sizeof(uint32_t) * (kMaxModuli + 1) * kLimbs);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2off, crt_off, sizeof(uint32_t) * (kMaxModuli + 1) * kLimbs);
  if (e != cudaSuccess) return e;
  float pinv[kMaxModuli + 1];
  int pb[kMaxModuli + 1];
  for (int m = 0; m <= kMaxModuli; ++m)
    if (!crt_estimate_constants(crt_P + m * kLimbs, 2.0 * m * kMat2WeightSum * kMat2HalfMax, m <= kMat2FourLimbs ? 4 : 5,
                                &pb[m], &pinv[m]))
      return cudaErrorInvalidValue;
  e = cudaMemcpyToSymbol(c_m2Pbase, pb, sizeof(pb));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_m2Pinv, pinv, sizeof(pinv));
}

cudaError_t launch_mat2_encode(const SplitJob* d_jobs, int njobs, int64_t units, int64_t first, cudaStream_t s,
                               unsigned char* ws, int max_bits) {
  if (units <= 0) return cudaSuccess;
  // the matrix entries are sums of two b-bit integers: three digits hold 2^47
  if (max_bits <= 46) mat2_encode_kernel<3><<<(unsigned)units, kThreads, 0, s>>>(d_jobs, njobs, ws, first);
  else mat2_encode_kernel<4><<<(unsigned)units, kThreads, 0, s>>>(d_jobs, njobs, ws, first);
  return cudaGetLastError();
}

cudaError_t launch_mat2_crt(const SplitJob* d_jobs, int njobs, int64_t units, cudaStream_t s, unsigned char* ws,
                            int max_nmod, bool all_wide) {
  if (units <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)units, block = 2 * kCrtCols;
  if (max_nmod <= kMat2FourLimbs) {
    if (all_wide) mat2_crt_kernel<4, true><<<grid, block, 0, s>>>(d_jobs, njobs, ws);
    else mat2_crt_kernel<4, false><<<grid, block, 0, s>>>(d_jobs, njobs, ws);
  } else {
    if (all_wide) mat2_crt_kernel<kLimbs, true><<<grid, block, 0, s>>>(d_jobs, njobs, ws);
    else mat2_crt_kernel<kLimbs, false><<<grid, block, 0, s>>>(d_jobs, njobs, ws);
  }
  return cudaGetLastError();
}

}  // namespace hmat
