// split_mat2.cu — the matrix form of split-mode products: encoder and CRT (the
// residue GEMM between them is split_gemm.cu's).
//
// Modulo an odd p all of whose prime factors are 1 modulo 4 there is an s with
// s^2 = -1.  Two consequences, each exact in integers modulo p:
//   * i -> s and i -> -s map the complex integers onto two copies of Z_p: a
//     complex product is two real ones (u: i -> s, v: i -> -s) instead of Gauss's
//     three;
//   * q1 + q2 i + q3 j + q4 k -> [[q1 + s q2, q3 + s q4], [-q3 + s q4, q1 - s q2]]
//     maps the quaternions over Z_p onto the 2 x 2 matrices over Z_p: a quaternion
//     product takes Strassen's seven multiplications, in Winograd's variant
//     (S. Winograd, "On multiplication of 2 x 2 matrices", 1971):
//       S1 = x21 + x22, S2 = S1 - x11, S3 = x11 - x21, S4 = x12 - S2,
//       T1 = y12 - y11, T2 = y22 - T1, T3 = y22 - y12, T4 = T2 - y21,
//       P1 = x11 y11, P2 = x12 y21, P3 = S4 y22, P4 = x22 T4, P5 = S1 T1, P6 = S2 T2, P7 = S3 T3,
//       c11 = P1 + P2, c12 = P1 + P6 + P5 + P3, c21 = P1 + P6 + P7 - P4, c22 = P1 + P6 + P7 + P5.
// Residue GEMMs per modulus, against the plan's (Eq. bilinearH with Gauss):
//   biquaternion x biquaternion                    14  (two copies of 7)   24
//   real (or i times real) quaternion x biquaternion  14                   16
//   real quaternion x real quaternion               7                      8
//   complex x biquaternion                          8  (two copies of 4)   12
//   complex x complex                               2                      3
// The moduli are smaller (15 of 111 bits where the plans' 14 have 109): a full
// product at tol 1e-12 takes 210 GEMMs instead of 336.  Every residue is exact,
// and the integers recovered are those of the plans' forms.
//
// Factor and product planes: the seven of Winograd's order (P1..P7; the left
// factors x11, x12, S4, x22, S1, S2, S3), copy u then copy v; complex x
// biquaternion: the four coefficients, copy u then copy v.  A real quaternion is
// the same in both copies and is encoded once.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <type_traits>

#include "split_device.cuh"

namespace hmat {

namespace {

// Per modulus: the digit weights w[d] = 2^(16 d) and s 2^(16 d), centred.
struct Mat2Mod {
  float npf, inv;       // -p, fl(1/p)
  float w[4], sw[4];
};
__constant__ Mat2Mod c_m2[kMat2MaxModuli];
// The CRT's tables by modulus count, all scaled by 2^shift (shift: so that the
// sums of up to kMat2FourLimbs moduli fill 128 bits and their leading limb alone
// gives the quotient; 0 for more moduli): the modulus product P, 2^128 - P, and per
// half and slot the offset N P, N = nmod * kMat2WeightSum * kMat2HalfMax, less the
// constants that the 128 added to every residue and the 2^31 added to every
// digit pair contribute.
__constant__ uint32_t c_m2P[kMat2MaxModuli + 1][kLimbs];
__constant__ uint4 c_m2negP[kMat2MaxModuli + 1];
// ([0]: matrix products, [1]: complex x biquaternion)
__constant__ long long c_m2off[kMat2MaxModuli + 1][2][2][4][kLimbs];   // per limb
__constant__ uint4 c_m2off4[kMat2MaxModuli + 1][2][2][4];              // modulo 2^128
__constant__ int c_m2shift[kMat2MaxModuli + 1];
__constant__ float c_m2Pinv[kMat2MaxModuli + 1];    // crt_estimate_constants
__constant__ float c_m2Pinv4[kMat2MaxModuli + 1];   // fl(2^96 / P)
__constant__ int c_m2Pbase[kMat2MaxModuli + 1];

// v - p round(v / p) on two lanes; v / p is off by at most |v| 2^-25 / p before
// the rounding, so |result| <= p / 2 + |v| 2^-25 + ... < 122 for |v| < 2^24
__device__ __forceinline__ float2 fmod2(float2 v, float2 npf, float2 inv) {
  const float2 q = __fadd2_rn(__ffma2_rn(v, inv, f2(12582912.0f)), f2(-12582912.0f));
  return __ffma2_rn(q, npf, v);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.0f), a); }

constexpr int kRows = 16, kK = 32, kThreads = 128, kPitch = kK + 2;
enum { kOpFull = 0, kOpQuat = 1, kOpCoef = 2, kOpCplx = 3 };   // what a side's operand is encoded as

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

// The left (SIDE 0) or right factors of one 2 x 2 product from the entries 11, 12, 21, 22.
template <int SIDE, class Put>
__device__ __forceinline__ void matrix_factors(const float2 (&x)[4], float2 npf, float2 inv, Put&& put) {
  if (SIDE == 0) {
    const float2 s1 = __fadd2_rn(x[2], x[3]);
    const float2 s2 = sub2(s1, x[0]);
    put(x[0]);
    put(x[1]);
    put(fmod2(sub2(x[1], s2), npf, inv));
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
}

// One thread's pair of k positions of one row: the digits stay in registers over
// the moduli; 4-byte stores, one per factor plane.
//   OPERAND kOpFull:  E = Re, Im of the entries 11, 12, 21, 22 (integers): 14 planes
//           kOpQuat:  E = the four real components: 7 planes
//           kOpCoef:  E = Re, Im of the four coefficients: 8 planes
//           kOpCplx:  E = Re, Im: 2 planes
template <int ND, int SIDE, int OPERAND>
__device__ __forceinline__ void encode_pair(const longlong2* E, int l0, int l1, unsigned char* out,
                                            uint32_t plane_bytes) {
  constexpr int kPairs = OPERAND == kOpQuat ? 2 : OPERAND == kOpCplx ? 1 : 4;   // (Re, Im) pairs
  float2 d[2 * kPairs][ND];
#pragma unroll
  for (int e = 0; e < 2 * kPairs; ++e) digits2<ND>(E[e], d[e]);
  for (int l = l0; l < l1; ++l) {
    const Mat2Mod& mc = c_m2[l];
    const float2 npf = f2(mc.npf), inv = f2(mc.inv);
    // |residue| <= 121 is exact in BF16, whose bits are the upper half of the float's
    auto put = [&](float2 x) {
      *reinterpret_cast<uint32_t*>(out) = __byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x7632);
      out += plane_bytes;
    };
    // Re + s Im and Re - s Im: |sum of weighted digits| < 2^24 (checked when the
    // root s is chosen)
    float2 u[4], v[4];
#pragma unroll
    for (int e = 0; e < kPairs; ++e) {
      float2 re = d[2 * e][0], im = __fmul2_rn(d[2 * e + 1][0], f2(mc.sw[0]));
#pragma unroll
      for (int q = 1; q < ND; ++q) {
        re = __ffma2_rn(d[2 * e][q], f2(mc.w[q]), re);
        im = __ffma2_rn(d[2 * e + 1][q], f2(mc.sw[q]), im);
      }
      u[e] = fmod2(__fadd2_rn(re, im), npf, inv);
      // (the copy v's entries 12 and 21 are s Im - Re of the other one)
      const bool neg = (OPERAND == kOpFull && (e == 1 || e == 2)) || (OPERAND == kOpQuat && e == 1);
      v[e] = fmod2(neg ? sub2(im, re) : sub2(re, im), npf, inv);
    }
    if constexpr (OPERAND == kOpFull) {
      const float2 vm[4] = {v[3], v[2], v[1], v[0]};
      matrix_factors<SIDE>(u, npf, inv, put);
      matrix_factors<SIDE>(vm, npf, inv, put);
    } else if constexpr (OPERAND == kOpQuat) {
      // 11: a1 + s a2, 12: a3 + s a4, 21: s a4 - a3, 22: a1 - s a2
      const float2 x[4] = {u[0], u[1], v[1], v[0]};
      matrix_factors<SIDE>(x, npf, inv, put);
    } else {
#pragma unroll
      for (int e = 0; e < kPairs; ++e) put(u[e]);
#pragma unroll
      for (int e = 0; e < kPairs; ++e) put(v[e]);
    }
  }
}

// One block per tile of 16 rows x 32 k of one side (op(A) rows or op(B)
// columns), every modulus.
//   phase 1: the present components of the tile are read (coalesced along
//            whichever index is contiguous in memory, all loads of a thread in
//            flight at once), scaled to integers, for a full operand combined to
//            the real and imaginary parts of its matrix entries, and staged in
//            shared memory;
//   phase 2: a thread takes two neighbouring k of one row, splits its eight
//            integers into float digits once, holds them in registers over the
//            moduli and stores one bfloat162 per factor plane: 16 lanes fill one
//            aligned half of a swizzled 128-byte row (or a row of a half block).
// Bound by its writes (28 bytes per modulus and element of a full operand: 65 GB in
// 10.2 ms at n = 8192, 0.94 of the copy bandwidth).
template <int ND, bool kOne>
__global__ void __launch_bounds__(kThreads, 4)
    mat2_encode_kernel(const __grid_constant__ JobParam<kOne> one, const SplitJob* jobs, int njobs,
                       unsigned char* ws, int64_t first) {
  __shared__ __align__(16) long long ent[8][kRows][kPitch];
  __shared__ int s_row[kRows];
  // One job, in the arguments: the operands are read before the wait for the exponents,
  // whose kernel has itself waited for whatever wrote the operands before it let this
  // one start.  A table on the device is memory like any other: wait first.
  if constexpr (!kOne) wait_for_previous_kernel();
  const int64_t blk = first + blockIdx.x;
  const SplitJob& sj = unit_job(one, jobs, njobs, blk, 5);
  const JobDesc& d = sj.d;
  const int ktiles = (d.k + kK - 1) / kK;
  const int64_t a_blocks = (int64_t)((d.m + kRows - 1) / kRows) * ktiles;
  int64_t within = blk - sj.enc2_begin;
  const int side = within >= a_blocks ? 1 : 0;
  if (side) within -= a_blocks;
  const uint32_t local = (uint32_t)within;               // a launch has fewer than 2^31 blocks
  const int tile_rows = side ? sj.bn : kTileM;
  const int rows_pad = (side ? sj.tiles_n : sj.tiles_m) * tile_rows;
  const uint32_t rowtile = local / (uint32_t)ktiles;
  const int r0 = (int)rowtile * kRows;
  const int k0 = (int)(local - rowtile * (uint32_t)ktiles) * kK;
  const int nout = side ? d.n : d.m;
  const uint32_t flags = side ? d.fb : d.fa;
  const double* base = side ? d.B : d.A;
  const int64_t ld = side ? d.ldb : d.lda, cs = side ? d.sB : d.sA;
  const int8_t* sign = side ? d.signB : d.signA;
  const bool contiguous = side ? (d.transB != 0) : (d.transA == 0);
  // block-uniform: fourteen planes a full operand, seven a quaternion, eight the
  // coefficients beside a complex one, two a complex one
  const int planes = side ? sj.nrf : sj.nlf;
  const int operand = planes == 14 ? kOpFull : planes == 7 ? kOpQuat : planes == 8 ? kOpCoef : kOpCplx;
  const int t = threadIdx.x;
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
        raw[u][c] = kOne ? load_coherent(src + (int64_t)c * cs)
                         : (unsigned long long)__double_as_longlong(__ldcs(src + (int64_t)c * cs));
    }
  }
  if constexpr (kOne) wait_for_previous_kernel();   // the exponents
  if (t < kRows) {
    const int r = r0 + t;
    s_row[t] = (r < nout) ? reinterpret_cast<const int32_t*>(ws + (side ? sj.off_texp : sj.off_sexp))[r] : 0;
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
    if (operand == kOpFull) {
      // a_e = X[e], b_e = X[e + 4]: Re and Im of the entries 11, 12, 21, 22 (copy u)
      ent[0][rr][kk] = X[0] - X[5];
      ent[1][rr][kk] = X[4] + X[1];
      ent[2][rr][kk] = X[2] - X[7];
      ent[3][rr][kk] = X[6] + X[3];
      ent[4][rr][kk] = -X[2] - X[7];
      ent[5][rr][kk] = X[3] - X[6];
      ent[6][rr][kk] = X[0] + X[5];
      ent[7][rr][kk] = X[4] - X[1];
    } else if (operand == kOpQuat) {         // one of the two halves is absent (zero)
#pragma unroll
      for (int e = 0; e < 4; ++e) ent[e][rr][kk] = X[e] + X[e + 4];
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e == 0 || operand == kOpCoef) {
          ent[2 * e][rr][kk] = X[e];
          ent[2 * e + 1][rr][kk] = X[e + 4];
        }
    }
  }
  __syncthreads();

  const int64_t tile_bytes = (int64_t)tile_rows * kTileK * 2;
  const uint32_t plane_bytes = (uint32_t)(side ? sj.encB_plane : sj.encA_plane);   // below 2^32 (checked on the host)
  unsigned char* enc = ws + (side ? sj.off_encB : sj.off_encA);
  // this block's moduli (small launches share a tile's moduli between blocks)
  const int l0 = (int)(blockIdx.y * (unsigned)sj.nmod / gridDim.y), l1 = (int)((blockIdx.y + 1) * (unsigned)sj.nmod / gridDim.y);
  enc += (int64_t)l0 * planes * plane_bytes;
#pragma unroll 1
  for (int pass = 0; pass < kRows * kK / 2 / kThreads; ++pass) {
    const int pos = t + pass * kThreads;
    const int rr = pos / (kK / 2), kp = 2 * (pos % (kK / 2));
    const int r = r0 + rr;
    if (r >= rows_pad) return;
    const int kg = k0 + kp;
    const int kb = kg / kTileK, c16 = (kg % kTileK) / 8, in16 = (kg % 8) * 2;
    const int rt = r / tile_rows, rin = r % tile_rows;
    const bool half = kb + 1 == sj.nkb && half_last_block(d.k);
    const int in_tile = half ? rin * 64 + ((c16 ^ ((rin >> 1) & 3)) << 4) : rin * 128 + ((c16 ^ (rin & 7)) << 4);
    unsigned char* out = enc + ((int64_t)rt * sj.nkb + kb) * tile_bytes + in_tile + in16;
    longlong2 E[8];
    auto load = [&](int count) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e < count) E[e] = *reinterpret_cast<const longlong2*>(&ent[e][rr][kp]);
    };
    if (operand == kOpFull) {
      load(8);
      if (side) encode_pair<ND, 1, kOpFull>(E, l0, l1, out, plane_bytes);
      else encode_pair<ND, 0, kOpFull>(E, l0, l1, out, plane_bytes);
    } else if (operand == kOpQuat) {
      load(4);
      if (side) encode_pair<ND, 1, kOpQuat>(E, l0, l1, out, plane_bytes);
      else encode_pair<ND, 0, kOpQuat>(E, l0, l1, out, plane_bytes);
    } else if (operand == kOpCoef) {
      load(8);
      encode_pair<ND, 0, kOpCoef>(E, l0, l1, out, plane_bytes);
    } else {
      load(2);
      encode_pair<ND, 0, kOpCplx>(E, l0, l1, out, plane_bytes);
    }
  }
}

// ------------------------------------------------------------------ CRT
// One warp per 32 consecutive elements of an output row; a block of four warps
// covers four rows of 32 columns, two of 64 or one of 128 (mat2_crt_width).
//
// Per element and modulus the outputs are sums of the product residues.  With cu,
// cv the entries of the two copies' 2 x 2 products:
//   half 0 (1/4):   t11 = cu11 + cv22, t22 = cu22 + cv11, t12 = cu12 - cv21, t21 = cu21 - cv12,
//   half 1 (1/4s):  t11 = cu11 - cv22, t22 = cu22 - cv11, t12 = cu12 + cv21, t21 = cu21 + cv12,
//   half 0: M1 = t11 + t22, M6 = t22 - t11, M3 = t12 - t21, M8 = -(t12 + t21)
//   half 1: M5 = t11 + t22, M2 = t11 - t22, M7 = t12 - t21, M4 = t12 + t21
// (real quaternions: one copy, t = 2 cu, M1 and M3 of half 0, M2 and M4 of half 1);
// complex x biquaternion: M_e = 2 (u_e + v_e) of half 0, M_{e+4} = 2 (u_e - v_e) of
// half 1.  S = N P + sum_l x_l d_l with d_l the CRT elements that carry 1/4 or
// 1/(4 s) is congruent to the output modulo P.  An operand that is i times a real
// quaternion was encoded as the real one; the outputs are turned by its i.
//
// The sum over the moduli is a contraction of depth nmod <= 16 (or two steps of
// it), and runs on the tensor cores: A[element][modulus] = the integers t (FP16,
// exact up to 2048), B[modulus][digit] = the balanced 8-bit digits of d_l, FP32
// sums below 2^22 (exact).  A thread holds the fragment elements of four columns
// and four moduli: it reads their residues as words from shared memory,
// interleaves two moduli by byte permutes into half2 (an unsigned byte is an FP16
// subnormal, so no conversion is needed: everything carries a factor 2^-24) and
// forms the sums with half2 additions.  The residues are stored with 128 added
// (unsigned bytes); what that adds to a sum is a constant, taken out of the
// offset N P.  Pairs of digit sums are packed to 32-bit integers of weight
// 2^(16 i), transposed through shared memory so that a lane owns one column, and
// finished there.
//
// Bound by instruction issue (2.6 of 4 per cycle, 54 instructions per element and
// warp lane; 64-bit multiply-adds per modulus, output and limb took 113): 1.2 ms
// for 4096 x 4096 (2.35 ms with those), 0.68 ms of which its 4.6 GB would take at
// the copy bandwidth; the 512-product batch 3.34 ms (6.1 ms).
constexpr int kCrtThreads = 128;
constexpr int mod_stride(int planes) {                // bytes; the four moduli pairs of a read fall on different banks
  return planes * kCrtCols + 16;
}
constexpr int kTrStride = 40;                         // words; likewise for the 16-byte stores of the transpose

// digits of the CRT elements in the B fragments' layout: [nmod][half][k step][n tile][register][lane]
__device__ uint32_t g_m2digits[kMat2MaxModuli + 1][2][2][2][2][32];

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2],
                                        const float (&c)[4]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
__device__ __forceinline__ uint32_t hadd2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t hsub2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// The accumulators start at kMagic: with an integer sum x, |x| < 2^22, the result
// kMagic + x 2^-24 lies in (0.5, 1), where a float's last bit is 2^-24, so its bits
// are kMagicBits + x and no conversion is needed.
constexpr float kMagic = 0.75f;
constexpr uint32_t kMagicBits = 0x3F400000u;
// the packed pair of digit sums x0 + 256 x1, plus this constant
constexpr uint32_t kPairBias = kMagicBits * 257u;
__device__ __forceinline__ uint32_t digit_pair(float x0, float x1) {
  return __float_as_uint(x0) + 256u * __float_as_uint(x1);
}

// A double's bits rounded from |X| = [x3 x2 x1 x0] 2^scale_exp for values the fast
// path leaves (zeros, magnitudes below 2^64, results outside the normal range).
__device__ __noinline__ double limbs4_slow(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3, int neg,
                                           int scale_exp) {
  const uint32_t x[4] = {x0, x1, x2, x3};
  return limbs4_to_double(x, neg, scale_exp);
}

// The output of one slot from its eight digit pairs (each with 2^31 added, pair i
// of weight 2^(16 i)): S = off + sum_i p_i 2^(16 i) modulo 2^128 lies in (0, 2 N P),
// X = S - q P with q the nearest integer to S / P, returned as X 2^scale_exp.  With
// 2 N P in (2^126, 2^128) the leading limb alone estimates S / P within 2^-15 (the
// limbs left out) + 2^-8 (its conversion) + 2^-8 (the reciprocal), far inside the
// 0.0796 that separates X from a half P.  Every lane of the warp calls it.
__device__ __forceinline__ double crt_value4(const uint32_t (&p)[8], uint4 off, uint4 negP, float pinv, int scale_exp) {
  uint32_t x0, x1, x2, x3;
  asm("{\n\t"
      "add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\taddc.cc.u32 %2, %6, %10;\n\taddc.u32 %3, %7, %11;\n\t"
      "add.cc.u32 %0, %0, %12;\n\taddc.cc.u32 %1, %1, %13;\n\taddc.cc.u32 %2, %2, %14;\n\taddc.u32 %3, %3, %15;\n\t}"
      : "=&r"(x0), "=&r"(x1), "=&r"(x2), "=&r"(x3)
      : "r"(p[0]), "r"(p[2]), "r"(p[4]), "r"(p[6]), "r"(p[1] << 16), "r"(__funnelshift_l(p[1], p[3], 16)),
        "r"(__funnelshift_l(p[3], p[5], 16)), "r"(__funnelshift_l(p[5], p[7], 16)), "r"(off.x), "r"(off.y),
        "r"(off.z), "r"(off.w));
  const uint32_t q = __float_as_uint(fmaf((float)x3, pinv, 12582912.0f)) - 0x4B400000u;
  asm("{\n\t"
      "mad.lo.cc.u32 %0, %4, %5, %0;\n\tmadc.lo.cc.u32 %1, %4, %6, %1;\n\tmadc.lo.cc.u32 %2, %4, %7, %2;\n\t"
      "madc.lo.u32 %3, %4, %8, %3;\n\t"
      "mad.hi.cc.u32 %1, %4, %5, %1;\n\tmadc.hi.cc.u32 %2, %4, %6, %2;\n\tmadc.hi.u32 %3, %4, %7, %3;\n\t}"
      : "+r"(x0), "+r"(x1), "+r"(x2), "+r"(x3)
      : "r"(q), "r"(negP.x), "r"(negP.y), "r"(negP.z), "r"(negP.w));
  const uint32_t flip = (uint32_t)((int)x3 >> 31);   // |X| = (x ^ flip) - flip
  asm("{\n\t.reg .u32 f;\n\tneg.s32 f, %4;\n\t"
      "xor.b32 %0, %0, %4;\n\txor.b32 %1, %1, %4;\n\txor.b32 %2, %2, %4;\n\txor.b32 %3, %3, %4;\n\t"
      "add.cc.u32 %0, %0, f;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.cc.u32 %2, %2, 0;\n\taddc.u32 %3, %3, 0;\n\t}"
      : "+r"(x0), "+r"(x1), "+r"(x2), "+r"(x3)
      : "r"(flip));
  // the 96 bits from the leading nonzero limb, the rest as a sticky word
  const bool three = x3 == 0;
  const uint32_t a = three ? x2 : x3, b = three ? x1 : x2, c = three ? x0 : x1, rest = three ? 0u : x0;
  const int lz = __clz(a);
  const uint32_t hi = __funnelshift_l(b, a, lz);
  uint32_t lo = __funnelshift_l(c, b, lz);
  if (((c << lz) | rest) != 0u) lo |= 1u;            // sticky bit: one correct rounding below
  // |X| = [hi lo] 2^E, hi's top bit set
  const int bexp = scale_exp - lz + (three ? 32 + 1086 : 64 + 1086);   // IEEE biased exponent
  if (!__all_sync(0xffffffffu, a != 0u && bexp >= 1 && bexp <= 2046))
    return limbs4_slow(x0, x1, x2, x3, (int)(flip & 1u), scale_exp);
  // nearest even: the 11 dropped bits above half, or at half with an odd last bit
  const uint32_t m0 = __funnelshift_r(lo, hi, 11), m1 = hi >> 11;
  const uint32_t up = ((lo << 21) + (m0 & 1u)) > 0x80000000u ? 1u : 0u;
  const unsigned long long bits = (((unsigned long long)m1 << 32) | m0) + up;
  return __hiloint2double((int)(((uint32_t)(bits >> 32) + ((uint32_t)(bexp - 1) << 20)) | (flip & 0x80000000u)),
                          (int)(uint32_t)bits);
}

struct Mat2Pair {          // a coefficient's real and imaginary part
  double re, im;
};

// x turned by i^rot; zeros stay +0
__device__ __forceinline__ Mat2Pair turn(Mat2Pair x, int rot) {
  auto neg = [](double v) {
    const long long b = __double_as_longlong(v);
    return __longlong_as_double((b << 1) == 0 ? b : b ^ (1ll << 63));
  };
  if (rot == 1) return {neg(x.im), x.re};
  if (rot == 2) return {neg(x.re), neg(x.im)};
  return x;
}

// The block's work for a job of kind KIND; L: limbs of the sums, KS: k steps (of 16 moduli).
template <int L, int KS, int KIND, bool kOne>
__device__ __forceinline__ void crt_block(const SplitJob& sj, uint32_t local, const unsigned char* ws,
                                          uint8_t* ring, uint32_t (*tr)[8][kTrStride]) {
  constexpr int NP = KIND == kMat2Full ? 14 : KIND == kMat2Quat ? 7 : KIND == kMat2Scaled ? 8 : 2;
  constexpr int kStride = mod_stride(NP);
  constexpr int kRingMods = KS == 1 ? 16 : kMat2MaxModuli + 1;
  const JobDesc& d = sj.d;
  const int nm = sj.nmod;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  // 128 / w rows of w columns, w = 128, 64 or 32; a launch has fewer than 2^31 blocks
  const int w = sj.crt_w, lw = 31 - __clz(w);
  const uint32_t colblocks = (uint32_t)(d.n + w - 1) >> lw;
  const uint32_t rowblock = local / colblocks;
  const int i0 = (int)rowblock * (kCrtCols >> lw);
  const int j0 = (int)(local - rowblock * colblocks) << lw;
  const int64_t group = (int64_t)sj.tiles_m * (kTileM * 32);   // bytes of 32 columns of residues
  // this thread's fragments of the digits (zero for moduli >= nmod)
  uint32_t b[2][KS][2][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int v = 0; v < 2; ++v) b[h][ks][nt][v] = __ldg(&g_m2digits[nm][h][ks][nt][v][lane]);
  if constexpr (kOne) wait_for_previous_kernel();          // the residues
  // copy: thread tid takes 16-byte chunk tid % 8 of one product's planes, of every
  // 16 / NP-th modulus (constant steps in both addresses)
  {
    constexpr int kStep = 16 / NP;
    const int cc = tid & 7, crow = cc >> (lw - 4), col = j0 + (cc & ((w >> 4) - 1)) * 16;
    const int r = (tid >> 3) % NP, l0 = (tid >> 3) / NP;
    if (l0 < kStep && i0 + crow < d.m && col < d.n) {
      const int64_t step = (int64_t)(kStep * NP) * sj.res_plane;
      const unsigned char* src = ws + sj.off_res + (int64_t)(l0 * NP + r) * sj.res_plane + (int64_t)(col >> 5) * group +
                                 (int64_t)(i0 + crow) * 32 + (col & 16);
      uint8_t* dst = ring + l0 * kStride + r * kCrtCols + cc * 16;
#pragma unroll
      for (int l = 0; l < kRingMods; l += kStep) {
        if (l0 + l >= nm) break;
        cp_async16(dst + l * kStride, src);
        src += step;
      }
    }
    cp_async_commit();
  }
  const int wi = i0 + (32 * warp >> lw), j = j0 + (32 * warp & (w - 1)) + lane;
  const bool valid = wi < d.m && j < d.n;
  int sc = -c_m2shift[nm];
  if (valid)
    sc -= reinterpret_cast<const int32_t*>(ws + sj.off_sexp)[wi] + reinterpret_cast<const int32_t*>(ws + sj.off_texp)[j];
  const int pb = c_m2Pbase[nm];
  const float pinv = L == 4 ? c_m2Pinv4[nm] : c_m2Pinv[nm];
  double* cbase = d.C + (int64_t)wi * d.ldc + j;
  // compared as bits: FP64 instructions are scarce, and these are uniform
  auto zero = [](double v) { return (__double_as_longlong(v) << 1) == 0; };
  const bool use_beta = !zero(d.beta_re) || !zero(d.beta_im);
  if (use_beta && valid)                                   // C is needed at the end: bring it near now
    for (int e = 0; e < 8; ++e) asm volatile("prefetch.global.L1 [%0];" ::"l"(cbase + (int64_t)e * d.sC));
  const bool plain = __double_as_longlong(d.alpha_re) == 0x3FF0000000000000ll && zero(d.alpha_im) && !use_beta;
  const int rot = sj.rot;
  const float start[4] = {kMagic, kMagic, kMagic, kMagic};
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();

  // cu: sums c11, c22, c12, c21 of copy u (or the four coefficients) for four
  // columns and 2 KS pairs of moduli; cv: what copy v adds to t11, t22, t12, t21
  // in half 0 and takes away in half 1
  constexpr int kSums = KIND == kMat2Complex ? 1 : 4;
  uint32_t cu[kSums][2 * KS][4], cv[kSums][2 * KS][4];     // [sum][pair][column]
#pragma unroll
  for (int kp = 0; kp < 2 * KS; ++kp) {
    const int l = 8 * kp + 2 * t;
    const bool have = KS == 1 || l + 1 < kRingMods;        // beyond the ring: moduli that do not exist
    uint32_t z[2 * NP];
#pragma unroll
    for (int r = 0; r < NP; ++r) {
      uint32_t w0 = 0, w1 = 0;
      if (have) {
        const uint8_t* at = ring + l * kStride + r * kCrtCols + 32 * warp + 4 * g;
        w0 = *reinterpret_cast<const uint32_t*>(at);
        w1 = *reinterpret_cast<const uint32_t*>(at + kStride);
      }
      z[2 * r] = __byte_perm(w0, w1, 0x5140);              // columns 0 and 1, moduli interleaved
      z[2 * r + 1] = __byte_perm(w0, w1, 0x7362);          // columns 2 and 3
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      uint32_t p[NP];
#pragma unroll
      for (int r = 0; r < NP; ++r) p[r] = __byte_perm(z[2 * r + (c >> 1)], 0u, (c & 1) ? 0x4342 : 0x4140);
      if constexpr (KIND == kMat2Full || KIND == kMat2Quat) {
        auto sums = [&](int o, uint32_t (&x)[4]) {         // c11, c22, c12, c21 of the products o .. o + 6
          const uint32_t u1 = hadd2(p[o], p[o + 5]), u2 = hadd2(u1, p[o + 6]);
          x[0] = hadd2(p[o], p[o + 1]);
          x[1] = hadd2(u2, p[o + 4]);
          x[2] = hadd2(hadd2(u1, p[o + 4]), p[o + 2]);
          x[3] = hsub2(u2, p[o + 3]);
        };
        uint32_t x[4];
        sums(0, x);
#pragma unroll
        for (int e = 0; e < 4; ++e) cu[e][kp][c] = x[e];
        if constexpr (KIND == kMat2Full) {
          sums(7, x);
          cv[0][kp][c] = x[1];
          cv[1][kp][c] = x[0];
          cv[2][kp][c] = x[3];                             // (entries 12 and 21 with the opposite sign)
          cv[3][kp][c] = x[2];
        }
      } else {
#pragma unroll
        for (int e = 0; e < kSums; ++e) {                  // twice the coefficient
          cu[e][kp][c] = hadd2(p[e], p[e]);
          cv[e][kp][c] = hadd2(p[kSums + e], p[kSums + e]);
        }
      }
    }
  }

#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {                         // coefficients 2 pr and 2 pr + 1
    // which slots (half, e) exist
    auto has = [](int pr_, int h, int e) {
      if (KIND == kMat2Quat) return h == e;
      if (KIND == kMat2Complex) return pr_ == 0 && e == 0;
      return true;
    };
    double val[2][2] = {};                                 // [half][slot]
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!has(pr, h, 0) && !has(pr, h, 1)) continue;
      uint32_t pair[2][2][4];                              // [sum][n tile][column]
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (KIND == kMat2Complex && e > 0) continue;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          float acc[2][4];
#pragma unroll
          for (int ks = 0; ks < KS; ++ks) {
            uint32_t a[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {                  // rows g, g + 8: columns 2 mt, 2 mt + 1; then the next pair
              const int si = KIND == kMat2Complex ? 0 : 2 * pr + e;
              const uint32_t x = cu[si][2 * ks + (v >> 1)][2 * mt + (v & 1)];
              if constexpr (KIND == kMat2Quat) {
                a[v] = hadd2(x, x);
              } else {
                const uint32_t y = cv[si][2 * ks + (v >> 1)][2 * mt + (v & 1)];
                const bool minus = (h == 1) != (KIND == kMat2Full && pr == 1);
                a[v] = minus ? hsub2(x, y) : hadd2(x, y);
              }
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
              if (ks == 0) mma_f16(acc[nt], a, b[h][ks][nt], start);
              else mma_f16(acc[nt], a, b[h][ks][nt], acc[nt]);
            }
          }
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            pair[e][nt][2 * mt] = digit_pair(acc[nt][0], acc[nt][1]);
            pair[e][nt][2 * mt + 1] = digit_pair(acc[nt][2], acc[nt][3]);
          }
        }
      }
      __syncwarp();                                        // the previous sums have been read
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        uint32_t s[2][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          // (2^31 added to make the pairs unsigned)
          constexpr uint32_t kPlus = 0x80000000u - 2u * kPairBias, kMinus = 0x80000000u + 2u * kPairBias;
          const uint32_t x = pair[0][nt][c];
          if constexpr (KIND == kMat2Scaled || KIND == kMat2Complex) {
            s[0][c] = x + (0x80000000u - kPairBias);
            if constexpr (KIND == kMat2Scaled) s[1][c] = pair[1][nt][c] + (0x80000000u - kPairBias);
          } else {
            // pr 0: slot 0 = t11 + t22, slot 1 = t22 - t11 (half 1: t11 - t22);
            // pr 1: slot 0 = t12 - t21, slot 1 = -(t12 + t21) (half 1: t12 + t21)
            const uint32_t y = pair[1][nt][c];
            s[0][c] = pr == 0 ? x + y + kPlus : x - y + 0x80000000u;
            s[1][c] = pr == 0 ? (h ? x - y : y - x) + 0x80000000u : (h ? x + y + kPlus : kMinus - (x + y));
          }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (has(pr, h, e))
            *reinterpret_cast<uint4*>(&tr[e][4 * nt + t][4 * g]) = make_uint4(s[e][0], s[e][1], s[e][2], s[e][3]);
      }
      __syncwarp();
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (!has(pr, h, e)) continue;
        constexpr int kTab = KIND == kMat2Scaled || KIND == kMat2Complex ? 1 : 0;
        uint32_t p[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) p[i] = tr[e][i][lane];
        if constexpr (L == 4) {
          val[h][e] = crt_value4(p, c_m2off4[nm][kTab][h][2 * pr + e], c_m2negP[nm], pinv, sc);
        } else {
          const long long* off = c_m2off[nm][kTab][h][2 * pr + e];
          long long s[L];
#pragma unroll
          for (int q = 0; q < L; ++q) {
            s[q] = off[q];
            if (q < 4) s[q] += (long long)p[2 * q] + (long long)p[2 * q + 1] * 65536ll;
          }
          val[h][e] = crt_value<L>(s, c_m2P[nm], pb, pinv, sc);
        }
      }
    }
    if (valid) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        // matrix products: slot 0 of half 0 and slot 1 of half 1 are real parts
        const bool swap = (KIND == kMat2Full || KIND == kMat2Quat) && e == 1;
        const Mat2Pair q = turn(swap ? Mat2Pair{val[1][e], val[0][e]} : Mat2Pair{val[0][e], val[1][e]}, rot);
        double* cr = cbase + (int64_t)(2 * pr + e) * d.sC;
        double* ci = cr + 4 * d.sC;
        if (plain) {                                       // block-uniform
          *cr = q.re;
          *ci = q.im;
          continue;
        }
        double x = 0.0, y = 0.0;
        if (use_beta) {
          x = *cr;
          y = *ci;
        }
        double vr = d.alpha_re * q.re + -1.0 * d.alpha_im * q.im;
        double vi = d.alpha_re * q.im + 1.0 * d.alpha_im * q.re;
        if (use_beta) {
          vr += d.beta_re * x + -1.0 * d.beta_im * y;
          vi += d.beta_re * y + 1.0 * d.beta_im * x;
        }
        *cr = vr;
        *ci = vi;
      }
    }
  }
}

template <int L, int KS, bool kOne>
__global__ void __launch_bounds__(kCrtThreads, 4)
    mat2_crt_kernel(const __grid_constant__ JobParam<kOne> one, const SplitJob* jobs, int njobs,
                    const unsigned char* ws) {
  __shared__ __align__(16) uint8_t ring[(KS == 1 ? 16 : kMat2MaxModuli + 1) * mod_stride(kMat2MaxPlanes)];
  __shared__ __align__(16) uint32_t tr[kCrtThreads / 32][2][8][kTrStride];
  if constexpr (!kOne) wait_for_previous_kernel();         // before anything is read from the table
  const int64_t blk = blockIdx.x;
  const SplitJob& sj = unit_job(one, jobs, njobs, blk, 6);
  const uint32_t local = (uint32_t)(blk - sj.crt2_begin);
  auto* mine = tr[threadIdx.x >> 5];
  switch (sj.mat2) {                                       // block-uniform
    case kMat2Full: crt_block<L, KS, kMat2Full, kOne>(sj, local, ws, ring, mine); break;
    case kMat2Quat: crt_block<L, KS, kMat2Quat, kOne>(sj, local, ws, ring, mine); break;
    case kMat2Scaled: crt_block<L, KS, kMat2Scaled, kOne>(sj, local, ws, ring, mine); break;
    default: crt_block<L, KS, kMat2Complex, kOne>(sj, local, ws, ring, mine); break;
  }
}

}  // namespace

// IEEE half of an integer |v| <= 128
static uint32_t half_bits(int v) {
  if (v == 0) return 0;
  const uint32_t sign = v < 0 ? 0x8000u : 0u;
  uint32_t m = (uint32_t)(v < 0 ? -v : v), e = 0;
  while ((m >> (e + 1)) != 0) ++e;                  // 2^e <= m < 2^(e + 1), e <= 7
  return sign | ((e + 15u) << 10) | ((m << (10u - e)) & 0x3FFu);
}

cudaError_t mat2_configure(const int* moduli, const int* root, int n, const int32_t* crt_d, const uint32_t* crt_P,
                           const uint32_t* crt_off, const int* shift) {
  constexpr int M = kMat2MaxModuli;
  Mat2Mod mc[M];
  if (n != M) return cudaErrorInvalidValue;
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
  // the CRT elements' digits in base 256, balanced, as the B fragments: lane (g, t)
  // holds column (digit) g of rows (moduli) 2t, 2t + 1 (register 0) and 2t + 8, 2t + 9
  // (register 1) of a 16 x 8 tile
  static uint32_t dig[M + 1][2][2][2][2][32];
  static long long off[M + 1][2][2][4][kLimbs];
  static uint4 off4[M + 1][2][2][4], negP[M + 1];
  std::memset(dig, 0, sizeof(dig));
  std::memset(off, 0, sizeof(off));
  float pinv[M + 1], pinv4[M + 1] = {};
  int pb[M + 1];
  for (int m = 0; m <= M; ++m) {
    for (int h = 0; h < 2; ++h) {
      double worst[16] = {};                        // bound of each digit's sum over the moduli
      long long total[kLimbs] = {};                 // sum of the elements, by limb
      for (int l = 0; l < m; ++l) {
        const int32_t* x = crt_d + (((int64_t)m * 2 + h) * M + l) * kLimbs;   // signed 32-bit digits
        long long carry = 0;
        for (int q = 0; q < 4 * kLimbs; ++q) {
          long long v = carry + (((long long)x[q / 4] >> (8 * (q % 4))) & 0xFF);
          if (q % 4 == 3) v = carry + ((long long)x[q / 4] >> 24);            // the signed top byte of the limb
          carry = (v + 128) >> 8;
          const int digit = (int)(v - 256 * carry);                            // in [-128, 127]
          if (q >= 16) {
            if (digit != 0) return cudaErrorInvalidValue;                      // the elements are below 2^127
            continue;
          }
          // sums of up to four of one copy's residues, each stored as residue + 128
          worst[q] += std::fabs((double)digit) * 2 * 4 * ((moduli[l] - 1) / 2 + 128);
          const int ks = l / 16, k = l % 16, nt = q / 8, g = q % 8;
          dig[m][h][ks][nt][k / 8][g * 4 + (k % 8) / 2] |= half_bits(digit) << (16 * (k & 1));
        }
        if (carry != 0) return cudaErrorInvalidValue;
        for (int q = 0; q < kLimbs; ++q) total[q] += x[q];
      }
      for (int q = 0; q < 16; ++q)                  // exact under the conversion's magic number, pairs within int32
        if (worst[q] >= 4194304.0 || (q % 2 && 2.0 * (worst[q - 1] + 256.0 * worst[q]) >= 2147483648.0))
          return cudaErrorInvalidValue;
      // 128 times the sum of the weights of the residues in each slot: matrix products, complex x biquaternion
      static const int bias[2][2][4] = {{{1536, 0, 512, 0}, {0, -512, 0, 1536}}, {{512, 512, 512, 512}, {0, 0, 0, 0}}};
      for (int tab = 0; tab < 2; ++tab)
        for (int s = 0; s < 4; ++s) {
          long long carry = 0;
          uint32_t w[kLimbs];
          for (int q = 0; q < kLimbs; ++q) {
            long long& o = off[m][tab][h][s][q];
            o = (long long)crt_off[m * kLimbs + q] - bias[tab][h][s] * total[q] - (q < 4 ? (1ll << 31) + (1ll << 47) : 0);
            carry += o;
            w[q] = (uint32_t)carry;
            carry >>= 32;
          }
          off4[m][tab][h][s] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    const uint32_t* P = crt_P + m * kLimbs;
    // both limb counts that can run m moduli (a call's deepest job picks its kernel's)
    for (int limbs = m <= kMat2FourLimbs ? 4 : kLimbs; limbs <= kLimbs; ++limbs)
      if (!crt_estimate_constants(P, 2.0 * m * kMat2WeightSum * kMat2HalfMax, limbs, &pb[m], &pinv[m]))
        return cudaErrorInvalidValue;
    unsigned long long carry = 1;                    // 2^128 - P
    uint32_t w[4];
    for (int q = 0; q < 4; ++q) {
      carry += (uint32_t)~P[q];
      w[q] = (uint32_t)carry;
      carry >>= 32;
    }
    negP[m] = make_uint4(w[0], w[1], w[2], w[3]);
    if (m >= 1 && m <= kMat2FourLimbs) {
      double p = 0.0, bound = 2.0 * m * kMat2WeightSum * kMat2HalfMax;
      for (int q = 3; q >= 0; --q) p = p * 4294967296.0 + (double)P[q];
      if (!(bound * p > std::ldexp(1.0, 126) && bound * p < std::ldexp(1.0, 128))) return cudaErrorInvalidValue;
      pinv4[m] = (float)(std::ldexp(1.0, 96) / p);
    }
  }
  e = cudaMemcpyToSymbol(g_m2digits, dig, sizeof(dig));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2off, off, sizeof(off));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2off4, off4, sizeof(off4));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2negP, negP, sizeof(negP));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2Pinv4, pinv4, sizeof(pinv4));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2shift, shift, sizeof(int) * (M + 1));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2P, crt_P, sizeof(uint32_t) * (M + 1) * kLimbs);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(c_m2Pbase, pb, sizeof(pb));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_m2Pinv, pinv, sizeof(pinv));
}

cudaError_t launch_mat2_encode(const SplitJobs& jobs, int64_t units, int64_t first, cudaStream_t s,
                               unsigned char* ws, int max_bits, int sm_count) {
  if (units <= 0) return cudaSuccess;
  // A launch whose tiles do not fill the GPU (four blocks an SM) splits each
  // tile's moduli over up to four blocks, which repeat phase 1: a whole product
  // at n = 256 (256 tiles) 43.1 -> 41.0 us, at n = 64 24.6 -> 20.5.
  const int64_t fill = 4 * (int64_t)sm_count;
  const unsigned groups = (unsigned)(units * 4 <= fill ? 4 : units * 2 <= fill ? 2 : 1);
  // the matrix entries are sums of two b-bit integers: three digits hold 2^47
  return with_jobs(jobs, [&](const auto& one) {
    constexpr bool kOne = std::is_same_v<std::decay_t<decltype(one)>, JobParam<true>>;
    return launch_dependent(max_bits <= 46 ? mat2_encode_kernel<3, kOne> : mat2_encode_kernel<4, kOne>,
                            dim3((unsigned)units, groups), dim3(kThreads), 0, s, one, jobs.table, jobs.n, ws, first);
  });
}

cudaError_t launch_mat2_crt(const SplitJobs& jobs, int64_t units, cudaStream_t s, unsigned char* ws,
                            int max_nmod) {
  if (units <= 0) return cudaSuccess;
  return with_jobs(jobs, [&](const auto& one) {
    constexpr bool kOne = std::is_same_v<std::decay_t<decltype(one)>, JobParam<true>>;
    return launch_dependent(max_nmod <= kMat2FourLimbs ? mat2_crt_kernel<4, 1, kOne> : mat2_crt_kernel<kLimbs, 2, kOne>,
                            dim3((unsigned)units), dim3(kCrtThreads), 0, s, one, jobs.table, jobs.n, ws);
  });
}

}  // namespace hmat
