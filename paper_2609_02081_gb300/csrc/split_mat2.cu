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
#include <cstring>

#include "split_device.cuh"

namespace hmat {

namespace {

constexpr int kPlanes = kMat2Planes;

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
__constant__ long long c_m2off[kMat2MaxModuli + 1][2][4][kLimbs];   // per limb
__constant__ uint4 c_m2off4[kMat2MaxModuli + 1][2][4];              // modulo 2^128
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
// One warp per 32 consecutive elements of an output row; a block of four warps
// covers one row of 128 columns, or four rows of 32 for narrow products.
//
// Per element the sums c11, c12, c21, c22 of both copies' product residues are
// formed per modulus, and with u, v the two copies and t = u + v (half 0) or
// u - v (half 1) of c:
//   half 0: M1 = (t11 + t22)/4, M6 = (t22 - t11)/4, M3 = (t12 - t21)/4, M8 = -(t12 + t21)/4
//   half 1: M5 = (t11 + t22)/4s, M2 = (t11 - t22)/4s, M7 = (t12 - t21)/4s, M4 = (t12 + t21)/4s.
// S = N P + sum_l x_l d_l with d_l the CRT elements that carry 1/4 or 1/(4 s) is
// congruent to the output modulo P.
//
// The sum over the moduli is a contraction of depth nmod <= 16 (or two steps of
// it), and runs on the tensor cores: A[element][modulus] = the integers t (FP16,
// exact up to 2048), B[modulus][digit] = the balanced 8-bit digits of d_l, FP32
// sums below 2^22 (exact).  A thread holds the fragment elements of four columns
// and four moduli: it reads its 4 x 14 words of residues from shared memory,
// interleaves two moduli by byte permutes into half2 (an unsigned byte is an FP16
// subnormal, so no conversion is needed: everything carries a factor 2^-24) and
// forms the sums with half2 additions.  The residues are stored with 128 added
// (unsigned bytes); what that adds to a sum is a constant, taken out of the
// offset N P.  Pairs of digit sums are packed to 32-bit integers of weight
// 2^(16 i), transposed through shared memory so that a lane owns one column, and
// finished there.
//
// Bound by instruction issue (2.7 of 4 per cycle, 57 instructions per element and
// warp lane; 64-bit multiply-adds per modulus, output and limb took 113): 1.25 ms
// for 4096 x 4096 (2.35 ms with those), 0.87 ms of which its 5.9 GB would take at
// the copy bandwidth; the 512-product batch 3.6 ms (6.1 ms).
constexpr int kCrtThreads = 128;
constexpr int kModStride = kPlanes * kCrtCols + 16;   // bytes; the four moduli pairs of a read fall on different banks
constexpr int kTrStride = 40;                         // words; likewise for the 16-byte stores of the transpose

// digits of the CRT elements in the B fragments' layout: [nmod][half][k step][n tile][register][lane]
__device__ uint32_t g_m2digits[kMat2MaxModuli + 1][2][2][2][2][32];

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
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

// The sums c11, c22, c12, c21 of one copy for one column and a pair of moduli,
// from its seven products.
__device__ __forceinline__ void copy_sums(const uint32_t (&p)[7], uint32_t (&c)[4]) {
  const uint32_t u1 = hadd2(p[0], p[5]), u2 = hadd2(u1, p[6]);
  c[0] = hadd2(p[0], p[1]);
  c[1] = hadd2(u2, p[4]);
  c[2] = hadd2(hadd2(u1, p[4]), p[2]);
  c[3] = hsub2(u2, p[3]);
}

// kMagic + x for an FP32 sum x 2^-24 of the products: its bits are kMagicBits + x
constexpr float kMagic = 12582912.0f;
constexpr uint32_t kMagicBits = 0x4B400000u;
// the packed pair of digit sums x0 + 256 x1, plus this constant
constexpr uint32_t kPairBias = kMagicBits * 257u;
__device__ __forceinline__ uint32_t digit_pair(float x0, float x1) {
  const float2 v = __ffma2_rn(make_float2(x0, x1), f2(16777216.0f), f2(kMagic));
  return __float_as_uint(v.x) + 256u * __float_as_uint(v.y);
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

// L: limbs of the sums, KS: k steps (of 16 moduli), kWide: every job's blocks are
// one row of 128 columns.
template <int L, int KS, bool kWide>
__global__ void __launch_bounds__(kCrtThreads, 4) mat2_crt_kernel(const SplitJob* __restrict__ jobs, int njobs,
                                                                  unsigned char* __restrict__ ws) {
  constexpr int kRingMods = KS == 1 ? 16 : kMat2MaxModuli + 1;
  __shared__ __align__(16) uint8_t ring[kRingMods][kModStride];
  __shared__ __align__(16) uint32_t tr[kCrtThreads / 32][2][8][kTrStride];
  const int64_t blk = blockIdx.x;
  const SplitJob& sj = jobs[find_split_job(jobs, njobs, blk, 6)];
  const JobDesc& d = sj.d;
  const int nm = sj.nmod;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int w = kWide ? kCrtCols : sj.crt_w;
  const int64_t local = blk - sj.crt2_begin;
  const int colblocks = (d.n + w - 1) / w;
  const int i0 = (int)(local / colblocks) * (kCrtCols / w);
  const int j0 = (int)(local % colblocks) * w;
  const int64_t ncols = (int64_t)sj.tiles_n * sj.bn;
  // copy: thread tid takes 16-byte chunk tid % 8 of planes tid / 8, tid / 8 + 16, ...
  {
    const int64_t plane = sj.res_plane;
    const int cc = tid & 7, cw = w / 16, crow = cc / cw, ccol = (cc % cw) * 16;
    if (i0 + crow < d.m && (int64_t)j0 + ccol < ncols) {
      int q = tid >> 3;                                    // plane: modulus l, product r
      const unsigned char* src = ws + sj.off_res + (int64_t)q * plane + (int64_t)(i0 + crow) * ncols + j0 + ccol;
      int l = q >= kPlanes ? 1 : 0, r = q - l * kPlanes;
      for (; q < nm * kPlanes; q += 16) {
        cp_async16(&ring[l][r * kCrtCols + cc * 16], src);
        src += 16 * plane;
        r += 2;
        l += r >= kPlanes ? 2 : 1;
        r -= r >= kPlanes ? kPlanes : 0;
      }
    }
    cp_async_commit();
  }
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
  const int wi = i0 + (kWide ? 0 : 32 * warp / w), j = j0 + (kWide ? 32 * warp : 32 * warp % w) + lane;
  const bool valid = wi < d.m && j < d.n;
  int sc = 0;
  if (valid)
    sc = -(reinterpret_cast<const int32_t*>(ws + sj.off_sexp)[wi] + reinterpret_cast<const int32_t*>(ws + sj.off_texp)[j]);
  sc -= c_m2shift[nm];
  const int pb = c_m2Pbase[nm];
  const float pinv = L == 4 ? c_m2Pinv4[nm] : c_m2Pinv[nm];
  double* cbase = d.C + (int64_t)wi * d.ldc + j;
  // compared as bits: FP64 instructions are scarce, and these are uniform
  auto zero = [](double v) { return (__double_as_longlong(v) << 1) == 0; };
  const bool use_beta = !zero(d.beta_re) || !zero(d.beta_im);
  if (use_beta && valid)                                   // C is needed at the end: bring it near now
    for (int e = 0; e < 8; ++e) asm volatile("prefetch.global.L1 [%0];" ::"l"(cbase + (int64_t)e * d.sC));
  const bool plain = __double_as_longlong(d.alpha_re) == 0x3FF0000000000000ll && zero(d.alpha_im) && !use_beta;
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();

  // sums c11, c22, c12, c21 of both copies for four columns and 2 KS pairs of moduli
  uint32_t cu[4][2 * KS][4], cv[4][2 * KS][4];             // [sum][pair][column]
#pragma unroll
  for (int kp = 0; kp < 2 * KS; ++kp) {
    const int l = 8 * kp + 2 * t;
    const bool have = KS == 1 || l + 1 < kRingMods;        // beyond the ring: moduli that do not exist
    uint32_t z[2 * kPlanes];
#pragma unroll
    for (int r = 0; r < kPlanes; ++r) {
      uint32_t w0 = 0, w1 = 0;
      if (have) {
        w0 = *reinterpret_cast<const uint32_t*>(&ring[l][r * kCrtCols + 32 * warp + 4 * g]);
        w1 = *reinterpret_cast<const uint32_t*>(&ring[l + 1][r * kCrtCols + 32 * warp + 4 * g]);
      }
      z[2 * r] = __byte_perm(w0, w1, 0x5140);              // columns 0 and 1, moduli interleaved
      z[2 * r + 1] = __byte_perm(w0, w1, 0x7362);          // columns 2 and 3
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      uint32_t pu[7], pv[7], su[4], sv[4];
#pragma unroll
      for (int r = 0; r < 7; ++r) {
        pu[r] = __byte_perm(z[2 * r + (c >> 1)], 0u, (c & 1) ? 0x4342 : 0x4140);
        pv[r] = __byte_perm(z[2 * (r + 7) + (c >> 1)], 0u, (c & 1) ? 0x4342 : 0x4140);
      }
      copy_sums(pu, su);
      copy_sums(pv, sv);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        cu[e][kp][c] = su[e];
        cv[e][kp][c] = sv[e];
      }
    }
  }

#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {                         // sums 11 and 22, then 12 and 21
    double val[2][2];                                      // [half][slot]
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t pair[2][2][4];                              // [sum][n tile][column]
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          float acc[2][4] = {};
#pragma unroll
          for (int ks = 0; ks < KS; ++ks) {
            uint32_t a[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {                  // rows g, g + 8: columns 2 mt, 2 mt + 1; then the next pair
              const uint32_t x = cu[2 * pr + e][2 * ks + (v >> 1)][2 * mt + (v & 1)];
              const uint32_t y = cv[2 * pr + e][2 * ks + (v >> 1)][2 * mt + (v & 1)];
              a[v] = h ? hsub2(x, y) : hadd2(x, y);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) mma_f16(acc[nt], a, b[h][ks][nt]);
          }
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            pair[e][nt][2 * mt] = digit_pair(acc[nt][0], acc[nt][1]);
            pair[e][nt][2 * mt + 1] = digit_pair(acc[nt][2], acc[nt][3]);
          }
        }
      __syncwarp();                                        // the previous sums have been read
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        uint32_t s0[4], s1[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t x = pair[0][nt][c], y = pair[1][nt][c];
          // pr 0: slot 0 = c11 + c22, slot 1 = c22 - c11 (half 1: c11 - c22);
          // pr 1: slot 0 = c12 - c21, slot 1 = -(c12 + c21) (half 1: c12 + c21)
          // (2^31 added to make the pairs unsigned)
          constexpr uint32_t kPlus = 0x80000000u - 2u * kPairBias, kMinus = 0x80000000u + 2u * kPairBias;
          s0[c] = pr == 0 ? x + y + kPlus : x - y + 0x80000000u;
          s1[c] = pr == 0 ? (h ? x - y : y - x) + 0x80000000u : (h ? x + y + kPlus : kMinus - (x + y));
        }
        *reinterpret_cast<uint4*>(&tr[warp][0][4 * nt + t][4 * g]) = make_uint4(s0[0], s0[1], s0[2], s0[3]);
        *reinterpret_cast<uint4*>(&tr[warp][1][4 * nt + t][4 * g]) = make_uint4(s1[0], s1[1], s1[2], s1[3]);
      }
      __syncwarp();
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        uint32_t p[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) p[i] = tr[warp][e][i][lane];
        if constexpr (L == 4) {
          val[h][e] = crt_value4(p, c_m2off4[nm][h][2 * pr + e], c_m2negP[nm], pinv, sc);
        } else {
          const long long* off = c_m2off[nm][h][2 * pr + e];
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
    // slot e of half h is component (4 h + 2 pr + e) with the half flipped for
    // odd e, so slot e's two values are the real (component 2 pr + e) and the
    // imaginary part of one coefficient
    if (valid) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const double re = e ? val[1][e] : val[0][e], im = e ? val[0][e] : val[1][e];
        double* cr = cbase + (int64_t)(2 * pr + e) * d.sC;
        double* ci = cr + 4 * d.sC;
        if (plain) {                                       // block-uniform
          *cr = re;
          *ci = im;
          continue;
        }
        double x = 0.0, y = 0.0;
        if (use_beta) {
          x = *cr;
          y = *ci;
        }
        double vr = d.alpha_re * re + -1.0 * d.alpha_im * im;
        double vi = d.alpha_re * im + 1.0 * d.alpha_im * re;
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
  static long long off[M + 1][2][4][kLimbs];
  static uint4 off4[M + 1][2][4], negP[M + 1];
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
      // 128 times the sum of the weights of the residues in each slot (half 1: u - v, none)
      static const int bias[4] = {1536, 512, 512, -1536};
      for (int s = 0; s < 4; ++s)
        for (int q = 0; q < kLimbs; ++q)
          off[m][h][s][q] = (long long)crt_off[m * kLimbs + q] - (h == 0 ? bias[s] * total[q] : 0) -
                            (q < 4 ? (1ll << 31) + (1ll << 47) : 0);
      for (int s = 0; s < 4; ++s) {
        uint32_t w[4];
        long long carry = 0;
        for (int q = 0; q < 4; ++q) {
          carry += off[m][h][s][q];
          w[q] = (uint32_t)carry;
          carry >>= 32;
        }
        off4[m][h][s] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    const uint32_t* P = crt_P + m * kLimbs;
    if (!crt_estimate_constants(P, 2.0 * m * kMat2WeightSum * kMat2HalfMax, m <= kMat2FourLimbs ? 4 : 5, &pb[m],
                                &pinv[m]))
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
  const unsigned grid = (unsigned)units;
  auto launch = [&](auto kernel) { kernel<<<grid, kCrtThreads, 0, s>>>(d_jobs, njobs, ws); };
  if (max_nmod <= kMat2FourLimbs) {
    if (all_wide) launch(mat2_crt_kernel<4, 1, true>);
    else launch(mat2_crt_kernel<4, 1, false>);
  } else {
    launch(mat2_crt_kernel<kLimbs, 2, false>);
  }
  return cudaGetLastError();
}

}  // namespace hmat
