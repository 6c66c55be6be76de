// split_host.cu — split-mode parameters, CRT constants, workspace layout and launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "split.hpp"

namespace hmat {

size_t split_gemm_smem_bytes();
cudaError_t split_gemm_configure(const int* moduli, int n);

// Odd, pairwise coprime moduli <= 255 (largest first): 255 = 3*5*17,
// 253 = 11*23, 247 = 13*19, 217 = 7*31, the rest prime.  Residues are centred
// in [-(p-1)/2, (p-1)/2] = [-127, 127] (exact in BF16, fit int8) and p >= 149.
static const int kModuli[kModTable] = {255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211,
                                       199, 197, 193, 191, 181, 179, 173, 167, 163, 157, 151, 149};

// Matrix form: odd, pairwise coprime moduli below 255 all of whose prime
// factors are 1 modulo 4 (221 = 13*17, 205 = 5*41, the rest prime), so that -1
// has a square root modulo each: the largest seventeen, 124.2 bits together.
// 257 is left out: its centred residues do not fit a byte.
static const int kMat2Moduli[kMat2MaxModuli] = {241, 233, 229, 221, 205, 197, 193, 181, 173,
                                                157, 149, 137, 113, 109, 101, 97,  89};

// Margin (bits) between the requested tolerance and the integer width: the
// scaling error of one operand element is <= 2^-b of its row/column maximum,
// and sums over k of such errors relative to the result stay well below 2^6.
static constexpr int kBitsMargin = 6;

hmat_status split_params(int64_t k, double tol, SplitParams* out) {
  if (tol == 0.0) tol = 1e-12;
  if (!(tol > 0.0) || !std::isfinite(tol)) return HMAT_STATUS_INVALID_VALUE;
  // k of up to 127 chunks of 1024: the running sums of the chunks' residues (twice as
  // many chunks in the four-multiplication form) stay exact
  if (k > (int64_t)127 * kChunkK) return HMAT_STATUS_UNSUPPORTED;
  SplitParams sp;
  const int want = (int)std::ceil(-std::log2(tol));
  // operands are rounded to at most 52-bit integers: below ~2^-50 nothing is promised
  if (want + 2 > 52) return HMAT_STATUS_TOLERANCE_UNREACHABLE;
  int bits = std::max(10, std::min(52, want + kBitsMargin));
  // the exact integer result of one output component is a sum of at most 8 real
  // products over k of b-bit integers: |Q| <= 8 k 2^(2b); CRT needs P > 2 |Q|,
  // and the extra 2^0.25 (|Q| < 0.42 P) lets the CRT kernel take the quotient
  // as the nearest integer to a float estimate of S / P, with no correction
  const double need = 2.0 * bits + std::log2((double)std::max<int64_t>(k, 1)) + 4.0 + 0.25;
  double acc = 0.0;
  int n = 0;
  while (acc <= need) {
    if (n >= kMaxModuli) return HMAT_STATUS_TOLERANCE_UNREACHABLE;
    sp.moduli[n] = kModuli[n];
    acc += std::log2((double)kModuli[n]);
    ++n;
  }
  sp.nmod = n;
  sp.bits = bits;
  sp.log2P = acc;
  *out = sp;
  return HMAT_STATUS_SUCCESS;
}

static int centred_mod(long long v, int p) {
  const int r = (int)(((v % p) + p) % p);
  return r > (p - 1) / 2 ? r - p : r;
}
// sum of the magnitudes of the weights 2^0, 2^16, 2^32 and their multiples by s modulo p
static long long mat2_digit_sum(int p, int s) {
  long long sum = 0;
  for (int d = 0; d < 3; ++d) {
    const int c = centred_mod(1ll << (16 * d), p);
    sum += std::abs(c) + std::abs(centred_mod((long long)c * s, p));
  }
  return sum;
}
// The square root of -1 modulo p with the smallest digit-weight sum (see
// mat2_digit_sum), up to sign, in [1, p); 0 if p has none within the bound.
static int mat2_root(int p) {
  int best = 0;
  long long best_sum = 0;
  for (int s = 1; s < p; ++s) {
    if ((s * s + 1) % p != 0) continue;
    const long long sum = mat2_digit_sum(p, s);
    if (best == 0 || sum < best_sum) {
      best = s;
      best_sum = sum;
    }
  }
  // u = sum_d x_d c_d + s y_d c_d stays an exact float: digits |x_d|, |y_d| <=
  // 2^15 + 1 (the fourth one <= 2^6) times the weights, below 2^24
  return best_sum < 500 ? best : 0;
}

int mat2_moduli(int64_t k, int bits) {
  // the same range as split_params: the recovered integers are the same
  const double need = 2.0 * bits + std::log2((double)std::max<int64_t>(k, 1)) + 4.0 + 0.25;
  double acc = 0.0;
  int n = 0;
  while (acc <= need) {
    if (n >= kMat2MaxModuli) return 0;
    acc += std::log2((double)kMat2Moduli[n++]);
  }
  return n;
}

bool crt_estimate_constants(const uint32_t* P, double max_quotient, int limbs, int* pb, float* pinv) {
  int top = 0;
  for (int q = 0; q < kLimbs; ++q)
    if (P[q]) top = q;
  *pb = top > 0 ? top - 1 : 0;
  double f = 0.0;                      // P / 2^(32 pb), then its float reciprocal
  for (int q = kLimbs - 1; q >= *pb; --q) f = f * 4294967296.0 + (double)P[q];
  *pinv = f > 0.0 ? (float)(1.0 / f) : 1.f;
  // the sums fit the limbs, and 2 + 2 (limbs - 1 - pb) + 2 float roundings of
  // relative size 2^-24 on S / P stay below the 0.0796 margin (1/2 - 2^-1.25)
  if (std::log2(f) + 32.0 * *pb + std::log2(std::max(max_quotient, 1.0)) >= 32.0 * limbs) return false;
  const double rounds = 4.0 + 2.0 * (limbs - 1 - *pb);
  return rounds * std::ldexp(1.0, -24) * max_quotient < 0.5 - std::exp2(-1.25);
}

// ----------------------------------------------------------------- tiny big integers (32-bit limbs)
namespace {

void big_mul_small(uint32_t* x, uint32_t m) {
  unsigned long long c = 0;
  for (int q = 0; q < kLimbs; ++q) {
    const unsigned long long t = (unsigned long long)x[q] * m + c;
    x[q] = (uint32_t)t;
    c = t >> 32;
  }
}
uint32_t big_mod_small(const uint32_t* x, uint32_t m) {
  unsigned long long r = 0;
  for (int q = kLimbs - 1; q >= 0; --q) r = ((r << 32) | x[q]) % m;
  return (uint32_t)r;
}
uint32_t inv_mod(uint32_t a, uint32_t m) {
  for (uint32_t x = 1; x < m; ++x)
    if ((unsigned long long)a * x % m == 1) return x;
  return 0;
}
// CRT basis element of moduli[l] among the first n: congruent to c modulo p_l
// and to 0 modulo the others, below P, in signed 32-bit digits (each word above
// 2^31 - 1 borrows from the next); times 2^shift
bool crt_element(const int* moduli, int n, int l, uint32_t c, int32_t* digits, int shift = 0) {
  const uint32_t p = (uint32_t)moduli[l];
  uint32_t Ml[kLimbs] = {1, 0, 0, 0, 0};
  for (int j = 0; j < n; ++j)
    if (j != l) big_mul_small(Ml, (uint32_t)moduli[j]);
  const uint32_t inv = inv_mod(big_mod_small(Ml, p), p);
  big_mul_small(Ml, (uint32_t)((unsigned long long)inv * (c % p) % p));
  for (int i = 0; i < shift; ++i) big_mul_small(Ml, 2u);
  long long carry = 0;
  for (int q = 0; q < kLimbs; ++q) {
    long long w = (long long)Ml[q] + carry;
    carry = 0;
    if (w >= (1ll << 31)) {
      w -= 1ll << 32;
      carry = 1;
    }
    digits[q] = (int32_t)w;
  }
  return carry == 0;   // the element is below P < 2^(32 kLimbs - 1)
}

// Tables of the matrix form: s with s^2 = -1 (mod p) per modulus, the CRT
// elements carrying 1/4 (outputs formed from the sums of the two matrix copies)
// and 1/(4 s) (from their differences), the products P and the offsets.
cudaError_t mat2_configure_tables() {
  static int32_t crt[kMat2MaxModuli + 1][2][kMat2MaxModuli][kLimbs];
  static uint32_t P[kMat2MaxModuli + 1][kLimbs], off[kMat2MaxModuli + 1][kLimbs];
  std::memset(crt, 0, sizeof(crt));
  std::memset(P, 0, sizeof(P));
  std::memset(off, 0, sizeof(off));
  int root[kMat2MaxModuli], shift[kMat2MaxModuli + 1] = {};
  for (int l = 0; l < kMat2MaxModuli; ++l) {
    root[l] = mat2_root(kMat2Moduli[l]);
    if (root[l] == 0) return cudaErrorInvalidValue;
  }
  for (int n = 1; n <= kMat2MaxModuli; ++n) {
    P[n][0] = 1;
    double log2P = 0.0;
    for (int l = 0; l < n; ++l) {
      big_mul_small(P[n], (uint32_t)kMat2Moduli[l]);
      log2P += std::log2((double)kMat2Moduli[l]);
    }
    if (n <= kMat2FourLimbs)                         // 2 N P in (2^126.9, 2^127.99)
      shift[n] = (int)std::floor(127.99 - log2P - std::log2(2.0 * n * kMat2WeightSum * kMat2HalfMax));
    for (int i = 0; i < shift[n]; ++i) big_mul_small(P[n], 2u);
    std::memcpy(off[n], P[n], sizeof(off[n]));
    big_mul_small(off[n], (uint32_t)(n * kMat2WeightSum * kMat2HalfMax));
    for (int l = 0; l < n; ++l) {
      const uint32_t p = (uint32_t)kMat2Moduli[l];
      if (!crt_element(kMat2Moduli, n, l, inv_mod(4u, p), crt[n][0][l], shift[n]) ||
          !crt_element(kMat2Moduli, n, l, inv_mod(4u * (uint32_t)root[l] % p, p), crt[n][1][l], shift[n]))
        return cudaErrorInvalidValue;
    }
  }
  return mat2_configure(kMat2Moduli, root, kMat2MaxModuli, &crt[0][0][0][0], &P[0][0], &off[0][0], shift);
}

}  // namespace

cudaError_t split_configure() {
  int32_t crt[kMaxModuli + 1][kMaxModuli][kLimbs];
  uint32_t P[kMaxModuli + 1][kLimbs];
  uint32_t off[kMaxModuli + 1][kLimbs];
  std::memset(crt, 0, sizeof(crt));
  std::memset(P, 0, sizeof(P));
  std::memset(off, 0, sizeof(off));
  for (int n = 1; n <= kMaxModuli; ++n) {
    P[n][0] = 1;
    for (int l = 0; l < n; ++l) big_mul_small(P[n], (uint32_t)kModuli[l]);
    // offset N P with N = n * kMaxWeightSum * 127 (the CRT sums stay positive)
    std::memcpy(off[n], P[n], sizeof(off[n]));
    big_mul_small(off[n], (uint32_t)(n * kMaxWeightSum * 127));
    for (int l = 0; l < n; ++l) {
      // d_l = (P / p_l) * ((P / p_l)^-1 4^-1 mod p_l): congruent to 4^-1 modulo
      // p_l and to 0 modulo the other moduli, below P
      if (!crt_element(kModuli, n, l, inv_mod(4u, (uint32_t)kModuli[l]), crt[n][l])) return cudaErrorInvalidValue;
    }
  }
  cudaError_t e = split_upload_constants(kModuli, kModTable, &crt[0][0][0], &P[0][0], &off[0][0]);
  if (e != cudaSuccess) return e;
  e = mat2_configure_tables();
  if (e != cudaSuccess) return e;
  // the GEMM's modulus table: the plans' moduli, then (from kModTable) the matrix form's
  int moduli[2 * kModTable];
  for (int l = 0; l < kModTable; ++l) {
    moduli[l] = kModuli[l];
    moduli[kModTable + l] = l < kMat2MaxModuli ? kMat2Moduli[l] : kMat2Moduli[0];
  }
  return split_gemm_configure(moduli, 2 * kModTable);
}

void split_release(SplitState& s) {
  for (SplitSlot& q : s.slots) {
    if (q.used && q.done) cudaEventSynchronize(q.done);
    if (q.done) cudaEventDestroy(q.done);
    if (q.uploaded) cudaEventDestroy(q.uploaded);
    if (q.h_jobs) cudaFreeHost(q.h_jobs);
    if (q.d_jobs) cudaFree(q.d_jobs);
    q = SplitSlot();
  }
  if (s.upload) cudaStreamDestroy(s.upload);
  s.upload = nullptr;
}

// ----------------------------------------------------------------- layout
// Built-in tile width: the fewest tiles of at most 256 columns, each as
// narrow as a multiple of 32 allows (tcgen05 takes any N that is a multiple of
// 16 with M = 128; the epilogue stores 32-column groups), so
// that padding columns stay below 32 per tile (n = 96: one tile of 96; n = 300:
// two of 160).
static int pick_bn(int64_t n) {
  const int64_t tiles = (n + 255) / 256;
  const int64_t per = (n + tiles - 1) / tiles;
  return (int)std::min<int64_t>(256, std::max<int64_t>(32, (per + 31) / 32 * 32));
}

static int ceil_log2(int64_t x) {
  int b = 0;
  while (((int64_t)1 << b) < x) ++b;
  return b;
}

int tile_bin(int64_t x) { return std::min(kTileBins - 1, ceil_log2(std::max<int64_t>(x, 1))); }

// Tile width for an m x n output: the tuned table entry for its (log2 m, log2 n)
// bin when one is set, else the default size rule.
static int choose_bn(const int8_t* table, int64_t m, int64_t n) {
  if (table) {
    const int v = table[tile_bin(m) * kTileBins + tile_bin(n)];   // 1, 2, 3 -> 64, 128, 256
    if (v >= 1 && v <= 3) return 32 << v;
  }
  return pick_bn(n);
}

static inline int64_t align256(int64_t x) { return (x + 255) & ~(int64_t)255; }

// Places the job's regions behind *offset (exponents, encoded factors, product residues).
static void place_job(SplitJob* sj, int64_t m, int64_t n, int64_t* offset) {
  int64_t off = *offset;
  sj->off_sexp = off;
  off = align256(off + 4 * m);
  sj->off_texp = off;
  off = align256(off + 4 * n);
  sj->off_encA = off;
  off = align256(off + (int64_t)sj->nmod * sj->nlf * sj->encA_plane);
  sj->off_encB = off;
  off = align256(off + (int64_t)sj->nmod * sj->nrf * sj->encB_plane);
  sj->off_res = off;
  off = align256(off + (int64_t)sj->nmod * sj->np * sj->res_plane);
  *offset = off;
}

Mat2Shape mat2_shape(uint32_t fa, uint32_t fb) {
  enum { kNone, kFull, kReal, kImag, kCplx };
  auto what = [](uint32_t f) {
    return f == 0xFFu ? kFull : f == 0x0Fu ? kReal : f == 0xF0u ? kImag : f == 0x11u ? kCplx : kNone;
  };
  const int a = what(fa), b = what(fb);
  const bool qa = a == kReal || a == kImag, qb = b == kReal || b == kImag;
  const int rot = (a == kImag ? 1 : 0) + (b == kImag ? 1 : 0);
  if ((a == kFull || qa) && (b == kFull || qb)) {
    if (qa && qb) return Mat2Shape{kMat2Quat, 7, 7, 7, rot};
    return Mat2Shape{kMat2Full, qa ? 7 : 14, qb ? 7 : 14, 14, rot};
  }
  if (a == kCplx && b == kFull) return Mat2Shape{kMat2Scaled, 2, 8, 8, 0};
  if (a == kFull && b == kCplx) return Mat2Shape{kMat2Scaled, 8, 2, 8, 0};
  if (a == kCplx && b == kCplx) return Mat2Shape{kMat2Complex, 2, 2, 2, 0};
  return Mat2Shape{};
}

// Turns a job laid out at offset0 into the matrix form, inside the bytes its plan's
// form occupies, when its operands have one.  The form wins wherever its planes
// (14 per modulus for a full product, one or two moduli more) do not outnumber the
// plan's (24, or 16 in the four-multiplication form), which also keeps it inside
// those bytes; that leaves out a few tiny k at loose tolerances (k <= 15 at tol
// 1e-3: 6 x 14 planes against 5 x 16).  Measured at tol 1e-12: full m = n = k =
// 8192, 15 x 14 planes against Gauss's 14 x 24: 226 -> 140 ms; the 512-product
// batch: 31.7 -> 18.7 ms; TRS x TRA m = n = k = 4096, 15 x 7 against 14 x 8: 14.4 -> 10.0 ms;
// complex x full 3000 x 1000 x 2000, 15 x 8 against 14 x 12: 2.49 -> 1.33 ms.
static void to_mat2(SplitJob* sj, int64_t offset0) {
  const Mat2Shape s = mat2_shape(sj->d.fa, sj->d.fb);
  if (s.kind == kMat2None) return;
  const int nm = mat2_moduli(sj->d.k, sj->bits);
  if (nm == 0 || nm * s.np > sj->nmod * sj->np || nm * s.nlf > sj->nmod * sj->nlf || nm * s.nrf > sj->nmod * sj->nrf)
    return;
  sj->mat2 = s.kind;
  sj->rot = s.rot;
  sj->mod_base = kModTable;
  sj->four_m = 0;
  sj->neg2 = 0;
  sj->nmod = nm;
  sj->np = s.np;
  sj->nlf = s.nlf;
  sj->nrf = s.nrf;
  // product p: the same plane of both sides; a side with half the planes has one
  // for both copies (a quaternion), a complex side one per copy
  for (int p = 0; p < kMaxProducts; ++p) {
    auto plane = [&](int planes) { return (int8_t)(p >= s.np ? 0 : planes == 2 ? p / (s.np / 2) : p % planes); };
    sj->pl[p] = plane(s.nlf);
    sj->pr[p] = plane(s.nrf);
    sj->pl2[p] = sj->pr2[p] = 0;
  }
  int64_t off = offset0;
  place_job(sj, sj->d.m, sj->d.n, &off);
}

// Accumulation chunks of the job's products: FP32 sums are exact up to 2^24, which is
// 1024 of k for residues up to 128 and 1088 for the matrix form's, up to 121.  Each
// chunk's drain runs beside the next chunk's MMAs, so the k-blocks are spread evenly: a
// short last chunk would leave the issuer waiting for the drain before it (1537 x 771 x
// 2049, three chunks of 16 + 16 + 1 k-blocks against two of 17 + 16: 867 -> 828 us).
static bool set_per_chunk(SplitJob* sj) {      // true when one chunk holds them all
  const int total = sj->four_m ? 2 * sj->nkb : sj->nkb;
  const int most = (sj->mat2 ? kMat2ChunkK : kChunkK) / kTileK;
  const int chunks = std::max(1, (total + most - 1) / most);
  sj->per_chunk = (total + chunks - 1) / chunks;
  return chunks == 1;
}
static_assert(kChunkK * 128 * 128 <= (1 << 24) && kMat2ChunkK * (kMat2HalfMax + 1) * (kMat2HalfMax + 1) <= (1 << 24),
              "exact FP32 accumulation of a chunk");

// plane skews: an odd multiple of 256 B (bulk copies need 16-byte alignment)
static constexpr int64_t kPlaneSkewEnc = 3 * 256;
static constexpr int64_t kPlaneSkewRes = 3 * 256;

// encode blocks: tiles of 16 rows x 32 k over the operand's rows rounded up to
// 16 (the residue GEMM copies whole 8-row groups of a tile and never reads the
// rows beyond them) and the inner dimension padded to whole k-blocks (zeros)
static inline int64_t enc_blocks(int64_t rows, int64_t nkb) { return ((rows + 15) / 16) * (nkb * kTileK / 32); }
// the matrix form's: the last k-block may be a half one
static inline int64_t mat2_enc_blocks(int64_t rows, int64_t k) { return ((rows + 15) / 16) * ((k + 31) / 32); }
static inline int64_t job_enc_blocks(const SplitJob& sj, int64_t rows) {
  return sj.mat2 ? mat2_enc_blocks(rows, sj.d.k) : enc_blocks(rows, sj.nkb);
}
// CRT blocks: one per `rows` output rows and kCrtCols consecutive columns
static inline int64_t crt_blocks(int64_t m, int64_t n, int rows) {
  return ((m + rows - 1) / rows) * ((n + kCrtCols - 1) / kCrtCols);
}
// CRT blocks of a job and its block width: the full-plan kernel's blocks are
// kCrtCols / crt_width(n) rows of crt_width(n) columns, the matrix form's likewise
// with mat2_crt_width, the other kernels' kCrtRows rows of kCrtCols columns
// Matrix form: 4 rows of 32 columns, which read 128 contiguous bytes of the residues (kept
// in groups of 32 columns), unless a wider block pads the output by 6 % less (few rows).
// The 512-product batch's CRT: 3.44 -> 3.27 ms against rows of residues with blocks of 32
// to 128 columns; rows of 128 columns here: 4.08 ms.
static int mat2_crt_width(int64_t m, int64_t n) {
  int best = 32;
  int64_t least = 0;
  for (int w = 32; w <= kCrtCols; w *= 2) {
    const int64_t rows = kCrtCols / w, elems = ((m + rows - 1) / rows * rows) * ((n + w - 1) / w * w);
    if (w == 32 || 106 * elems < 100 * least) {
      best = w;
      least = elems;
    }
  }
  return best;
}
static inline int64_t crt_job_blocks(SplitJob& sj, bool all_full) {
  if (!all_full && !sj.mat2) {
    sj.crt_w = kCrtCols;
    return crt_blocks(sj.d.m, sj.d.n, kCrtRows);
  }
  sj.crt_w = sj.mat2 ? mat2_crt_width(sj.d.m, sj.d.n) : crt_width(sj.d.n);
  const int64_t rows = kCrtCols / sj.crt_w;
  return ((sj.d.m + rows - 1) / rows) * ((sj.d.n + sj.crt_w - 1) / sj.crt_w);
}

// Fill the layout fields of sj (everything except the JobDesc and the unit prefixes).
static hmat_status layout_job(const SplitShape& sh, const KPlan* plan, double tol, const TileTables& tables, SplitJob* sj,
                              int64_t* offset) {
  if (plan) {                      // the CRT's integer residue step needs |4Q| <= kMaxWeightSum * 127
    for (int e = 0; e < 8; ++e) {
      int wsum = 0;
      for (int q = 0; q < plan->np; ++q) wsum += std::abs((int)plan->w4[e][q]);
      if (wsum > kMaxWeightSum) return HMAT_STATUS_INTERNAL;
    }
  }
  SplitParams sp;
  hmat_status st = split_params(sh.k, tol, &sp);
  if (st != HMAT_STATUS_SUCCESS) return st;
  sj->nmod = sp.nmod;
  sj->bits = sp.bits;
  sj->bn = choose_bn(tables.lookup(sh.fa, sh.fb), sh.m, sh.n);
  sj->tiles_m = (int32_t)((sh.m + kTileM - 1) / kTileM);
  sj->tiles_n = (int32_t)((sh.n + sj->bn - 1) / sj->bn);
  sj->nkb = (int32_t)((sh.k + kTileK - 1) / kTileK);
  sj->np = sh.np;
  sj->nlf = sh.nlf;
  sj->nrf = sh.nrf;
  sj->full = (plan ? plan->bilinear_full != 0 : sh.full != 0) ? 1 : 0;
  sj->four_m = (plan ? plan->four_m != 0 : sh.four_m != 0) ? 1 : 0;
  if (plan) {
    // every factor slot a product names lies inside the job's planes
    for (int p = 0; p < plan->np; ++p) {
      if (plan->pl[p] < 0 || plan->pl[p] >= sh.nlf || plan->pr[p] < 0 || plan->pr[p] >= sh.nrf)
        return HMAT_STATUS_INTERNAL;
      if (plan->four_m && (plan->pl2[p] < 0 || plan->pl2[p] >= sh.nlf || plan->pr2[p] < 0 || plan->pr2[p] >= sh.nrf))
        return HMAT_STATUS_INTERNAL;
    }
    for (int p = 0; p < kMaxProducts; ++p) {
      sj->pl[p] = plan->pl[p];
      sj->pr[p] = plan->pr[p];
      sj->pl2[p] = plan->four_m ? plan->pl2[p] : 0;
      sj->pr2[p] = plan->four_m ? plan->pr2[p] : 0;
    }
    sj->neg2 = plan->four_m ? plan->neg2 : 0;
  }
  // Plane strides get a skew so that the many planes a single encode / CRT
  // thread touches do not sit at power-of-two distances (which maps them onto
  // the same memory channels and cache sets).
  sj->encA_plane = (int64_t)sj->tiles_m * sj->nkb * kTileM * kTileK * 2 + kPlaneSkewEnc;
  sj->encB_plane = (int64_t)sj->tiles_n * sj->nkb * sj->bn * kTileK * 2 + kPlaneSkewEnc;
  // the encoder addresses a factor plane with a 32-bit stride (m k or k n below 2^31)
  if (sj->encA_plane >= ((int64_t)1 << 32) || sj->encB_plane >= ((int64_t)1 << 32)) return HMAT_STATUS_UNSUPPORTED;
  sj->res_plane = ((int64_t)sj->tiles_m * kTileM) * ((int64_t)sj->tiles_n * sj->bn) + kPlaneSkewRes;
  place_job(sj, sh.m, sh.n, offset);
  return HMAT_STATUS_SUCCESS;
}

hmat_status split_b_region_bytes(const SplitShape& sh, double tol, const TileTables& tables, int64_t* bytes) {
  SplitJob sj;
  std::memset(&sj, 0, sizeof(sj));
  int64_t off = 0;
  hmat_status st = layout_job(sh, nullptr, tol, tables, &sj, &off);
  if (st != HMAT_STATUS_SUCCESS) return st;
  *bytes = align256(4 * sh.n) + align256((int64_t)sj.nmod * sj.nrf * sj.encB_plane);
  return HMAT_STATUS_SUCCESS;
}

void split_place_b(SplitJob& sj, int64_t offset) {
  sj.off_texp = offset;
  sj.off_encB = offset + align256(4 * (int64_t)sj.d.n);
}

hmat_status split_workspace_bytes(const std::vector<SplitShape>& shapes, double tol, const TileTables& tables,
                                  size_t* bytes) {
  int64_t off = 0;
  for (const SplitShape& sh : shapes) {
    SplitJob sj;
    std::memset(&sj, 0, sizeof(sj));
    hmat_status st = layout_job(sh, nullptr, tol, tables, &sj, &off);
    if (st != HMAT_STATUS_SUCCESS) return st;
  }
  *bytes = (size_t)off;
  return HMAT_STATUS_SUCCESS;
}

hmat_status split_prepare(const std::vector<JobDesc>& jobs, const KPlan* h_plans, double tol, size_t ws_bytes,
                          const TileTables& tables, bool mat2, SplitPrep* out) {
  SplitPrep sp;
  int64_t off = 0;
  for (const JobDesc& d : jobs) {
    const KPlan& P = h_plans[d.plan];
    SplitJob sj;
    std::memset(&sj, 0, sizeof(sj));
    sj.d = d;
    SplitShape sh{d.m, d.n, d.k, P.np, P.nlf, P.nrf, P.bilinear_full, d.fa, d.fb, P.four_m};
    const int64_t off0 = off;
    hmat_status st = layout_job(sh, &P, tol, tables, &sj, &off);
    if (st != HMAT_STATUS_SUCCESS) return st;
    // the residue GEMM decodes a job's items with 32-bit arithmetic
    const int64_t plan_items = (int64_t)sj.nmod * sj.np * sj.tiles_m * sj.tiles_n;
    if (plan_items >= ((int64_t)1 << 31)) return HMAT_STATUS_UNSUPPORTED;
    if (mat2) to_mat2(&sj, off0);
    sj.exp_begin = sp.exp_units;
    sp.exp_units += (d.m + 31) / 32 + (d.n + 31) / 32;
    const int64_t ea = job_enc_blocks(sj, d.m), eb = job_enc_blocks(sj, d.n);
    sj.encA_begin = sp.encA_units;
    sj.encB_begin = sp.encB_units;
    sj.enc2_begin = sp.enc2_units;
    if (sj.mat2) {
      sp.enc2_units += ea + eb;
      sp.max_bits2 = std::max(sp.max_bits2, sj.bits);
      sp.max_nmod2 = std::max(sp.max_nmod2, sj.nmod);
    } else {
      sp.encA_units += ea;
      sp.encB_units += eb;
      sp.max_bits = std::max(sp.max_bits, sj.bits);
      sp.max_nmod = std::max(sp.max_nmod, sj.nmod);
      sp.max_np = std::max(sp.max_np, sj.np);
      sp.all_full = sp.all_full && sj.full;
      ++sp.n_plan;
    }
    sj.item_begin = sp.items;
    sp.items += (int64_t)sj.nmod * sj.np * sj.tiles_m * sj.tiles_n;
    if (!set_per_chunk(&sj)) sp.one_chunk = false;
    sp.n_four_m += sj.four_m ? 1 : 0;
    sp.jobs.push_back(sj);
  }
  // the CRT kernel, and with it the block shape, depends on every job's plan
  for (SplitJob& sj : sp.jobs) {
    const int64_t blocks = crt_job_blocks(sj, sp.all_full);
    sj.crt_begin = sp.crt_units;
    sj.crt2_begin = sp.crt2_units;
    (sj.mat2 ? sp.crt2_units : sp.crt_units) += blocks;
    if (!sj.mat2) sp.all_wide = sp.all_wide && sj.crt_w == kCrtCols;
  }
  if ((size_t)off > ws_bytes) return HMAT_STATUS_WORKSPACE_TOO_SMALL;
  sp.ws_needed = off;
  *out = std::move(sp);
  return HMAT_STATUS_SUCCESS;
}

hmat_status split_layout_single(const JobDesc& d, const KPlan& P, double tol, const TileTables& tables, bool mat2,
                                SplitJob* out, SplitUnits* units) {
  SplitJob sj;
  std::memset(&sj, 0, sizeof(sj));
  sj.d = d;
  SplitShape sh{d.m, d.n, d.k, P.np, P.nlf, P.nrf, P.bilinear_full, d.fa, d.fb, P.four_m};
  int64_t off = 0;
  hmat_status st = layout_job(sh, &P, tol, tables, &sj, &off);
  if (st != HMAT_STATUS_SUCCESS) return st;
  if ((int64_t)sj.nmod * sj.np * sj.tiles_m * sj.tiles_n >= ((int64_t)1 << 31)) return HMAT_STATUS_UNSUPPORTED;
  if (mat2) to_mat2(&sj, 0);
  units->exp = (d.m + 31) / 32 + (d.n + 31) / 32;
  units->encA = job_enc_blocks(sj, d.m);
  units->encB = job_enc_blocks(sj, d.n);
  units->items = (int64_t)sj.nmod * sj.np * sj.tiles_m * sj.tiles_n;
  units->crt = crt_job_blocks(sj, sj.full != 0);
  units->max_bits = sj.bits;
  units->max_nmod = sj.nmod;
  units->max_np = sj.np;
  units->one_chunk = set_per_chunk(&sj);
  units->all_full = sj.full != 0;
  units->four_m = sj.four_m != 0;
  units->ws_bytes = off;
  *out = sj;
  return HMAT_STATUS_SUCCESS;
}

hmat_status split_launch(hmat_context* h, const SplitPrep& sp, const SplitJob* d_jobs, const KPlan* d_plans,
                         unsigned char* ws, cudaStream_t stream) {
  const int njobs = (int)sp.jobs.size();
  SplitJobs jobs;
  jobs.table = d_jobs;
  jobs.n = njobs;
  jobs.one = &sp.jobs[0];
  cudaError_t e;
  // with reuse_a / reuse_b (one job) the A units, which come first in the
  // exponent stage, or the B units after them, are skipped, and so is that
  // side's encoder launch
  const bool skip_a = sp.reuse_a && njobs == 1, skip_b = sp.reuse_b && njobs == 1;
  {
    ProfScope ps(h, 1, stream);
    const int64_t a_units = njobs == 1 ? (sp.jobs[0].d.m + 31) / 32 : 0;
    const int64_t first = skip_a ? a_units : 0, end = skip_b ? a_units : sp.exp_units;
    e = launch_split_exponents(jobs, end, first, stream, ws, handle_sm_count(h));
  }
  if (e != cudaSuccess) return split_cuda_error(e);
  {
    ProfScope ps(h, 2, stream);
    if (!skip_a) e = launch_split_encode(jobs, d_plans, 0, sp.encA_units, stream, ws, sp.max_bits);
    if (e == cudaSuccess && !skip_b)
      e = launch_split_encode(jobs, d_plans, 1, sp.encB_units, stream, ws, sp.max_bits);
    // the matrix form's blocks: A side first, then B side
    const int64_t a_blocks = njobs == 1 ? mat2_enc_blocks(sp.jobs[0].d.m, sp.jobs[0].d.k) : 0;
    const int64_t first = skip_a ? a_blocks : 0, end = skip_b ? std::min(a_blocks, sp.enc2_units) : sp.enc2_units;
    if (e == cudaSuccess && end > first)
      e = launch_mat2_encode(jobs, end - first, first, stream, ws, sp.max_bits2, handle_sm_count(h));
  }
  if (e != cudaSuccess) return split_cuda_error(e);
  {
    ProfScope ps(h, 3, stream);
    const int grid = (int)std::min<int64_t>(sp.items, handle_sm_count(h));
    e = launch_split_gemm(jobs, sp.items, grid, stream, ws, sp.one_chunk);
  }
  if (e != cudaSuccess) return split_cuda_error(e);
  {
    ProfScope ps(h, 4, stream);
    const int full_form = sp.n_four_m == 0 ? 0 : (sp.n_four_m == sp.n_plan ? 1 : 2);
    e = launch_split_crt(jobs, d_plans, sp.crt_units, stream, ws, sp.max_nmod, sp.max_np, sp.all_full,
                         full_form, sp.all_wide);
    if (e == cudaSuccess && sp.crt2_units > 0)
      e = launch_mat2_crt(jobs, sp.crt2_units, stream, ws, sp.max_nmod2);
  }
  return e == cudaSuccess ? HMAT_STATUS_SUCCESS : split_cuda_error(e);
}

// Upload the job table through the handle's staging buffer and launch.
hmat_status run_split(hmat_context* h, const SplitPrep& sp, const KPlan* d_plans, void* workspace,
                      cudaStream_t stream) {
  // one matrix-form job travels in the kernel arguments: nothing to stage, copy or wait for
  if (sp.jobs.size() == 1 && sp.jobs[0].mat2)
    return split_launch(h, sp, nullptr, d_plans, static_cast<unsigned char*>(workspace), stream);
  SplitState& st_all = handle_split(h);
  SplitSlot& s = st_all.slots[st_all.next];
  st_all.next = (st_all.next + 1) % kSplitSlots;
  if (s.used) {   // the slot's previous call has finished reading its table
    if (cudaEventSynchronize(s.done) != cudaSuccess) return HMAT_STATUS_CUDA_ERROR;
  }
  if (!s.done && cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming) != cudaSuccess)
    return HMAT_STATUS_CUDA_ERROR;
  if (s.cap < sp.jobs.size()) {
    if (s.h_jobs) cudaFreeHost(s.h_jobs);
    if (s.d_jobs) cudaFree(s.d_jobs);
    s.h_jobs = nullptr;
    s.d_jobs = nullptr;
    s.cap = 0;
    const size_t cap = std::max<size_t>(sp.jobs.size(), 16);
    if (cudaMallocHost(&s.h_jobs, cap * sizeof(SplitJob)) != cudaSuccess) return HMAT_STATUS_CUDA_ERROR;
    if (cudaMalloc(&s.d_jobs, cap * sizeof(SplitJob)) != cudaSuccess) return HMAT_STATUS_CUDA_ERROR;
    s.cap = cap;
  }
  std::memcpy(s.h_jobs, sp.jobs.data(), sp.jobs.size() * sizeof(SplitJob));
  // The table is copied on the handle's upload stream when the call is made
  // (the slot's previous call has finished, synchronised above) and `stream`
  // waits for it.  A copy in the order of `stream` would be issued only when
  // the stream reaches it and could then wait behind bulk copies of other
  // streams on the same copy engine (the operand blocks of a streamed
  // product), holding up the kernels.  Under stream capture the copy stays
  // on `stream`.
  const size_t bytes = sp.jobs.size() * sizeof(SplitJob);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) return HMAT_STATUS_CUDA_ERROR;
  if (capture == cudaStreamCaptureStatusNone) {
    if (!st_all.upload && cudaStreamCreateWithFlags(&st_all.upload, cudaStreamNonBlocking) != cudaSuccess)
      return HMAT_STATUS_CUDA_ERROR;
    if (!s.uploaded && cudaEventCreateWithFlags(&s.uploaded, cudaEventDisableTiming) != cudaSuccess)
      return HMAT_STATUS_CUDA_ERROR;
    if (cudaMemcpyAsync(s.d_jobs, s.h_jobs, bytes, cudaMemcpyHostToDevice, st_all.upload) != cudaSuccess ||
        cudaEventRecord(s.uploaded, st_all.upload) != cudaSuccess ||
        cudaStreamWaitEvent(stream, s.uploaded, 0) != cudaSuccess)
      return HMAT_STATUS_CUDA_ERROR;
  } else if (cudaMemcpyAsync(s.d_jobs, s.h_jobs, bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess) {
    return HMAT_STATUS_CUDA_ERROR;
  }
  hmat_status st = split_launch(h, sp, s.d_jobs, d_plans, static_cast<unsigned char*>(workspace), stream);
  if (st != HMAT_STATUS_SUCCESS) return st;
  if (cudaEventRecord(s.done, stream) != cudaSuccess) return HMAT_STATUS_CUDA_ERROR;
  s.used = true;
  return HMAT_STATUS_SUCCESS;
}

}  // namespace hmat
