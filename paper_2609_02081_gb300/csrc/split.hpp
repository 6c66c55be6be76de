// split.hpp — split-precision (integer modular, Ozaki-type) mode: host-side interface.
//
// The exact integer products behind the bilinear scheme are computed on the
// BF16 tensor cores:
//   1. exponents : per row i of op(A) a power of two 2^s_i, per column j of
//                  op(B) 2^t_j, so that every component scaled by it is < 2^b
//                  in magnitude (one exponent shared by all eight components,
//                  so the pre-additions of the bilinear scheme stay exact);
//   2. encode    : X = round(op(A) 2^s) as integers, and for every modulus p
//                  the residues of the plan's left factors (the Hadamard and
//                  Gauss sums of Eq. bilinearH / Eq. cmplx-3-real-mult) in
//                  [-128, 128], stored as BF16 in the tensor-core tile layout;
//                  likewise the right factors of op(B);
//   3. residue GEMM (tcgen05): every real product of the plan for every
//                  modulus, BF16 x BF16 -> FP32 in tensor memory; FP32 sums of
//                  integers below 2^24 are exact, so the accumulator is drained
//                  every 1024 inner steps into int32 and reduced mod p at the end;
//   4. CRT       : per output element the plan's recombination (weights 2,
//                  -1/4, ... taken mod p), the Chinese remainder theorem over
//                  the moduli (exact integer of up to ~140 bits), conversion to
//                  FP64, the 2^-(s_i + t_j) rescaling and the complex alpha/beta
//                  update (Sec. III scaling and addition).
// Most products run by default in the matrix form (split_mat2.cu), which
// replaces the plan's products by fewer ones that exist only modulo suitable p:
// with s^2 = -1 (mod p) the biquaternions modulo p are two copies of the 2 x 2
// matrices modulo p (i -> s and i -> -s), and each 2 x 2 product takes seven
// multiplications (Strassen's, in Winograd's variant): 14 residue GEMMs per
// modulus instead of 24.  The integers that the CRT recovers, and so the results,
// are the same.
// The only rounding is step 2's scaling to b-bit integers; b and the modulus
// count follow from the requested tolerance and k.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>
#include <vector>

#include "../../include/hmat.h"
#include "common.cuh"

struct hmat_context;

namespace hmat {

constexpr int kMaxModuli = 18;
constexpr int kModTable = 24;
constexpr int kLimbs = 5;          // 160-bit CRT accumulators (32-bit limbs)
constexpr int kTileM = 128;        // tcgen05 M (one TMEM lane per output row)
constexpr int kTileK = 64;         // BF16 elements per 128-byte swizzled row
constexpr int kChunkK = 1024;      // inner steps per exact FP32 accumulation chunk
constexpr int kTileBins = 16;      // tile-width table: bins of ceil(log2 m) x ceil(log2 n)
constexpr int kCrtCols = 128;      // CRT output columns per block (two threads per element)
// CRT output rows per block: kCrtRows for the plan and generic kernels; the
// full-plan kernel (launches whose jobs all use the paper's full plan) takes
// kCrtCols / crt_width(n) rows of crt_width(n) columns: one row of 128 for
// wide products, four rows of 32 for narrower ones, whose ragged column
// blocks would leave threads idle
constexpr int kCrtRows = 4;
inline int crt_width(int64_t n) { return n >= 1024 ? kCrtCols : 32; }
// Largest sum_p |w4[e][p]| of a plan (the paper's full plan: 8 + 4 x 1 on the
// three Gauss terms); with centred product residues |T| <= 127 every output
// residue sum satisfies |4Q| <= 36 * 127 = 4572, which the CRT's integer
// residue step relies on.  Plans above it are refused.
constexpr int kMaxWeightSum = 36;
// Matrix form (split_mat2.cu).  What a job multiplies (SplitJob::mat2), by the
// operands' component flags: a pair of 2 x 2 products (full biquaternions, or one of
// them a real or i times a real quaternion), one 2 x 2 product (two such
// quaternions), a complex operand times the four coefficients of a full one, two
// complex operands.
enum { kMat2None = 0, kMat2Full = 1, kMat2Quat = 2, kMat2Scaled = 3, kMat2Complex = 4 };
struct Mat2Shape {
  int kind = kMat2None;
  int nlf = 0, nrf = 0, np = 0;      // factor planes per side and products per modulus
  int rot = 0;                       // the product is i^rot times that of the operands as encoded
};
Mat2Shape mat2_shape(uint32_t fa, uint32_t fb);
constexpr int kMat2MaxPlanes = 14;
// the largest sum of product residues in one output: |sum| <= 16 (p - 1)/2
constexpr int kMat2WeightSum = 16;
constexpr int kMat2ChunkK = 1088;  // its chunk (set_per_chunk)
constexpr int kMat2HalfMax = 120;  // (p - 1)/2 of its largest modulus, 241
// Most moduli whose sums S < 2 N P fit four 32-bit limbs (P < 2^111.1 and N =
// 15 * 16 * 120 < 2^14.9; checked when the tables are built)
constexpr int kMat2FourLimbs = 15;
constexpr int kMat2MaxModuli = 17; // whose CRT elements (P < 2^124.2) have sixteen 8-bit digits
// Largest inner dimension for which HMAT_CFORM_AUTO falls back from the matrix
// form to the four-multiplication form (and whose workspace it reports), not to
// Gauss's: its products (two terms of depth k) then fit one
// 1024-deep exact chunk of the residue GEMM.
constexpr int64_t kFourMMaxK = kChunkK / 2;

struct SplitParams {
  int nmod = 0;
  int bits = 0;
  int moduli[kMaxModuli];
  double log2P = 0.0;
};

// Moduli count and integer width for inner dimension k and target tolerance.
hmat_status split_params(int64_t k, double tol, SplitParams* out);
// Modulus count of the matrix form for inner dimension k and integer width
// bits; 0 when its moduli do not reach far enough.
int mat2_moduli(int64_t k, int bits);

struct SplitShape {
  int64_t m, n, k;
  int np, nlf, nrf;
  int full = 0;                     // the plan is the paper's full plan (KPlan::bilinear_full), either form
  uint32_t fa = 0xFFu, fb = 0xFFu;  // component flags of op(A), op(B) (the tile table may depend on them)
  int four_m = 0;                   // two-term products (KPlan::four_m): the GEMM runs over 2 k
};

// Split-mode tile-width tables: kTileBins x kTileBins codes (0 = built-in
// rule, 1/2/3 = 64/128/256 columns) for every product and, optionally, per
// (flagsA, flagsB) pair; a pair's own table wins for its products.
constexpr int kMaxFlagTables = 16;
struct TileTables {
  const int8_t* general = nullptr;  // null: the built-in rule
  const int8_t* by_flags = nullptr; // n_flags tables, kTileBins^2 codes each
  const uint16_t* keys = nullptr;   // (flagsA << 8) | flagsB of each
  int n_flags = 0;
  const int8_t* lookup(uint32_t fa, uint32_t fb) const {
    const uint16_t key = (uint16_t)(((fa & 0xFFu) << 8) | (fb & 0xFFu));
    for (int i = 0; i < n_flags; ++i)
      if (keys[i] == key) return by_flags + (size_t)i * kTileBins * kTileBins;
    return general;
  }
};

// A matrix-form operand whose last k-block holds at most 32 of k keeps it as a half
// block: rows of 64 bytes in the 64-byte swizzle instead of 128, at the start of the
// block's place, so that neither the encoder nor the GEMM moves the other half's zeros
// (64 products of 32 to 160: 307 -> 296 us, 512 of 32 to 1024: 20.2 -> 19.6 ms).
__host__ __device__ constexpr bool half_last_block(int k) { return ((k - 1) & 63) < 32; }

// Per-problem layout inside the caller's workspace.
struct SplitJob {
  JobDesc d;
  int32_t nmod, bits, bn;           // moduli, integer width, tile N
  int32_t tiles_m, tiles_n, nkb;    // 128-row tiles, bn-column tiles, 64-wide k blocks
  int32_t per_chunk;                // k-blocks of an accumulation chunk (set_per_chunk)
  int32_t np, nlf, nrf;
  int32_t full;                     // the plan is the paper's full plan (KPlan::bilinear_full), either form
  int32_t four_m;                   // two-term products: p is pl pr + (-1 if bit p of neg2) pl2 pr2
  int32_t crt_w;                    // full-plan and matrix-form CRT: columns per block row (kCrtCols / crt_w rows)
  int8_t pl[kMaxProducts], pr[kMaxProducts];
  int8_t pl2[kMaxProducts], pr2[kMaxProducts];
  uint64_t neg2;
  int64_t off_sexp, off_texp;       // int32 exponents (bytes into workspace)
  int64_t off_encA, off_encB;       // BF16 factor tiles
  int64_t off_res;                  // int8 product residues
  int64_t encA_plane, encB_plane;   // bytes between consecutive (modulus, factor) tile planes
  // bytes between consecutive (modulus, product) residue planes: rows of tiles_n bn bytes, in
  // the matrix form groups of 32 columns, each the tiles_m * 128 rows of 32 bytes
  int64_t res_plane;
  int32_t mat2, rot;                // matrix form (kMat2None: a plan's products): kind, power of i of the result
  int32_t mod_base;                 // first modulus in the GEMM's table (kModTable: the matrix form's moduli)
  int64_t item_begin;               // residue-GEMM work items before this job
  int64_t encA_begin, encB_begin;   // encode blocks before this job (matrix-form jobs have none)
  int64_t crt_begin;                // CRT blocks before this job (likewise)
  int64_t enc2_begin, crt2_begin;   // matrix form: encode blocks (A side, then B side) and CRT blocks before this job
  int64_t exp_begin;                // exponent work units before this job
};

// The job table as the launchers take it: a device array of n jobs, or one
// matrix-form job in host memory that travels in the kernels' arguments (table
// null), with nothing to stage, copy or wait for before the launch.
struct SplitJobs {
  const SplitJob* table = nullptr;
  int32_t n = 0;
  const SplitJob* one = nullptr;
};
// Kernel argument of the kernels that come in both versions.
template <bool kOne>
struct JobParam {};
template <>
struct JobParam<true> {
  SplitJob job;
};
static_assert(sizeof(SplitJob) <= 3800, "a job must fit the kernel argument space");

// Workspace bytes for a set of problems (sum of the per-problem layouts).
hmat_status split_workspace_bytes(const std::vector<SplitShape>& shapes, double tol, const TileTables& tables,
                                  size_t* bytes);
// Bin index of a dimension in the tile-width table.
int tile_bin(int64_t x);

// Handle-owned state of the split path (job-table staging).
// Job-table staging for split-mode calls: a ring of slots, so the host can
// queue the next call while the previous one still reads its table.  Two
// slots measured best for streamed products (n = 8192, 16 blocks: 283-285 ms
// per product against 284-292 with one slot and 292-295 with four, whose
// copies queued far ahead of the products).
struct SplitSlot {
  SplitJob* h_jobs = nullptr;
  SplitJob* d_jobs = nullptr;
  size_t cap = 0;
  cudaEvent_t done = nullptr;       // recorded on the call's stream after its last kernel
  cudaEvent_t uploaded = nullptr;   // recorded on the upload stream after the table copy
  bool used = false;
};
constexpr int kSplitSlots = 2;

struct SplitState {
  SplitSlot slots[kSplitSlots];
  int next = 0;
  cudaStream_t upload = nullptr;    // job-table copies, issued when the call is made
  bool has_table = false;
  int8_t tile_table[kTileBins * kTileBins] = {};   // tuned tile widths (0: default rule)
  int n_flag_tables = 0;                            // per flag pair tables, first n_flag_tables used
  uint16_t flag_keys[kMaxFlagTables] = {};
  int8_t flag_tables[kMaxFlagTables][kTileBins * kTileBins] = {};
};

cudaError_t split_configure();
void split_release(SplitState& s);

// Split-mode jobs of one call with their layouts and per-stage unit counts.
struct SplitPrep {
  std::vector<SplitJob> jobs;
  int64_t exp_units = 0, encA_units = 0, encB_units = 0, items = 0, crt_units = 0;
  int64_t enc2_units = 0, crt2_units = 0;   // matrix-form jobs
  int max_bits2 = 0, max_nmod2 = 0;         // matrix-form jobs (max_bits, max_nmod, max_np: the others)
  int64_t ws_needed = 0;
  int max_bits = 0, max_nmod = 0, max_np = 0;
  bool one_chunk = true;              // every job's products fit one accumulation chunk
  bool all_full = true;             // every job outside the matrix form uses the paper's full plan (either form)
  int n_four_m = 0;                 // jobs in the four-multiplication form
  int n_plan = 0;                   // jobs outside the matrix form
  bool all_wide = true;             // every job's full-plan CRT blocks are one row of kCrtCols columns
  // one job whose A-side exponents and encoded factor tiles are already in the
  // workspace from the previous call with the same A block and the same shape
  bool reuse_a = false;
  // one job whose B-side exponents and encoded tiles (at the job's off_texp /
  // off_encB, see split_place_b) are already there from an earlier call with
  // the same B block and the same shape
  bool reuse_b = false;
};

// Bytes of a job's B side (column exponents and encoded right factors), the
// region split_place_b points a job at.
hmat_status split_b_region_bytes(const SplitShape& sh, double tol, const TileTables& tables, int64_t* bytes);
// Point the job's B side at `offset` (bytes into the split workspace) instead
// of its own layout slot.
void split_place_b(SplitJob& sj, int64_t offset);

// Lay the jobs out in a workspace of ws_bytes (WORKSPACE_TOO_SMALL if it does not fit).
// mat2: products that have a matrix form run in it inside the bytes that
// their plan's form occupies (the workspace a caller must bring does not depend
// on it); products for which it has no advantage keep the plan's form.
hmat_status split_prepare(const std::vector<JobDesc>& jobs, const KPlan* h_plans, double tol, size_t ws_bytes,
                          const TileTables& tables, bool mat2, SplitPrep* out);
// Layout of one job at workspace offset 0 with its per-stage unit counts;
// uses no heap memory (for the entry point that allocates nothing).
struct SplitUnits {
  int64_t exp = 0, encA = 0, encB = 0, items = 0, crt = 0, ws_bytes = 0;
  int max_bits = 0, max_nmod = 0, max_np = 0;
  bool one_chunk = true;              // every job's products fit one accumulation chunk
  bool all_full = false;
  bool four_m = false;
};
hmat_status split_layout_single(const JobDesc& d, const KPlan& P, double tol, const TileTables& tables, bool mat2,
                                SplitJob* out, SplitUnits* units);
// Launch the four stages reading the device job table d_jobs (null: sp's one
// matrix-form job, in the kernel arguments).
hmat_status split_launch(hmat_context* h, const SplitPrep& sp, const SplitJob* d_jobs, const KPlan* d_plans,
                         unsigned char* ws, cudaStream_t stream);
// Upload the job table through the handle's staging buffer (unless it is one
// matrix-form job), then split_launch.
hmat_status run_split(hmat_context* h, const SplitPrep& sp, const KPlan* d_plans, void* workspace,
                      cudaStream_t stream);

// Profiling bracket around one kernel launch (no-op unless profiling is on).
class ProfScope {
 public:
  ProfScope(hmat_context* h, int kernel, cudaStream_t stream);
  ~ProfScope();

 private:
  hmat_context* h_;
  int kernel_;
  cudaStream_t stream_;
  cudaEvent_t a_ = nullptr, b_ = nullptr;
};

int handle_sm_count(hmat_context* h);
// Record a CUDA error for hmat_last_cuda_error() and return HMAT_STATUS_CUDA_ERROR.
hmat_status split_cuda_error(cudaError_t e);
SplitState& handle_split(hmat_context* h);


// Device-side kernel launchers (split_kernels.cu).
cudaError_t launch_split_exponents(const SplitJobs& jobs, int64_t units, int64_t first_unit,
                                   cudaStream_t s, unsigned char* ws, int sm_count);
// units are blocks: encode tiles of 32 rows x 32 k, CRT blocks of 256 elements
cudaError_t launch_split_encode(const SplitJobs& jobs, const KPlan* d_plans, int side, int64_t units,
                                cudaStream_t s, unsigned char* ws, int max_bits);
// one_chunk: every job's products fit one accumulation chunk (the one-chunk kernel form)
cudaError_t launch_split_gemm(const SplitJobs& jobs, int64_t items, int grid, cudaStream_t s,
                              unsigned char* ws, bool one_chunk);
// all_full: every job uses the paper's full plan (structured recombination),
// full_form: 0 all in Gauss's form, 1 all in the four-multiplication form, 2
// both; all_wide: every job's full-plan CRT blocks are one row of kCrtCols
// columns; else plans of at most 24 products take the packed-weight kernel with
// the same layout, larger ones (the component-wise comparison plan) the
// generic one
cudaError_t launch_split_crt(const SplitJobs& jobs, const KPlan* d_plans, int64_t units,
                             cudaStream_t s, unsigned char* ws, int max_nmod, int max_np, bool all_full,
                             int full_form, bool all_wide);
// Matrix form (split_mat2.cu).  Encode blocks [first, first + units) of the
// A and B sides of its jobs; jobs of other forms have no blocks.
cudaError_t launch_mat2_encode(const SplitJobs& jobs, int64_t units, int64_t first, cudaStream_t s,
                               unsigned char* ws, int max_bits, int sm_count);
cudaError_t launch_mat2_crt(const SplitJobs& jobs, int64_t units, cudaStream_t s, unsigned char* ws,
                            int max_nmod);
// n (kMat2MaxModuli) moduli, root[l]^2 = -1 mod moduli[l], and by modulus count
// the CRT tables [n + 1][2][n][kLimbs], [n + 1][kLimbs], [n + 1][kLimbs], all
// times 2^shift[count]
cudaError_t mat2_configure(const int* moduli, const int* root, int n, const int32_t* crt_d, const uint32_t* crt_P,
                           const uint32_t* crt_off, const int* shift);
// Constants of the CRT's quotient estimate for the modulus product P: pb the
// limb below its top one, pinv = fl(2^(32 pb) / P).  False when the estimate's
// error on sums below max_quotient P could miss the quotient with `limbs` limbs.
bool crt_estimate_constants(const uint32_t* P, double max_quotient, int limbs, int* pb, float* pinv);
cudaError_t split_upload_constants(const int* moduli, int nmod_table, const int32_t* crt_d, const uint32_t* crt_P,
                                   const uint32_t* crt_off);

}  // namespace hmat
