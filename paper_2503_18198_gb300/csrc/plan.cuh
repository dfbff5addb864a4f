// plan.cuh -- the plan object and the internal entry points between the
// library's translation units.
#pragma once

#include "common.cuh"

// Work unit of a fibre-layout copy: its range of stream entries (from its
// first nonzero to its last, headers between them included) and the fibre
// header of its first nonzero, which may lie before the range.
struct FibreUnit {
  int64_t sbeg, send;  // stream entries [sbeg, send); empty unit: sbeg == send
  int cd_first;        // output row of the unit's first nonzero
  int ca_first;        // first input-mode index of that nonzero's fibre
  int cd_last;         // output row of the nonzero before the unit's end (-1: none)
  int pad;
};

struct spm_mode_copy {
  int4* rec = nullptr;       // records, record_int4s(N) int4 per nonzero (null: lean or fibre copy)
  int2* fstream = nullptr;   // fibre copy: header entries {c_a | 2^31, c_d} each followed by
                             // the fibre's nonzero entries {c_b, value bits}; 2 entries of padding
  FibreUnit* funits = nullptr;  // fibre copy: [kappa * nu] work units
  int64_t nfib = 0;          // fibre copy: number of fibres (headers)
  int32_t* perm = nullptr;   // input position of each copy position (null: lean copy)
  int32_t* src = nullptr;    // lean copy: position in copy 0 of each copy position
  int64_t* off = nullptr;    // device int64[kappa+1] partition offsets
  int64_t* woff = nullptr;   // device int64[kappa*nu+1] work-unit offsets
  int kx = 0, nx = 0;        // thread blocks and units per block with which the kernel runs it
  uint32_t* rowmask = nullptr;  // bit i set: output row i has a nonzero
  int64_t empty_rows = 0;    // rows without nonzeros
  int scheme = 0;            // 0 cost-balanced, 1 or 2 (Sec. III-B)
};

// Ranks of the tensor-core row solve.
#ifndef SPM_ALS_TC
#define SPM_ALS_TC 1  // 0: every rank takes the CUDA-core (double-float) row solve
#endif
__host__ __device__ constexpr bool tc_solve_rank(int R) {
  return SPM_ALS_TC && (R == 16 || R == 32 || R == 64);
}
// Bytes of the solve's W digit tiles: the BF16 digit stack (7 digits x R x R) and
// R column exponents.  Where there is none the system kernel writes V^{-1} for
// the CUDA-core solve in its place.
inline constexpr size_t als_wdig_bytes(int R) {
  return tc_solve_rank(R) ? (size_t)7 * 2 * R * R + 4 * (size_t)R : 0;
}

constexpr int ALS_MAX_RANK = 64;  // of CP-ALS sweeps

struct spm_als_state {
  bool ready = false;                 // Gram cache valid for `fac_ptr`
  const void* fac_ptr[SPM_MAX_MODES] = {};
  double* gram = nullptr;             // [N][R*R] Grams of the stored factors
  double* gram_part = nullptr;        // [gram_blocks][R*R] block partials
  int gram_blocks = 0;
  float* winv = nullptr;              // 2*R*R: V^{-1} as hi/lo float pairs
  double* colsq_part = nullptr;       // [gram_blocks][R] column sums of Z^2
  float* colmax_part = nullptr;       // [gram_blocks][R] column maxima of |Z|
  unsigned char* wdig = nullptr;      // W = V^{-1} as BF16 digit tiles (tensor-core solve)
  double* inner_part = nullptr;       // [gram_blocks][R] sums of M .* Y
  double* lambda_ws = nullptr;        // R
  float* M = nullptr;                 // Imax*R MTTKRP output
  float* Z = nullptr;                 // Imax*R unnormalised update
  // plan-order MTTKRP with several blocks per partition: unit boundary partials
  // [kappa*nu][2][R], their rows, finished blocks per partition (else null)
  float* upart = nullptr;
  int* urow = nullptr;
  int* pdone = nullptr;
  int split_cap = 0;  // partitions those hold
  // the Gram of a mode and the normal-equation system of the next depend only on
  // factors already written, so they are formed on a side stream while the next
  // mode's MTTKRP runs
  cudaStream_t side = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
};

struct spmttkrp_plan_s {
  int device = 0;
  int N = 0;
  int R = 0;
  int64_t dims[SPM_MAX_MODES] = {};
  int64_t nnz = 0;
  uint32_t flags = 0;
  bool bf16 = false;
  bool lean = false;  // SPM_PLAN_LEAN: copies 1..N-1 are positions into copy 0
  bool fibre = false; // SPM_PLAN_FIBRE: every copy in the fibre layout (3 modes)
  int kappa = 0;
  int kappa_cap = 0;  // partitions the off/woff/cta arrays are sized for
  int nu = 0;      // work units per partition
  int policy = 0;  // SPM_POLICY_* >> 4
  spm_mode_copy mode[SPM_MAX_MODES];
  // MTTKRP workspace: per-partition boundary-row partial sums.
  float* cta_part = nullptr;   // [boundary_blocks][2][R]
  int* cta_meta = nullptr;     // [boundary_blocks][4]
  // Device scalars.
  int* dev_err = nullptr;      // [0] sticky error flags (spm::DEV_ERR_*), [1] finished blocks
                               // of the running MTTKRP (zero between runs)
  double* normX2 = nullptr;    // |X|_F^2 (duplicates summed)
  double* norm_part = nullptr; // partials for normX2
  spm_als_state als;
  // host-buffer entry point: device staging of factors and outputs, and the
  // side streams / events that overlap its copies with the modes' kernels
  void* h_fac[SPM_MAX_MODES] = {};
  float* h_out[SPM_MAX_MODES] = {};
  cudaStream_t copy_in = nullptr, copy_out = nullptr;
  cudaEvent_t ev[2 * SPM_MAX_MODES + 2] = {};
  size_t bytes = 0;
  // record-copy wait bound of the MTTKRP kernel (0 = default; failure tests
  // set ~0u so the first wait gives up at once)
  uint32_t wait_limit = 0;
  // allocation bookkeeping
  void* allocs[96] = {};
  size_t alloc_bytes[96] = {};
  int nallocs = 0;
};

namespace spm {

// Device memory (dev_alloc.cu).  dev_free: with the size it was allocated with,
// once no queued work uses it; dev_drain(device) waits for all work of the
// memory's device, which need not be the current one (false: it could not, for
// instance during a stream capture, and the memory must not be handed back).
spm_status dev_alloc(void** ptr, size_t bytes);
void dev_free(void* ptr, size_t bytes);
bool dev_drain(int device);
// Bytes that are kept for reuse on `device` and belong to no buffer, and giving
// them back if they are more than `keep`.
size_t dev_held(int device);
void dev_trim(int device, size_t keep);
// dev_free of scratch that only work on `s` uses, whatever else is queued.
void scratch_free(void* ptr, size_t bytes, cudaStream_t s);

// Allocation owned by the plan (recorded for destroy and for plan_bytes).
spm_status plan_alloc(spmttkrp_plan_s* p, void** ptr, size_t bytes);

// Replace an allocation made by plan_alloc with a new one of `bytes`
// (contents not kept).
spm_status plan_realloc(spmttkrp_plan_s* p, void** ptr, size_t bytes);

// Release one allocation made by plan_alloc (after a device synchronisation
// of the caller's stream, or stream-ordered work that no longer reads it).
void plan_free(spmttkrp_plan_s* p, void** ptr);

// Slots (work units a warp takes side by side) of the fibre-layout kernel for
// rank R: each lane holds SPM_FB_VEC ranks of a unit's rows (4: one 16-byte
// FP32 or 8-byte BF16 load per row; 8: two 16-byte FP32 loads or one 16-byte
// BF16 load), R / SPM_FB_VEC lanes per unit; 0 when the rank has no fibre
// kernel.  With 8 the per-step control work is shared by twice the slots but
// a batch more often holds a row change; 4 measured faster.
#ifndef SPM_FB_VEC
#define SPM_FB_VEC 4
#endif
inline int fibre_slots(int R) {
  return (R == 16 || R == 32 || R == 64) ? 32 * SPM_FB_VEC / R : 0;
}

// Device bytes a plan holds (resident: copies, partitions, workspace, and
// with `als` the CP-ALS state) and the most its build adds for a while
// (transient scratch), for the given shape.
void plan_bytes_estimate(int N, const int64_t* dims, int64_t nnz, int R, int kappa, bool als,
                         bool lean, size_t* resident, size_t* transient, bool fibre = false,
                         int policy = 0, bool bf16 = false);

// Thread blocks and work units per block with which a record copy of nnz
// nonzeros is run.  The partitions B_{d,z} that the caller sees (kappa, nu)
// are kept, one block of 32 warps each, where there are enough of them for the
// device -- or a whole number per SM was asked for, as in the paper -- and each
// holds 4096 nonzeros; otherwise the copy is cut for the device:
//  * a block per 1024 nonzeros up to two per SM.  One tensor of 4,096
//    nonzeros on the default 304 partitions of 128 units ran 31 us per mode
//    (cold caches), 300,000 nonzeros 50 us; in this shape 14 and 11 us;
//  * units of at least 128 nonzeros (two record tiles), 16 to nu per block.
// The kernel reads its unit boundaries off the plan's: unit j of kx * nx begins
// j / (kx * nx) of the way through the plan's units, inside one by its length.
// Scheme 1 keeps its partitions: their rows are not in order across them.
// (One per SM: 20M uniform nonzeros, three modes 0.80 ms, two per SM 0.83; on
// skewed tensors two are faster, which the autotuner finds out.)
// A plan with fewer partitions than that was asked for few (the batch's autotuner
// and the server choose about 131,072 nonzeros each, to share the device among
// many tensors): MTTKRP_CUT blocks per partition.  96 FP32 tensors up to 2M
// nonzeros, two sweeps: 5.40 ms cut for the device, 4.47 / 4.40 / 4.83 ms with
// 16 / 8 / 2; ten served jobs of up to 3M: 13.9 cut for the device, 14.1 / 15.0
// / 18.5 ms.
constexpr int MTTKRP_CUT = 16;
struct MttkrpShape {
  int kx, nx;
};
inline constexpr int mttkrp_fine_blocks(int64_t nnz, int sms) {
  const int64_t b = (nnz + 1023) / 1024;
  return (int)(b < 1 ? 1 : b > 2 * sms ? 2 * sms : b);
}
inline constexpr MttkrpShape mttkrp_shape(int scheme, int64_t nnz, int kappa, int nu, int sms) {
  if (scheme == 1) return {kappa, nu};
  const int fine = mttkrp_fine_blocks(nnz, sms);
  const bool keep = kappa >= fine || kappa % sms == 0;
  const int kx = !keep ? std::min(fine, MTTKRP_CUT * kappa) : nnz / kappa >= 4096 ? kappa : fine;
  int nx = 16;
  while (2 * nx <= nu && nnz / kx >= (int64_t)nx * 256) nx *= 2;
  return {kx, nx};
}
// Blocks per partition of a run in plan order (BF16 CP-ALS, see run_mttkrp): a
// partition's units are shared by up to nu / 16 blocks (16 warps take one each)
// while there are fewer than two blocks per SM and 1024 nonzeros for each.
inline constexpr int mttkrp_split(int64_t nnz, int kappa, int nu, int sms) {
  int s = 1;
  while (32 * s <= nu && nu % (2 * s) == 0 && kappa * s < 2 * sms && nnz / kappa >= 2048 * (int64_t)s) s *= 2;
  return s;
}

// Whether a plan's CP-ALS keeps the buffers of such a run (fibre copies have their
// own kernel).
inline constexpr bool als_splits(bool bf16, bool fibre, int64_t nnz, int kappa, int nu, int sms) {
  return bf16 && !fibre && mttkrp_split(nnz, kappa, nu, sms) > 1;
}

// Warps of a block: short unit lists leave half of the SM to a second block,
// whose start and merge overlap the first one's gathers.
inline int mttkrp_warps(int nx) { return nx >= 32 ? 32 : 16; }

// Blocks for which boundary partials are held.
inline int boundary_blocks(int64_t nnz, int kappa, int sms) {
  const int fine = mttkrp_fine_blocks(nnz, sms);
  return kappa > fine ? kappa : fine;
}

// Set every copy's kx and nx from the plan's kappa.
void plan_shapes(spmttkrp_plan_s* p);

// P2 again for a new partition count (cost-balanced and Scheme 2 policies).
spm_status plan_repartition(spmttkrp_plan_s* p, int kappa, cudaStream_t s);

// P1 + P2: build every mode copy and its partition (plan.cu).
spm_status build_copies(spmttkrp_plan_s* p, const int32_t* const* idx,
                        const float* vals, cudaStream_t s);

// P3 + P4: one MTTKRP launch sequence for mode d (mttkrp.cu).
// plan_order (BF16 factors, R <= 64): sum in the order that the plan's
// partitions define, whatever the launch shape.  A decomposition with BF16
// factors asks for it: each update is rounded to 8 bits, so one flipped last bit
// of M becomes another factor, and its result would depend on how the device is
// filled.  (Any fixed order is as near to the exact sums: this is about results
// that stay the same, not about accuracy.  It bounds the launch shapes, see
// mttkrp_split.)
spm_status run_mttkrp(spmttkrp_plan_s* p, int mode, const void* const* factors,
                      float* out, cudaStream_t s, bool plan_order = false);

// Kernels that run_mttkrp launches (any order), and the blocks of the spMTTKRP
// kernel among them; the same conditions as there.
int mttkrp_launches(const spmttkrp_plan_s* p, int mode, int* blocks);

// The launch shape and plan-order fields of `a` for mode d of plan p.
struct MttkrpArgs;
void mttkrp_set_shape(const spmttkrp_plan_s* p, int d, bool plan_order, MttkrpArgs* a);

// P6: one CP-ALS sweep (als.cu).
spm_status als_sweep(spmttkrp_plan_s* p, void* const* factors, double* lambda,
                     double* fit, cudaStream_t s);

// G = Y^T Y (FP64, R x R) of a stored factor with the plan's block split (als.cu).
// With `mask`, rows whose bit is clear are known to be zero and are skipped.
spm_status gram(spmttkrp_plan_s* p, const void* Y, int64_t I, double* G, cudaStream_t s,
                const uint32_t* mask = nullptr);

// Allocate the plan's CP-ALS workspace on first use (als.cu).
spm_status ensure_als_state(spmttkrp_plan_s* p, cudaStream_t s);

int sm_count();

// True when an allocation failure injected by spm_inject_alloc_failure is
// due now (diag.cu).
bool alloc_fault_due();

// Partition count of a plan made with SPM_KAPPA(0): SPM_PARTITIONS_PER_SM
// per SM (-1 when the device cannot be queried).
int default_kappa();

}  // namespace spm
