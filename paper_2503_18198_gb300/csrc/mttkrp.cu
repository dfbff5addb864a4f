// mttkrp.cu -- launch of one spMTTKRP along mode d (Algorithm 1's body for one
// mode): one kernel over the copy's blocks, which also zeroes the rows without
// nonzeros and adds the rows cut by block boundaries.  Fibre copies take
// separate zeroing and fix-up launches, Scheme 1 copies a cleared output.
#include <algorithm>

#include "mttkrp_kernel.cuh"

namespace spm {

using MttkrpKernelFn = void (*)(const MttkrpArgs);
MttkrpKernelFn pick_mttkrp_f32_a(int nin, int R);
MttkrpKernelFn pick_mttkrp_f32_b(int nin, int R);
MttkrpKernelFn pick_mttkrp_bf16_a(int nin, int R);
MttkrpKernelFn pick_mttkrp_bf16_b(int nin, int R);
MttkrpKernelFn pick_mttkrp_f32_c(int R);
MttkrpKernelFn pick_mttkrp_bf16_c(int R);
MttkrpKernelFn pick_mttkrp_bf16_plan_a(int nin, int R);
MttkrpKernelFn pick_mttkrp_bf16_plan_b(int nin, int R);
MttkrpKernelFn pick_mttkrp_bf16_plan_lean(int nin, int R);
MttkrpKernelFn pick_mttkrp_f32_lean(int nin, int R);
MttkrpKernelFn pick_mttkrp_bf16_lean(int nin, int R);

spm_status launch_mttkrp_fibre(spmttkrp_plan_s* p, int mode, const void* const* factors,
                               float* out, cudaStream_t s);  // mttkrp_fibre.cu

MttkrpKernelFn pick_mttkrp_f32_between3(int R);
MttkrpKernelFn pick_mttkrp_f32_between4(int R);
MttkrpKernelFn pick_mttkrp_f32_between5(int R);
MttkrpKernelFn pick_mttkrp_bf16_between3(int R);
MttkrpKernelFn pick_mttkrp_bf16_between4(int R);
MttkrpKernelFn pick_mttkrp_bf16_between5(int R);
MttkrpKernelFn pick_mttkrp_f32_lean_between3(int R);
MttkrpKernelFn pick_mttkrp_f32_lean_between4(int R);
MttkrpKernelFn pick_mttkrp_f32_lean_between5(int R);
MttkrpKernelFn pick_mttkrp_bf16_lean_between3(int R);
MttkrpKernelFn pick_mttkrp_bf16_lean_between4(int R);
MttkrpKernelFn pick_mttkrp_bf16_lean_between5(int R);

// 3 to 5 modes and a rank without a fast shape: the shape between, or null.
static MttkrpKernelFn pick_mttkrp_between(bool bf16, bool lean, int nin, int R) {
  const int W = bf16 ? 8 : 4, l = R / W;
  const bool fast = (R % W == 0 && l <= 64 && (l & (l - 1)) == 0) || (bf16 && nin == 2 && R == 4);
  if (fast) return nullptr;
  if (lean) switch (nin) {
    case 2: return bf16 ? pick_mttkrp_bf16_lean_between3(R) : pick_mttkrp_f32_lean_between3(R);
    case 3: return bf16 ? pick_mttkrp_bf16_lean_between4(R) : pick_mttkrp_f32_lean_between4(R);
    case 4: return bf16 ? pick_mttkrp_bf16_lean_between5(R) : pick_mttkrp_f32_lean_between5(R);
    default: return nullptr;
  }
  switch (nin) {
    case 2: return bf16 ? pick_mttkrp_bf16_between3(R) : pick_mttkrp_f32_between3(R);
    case 3: return bf16 ? pick_mttkrp_bf16_between4(R) : pick_mttkrp_f32_between4(R);
    case 4: return bf16 ? pick_mttkrp_bf16_between5(R) : pick_mttkrp_f32_between5(R);
    default: return nullptr;
  }
}

MttkrpKernelFn pick_mttkrp(bool bf16, int nin, int R) {
  if (MttkrpKernelFn fn = pick_mttkrp_between(bf16, false, nin, R)) return fn;
  if (nin == 4) return bf16 ? pick_mttkrp_bf16_c(R) : pick_mttkrp_f32_c(R);
  if (bf16) return nin <= 2 ? pick_mttkrp_bf16_a(nin, R) : pick_mttkrp_bf16_b(nin, R);
  return nin <= 2 ? pick_mttkrp_f32_a(nin, R) : pick_mttkrp_f32_b(nin, R);
}

namespace {

// Rows without nonzeros (bit clear in `mask`) are written as zeros.
__global__ void __launch_bounds__(256)
    zero_empty_rows_kernel(const uint32_t* __restrict__ mask, int64_t I, int R,
                           float* __restrict__ out) {
  zero_empty_rows_body(mask, I, R, out, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                       (I + 31) / 32, (int)(gridDim.x * (blockDim.x >> 5)), threadIdx.x & 31);
}

// One warp per block z of the MTTKRP (see mttkrp_fixup_body).
__global__ void __launch_bounds__(256)
    mttkrp_fixup_kernel(const float* cta_part, const int* cta_meta, int nblocks, int R,
                        float* __restrict__ out) {
  const int z = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (z < nblocks) mttkrp_fixup_body(cta_part, cta_meta, nblocks, R, out, z, threadIdx.x & 31);
}

}  // namespace

// Launch the boundary fix-up on given partials (no finished-block counter).
spm_status launch_mttkrp_fixup(const float* cta_part, const int* cta_meta, int kappa, int R,
                               float* out, cudaStream_t s) {
  if (kappa <= 1) return SPM_OK;
  const int threads = 256;
  const int blocks = (int)ceil_div<int64_t>((int64_t)kappa * 32, threads);
  mttkrp_fixup_kernel<<<blocks, threads, 0, s>>>(cta_part, cta_meta, kappa, R, out);
  SPM_CUDA_TRY(cudaGetLastError());
  return SPM_OK;
}

void mttkrp_set_shape(const spmttkrp_plan_s* p, int d, bool plan_order, MttkrpArgs* a) {
  const spm_mode_copy& c = p->mode[d];
  a->words = 4 * record_int4s(p->N);
  a->nplan = p->kappa * p->nu;
  a->woff = c.woff;
  if (!plan_order) {
    a->split = 0;
    a->nu = c.nx;
    a->nblocks = c.kx;
    return;
  }
  a->split = 1;
  if (p->als.split_cap >= p->kappa && c.scheme != 1) {
    a->split = mttkrp_split(p->nnz, p->kappa, p->nu, sm_count());
    a->upart = p->als.upart;
    a->urow = p->als.urow;
    a->pdone = p->als.pdone;
  }
  a->nu = p->nu / a->split;
  a->nblocks = p->kappa * a->split;
}

int mttkrp_launches(const spmttkrp_plan_s* p, int mode, int* blocks) {
  const spm_mode_copy& c = p->mode[mode];
  MttkrpArgs a{};
  mttkrp_set_shape(p, mode, false, &a);
  *blocks = p->nnz == 0 ? 0 : c.fstream ? p->kappa : a.nblocks;
  if (p->nnz == 0) return 0;
  if (c.fstream) return (c.empty_rows > 0 ? 1 : 0) + 1 + (p->kappa > 1 ? 1 : 0);
  return 1 + (c.scheme != 1 && !mttkrp_few_parts(a) ? 1 : 0);
}

spm_status run_mttkrp(spmttkrp_plan_s* p, int mode, const void* const* factors, float* out,
                      cudaStream_t s, bool plan_order) {
  if (!p || mode < 0 || mode >= p->N || !factors || !out) return SPM_ERR_INVALID_ARG;
  const int R = p->R;
  const spm_mode_copy& c = p->mode[mode];
  MttkrpArgs a{};
  const bool lean = c.src != nullptr;  // lean copy: records gathered from copy 0
  a.rec = lean ? p->mode[0].rec : c.rec;
  a.src = c.src;
  a.fmode = mode;
  int m = 0;
  for (int w = 0; w < p->N; ++w) {
    if (w == mode) continue;
    if (!factors[w] || (reinterpret_cast<uintptr_t>(factors[w]) & 15u)) return SPM_ERR_INVALID_ARG;
    a.fac[m++] = factors[w];
  }
  if (reinterpret_cast<uintptr_t>(out) & 15u) return SPM_ERR_INVALID_ARG;
  a.out = out;
  a.cta_part = p->cta_part;
  a.cta_meta = p->cta_meta;
  a.nnz = p->nnz;
  a.I = p->dims[mode];
  a.R = R;
  a.nin = p->N - 1;
  mttkrp_set_shape(p, mode, plan_order, &a);
  a.err = p->dev_err;
  a.wait_limit = p->wait_limit;
  const size_t out_bytes = sizeof(float) * (size_t)a.I * (size_t)R;
  if (p->nnz == 0) {
    SPM_CUDA_TRY(cudaMemsetAsync(out, 0, out_bytes, s));
    return SPM_OK;
  }
  if (c.fstream) {
    if (c.empty_rows > 0) {
      const int blocks = (int)std::min<int64_t>(ceil_div<int64_t>((a.I + 31) / 32, 8), 152 * 8);
      zero_empty_rows_kernel<<<blocks, 256, 0, s>>>(c.rowmask, a.I, R, out);
      SPM_CUDA_TRY(cudaGetLastError());
    }
    SPM_TRY(launch_mttkrp_fibre(p, mode, factors, out, s));
    return launch_mttkrp_fixup(p->cta_part, p->cta_meta, p->kappa, R, out, s);
  }
  if (c.scheme == 1) {  // no row spans two partitions
    SPM_CUDA_TRY(cudaMemsetAsync(out, 0, out_bytes, s));
  } else {
    if (mttkrp_few_parts(a)) a.done = p->dev_err + 1;
    if (c.empty_rows > 0) a.rowmask = c.rowmask;
  }
  const int nin = p->N - 1;
  MttkrpKernelFn fn;
  if (a.split > 0)  // BF16 (run_mttkrp's plan order)
    fn = lean ? pick_mttkrp_bf16_plan_lean(nin, R)
              : (nin <= 2 ? pick_mttkrp_bf16_plan_a(nin, R) : pick_mttkrp_bf16_plan_b(nin, R));
  else if (lean) {
    fn = pick_mttkrp_between(p->bf16, true, nin, R);  // the full plan's lanes: the same sums
    if (!fn) fn = p->bf16 ? pick_mttkrp_bf16_lean(nin, R) : pick_mttkrp_f32_lean(nin, R);
  } else
    fn = pick_mttkrp(p->bf16, nin, R);
  if (!fn) return SPM_ERR_UNSUPPORTED;
  // a block that is full of short units leaves room for a second one
  const int warps = a.split > 1 || (a.split == 1 && p->nnz / p->kappa < 4096) ? 16
                    : a.split == 1 ? 32 : mttkrp_warps(a.nu);
  const size_t smem = mttkrp_smem_bytes(R, a.split > 1 ? p->nu : a.nu, warps);
  SPM_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // Smallest shared-memory carve-out that fits the resident blocks: the rest
  // of the unified array is L1 for the gathered factor rows.
  const size_t used = (smem + 2048) * (warps == 32 ? 1 : 2);
  const int carve = (int)std::min<size_t>(100, (used + 2048) * 100 / (228 * 1024) + 1);
  SPM_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, carve));
  fn<<<a.nblocks, warps * 32, smem, s>>>(a);
  SPM_CUDA_TRY(cudaGetLastError());
  if (c.scheme != 1 && !a.done)
    return launch_mttkrp_fixup(p->cta_part, p->cta_meta, mttkrp_parts(a), R, out, s);
  return SPM_OK;
}

}  // namespace spm
