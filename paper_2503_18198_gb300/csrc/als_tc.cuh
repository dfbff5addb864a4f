// als_tc.cuh -- the CP-ALS row passes on the tensor cores, with FP64-level
// accuracy from BF16 x BF16 -> FP32 MMAs (exact operand splitting).
//
// Row solve Z = M V^{-1}.  V is the Hadamard product of the Grams (Sec. II-A5) in
// FP64; W = V^{-1} comes from L D L^T in FP32 pairs with a correction from the
// FP64 residual, or in FP64 where V is ill-conditioned (system_body).  Splitting:
//  * each row i of M (FP32) is scaled by 2^-e_i (e_i the exponent of its
//    largest magnitude) and cut into SM_DIG integer digits of 7 bits,
//    m_i = 2^e_i * sum_p k_p(i) 2^{-7(p+1)}, |k_p| <= 128;
//  * each column c of W likewise into SW_DIG digits with scale 2^f_c (done
//    once per mode by system_body, not per block).
// A digit is an integer of at most 8 bits, exact in BF16; a product of two
// digits is at most 2^14, and a sum of at most SM_DIG * R such products stays
// below 2^24, so the MMA accumulates it exactly in FP32.  Products of the
// same total weight p + q = L share the scale 2^(e_i + f_c - 7(L+2)), so one
// TMEM accumulator per level L collects all of them exactly:
//   D_L = sum_{p + q = L} Kp(M) Kq(W),   Z = sum_L 2^(e_i + f_c - 7(L+2)) D_L.
// One MMA per digit p of M covers every level it feeds: its B operand is the
// stack of W's digit tiles q = 0 .. LMAX - p (N = (LMAX + 1 - p) R columns)
// and its accumulator starts at level p's columns.  Levels L <= LMAX are kept
// (the dropped ones weigh 2^-49 of level 0); levels LMAX .. 2 are summed in
// FP32 (their weight is at most 2^-14 of level 0, so the rounding of that sum
// is below 2^-36 of the scale below), levels 1 and 0 in double-float with
// exact power-of-two scalings, then the sum is rounded once to FP32.
// The error against exact arithmetic is below 2^-34 of
// max_s |M(i,s)| * sum_s |W(s,c)| -- far under the FP32 rounding of Z.
//
// One CTA of 256 threads per virtual block: threads t and t + 128 own row t
// of each 128-row tile (TMEM lane t), half of its columns each; the tile of M
// comes in by one bulk copy, the
// digits are written to shared memory in the K-major layout of the MMA, one
// thread issues the MMAs and commits them to an mbarrier.  Rows without
// nonzeros (bit clear in `mask`) are not written, as in solve_body.
#pragma once

#include "als_kernels.cuh"
#include "tc_common.cuh"

namespace spm {

constexpr int TC_ROWS = 128;   // rows per tile (TMEM lanes)
constexpr int TC_THREADS = 256;  // two threads per row / lane (warps w and w + 4 share lanes)
constexpr int SM_DIG = 5;      // digits of a row of M  (35 bits)
constexpr int SW_DIG = 7;      // digits of a column of W (49 bits)
constexpr int TC_LMAX = 6;     // highest digit level kept
static_assert(TC_LMAX + 1 == SW_DIG, "W's digit stack covers every kept level");


// Virtual blocks of the row solve over I rows: one tile of the tensor-core
// solve each while the partial buffers last.
inline int solve_blocks(int R, int64_t I, int cap) {
  return tc_solve_rank(R) ? work_blocks(I, TC_ROWS, cap) : als_row_blocks(I, cap);
}

// Shapes of the solve's shared-memory tiles (bytes) for rank R.
template <int R>
struct TcSolveShape {
  static constexpr int KA = SM_DIG * R;        // K of the M-digit tile (digit p at K block p)
  static constexpr int NB = SW_DIG * R;        // rows of the W-digit stack (row q R + c)
  static constexpr int A_BYTES = TC_ROWS * KA * 2;
  static constexpr int B_BYTES = NB * R * 2;   // K = R
  static constexpr int WD_BYTES = B_BYTES + R * 4;  // + the column exponents f_c
  static constexpr int MT_BYTES = TC_ROWS * R * 4;  // one tile of M (FP32)
  static constexpr int ZS_STRIDE = R + 1;           // staged Z row (floats)
  static constexpr int NCOLS_USED = (TC_LMAX + 1) * R;
  static constexpr uint32_t NCOLS = NCOLS_USED <= 32 ? 32 : NCOLS_USED <= 64 ? 64
                                  : NCOLS_USED <= 128 ? 128 : NCOLS_USED <= 256 ? 256 : 512;
  // the staged Z tile reuses the digit tile once the MMAs have read it
  static_assert(TC_ROWS * ZS_STRIDE * 4 <= A_BYTES, "Z staging fits in the digit tile");
  static_assert(WD_BYTES % 16 == 0 && A_BYTES % 16 == 0, "bulk copy sizes");
  static constexpr size_t SMEM = (size_t)A_BYTES + WD_BYTES + 2 * MT_BYTES;
};

// Bytes of the per-mode W digit tile for rank R (0 when R takes no tensor-core solve).
__host__ __device__ constexpr int tc_wdig_bytes(int R) {
  return R == 16 ? TcSolveShape<16>::WD_BYTES
         : R == 32 ? TcSolveShape<32>::WD_BYTES
         : R == 64 ? TcSolveShape<64>::WD_BYTES : 0;
}

static_assert(!SPM_ALS_TC || (tc_wdig_bytes(16) == als_wdig_bytes(16) &&
                              tc_wdig_bytes(32) == als_wdig_bytes(32) &&
                              tc_wdig_bytes(64) == als_wdig_bytes(64)),
              "plan accounting of the W digit tiles");

// 2^k as a float for -126 <= k <= 127 (exact).
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

// Exponent e with |x| < 2^e for the largest |x| seen (float bits; 0 for zero).
__device__ __forceinline__ int scale_expf(float amax) {
  if (!(amax > 0.f)) return 0;
  int e;
  (void)frexpf(amax, &e);  // amax = m 2^e, 0.5 <= m < 1
  return e;
}

// ---- pairs of FP32 values in one instruction (f32x2): the same roundings as
// the scalar operations, half the issue slots, which bound the row passes
// (solve of 567,000 rows of R = 32: 86 -> 73 us, normalisation and Gram 97 ->
// 90 us, on average over the modes of the scale workload; then see
// tc_scale_gram_body's last sums).
__device__ __forceinline__ uint64_t f2_const(float x) { return f2_pack(x, x); }
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {  // a - b, rounded once
  return f2_fma(b, f2_const(-1.f), a);
}
// rint of both for abs <= 2^22 by the 1.5 * 2^23 shift (round half to even, like
// rintf; two adds on the FMA pipe instead of the conversion pipe).
__device__ __forceinline__ uint64_t f2_round_int(uint64_t y) {
  return f2_add(f2_add(y, f2_const(12582912.f)), f2_const(-12582912.f));
}
// Two integer-valued floats of magnitude <= 256 as a BF16 pair (lo = a): their
// low 16 bits are zero, so the BF16 value is the high half, exactly.
__device__ __forceinline__ uint32_t f2_pack_bf16_int(uint64_t k) {
  return __byte_perm((uint32_t)k, (uint32_t)(k >> 32), 0x7632);
}
struct df2 {  // two double-floats
  uint64_t hi, lo;
};
__device__ __forceinline__ void df2_add(df2& a, uint64_t x) {  // a += x (error-free two-sum)
  const uint64_t s = f2_add(a.hi, x);
  const uint64_t bb = f2_sub(s, a.hi);
  const uint64_t err = f2_add(f2_sub(a.hi, f2_sub(s, bb)), f2_sub(x, bb));
  a.hi = s;
  a.lo = f2_add(a.lo, err);
}
__device__ __forceinline__ void df2_add_square(df2& a, uint64_t z) {  // a += z z
  const uint64_t p = f2_mul(z, z);
  const uint64_t e = f2_fma(z, z, f2_mul(p, f2_const(-1.f)));
  const uint64_t s = f2_add(a.hi, p);
  const uint64_t bb = f2_sub(s, a.hi);
  const uint64_t err = f2_add(f2_sub(a.hi, f2_sub(s, bb)), f2_sub(p, bb));
  a.hi = s;
  a.lo = f2_add(a.lo, f2_add(err, e));
}


// ---------------------------------------------------------------------------
// The normal-equation system of one mode and columns of its inverse.
//
// V = the Hadamard product of the Grams of every mode but d (Sec. II-A5), FP64;
// V = L D L^T (L unit lower triangular), X = L^{-1}, W = V^{-1} = X^T D^{-1} X.
// L and X come out of one in-place elimination of the lower triangle T: step j
// takes the pivot d_j = T(j, j) and, for every row i > j with l = T(i, j) / d_j,
//   T(i, k) -= l T(k, j)  (j < k <= i, the Schur complement),
//   T(i, k) -= l T(j, k)  (k < j, rows of X),   T(i, j) = -l,
// so when step j is done row j + 1 holds X(j + 1, :).  A column of W is then
// R dot products: no substitution chains.
//
// Every entry of T lives in a register of the thread that owns it for the whole
// elimination (entry e of the triangle, row-major, belongs to thread e mod 256:
// the entries still active at step j are a contiguous tail, spread evenly over
// the warps), the pivot row and column go through shared memory once per step,
// and one warp forms the reciprocal (in double-float up to R = 32, every thread).
//
// Bound: the chain pivot -> reciprocal -> column -> next pivot, and in FP64 its
// throughput (2 fused multiply-adds per cycle and SM, 64 cycles each).  So the
// elimination and the dot products run in double-float (FP32 pairs, 2^-46) on
// V scaled by powers of two to a diagonal in [1, 4), and each column then takes
// one step of iterative refinement: its residual e_c - V w in FP64 (R^2
// multiply-adds), the correction X^T D^{-1} X r in FP32.  That leaves an error
// no larger than that of an FP64 factorisation while cond(V) is moderate: it is
// taken when every pivot is at least 2^-16 and trace(V^{-1}) of the scaled system
// at most 2^7 + 2 R (systems of the timed decompositions, R = 8 to 64: 5 to 57);
// otherwise the same elimination runs in FP64, which also decides whether V is
// positive definite.  Error of W against extended precision, relative to that of
// an FP64 Cholesky factor with two substitutions (geometric means over nine ranks
// from 3 to 64): cond(V) = 3 .. 300 0.90 - 0.96, 1e3 .. 4e3 0.92 - 0.96, 1e4 ..
// 1e8 0.95 - 1.02.  (With a limit of 2^12 the pairs served conditions up to 1e4,
// at 1.04 - 1.08 from 2e3 on.)  Rows solved with it: tests/test_gpu_system.py and
// tests/test_gpu_system_ranks.py.
// One system, one column per block, alone on the GPU, R = 16 / 32 / 64: 10 /
// 18 / 51 us (the same elimination in FP64 12.3 / 25.6 / 78 us; before it, a
// Cholesky factor and two substitution chains per column, 20 / 46 / 139 us).
// ---------------------------------------------------------------------------
constexpr int SYS_THREADS = 256;
constexpr int SYS_RMAX = 64;
constexpr int SYS_COLS = 8;  // most columns of W per block
constexpr int SYS_TRI = SYS_RMAX * (SYS_RMAX + 1) / 2;

// Shared memory of a system block.
struct SystemSmem {
  union {
    double X[SYS_RMAX * (SYS_RMAX + 1)];  // FP64: X(k, c) at k (R | 1) + c
    struct {                              // pairs: lower triangles, entry i (i + 1) / 2 + k
      double A[SYS_TRI];                  // V scaled
      float2 XF[SYS_TRI];                 // X as (hi, lo)
    };
  };
  double W[SYS_COLS * SYS_RMAX];          // per column c: D^{-1} X(:, c) (FP64), then W(:, c)
  union {
    float2 y[SYS_COLS * SYS_RMAX];        // pairs: D^{-1} X(:, c)
    float ru[2][SYS_COLS * SYS_RMAX];     // then the residual and D^{-1} X r
  };
  union {                                 // step j: T(k, j) for k >= j, X(j, k) for k < j
    double piv[2][SYS_RMAX];
    float2 pivf[2][SYS_RMAX];
  };
  union {                                 // step j: -T(i, j) / d_j for i > j
    double nl[SYS_RMAX];
    float2 nlf[SYS_RMAX];
  };
  union {                                 // 1 / d_k
    double rd[SYS_RMAX];
    float2 rdf[SYS_RMAX];
  };
  int ex[SYS_RMAX];                       // row i of V is scaled by 2^-ex[i]
  float red[SYS_THREADS / 32];
  int bad;
};

// 2^k as a double for -1022 <= k <= 1023 (exact), else via scalbn.
__device__ __forceinline__ double times_pow2(double x, int k) {
  if (k >= -1022 && k <= 1023) return __dmul_rn(x, __longlong_as_double((long long)(k + 1023) << 52));
  return scalbn(x, k);
}

// Reciprocal of a positive finite d in pieces that keep the chain behind it
// short: d = m 2^(ex - 1023) with 1 <= m < 2, r0 = the FP32 reciprocal of m
// (e = 1 - m r0 is below 2^-22) and the cubic Newton factor 1 + e + e^2, whose
// error is e^3; x / d = (x r0 s) (1 + t) with t = e + e^2, s = 2^(1023 - ex).
// Exponents at the ends of the range take the division.
struct RecipPos {
  double r0, t;  // 1 / d = r0 (1 + t)
};
__device__ __forceinline__ RecipPos recip_pos(double d) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  const int ex = hi >> 20;  // biased exponent
  if (ex < 64 || ex > 1982) return {1.0 / d, 0.0};
  const int mant = hi & 0xfffff;
  float rf;  // in [0.5, 1]; widened by its bits below
  asm("rcp.approx.ftz.f32 %0, %1;"
      : "=f"(rf)
      : "f"(__int_as_float(0x3f800000 | (mant << 3) | (int)((unsigned)lo >> 29))));
  const int rb = __float_as_int(rf);
  const int rh = (rb >> 3) + ((1023 - 127) << 20), rl = rb << 29;
  const double e = fma(-__hiloint2double(mant | 0x3ff00000, lo), __hiloint2double(rh, rl), 1.0);
  return {__hiloint2double(rh + ((1023 - ex) << 20), rl), fma(e, e, e)};
}

// W(:, c0 .. c0 + nc - 1) out of shared memory: w = W(:, c) goes to winv as FP32
// (hi, lo) pairs (W(s, c) at s R + c and R R + s R + c), or, when wdig is
// non-null, into the digit tile of the tensor-core solve: w is scaled by 2^-f_c
// (|w_s| < 2^f_c), rounded to 49 fractional bits and recoded from the least
// significant end into SW_DIG balanced 7-bit digits (|k_q| <= 64 below the
// leading digit, |k_0| <= 128), w_s 2^-f_c ~ sum_q k_q 2^{-7(q+1)}; digit q of
// w_s goes to row q R + c, column s of a K-major (K = R) BF16 tile, f_c to the
// int array after it.
__device__ __forceinline__ void system_store(const SystemSmem& sm, int R, int c0, int nc,
                                             float* __restrict__ winv,
                                             unsigned char* __restrict__ wdig) {
  const int t = threadIdx.x, RR = R * R;
  const int l = t & 31;
  for (int cc = t >> 5; cc < nc; cc += SYS_THREADS / 32) {
    const int c = c0 + cc;
    int fx = INT_MIN;  // exponent bound of the column
    for (int h = 0; h < 2; ++h) {
      const int s = l + 32 * h;
      if (s >= R) continue;
      const double w = sm.W[cc * SYS_RMAX + s];
      if (!wdig) {
        const float hi = (float)w;
        winv[s * R + c] = hi;
        winv[RR + s * R + c] = (float)__dsub_rn(w, (double)hi);
      }
      const unsigned long long bits = __double_as_longlong(w) & 0x7FFFFFFFFFFFFFFFull;
      if (bits != 0) {
        const int be = (int)(bits >> 52);
        fx = max(fx, be == 0 ? -1021 : be - 1022);  // |w| < 2^(be - 1022)
      }
    }
    if (!wdig) continue;
    fx = __reduce_max_sync(SPM_FULL_MASK, fx);
    if (fx == INT_MIN) fx = 0;
    if (l == 0) reinterpret_cast<int*>(wdig + SW_DIG * RR * 2)[c] = fx;
    for (int h = 0; h < 2; ++h) {
      const int s = l + 32 * h;
      if (s >= R) continue;
      long long n = __double2ll_rn(times_pow2(sm.W[cc * SYS_RMAX + s], 49 - fx));  // |n| <= 2^49
#pragma unroll
      for (int q = SW_DIG - 1; q >= 0; --q) {
        long long dg = n;
        if (q > 0) {
          dg = ((n + 64) & 127) - 64;  // balanced remainder mod 128
          n = (n - dg) >> 7;           // exact
        }
        *reinterpret_cast<__nv_bfloat16*>(wdig + tc::kmajor_offset(q * R + c, s, R)) =
            __float2bfloat16_rn((float)(int)dg);
      }
    }
  }
}

// Columns c0 .. c1-1 (at most SYS_COLS) of W by one block of SYS_THREADS
// threads; NS >= R (R + 1) / 2 / SYS_THREADS entries of T per thread.  Every
// block that takes columns of the same system computes the same L and X, and
// an entry of W does not depend on which block or thread forms it, so any
// split of the columns gives the same bits.
// A pivot that is not positive and finite sets DEV_ERR_NUMERIC.
template <int NS>
__device__ __forceinline__ void system_body_ns(SystemSmem& sm, const double* __restrict__ grams,
                                               int N, int d, int R, int c0, int c1,
                                               float* __restrict__ winv,
                                               unsigned char* __restrict__ wdig,
                                               int* __restrict__ err) {
  const int t = threadIdx.x;
  if (t == 0) sm.bad = *(volatile int*)err ? 1 : 0;
  __syncthreads();
  if (sm.bad) return;
  const int RR = R * R, T = R * (R + 1) / 2;
  int ei[NS], ek[NS], last[NS];  // row, column, last row of the warp's entries
  double v[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    const int e = q * SYS_THREADS + t;  // e = i (i + 1) / 2 + k, k <= i
    int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while (i * (i + 1) / 2 > e) --i;
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    ei[q] = e < T ? i : -1;
    ek[q] = e < T ? e - i * (i + 1) / 2 : 0;
    last[q] = __reduce_max_sync(SPM_FULL_MASK, ei[q]);
    v[q] = 1.0;
  }
  const int w0 = d == 0 ? 1 : 0;  // the first mode of the product (none: V = 1)
  for (int w = w0; w < N; ++w)
    if (w != d) {
      double g[NS];
#pragma unroll
      for (int q = 0; q < NS; ++q)
        g[q] = ei[q] >= 0 ? grams[(int64_t)w * RR + ei[q] * R + ek[q]] : 0.0;
#pragma unroll
      for (int q = 0; q < NS; ++q) v[q] = w == w0 ? g[q] : __dmul_rn(v[q], g[q]);
    }
  for (int j = 0; j < R; ++j) {
    const int b = j & 1;
#pragma unroll
    for (int q = 0; q < NS; ++q)
      if (ei[q] >= j && (ek[q] == j || ei[q] == j)) sm.piv[b][ek[q] == j ? ei[q] : ek[q]] = v[q];
    __syncthreads();
    if (t < 32) {
      const double piv = sm.piv[b][j];
      const int hi = __double2hiint(piv);
      // positive and finite, by its bits
      const bool good = hi >= 0 && hi < 0x7ff00000 && (hi | __double2loint(piv)) != 0;
      const RecipPos r = good ? recip_pos(piv) : RecipPos{0.0, 0.0};
      for (int i = j + 1 + t; i < R; i += 32) {
        const double x = __dmul_rn(sm.piv[b][i], -r.r0);
        sm.nl[i] = fma(x, r.t, x);
      }
      if (t == 0) {
        sm.rd[j] = fma(r.r0, r.t, r.r0);
        if (!good) sm.bad = 1;
      }
    }
    __syncthreads();
    if (sm.bad) break;
    // Operands of every slot first (rows up to j: a zero multiplier; column j:
    // -l = fma(-l, 1, 0)), then the multiply-adds of the slots that hold a row
    // beyond j anywhere in the warp: no divergent branch, no slot waits for
    // the one before it.
    double l[NS], pv[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      l[q] = ei[q] > j ? sm.nl[ei[q]] : 0.0;
      pv[q] = ek[q] == j ? 1.0 : sm.piv[b][ek[q]];
      if (ei[q] > j && ek[q] == j) v[q] = 0.0;
    }
#pragma unroll
    for (int q = 0; q < NS; ++q)
      if (last[q] > j) v[q] = fma(l[q], pv[q], v[q]);
  }
  if (sm.bad) {
    if (t == 0) atomicOr(err, DEV_ERR_NUMERIC);
    return;
  }
  const int LD = R | 1;
#pragma unroll
  for (int q = 0; q < NS; ++q)
    if (ei[q] >= 0) sm.X[ei[q] * LD + ek[q]] = ei[q] == ek[q] ? 1.0 : v[q];
  __syncthreads();
  const int nc = c1 - c0;
  for (int x = t; x < nc * R; x += SYS_THREADS) {
    const int cc = x / R, k = x - cc * R;
    sm.W[cc * SYS_RMAX + k] = k >= c0 + cc ? __dmul_rn(sm.X[k * LD + c0 + cc], sm.rd[k]) : 0.0;
  }
  __syncthreads();
  // W(s, c) = sum over k >= max(s, c) of X(k, s) X(k, c) / d_k: four threads
  // per entry (k mod 4), added by shuffles
  constexpr int NW = SYS_COLS * SYS_RMAX * 4 / SYS_THREADS;  // rounds at most
  double wv[NW];
#pragma unroll
  for (int p = 0; p < NW; ++p) {
    const int x = p * (SYS_THREADS / 4) + (t >> 2);
    if (p * (SYS_THREADS / 4) >= nc * R) break;
    double a = 0.0;
    if (x < nc * R) {
      const int cc = x / R, s = x - cc * R;
      for (int k = (max(s, c0 + cc) & ~3) + (t & 3); k < R; k += 4)
        if (k >= s) a = fma(sm.X[k * LD + s], sm.W[cc * SYS_RMAX + k], a);
    }
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 1);
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 2);
    wv[p] = a;
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < NW; ++p) {
    const int x = p * (SYS_THREADS / 4) + (t >> 2);
    if (x < nc * R && (t & 3) == 0) sm.W[(x / R) * SYS_RMAX + x % R] = wv[p];
  }
  __syncthreads();
  system_store(sm, R, c0, nc, winv, wdig);
}

// ---- the same in double-float with refinement ----
__device__ __forceinline__ float2 ff_norm(float h, float l) {  // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return make_float2(s, __fsub_rn(l, __fsub_rn(s, h)));
}
__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  return ff_norm(p, e);
}
__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float bb = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(b.x, bb));
  return ff_norm(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 ff_fma(float2 a, float2 b, float2 c) {  // a b + c
  const float p = __fmul_rn(a.x, b.x);
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  const float s = __fadd_rn(c.x, p);
  const float bb = __fsub_rn(s, c.x);
  const float t = __fadd_rn(__fsub_rn(c.x, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  return ff_norm(s, __fadd_rn(t, __fadd_rn(c.y, e)));
}

// Columns c0 .. c1-1 of W; false (nothing written) when V is not well enough
// conditioned for it.  Every block of a system takes the same decision.
template <int NS>
__device__ __forceinline__ bool system_pairs_ns(SystemSmem& sm, const double* __restrict__ grams,
                                                int N, int d, int R, int c0, int c1,
                                                float* __restrict__ winv,
                                                unsigned char* __restrict__ wdig) {
  constexpr int QG = NS % 3 == 0 ? 3 : 1;
  // Up to three slots every thread forms the reciprocal and its rows'
  // multipliers: one barrier per step, no wait for a warp (R = 16 / 32: 11.1 /
  // 21.9 -> 9.7 / 21.1 us from cold caches).  With nine slots the extra issue
  // costs more (R = 64: 63.5 -> 69 us).
  constexpr bool OWN = NS <= 3;
  const int t = threadIdx.x, lane = t & 31;
  const int RR = R * R, T = R * (R + 1) / 2;
  int ei[NS], ek[NS], last[NS];  // last: the warp's entries' last row, so far
  float2 v[NS];
  if (t == 0) sm.bad = 0;
  {
    double a[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      const int e = q * SYS_THREADS + t;  // e = i (i + 1) / 2 + k, k <= i
      int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while (i * (i + 1) / 2 > e) --i;
      while ((i + 1) * (i + 2) / 2 <= e) ++i;
      ei[q] = e < T ? i : -1;
      ek[q] = e < T ? e - i * (i + 1) / 2 : 0;
      last[q] = __reduce_max_sync(SPM_FULL_MASK, ei[q]);
      if (q > 0) last[q] = max(last[q], last[q - 1]);  // past the triangle
      a[q] = 1.0;
    }
    const int w0 = d == 0 ? 1 : 0;  // the first mode of the product (none: V = 1)
    for (int w = w0; w < N; ++w)
      if (w != d) {
        double g[NS];
#pragma unroll
        for (int q = 0; q < NS; ++q)
          g[q] = ei[q] >= 0 ? grams[(int64_t)w * RR + ei[q] * R + ek[q]] : 0.0;
#pragma unroll
        for (int q = 0; q < NS; ++q) a[q] = w == w0 ? g[q] : __dmul_rn(a[q], g[q]);
      }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NS; ++q)
      if (ei[q] >= 0 && ei[q] == ek[q]) {
        const int hi = __double2hiint(a[q]);
        const int ex = (hi >> 20) - 1023;
        if (hi < 0 || ex < -900 || ex > 900) sm.bad = 1;
        sm.ex[ei[q]] = ex >> 1;
      }
    __syncthreads();
    if (sm.bad) return false;
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      v[q] = make_float2(0.f, 0.f);
      if (ei[q] >= 0) {
        const double x = times_pow2(a[q], -(sm.ex[ei[q]] + sm.ex[ek[q]]));
        sm.A[q * SYS_THREADS + t] = x;
        v[q].x = (float)x;
        v[q].y = (float)__dsub_rn(x, (double)v[q].x);
      }
    }
  }
  for (int j = 0; j < R; ++j) {
    const int b = j & 1;
#pragma unroll
    for (int q = 0; q < NS; ++q)
      if (ei[q] >= j && (ek[q] == j || ei[q] == j)) sm.pivf[b][ek[q] == j ? ei[q] : ek[q]] = v[q];
    __syncthreads();  // the buffers alternate
    float2 nr = make_float2(0.f, 0.f);
    if (OWN || t < 32) {
      const float2 p = sm.pivf[b][j];
      const bool good = p.x >= 1.52587890625e-5f && p.x <= 16.f;  // 2^-16; false for NaN
      if (OWN && !good) return false;
      float r0;
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(good ? p.x : 1.f));
      float e = fmaf(-p.x, r0, 1.f);
      e = fmaf(-p.y, r0, e);
      const float2 r = ff_norm(r0, __fmul_rn(r0, fmaf(e, e, e)));
      nr = make_float2(-r.x, -r.y);
      if (!OWN)
        for (int i = j + 1 + t; i < R; i += 32) sm.nlf[i] = ff_mul(sm.pivf[b][i], nr);
      if (t == 0) {
        sm.rdf[j] = r;
        if (!good) sm.bad = 1;
      }
    }
    if (!OWN) {
      __syncthreads();
      if (sm.bad) break;
    }
    // Three slots at a time while the warp has a row beyond j in them; rows up
    // to j: a zero multiplier; column j: -l = fma(-l, 1, 0).
#pragma unroll
    for (int q0 = 0; q0 < NS; q0 += QG) {
      if (last[q0 + QG - 1] <= j) continue;
      float2 l[QG], pv[QG];
#pragma unroll
      for (int u = 0; u < QG; ++u) {
        const int q = q0 + u;
        const float2 z = make_float2(0.f, 0.f);
        l[u] = ei[q] <= j ? z : OWN ? ff_mul(sm.pivf[b][ei[q]], nr) : sm.nlf[ei[q]];
        pv[u] = ek[q] == j ? make_float2(1.f, 0.f) : sm.pivf[b][ek[q]];
        if (ei[q] > j && ek[q] == j) v[q] = z;
      }
#pragma unroll
      for (int u = 0; u < QG; ++u) v[q0 + u] = ff_fma(l[u], pv[u], v[q0 + u]);
    }
  }
  if (OWN) __syncthreads();  // the last 1 / d_k
  if (sm.bad) return false;
  // X, and trace(W) = sum of X(k, c)^2 / d_k, summed in a fixed order
  float tr = 0.f;
#pragma unroll
  for (int q = 0; q < NS; ++q)
    if (ei[q] >= 0) {
      const float2 x = ei[q] == ek[q] ? make_float2(1.f, 0.f) : v[q];
      sm.XF[q * SYS_THREADS + t] = x;
      tr = fmaf(__fmul_rn(x.x, x.x), sm.rdf[ei[q]].x, tr);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(SPM_FULL_MASK, tr, o);
  if (lane == 0) sm.red[t >> 5] = tr;
  __syncthreads();
  float trace = 0.f;
#pragma unroll
  for (int w = 0; w < SYS_THREADS / 32; ++w) trace += sm.red[w];
  if (!(trace <= (float)(128 + 2 * R))) return false;
  auto X = [&](int k, int c) -> float2 { return sm.XF[k * (k + 1) / 2 + c]; };
  const int nc = c1 - c0;
  const unsigned rinv = (65535u + R) / R;  // x / R = x rinv >> 16 for x < 1024
  for (int x = t; x < nc * R; x += SYS_THREADS) {
    const int cc = (int)((unsigned)x * rinv >> 16), k = x - cc * R;
    sm.y[cc * SYS_RMAX + k] = k >= c0 + cc ? ff_mul(X(k, c0 + cc), sm.rdf[k]) : make_float2(0.f, 0.f);
  }
  __syncthreads();
  // every sum below: four threads per entry (index mod 4), added by shuffles
  const int sub = t & 3, ntask = nc * R, step = SYS_THREADS / 4;
  // w = X^T (D^{-1} X(:, c))
  for (int x0 = 0; x0 < ntask; x0 += step) {
    const int x = x0 + (t >> 2);
    float2 a = make_float2(0.f, 0.f);
    int cc = 0, s = 0;
    if (x < ntask) {
      cc = (int)((unsigned)x * rinv >> 16);
      s = x - cc * R;
      for (int k = (max(s, c0 + cc) & ~3) + sub; k < R; k += 4)
        if (k >= s) a = ff_fma(X(k, s), sm.y[cc * SYS_RMAX + k], a);
    }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1)
      a = ff_add(a, make_float2(__shfl_xor_sync(SPM_FULL_MASK, a.x, o),
                                __shfl_xor_sync(SPM_FULL_MASK, a.y, o)));
    if (x < ntask && sub == 0) sm.W[cc * SYS_RMAX + s] = __dadd_rn((double)a.x, (double)a.y);
  }
  __syncthreads();
  // r = e_c - V w in FP64
  for (int x0 = 0; x0 < ntask; x0 += step) {
    const int x = x0 + (t >> 2);
    double a = 0.0;
    int cc = 0, i = 0;
    if (x < ntask) {
      cc = (int)((unsigned)x * rinv >> 16);
      i = x - cc * R;
      if (sub == 0 && i == c0 + cc) a = -1.0;
      for (int k = sub; k < R; k += 4)
        a = fma(k <= i ? sm.A[i * (i + 1) / 2 + k] : sm.A[k * (k + 1) / 2 + i],
                sm.W[cc * SYS_RMAX + k], a);
    }
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 1);
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 2);
    if (x < ntask && sub == 0) sm.ru[0][cc * SYS_RMAX + i] = -(float)a;
  }
  __syncthreads();
  // D^{-1} X r
  for (int x0 = 0; x0 < ntask; x0 += step) {
    const int x = x0 + (t >> 2);
    float a = 0.f;
    int cc = 0, k = 0;
    if (x < ntask) {
      cc = (int)((unsigned)x * rinv >> 16);
      k = x - cc * R;
      for (int i = sub; i <= k; i += 4) a = fmaf(X(k, i).x, sm.ru[0][cc * SYS_RMAX + i], a);
    }
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 1);
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 2);
    if (x < ntask && sub == 0) sm.ru[1][cc * SYS_RMAX + k] = __fmul_rn(a, sm.rdf[k].x);
  }
  __syncthreads();
  // w += X^T of that; the scaling undone
  for (int x0 = 0; x0 < ntask; x0 += step) {
    const int x = x0 + (t >> 2);
    float a = 0.f;
    int cc = 0, s = 0;
    if (x < ntask) {
      cc = (int)((unsigned)x * rinv >> 16);
      s = x - cc * R;
      for (int k = (s & ~3) + sub; k < R; k += 4)
        if (k >= s) a = fmaf(X(k, s).x, sm.ru[1][cc * SYS_RMAX + k], a);
    }
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 1);
    a += __shfl_xor_sync(SPM_FULL_MASK, a, 2);
    if (x < ntask && sub == 0)
      sm.W[cc * SYS_RMAX + s] = times_pow2(__dadd_rn(sm.W[cc * SYS_RMAX + s], (double)a),
                                           -(sm.ex[s] + sm.ex[c0 + cc]));
  }
  __syncthreads();
  system_store(sm, R, c0, nc, winv, wdig);
  return true;
}

template <int NS>
__device__ __forceinline__ void system_body_n(SystemSmem& sm, const double* __restrict__ grams, int N,
                                              int d, int R, int c0, int c1, float* __restrict__ winv,
                                              unsigned char* __restrict__ wdig,
                                              int* __restrict__ err) {
  if (__syncthreads_or(threadIdx.x == 0 && *(volatile int*)err)) return;
  if (system_pairs_ns<NS>(sm, grams, N, d, R, c0, c1, winv, wdig)) return;
  __syncthreads();  // shared memory is reused
  system_body_ns<NS>(sm, grams, N, d, R, c0, c1, winv, wdig, err);
}

__device__ __forceinline__ void system_body(SystemSmem& sm, const double* __restrict__ grams, int N,
                                            int d, int R, int c0, int c1, float* __restrict__ winv,
                                            unsigned char* __restrict__ wdig,
                                            int* __restrict__ err) {
  if (R <= 16) system_body_n<1>(sm, grams, N, d, R, c0, c1, winv, wdig, err);
  else if (R <= 32) system_body_n<3>(sm, grams, N, d, R, c0, c1, winv, wdig, err);
  else system_body_n<9>(sm, grams, N, d, R, c0, c1, winv, wdig, err);
}

// Z = M W for rows tile vb, vb + nvb, ... (see the head of this file), with
// the column sums of Z^2 and the column maxima of |Z| of those rows into
// colsq_part / colmax_part (block vb's slots).  `wdig` is the mode's W digit
// tile (system_body).
template <int R>
__device__ __forceinline__ void tc_solve_body(const float* __restrict__ M,
                                              const unsigned char* __restrict__ wdig, int64_t I,
                                              float* __restrict__ Z, double* __restrict__ colsq_part,
                                              float* __restrict__ colmax_part,
                                              const int* __restrict__ err, int vb, int nvb,
                                              const uint32_t* __restrict__ mask) {
  using S = TcSolveShape<R>;
  extern __shared__ __align__(1024) unsigned char smem_tc[];
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t bars[4];  // [0]: MMAs done; [1], [2]: M tiles; [3]: W digits
  __shared__ double red[TC_THREADS];
  __shared__ float redm[TC_THREADS];
  __shared__ float amax_s[2][TC_ROWS];
  if (*(volatile const int*)err) return;
  constexpr int H = R / 2;  // columns per thread

  unsigned char* sA = smem_tc;
  unsigned char* sB = sA + S::A_BYTES;
  const int* fexp = reinterpret_cast<const int*>(sB + S::B_BYTES);
  float* sM = reinterpret_cast<float*>(sB + S::WD_BYTES);  // 2 stages
  float* sZ = reinterpret_cast<float*>(sA);                // after the MMAs of a tile
  const int t = threadIdx.x;
  const int warp = t >> 5;
  const int rl = t & (TC_ROWS - 1), half = t / TC_ROWS;  // row of the tile, column half
  const int64_t ntiles = (I + TC_ROWS - 1) / TC_ROWS;

  if (warp == 0) tc::tmem_alloc(&tmem_slot, S::NCOLS);
  if (t == 0) {
    for (int b = 0; b < 4; ++b) mbar_init(&bars[b], 1);
    fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;

  // bulk copy of tile `tile` of M into stage `st` (thread 0)
  auto fetch = [&](int64_t tile, int st) {
    fence_proxy_async_smem();  // the stage's earlier reads before the copy's writes
    const int64_t r0 = tile * TC_ROWS;
    const int64_t rows = I - r0 < TC_ROWS ? I - r0 : TC_ROWS;
    const uint32_t bytes = (uint32_t)(rows * R * 4);
    mbar_arrive_expect_tx(&bars[1 + st], bytes);
    bulk_g2s(sM + st * TC_ROWS * R, M + r0 * R, bytes, &bars[1 + st]);
  };
  bool ok = true;
  int fetched = 0;  // tiles whose copies were issued (thread 0's count)
  int mmas = 0;     // tiles whose MMAs were committed
  if (t == 0) {
    mbar_arrive_expect_tx(&bars[3], S::WD_BYTES);
    bulk_g2s(sB, wdig, S::WD_BYTES, &bars[3]);
    if (vb < ntiles) { fetch(vb, 0); fetched = 1; }
  }
  ok = mbar_wait_bounded(&bars[3], 0u);
  df2 sq = {0ull, 0ull};  // column (t % R) sums of Z^2 over this block's rows, two at a time
  float mx = 0.f;      // and max |Z|
  int it = 0;
  if (__syncthreads_and(ok))
    for (int64_t tile = vb; tile < ntiles && ok; tile += nvb, ++it) {
      const int st = it & 1;
      if (t == 0 && tile + nvb < ntiles) { fetch(tile + nvb, st ^ 1); ++fetched; }  // prefetch
      ok = mbar_wait_bounded(&bars[1 + st], (uint32_t)((it >> 1) & 1));
      if (!__syncthreads_and(ok)) break;
      const int64_t row = tile * TC_ROWS + rl;
      const bool in = row < I;
      // this thread's half of row rl of the staged tile, read in a per-row
      // rotation of its 16-byte chunks (rows are 4R bytes apart: unrotated,
      // a warp's reads would share banks)
      const float* mr = sM + st * TC_ROWS * R + rl * R + half * H;
      float amax = 0.f;
      if (in)
#pragma unroll
        for (int c = 0; c < H / 4; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(mr + ((c + rl) % (H / 4)) * 4);
          amax = fmaxf(amax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
        }
      amax_s[half][rl] = amax;
      __syncthreads();
      amax = fmaxf(amax_s[0][rl], amax_s[1][rl]);
      const int e_row = scale_expf(amax);  // |M(row, s)| < 2^e_row
      const bool fast = e_row >= -125 && e_row <= 126;
      const float inv = fast ? pow2f(-e_row) : 1.f;
#pragma unroll
      for (int g = 0; g < H / 8; ++g) {
        const int gg = (g + rl) % (H / 8);
        uint64_t x[4];
        if (in) {
          const float4 a = *reinterpret_cast<const float4*>(mr + gg * 8);
          const float4 b = *reinterpret_cast<const float4*>(mr + gg * 8 + 4);
          if (fast) {
            const uint64_t iv = f2_const(inv);
            x[0] = f2_mul(f2_pack(a.x, a.y), iv);
            x[1] = f2_mul(f2_pack(a.z, a.w), iv);
            x[2] = f2_mul(f2_pack(b.x, b.y), iv);
            x[3] = f2_mul(f2_pack(b.z, b.w), iv);
          } else {
            x[0] = f2_pack(ldexpf(a.x, -e_row), ldexpf(a.y, -e_row));
            x[1] = f2_pack(ldexpf(a.z, -e_row), ldexpf(a.w, -e_row));
            x[2] = f2_pack(ldexpf(b.x, -e_row), ldexpf(b.y, -e_row));
            x[3] = f2_pack(ldexpf(b.z, -e_row), ldexpf(b.w, -e_row));
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = 0ull;
        }
        // digit p of each value: rint of the remainder scaled by 2^7 (exact steps)
#pragma unroll
        for (int p = 0; p < SM_DIG; ++p) {
          uint32_t k[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint64_t y = f2_mul(x[j], f2_const(128.f));
            const uint64_t kk = f2_round_int(y);
            x[j] = f2_sub(y, kk);
            k[j] = f2_pack_bf16_int(kk);
          }
          *reinterpret_cast<uint4*>(sA + tc::kmajor_offset(rl, p * R + half * H + gg * 8, S::KA)) =
              make_uint4(k[0], k[1], k[2], k[3]);
        }
      }
      fence_proxy_async_smem();  // digits visible to the tensor core
      tc::fence_before_sync();
      __syncthreads();
      tc::fence_after_sync();
      if (t == 0) {
        // digit p of M against W's digits q = 0 .. LMAX - p, into levels p ..
        // LMAX (columns p R ..), N split in pieces of at most 256 columns
        for (int p = 0; p < SM_DIG; ++p) {
          const int nq = TC_LMAX + 1 - p;
#pragma unroll
          for (int k16 = 0; k16 < R; k16 += 16) {
            const uint64_t da = tc::smem_desc(smem_addr(sA) + ((p * R + k16) / 8) * 128, 128,
                                              (S::KA / 8) * 128);
            for (int q0 = 0; q0 < nq; q0 += 256 / R) {
              const int n = (nq - q0 < 256 / R ? nq - q0 : 256 / R) * R;
              const uint64_t db = tc::smem_desc(
                  smem_addr(sB) + (q0 * R / 8) * (R / 8) * 128 + (k16 / 8) * 128, 128, (R / 8) * 128);
              tc::mma_bf16(tmem + (uint32_t)((p + q0) * R), da, db, tc::idesc_bf16(TC_ROWS, n),
                           p > 0 || k16 > 0);
            }
          }
        }
        tc::commit(&bars[0]);
      }
      ++mmas;
      ok = mbar_wait_bounded(&bars[0], (uint32_t)(it & 1));
      tc::fence_after_sync();
      if (!__syncthreads_and(ok)) break;
      // Z(row, c) from the levels: LMAX .. 2 in FP32 (Horner), 1 and 0 in
      // double-float, then the scale 2^(e_row + f_c - 14) of level 0
      const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
      for (int c0 = half * H; c0 < half * H + H; c0 += 8) {
        uint32_t v[TC_LMAX + 1][8];
#pragma unroll
        for (int L = 0; L <= TC_LMAX; ++L) tc::ld8(lane_addr + (uint32_t)(L * R + c0), v[L]);
        tc::wait_ld();
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
          auto lev = [&](int L) -> uint64_t {
            return f2_pack(__uint_as_float(v[L][j]), __uint_as_float(v[L][j + 1]));
          };
          const uint64_t w7 = f2_const(0.0078125f);
          uint64_t h = lev(TC_LMAX);
#pragma unroll
          for (int L = TC_LMAX - 1; L >= 2; --L) h = f2_fma(h, w7, lev(L));
          df2 z = {lev(1), 0ull};
          df2_add(z, f2_mul(h, w7));
          z.hi = f2_mul(z.hi, w7);
          z.lo = f2_mul(z.lo, w7);
          df2_add(z, lev(0));
          const int k0 = e_row + fexp[c0 + j] - 14, k1 = e_row + fexp[c0 + j + 1] - 14;
          float z0, z1;
          if (min(k0, k1) >= -126 && max(k0, k1) <= 127) {
            const uint64_t sc = f2_pack(pow2f(k0), pow2f(k1));
            f2_unpack(f2_add(f2_mul(z.hi, sc), f2_mul(z.lo, sc)), z0, z1);
          } else {
            float h0, h1, l0, l1;
            f2_unpack(z.hi, h0, h1);
            f2_unpack(z.lo, l0, l1);
            z0 = __fadd_rn(ldexpf(h0, k0), ldexpf(l0, k0));
            z1 = __fadd_rn(ldexpf(h1, k1), ldexpf(l1, k1));
          }
          sZ[rl * S::ZS_STRIDE + c0 + j] = z0;
          sZ[rl * S::ZS_STRIDE + c0 + j + 1] = z1;
        }
      }
      tc::fence_before_sync();
      __syncthreads();
      // column sums of Z^2 and maxima of |Z| (fixed order), and the tile of Z
      // out (rows with nonzeros only)
      {
        constexpr int PER = TC_THREADS / R;  // threads per column
        static_assert(TC_ROWS % (2 * PER) == 0, "rows in pairs");
        const int c = t % R, g = t / R;
#pragma unroll 4
        for (int rr = g; rr < TC_ROWS; rr += 2 * PER) {
          const float za = sZ[rr * S::ZS_STRIDE + c], zb = sZ[(rr + PER) * S::ZS_STRIDE + c];
          df2_add_square(sq, f2_pack(za, zb));
          mx = fmaxf(mx, fmaxf(fabsf(za), fabsf(zb)));
        }
      }
      for (int x = t; x < TC_ROWS * R / 4; x += TC_THREADS) {
        const int rr = x / (R / 4), c4 = (x % (R / 4)) * 4;
        const int64_t gr = tile * TC_ROWS + rr;
        if (gr < I && row_live(mask, gr)) {
          const float* zs = sZ + rr * S::ZS_STRIDE + c4;
          *reinterpret_cast<float4*>(Z + gr * R + c4) = make_float4(zs[0], zs[1], zs[2], zs[3]);
        }
      }
      __syncthreads();  // sZ and the stage are reused by the next tile
    }
  if (!ok) {
    // a wait gave up: let the copies and MMAs still in flight finish before
    // tensor memory is released and the block exits
    if (t == 0) {
      (void)mbar_wait_bounded(&bars[3], 0u, 1u << 20);
      for (int k = it; k < fetched; ++k)
        (void)mbar_wait_bounded(&bars[1 + (k & 1)], (uint32_t)((k >> 1) & 1), 1u << 20);
      if (mmas > 0) (void)mbar_wait_bounded(&bars[0], (uint32_t)((mmas - 1) & 1), 1u << 20);
      atomicOr(const_cast<int*>(err), DEV_ERR_TIMEOUT);
    }
    __syncthreads();
  }
  {
    df sa, sb;
    f2_unpack(sq.hi, sa.hi, sb.hi);
    f2_unpack(sq.lo, sa.lo, sb.lo);
    red[t] = __dadd_rn(df_value(sa), df_value(sb));
  }
  redm[t] = mx;
  tc::fence_before_sync();
  __syncthreads();
  if (t < R) {
    double s = 0.0;
    float m = 0.f;
    for (int g = 0; g < TC_THREADS / R; ++g) {
      s += red[g * R + t];
      m = fmaxf(m, redm[g * R + t]);
    }
    colsq_part[(int64_t)vb * R + t] = s;
    if (colmax_part) colmax_part[(int64_t)vb * R + t] = m;
  }
  if (warp == 0) tc::tmem_dealloc(tmem, S::NCOLS);
  if (t == 0 && ok)
    for (int b = 0; b < 4; ++b) mbar_inval(&bars[b]);
}

// ---------------------------------------------------------------------------
// Normalisation and Gram of the new factor on the tensor cores (R = 16, 32):
// Y = Z / lambda (stored type FT), G = Y^T Y from the STORED Y, and (last mode
// of a sweep) the column sums of M .* Y.
//
// Column r of Y is scaled by 2^-g_r (|Y(i, r)| < 2^(g_r - 1) for every row,
// from the column maxima of |Z| and lambda) and cut into NDIG = 128 / R
// balanced integer digits of 7 bits, Y(i, r) 2^-g_r ~ sum_p k_p 2^{-7(p+1)},
// |k_p| <= 64.  Digit p of column r is row m = p R + r of a 128 x 128 BF16
// tile A whose K index is the row of Y within a 128-row tile; one MMA chain
// D += A A^T per tile sums, for every pair of digit rows (p, r), (q, s),
//   D(pR + r, qR + s) = sum_i k_p(i, r) k_q(i, s)
// exactly in FP32 (products <= 2^12, at most GT_FLUSH * 128 rows between
// reads: sums < 2^22).  Every GT_FLUSH tiles the accumulator is read and
// folded into double-float sums acc_{p,r}(s) += sum_q 2^-7q D(pR+r, qR+s);
// at the end G(r, s) = 2^(g_r + g_s - 14) sum_p 2^-7p acc_{p,r}(s).  With
// NDIG >= 4 digits (>= 29 bits below the column maximum) the stored FP32
// values within 2^-5 of their column's maximum are represented exactly and
// the others to 2^-29 of it: the Gram error is far below the FP32 rounding
// of the factor itself.
// ---------------------------------------------------------------------------
constexpr int GT_ROWS = 128;    // rows of Y per tile (K of the MMAs)
constexpr int GT_STAGES = 2;    // Z tiles in flight (two blocks fit an SM)
constexpr int GT_FLUSH = 8;     // tiles between accumulator reads (1024 rows)

__host__ __device__ constexpr bool tc_gram_rank(int R) { return tc_solve_rank(R) && R <= 32; }

template <int R>
struct TcGramShape {
  static constexpr int NDIG = 128 / R;
  static constexpr int NQ = TC_THREADS / R;          // row slices of a tile
  static constexpr int SLICE = GT_ROWS / NQ;         // rows per slice (multiple of 8)
  static constexpr int Z_BYTES = GT_ROWS * R * 4;
  static constexpr int A_BYTES = 128 * GT_ROWS * 2;  // one digit tile
  static constexpr int RED_LD = R + 1;               // row stride of the final per-digit parts
  static constexpr int RED_BYTES = 128 * RED_LD * 8;
  static_assert(RED_BYTES <= 2 * A_BYTES, "final reduction fits in the digit tiles");
  static_assert(SLICE % 8 == 0, "digit groups of 8 rows");
  static constexpr size_t SMEM = (size_t)GT_STAGES * Z_BYTES + 2 * A_BYTES;
};

// Virtual blocks of the tensor-core normalisation/Gram pass over I rows (a
// function of I and the partial-buffer size only: batched and single-tensor
// sweeps split alike).
inline int tc_gram_blocks(int64_t I, int cap) {
  const int64_t tiles = (I + GT_ROWS - 1) / GT_ROWS;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, cap / 2));
}

// What a short mode's pass takes over from the kernels beside it: the column
// norms (lambda_body) from `nb` > 0 partials of the solve, every block for
// itself and block 0 for `lam`; the whole Gram in place of a partial, when there
// is one block.  Such a launch costs more than its work: three modes of up to
// 128 rows at R = 16, 137 -> 107 us per sweep.  A longer mode has too many
// partials for every block to sum them.
struct TcFuse {
  int nb = 0;
  const double* colsq = nullptr;
  const float* colmax = nullptr;
  double* lam = nullptr;  // as `lam` of the pass
  double* G = nullptr;
};
// Up to this many partials the sum is a chain of additions shorter than a launch.
constexpr int TC_FUSE_PARTS = 8;

// The pass over tiles vb, vb + nvb, ... of Z (see above).  `lam` holds
// lambda (R values) then the column scale exponents g_r (R values, from
// lambda_body).  Writes Y, gram_part[vb] (R x R, lower triangle) and, when M is non-null,
// inner_part[vb] (R).  Rows without nonzeros (bit clear in `mask`) get Y = 0.
template <typename FT, int R>
__device__ __forceinline__ void tc_scale_gram_body(const float* __restrict__ Z,
                                                   const double* __restrict__ lam, int64_t I,
                                                   FT* __restrict__ Y, const float* __restrict__ M,
                                                   double* __restrict__ gram_part,
                                                   double* __restrict__ inner_part,
                                                   const int* __restrict__ err, int vb, int nvb,
                                                   const uint32_t* __restrict__ mask,
                                                   const TcFuse& fuse) {
  using S = TcGramShape<R>;
  extern __shared__ __align__(1024) unsigned char smem_tc[];
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t bars[GT_STAGES + 2];  // Z stages; MMAs of digit tile 0 / 1
  __shared__ double red_in[TC_THREADS];
  __shared__ int gx[R];
  __shared__ float linv[R];
  if (*(volatile const int*)err) return;

  float* sZ = reinterpret_cast<float*>(smem_tc);
  unsigned char* sA = smem_tc + GT_STAGES * S::Z_BYTES;
  const int t = threadIdx.x;
  const int warp = t >> 5;
  const int r = t % R, kq = t / R;  // digitising: column r, rows kq * SLICE .. of a tile
  // reading D: thread t < 128 owns accumulator lane t = digit row (p, r) = (t / R, t % R)
  const int64_t ntiles = (I + GT_ROWS - 1) / GT_ROWS;
  const int nloc = vb < ntiles ? (int)((ntiles - 1 - vb) / nvb + 1) : 0;

  if (t < R) {  // one FP64 division per column, not per thread
    double lr;
    if (fuse.nb > 0) {  // as lambda_body
      double v = 0.0;
      int mb = 0;
      for (int b = 0; b < fuse.nb; ++b) {
        v += fuse.colsq[b * R + t];
        mb = max(mb, __float_as_int(fuse.colmax[b * R + t]));
      }
      lr = sqrt(v);
      gx[t] = gram_scale_exp(__int_as_float(mb), lr);
      if (vb == 0) {
        fuse.lam[t] = lr;
        fuse.lam[R + t] = (double)gx[t];
      }
    } else {
      lr = lam[t];
      gx[t] = (int)lam[R + t];
    }
    linv[t] = lr > 0.0 ? (float)(1.0 / lr) : 1.f;
  }
  if (warp == 0) tc::tmem_alloc(&tmem_slot, 128);
  if (t == 0) {
    for (int b = 0; b < GT_STAGES + 2; ++b) mbar_init(&bars[b], 1);
    fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const float inv = linv[r];  // 1 for a column of zeros: z * 1 = z
  const int g = gx[r];
  const bool gfast = g >= -125 && g <= 126;
  const float gs = gfast ? pow2f(-g) : 1.f;

  auto fetch = [&](int j) {  // local tile j into stage j % GT_STAGES (thread 0)
    fence_proxy_async_smem();
    const int64_t r0 = ((int64_t)vb + (int64_t)j * nvb) * GT_ROWS;
    const int64_t rows = I - r0 < GT_ROWS ? I - r0 : GT_ROWS;
    const uint32_t bytes = (uint32_t)(rows * R * 4);
    mbar_arrive_expect_tx(&bars[j % GT_STAGES], bytes);
    bulk_g2s(sZ + (j % GT_STAGES) * GT_ROWS * R, Z + r0 * R, bytes, &bars[j % GT_STAGES]);
  };
  int fetched = 0;  // thread 0's count of issued tile copies
  if (t == 0)
    for (; fetched < nloc && fetched < GT_STAGES; ++fetched) fetch(fetched);

  df2 acc[R / 2];  // digit row t of D folded over q: acc(s) = sum_q 2^-7q D(t, qR + s)
#pragma unroll
  for (int s = 0; s < R / 2; ++s) acc[s] = {0ull, 0ull};
  df inn = {0.f, 0.f};
  bool ok = true;
  int j = 0, committed = 0;
  for (; j < nloc && ok; ++j) {
    const int st = j % GT_STAGES, b = j & 1;
    const int64_t row0 = ((int64_t)vb + (int64_t)j * nvb) * GT_ROWS;
    ok = mbar_wait_bounded(&bars[st], (uint32_t)((j / GT_STAGES) & 1));
    if (ok && j >= 2) ok = mbar_wait_bounded(&bars[GT_STAGES + b], (uint32_t)(((j - 2) >> 1) & 1));
    if (!__syncthreads_and(ok)) break;
    const float* zs = sZ + st * GT_ROWS * R;
    unsigned char* A = sA + b * S::A_BYTES;
#pragma unroll 1
    for (int k0 = kq * S::SLICE; k0 < (kq + 1) * S::SLICE; k0 += 8) {
      // rows row0 + k0 .. + 7 share one word of the mask (row0 + k0 is a multiple of 8)
      const uint32_t live8 =
          mask ? (__ldg(&mask[(row0 + k0) >> 5]) >> ((row0 + k0) & 31)) & 0xFFu : 0xFFu;
      float y8[8];
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int64_t row = row0 + k0 + jj;
        float y = 0.f;
        if (row < I) {
          const bool lv = (live8 >> jj) & 1u;
          const float z = lv ? zs[(k0 + jj) * R + r] : 0.f;
          const FT ys = store_cvt<FT>(__fmul_rn(z, inv));
          Y[row * R + r] = ys;
          y = load_f<FT>(&ys, 0);
          if (M && lv) df_add_prod(inn, M[row * R + r], y);
        }
        y8[jj] = y;
      }
      uint64_t x[4];
#pragma unroll
      for (int jj = 0; jj < 4; ++jj)
        x[jj] = gfast ? f2_mul(f2_pack(y8[2 * jj], y8[2 * jj + 1]), f2_const(gs))
                      : f2_pack(ldexpf(y8[2 * jj], -g), ldexpf(y8[2 * jj + 1], -g));
#pragma unroll
      for (int p = 0; p < S::NDIG; ++p) {
        uint32_t k[4];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const uint64_t yy = f2_mul(x[jj], f2_const(128.f));
          const uint64_t kk = f2_round_int(yy);
          x[jj] = f2_sub(yy, kk);
          k[jj] = f2_pack_bf16_int(kk);
        }
        *reinterpret_cast<uint4*>(A + tc::kmajor_offset(p * R + r, k0, GT_ROWS)) =
            make_uint4(k[0], k[1], k[2], k[3]);
      }
    }
    fence_proxy_async_smem();  // digits visible to the tensor core
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (t == 0) {
      if (fetched < nloc) { fetch(fetched); ++fetched; }  // into stage st, read by now
      const bool first = (j % GT_FLUSH) == 0;
      const uint32_t a0 = smem_addr(A);
#pragma unroll
      for (int k16 = 0; k16 < GT_ROWS; k16 += 16) {
        const uint64_t da = tc::smem_desc(a0 + (k16 / 8) * 128, 128, (GT_ROWS / 8) * 128);
        tc::mma_bf16(tmem, da, da, tc::idesc_bf16(128, 128), !(first && k16 == 0));
      }
      tc::commit(&bars[GT_STAGES + b]);
    }
    committed = j + 1;
    if ((j % GT_FLUSH) == GT_FLUSH - 1 || j == nloc - 1) {
      ok = mbar_wait_bounded(&bars[GT_STAGES + b], (uint32_t)((j >> 1) & 1));
      tc::fence_after_sync();
      if (!__syncthreads_and(ok)) break;
      if (t < 128) {  // warps 0 .. 3: one accumulator lane each
        const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int q = 0; q < S::NDIG; ++q) {
          uint32_t v[R / 8][8];
#pragma unroll
          for (int c8 = 0; c8 < R / 8; ++c8) tc::ld8(lane_addr + (uint32_t)(q * R + c8 * 8), v[c8]);
          tc::wait_ld();
          const uint64_t wq = f2_const(pow2f(-7 * q));
#pragma unroll
          for (int s = 0; s < R; s += 2)
            df2_add(acc[s / 2], f2_mul(f2_pack(__uint_as_float(v[s / 8][s % 8]),
                                               __uint_as_float(v[s / 8][s % 8 + 1])), wq));
        }
      }
      tc::fence_before_sync();
      __syncthreads();  // every read done before the next MMA overwrites D
    }
  }
  if (!ok) {
    // a wait gave up: let the copies and MMAs in flight finish before the
    // shared and tensor memory are reused or released
    if (t == 0) {
      for (int k = j; k < fetched; ++k)
        (void)mbar_wait_bounded(&bars[k % GT_STAGES], (uint32_t)((k / GT_STAGES) & 1), 1u << 20);
      if (committed > 0) {
        const int jc = committed - 1;
        (void)mbar_wait_bounded(&bars[GT_STAGES + (jc & 1)], (uint32_t)((jc >> 1) & 1), 1u << 20);
      }
      atomicOr(const_cast<int*>(err), DEV_ERR_TIMEOUT);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  // Per-digit parts of the Gram, weighted, into the digit tiles (all MMAs have
  // completed).  They stay FP32 pairs up to the last sum: FP64 issues at 1/64
  // of FP32's rate, and this epilogue in FP64 was most of a short tensor's
  // pass (96 tensors: 113 and 76 us per mode at R = 32 and 16; now 64 and
  // 54; one tile of R = 16: 12.1 -> 9.1 us).  The weights are powers of two.
  // The sum over the digits is kept in three parts, of which the last pair
  // collects what the first loses: at R = 16, where the digits hold every bit,
  // a sum in one pair was 20 times as far from the exact Gram as one in FP64.
  float2* red = reinterpret_cast<float2*>(sA);
  if (t < 128) {
    const uint64_t wp = f2_const(pow2f(-7 * (t / R)));
#pragma unroll
    for (int s = 0; s < R; s += 2) {
      float2 a, b;
      f2_unpack(f2_mul(acc[s / 2].hi, wp), a.x, b.x);
      f2_unpack(f2_mul(acc[s / 2].lo, wp), a.y, b.y);
      red[t * S::RED_LD + s] = a;
      red[t * S::RED_LD + s + 1] = b;
    }
  }
  if (M) red_in[t] = df_value(inn);
  __syncthreads();
  if (ok) {
    // lower triangle, folded into R / 2 rows of R + 1 entries
    for (int e = t; e < R / 2 * (R + 1); e += TC_THREADS) {
      const int i = e / (R + 1) + R / 2, k = e % (R + 1);
      const int rr = k <= i ? i : R - 1 - i, ss = k <= i ? k : k - i - 1;
      float h = 0.f;
      df lost = {0.f, 0.f}, low = {0.f, 0.f};  // two chains side by side
#pragma unroll
      for (int p = S::NDIG - 1; p >= 0; --p) {
        const float2 x = red[(p * R + rr) * S::RED_LD + ss];
        const float s = __fadd_rn(h, x.x);
        const float bb = __fsub_rn(s, h);
        df_add(lost, __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(x.x, bb)));
        df_add(low, x.y);
        h = s;
      }
      df_add(low, lost.hi);
      low.lo = __fadd_rn(low.lo, lost.lo);
      const double x = times_pow2(__dadd_rn((double)h, df_value(low)), gx[rr] + gx[ss] - 14);
      if (fuse.G) {
        fuse.G[rr * R + ss] = x;
        fuse.G[ss * R + rr] = x;
      } else {
        gram_part[(int64_t)vb * R * R + rr * R + ss] = x;
      }
    }
    if (M && t < R) {
      double sum = 0.0;
      for (int q = 0; q < S::NQ; ++q) sum += red_in[q * R + t];
      inner_part[(int64_t)vb * R + t] = sum;
    }
  }
  if (warp == 0) tc::tmem_dealloc(tmem, 128);
  if (t == 0 && ok)
    for (int b = 0; b < GT_STAGES + 2; ++b) mbar_inval(&bars[b]);
}

}  // namespace spm
