// Reduced-precision V-cycle inside FP64 CG.
//
// The hierarchy is built in FP64 (amg_setup); this file stores a copy of
// every level's A, P and R values in FP32 -- or, for level_precision 2, the
// finest level's A in BF16 -- and runs the V-cycle with FP32 vectors and FP32
// accumulation.  The V-cycle reads the FP64 CG residual and writes the FP64
// preconditioned residual; the coarsest dense solve stays FP64.  The outer
// CG (its SpMV with K, residuals, dot products, stopping test) is untouched.
//
// Why: GB300 runs FP64 FMAs at ~2/clk/SM but FP32 at 128/clk/SM, so the
// FP64 SpMV is bound by the FP64 pipe; in FP32 (40 bytes per 3x3 block instead
// of 76) or BF16 values (22 bytes) the smoother SpMVs become HBM-bound and
// move half or less of the bytes.  A preconditioner only has to be a fixed
// SPD-like operator, so its rounding error costs at most a few iterations.
#include <algorithm>
#include <type_traits>

#include "handles.cuh"

namespace tam {
namespace {

constexpr int TPB = 256;

template <typename T>
__device__ __forceinline__ float f32(T v) { return (float)v; }

// x: records of f32_pitch(BS) floats per node; the other vectors packed
template <int BS, typename TB>
__global__ void cheb_first_zero_f32_kernel(const TB* __restrict__ b, const float* __restrict__ dinv,
                                           const float* __restrict__ consts, float* __restrict__ d,
                                           float* __restrict__ x, int n_rows, const int* __restrict__ stop) {
  if (stop && *stop) return;
  const float cr = consts[3];
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n_rows; row += gridDim.x * blockDim.x) {
    float v[BS];
#pragma unroll
    for (int r = 0; r < BS; ++r) {
      const size_t i = (size_t)row * BS + r;
      v[r] = cr * dinv[i] * f32(b[i]);
      d[i] = v[r];
    }
    store_record<BS>(x, row, v);
  }
}

// One Chebyshev step fused into the FP32 SpMV of x (records; xn: records in
// FP32, packed in FP64 -- the V-cycle's result on level 0).
template <int BR, typename TB, typename TO>
struct EpiChebF {
  const TB* b;
  const float* x;
  const float* dinv;
  const float* coef;
  float* d;
  TO* xn;
  int n_rows;
  const int* stop;
  __device__ bool skip() const { return stop && *stop; }
  __device__ void operator()(int row, const float (&acc)[BR], double*) const {
    if (row >= n_rows) return;
    const float cd = coef[0], cr = coef[1];
    const size_t i0 = (size_t)row * BR;
    // the row's operands first: behind the stores of d (which may alias them,
    // as far as the compiler can tell) each load would wait for the last (a
    // 1,280-row level of 6 x 6 blocks: 18-20 us a step that way)
    float v[BR], res[BR], dv[BR];
    load_record<BR>(x, row, v);
#pragma unroll
    for (int r = 0; r < BR; ++r) res[r] = dinv[i0 + r] * (f32(b[i0 + r]) - acc[r]);
    if (cd != 0.f) {
#pragma unroll
      for (int r = 0; r < BR; ++r) dv[r] = d[i0 + r];
#pragma unroll
      for (int r = 0; r < BR; ++r) dv[r] = cd * dv[r] + cr * res[r];
    } else {
#pragma unroll
      for (int r = 0; r < BR; ++r) dv[r] = cr * res[r];
    }
#pragma unroll
    for (int r = 0; r < BR; ++r) {
      d[i0 + r] = dv[r];
      v[r] += dv[r];
    }
    if constexpr (std::is_same<TO, float>::value) {
      store_record<BR>(xn, row, v);
    } else {
#pragma unroll
      for (int r = 0; r < BR; ++r) xn[(size_t)row * BR + r] = (TO)v[r];
    }
  }
};

// t = b - A x (t: records)
template <int BR, typename TB>
struct EpiResidualF {
  const TB* b;
  float* t;
  int n_rows;
  const int* stop;
  __device__ bool skip() const { return stop && *stop; }
  __device__ void operator()(int row, const float (&acc)[BR], double*) const {
    if (row >= n_rows) return;
    float v[BR];
#pragma unroll
    for (int r = 0; r < BR; ++r) v[r] = f32(b[(size_t)row * BR + r]) - acc[r];
    store_record<BR>(t, row, v);
  }
};

// y = A x (y packed: the next level's right-hand side)
template <int BR>
struct EpiStoreF {
  float* y;
  int n_rows;
  const int* stop;
  __device__ bool skip() const { return stop && *stop; }
  __device__ void operator()(int row, const float (&acc)[BR], double*) const {
    if (row < n_rows)
#pragma unroll
      for (int r = 0; r < BR; ++r) y[(size_t)row * BR + r] = acc[r];
  }
};

// y += A x (y: records)
template <int BR>
struct EpiAddF {
  float* y;
  int n_rows;
  const int* stop;
  __device__ bool skip() const { return stop && *stop; }
  __device__ void operator()(int row, const float (&acc)[BR], double*) const {
    if (row >= n_rows) return;
    float v[BR];
    load_record<BR>(y, row, v);
#pragma unroll
    for (int r = 0; r < BR; ++r) v[r] += acc[r];
    store_record<BR>(y, row, v);
  }
};

// coarsest level: FP64 dense inverse applied to an FP32 (or FP64) vector, FP64
// dot products; y: records of bs entries in FP32, packed in FP64
template <typename TI, typename TO>
__global__ void dense_gemv_mixed_kernel(const double* __restrict__ A, const TI* __restrict__ b, TO* __restrict__ y,
                                        int N, int ld, int bs, const int* __restrict__ stop) {
  if (stop && *stop) return;
  int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= N) return;
  const double* a = A + (size_t)row * ld;
  double s = 0.0;
  for (int j = lane; j < N; j += 32) s = fma(a[j], (double)b[j], s);
  s = warp_sum(s);
  if (lane == 0) {
    const int i = row / bs;
    y[std::is_same<TO, float>::value ? i * f32_pitch(bs) + (row - i * bs) : row] = (TO)s;
  }
}

__global__ void to_f32_kernel(const double* __restrict__ in, float* __restrict__ out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

unsigned vgrid(long long N) { return stride_grid(N, TPB, 8); }

// A x with the level's reduced-precision values: BF16 on the finest level in
// mode 2, FP32 otherwise.
template <int BS, class Epi>
void level_spmv(const Level& L, const float* x, Epi epi, cudaStream_t s) {
  if (L.A16.vals) spop_apply_f32<BS, BS, __nv_bfloat16>(L.A16, x, epi, s);
  else spop_apply_f32<BS, BS, float>(L.A32, x, epi, s);
}

template <typename TB, typename TO>
void cheb_step_f(const Level& L, const TB* b, const float* x, TO* xn, int step, const int* stop, cudaStream_t s) {
  const float* coef = L.consts32.p + 2 + 2 * step;
  if (L.bs == 3)
    level_spmv<3>(L, x, EpiChebF<3, TB, TO>{b, x, L.dinv32.p, coef, L.d32.p, xn, L.n_rows, stop}, s);
  else
    level_spmv<6>(L, x, EpiChebF<6, TB, TO>{b, x, L.dinv32.p, coef, L.d32.p, xn, L.n_rows, stop}, s);
}

template <typename TB>
void residual_f(const Level& L, const TB* b, const float* x, float* t, const int* stop, cudaStream_t s) {
  if (L.bs == 3) level_spmv<3>(L, x, EpiResidualF<3, TB>{b, t, L.n_rows, stop}, s);
  else level_spmv<6>(L, x, EpiResidualF<6, TB>{b, t, L.n_rows, stop}, s);
}

void restrict_f(const Level& L, const float* t, float* bc, const int* stop, cudaStream_t s) {
  const int nr = L.R.n_rows;
  if (L.kdim == 6 && L.bs == 3) spop_apply_f32<6, 3, float>(L.R32, t, EpiStoreF<6>{bc, nr, stop}, s);
  else if (L.kdim == 6) spop_apply_f32<6, 6, float>(L.R32, t, EpiStoreF<6>{bc, nr, stop}, s);
  else spop_apply_f32<3, 3, float>(L.R32, t, EpiStoreF<3>{bc, nr, stop}, s);
}

void prolong_f(const Level& L, const float* xc, float* x, const int* stop, cudaStream_t s) {
  const int nr = L.P.n_rows;
  if (L.kdim == 6 && L.bs == 3) spop_apply_f32<3, 6, float>(L.P32, xc, EpiAddF<3>{x, nr, stop}, s);
  else if (L.kdim == 6) spop_apply_f32<6, 6, float>(L.P32, xc, EpiAddF<6>{x, nr, stop}, s);
  else spop_apply_f32<3, 3, float>(L.P32, xc, EpiAddF<3>{x, nr, stop}, s);
}

template <typename TB, typename TO>
void vcycle_low(tam_amg_s* H, int l, const TB* b, TO* out, const int* stop, cudaStream_t s) {
  Level& L = H->levels[l];
  if (l == (int)H->levels.size() - 1) {
    dense_gemv_mixed_kernel<TB, TO><<<grid_for((long long)H->n_coarse * 32, TPB), TPB, 0, s>>>(
        H->coarse_inv.p, b, out, H->n_coarse, H->coarse_ld, L.bs, stop);
    TAM_LAUNCH_CHECK();
    return;
  }
  const int deg = L.deg;
  float* xa = L.xa32.p;
  float* xb = L.xb32.p;
  if (L.bs == 3)
    cheb_first_zero_f32_kernel<3, TB><<<vgrid(L.n_rows), TPB, 0, s>>>(b, L.dinv32.p, L.consts32.p, L.d32.p, xa,
                                                                     L.n_rows, stop);
  else
    cheb_first_zero_f32_kernel<6, TB><<<vgrid(L.n_rows), TPB, 0, s>>>(b, L.dinv32.p, L.consts32.p, L.d32.p, xa,
                                                                     L.n_rows, stop);
  TAM_LAUNCH_CHECK();
  for (int k = 1; k < deg; ++k) {
    cheb_step_f<TB, float>(L, b, xa, xb, k, stop, s);
    std::swap(xa, xb);
  }
  residual_f<TB>(L, b, xa, L.t32.p, stop, s);
  Level& C = H->levels[l + 1];
  restrict_f(L, L.t32.p, C.b32.p, stop, s);
  vcycle_low<float, float>(H, l + 1, C.b32.p, C.y32.p, stop, s);
  prolong_f(L, C.y32.p, xa, stop, s);
  for (int k = 0; k < deg; ++k) {
    if (k == deg - 1) {
      cheb_step_f<TB, TO>(L, b, xa, out, k, stop, s);
    } else {
      cheb_step_f<TB, float>(L, b, xa, xb, k, stop, s);
      std::swap(xa, xb);
    }
  }
}

}  // namespace

void vcycle_apply_low(tam_amg_s* H, const double* r, double* z, const int* stop, cudaStream_t s) {
  vcycle_low<double, double>(H, 0, r, z, stop, s);
}

void build_low_precision(tam_amg_s* H, cudaStream_t s) {
  const int mode = H->prm.level_precision;
  // level_precision 0: for the batched solve alone, which reads block-CSR order
  auto order = [&](const SpOp& op) { return mode == 0 ? in_block_csr(op) : op; };
  auto low_copy = [&](const SpOp& op, DBuf<float>& v) {
    convert_values_f32(op, v, s);
    return SpOpLow<float>{op, v.p};
  };
  for (size_t l = 0; l < H->levels.size(); ++l) {
    Level& L = H->levels[l];
    const size_t N = (size_t)L.n_rows * L.bs;
    const bool coarsest = (l + 1 == H->levels.size());
    L.dinv32 = DBuf<float>(N, s);
    to_f32_kernel<<<vgrid((long long)N), TPB, 0, s>>>(L.dinv.p, L.dinv32.p, (long long)N);
    TAM_LAUNCH_CHECK();
    const size_t nc = 2 + 2 * (size_t)std::max(L.deg, 1);
    L.consts32 = DBuf<float>(nc, s);
    to_f32_kernel<<<1, 32, 0, s>>>(L.consts.p, L.consts32.p, (long long)nc);
    TAM_LAUNCH_CHECK();
    const size_t NP = (size_t)L.n_rows * f32_pitch(L.bs);  // vectors of records
    L.b32 = DBuf<float>(N, s);
    L.y32 = DBuf<float>(NP, s);
    if (coarsest) continue;
    L.xa32 = DBuf<float>(NP, s);
    L.xb32 = DBuf<float>(NP, s);
    L.d32 = DBuf<float>(N, s);
    L.t32 = DBuf<float>(NP, s);
    if (l == 0 && mode == 2) {
      convert_values_bf16(L.Aop, L.A16v, s);
      L.A16 = SpOpLow<__nv_bfloat16>{L.Aop, L.A16v.p};
    } else {
      L.A32 = low_copy(order(L.Aop), L.A32v);
    }
    L.P32 = low_copy(order(L.Pop), L.P32v);
    L.R32 = low_copy(order(L.Rop), L.R32v);
  }
  H->low_ready = true;
}

void build_batch_operators(tam_amg_s* H, cudaStream_t s) {
  for (size_t l = 0; l + 1 < H->levels.size(); ++l) {
    Level& L = H->levels[l];
    auto own = [&](const SpOpLow<float>& o, DBuf<float>& v) {
      if (!o.vals || !low_in_store(o.op)) return o;
      convert_values_f32(in_block_csr(o.op), v, s);
      return SpOpLow<float>{in_block_csr(o.op), v.p};
    };
    L.A32m = own(L.A32, L.A32mv);
    L.P32m = own(L.P32, L.P32mv);
    L.R32m = own(L.R32, L.R32mv);
    L.A16m = L.A16;
    if (L.A16.vals && low_in_store(L.A16.op)) {
      convert_values_bf16(in_block_csr(L.A16.op), L.A16mv, s);
      L.A16m = SpOpLow<__nv_bfloat16>{in_block_csr(L.A16.op), L.A16mv.p};
    }
  }
  H->batch_ready = true;
}

void release_low_precision(tam_amg_s* H) {
  for (Level& L : H->levels) {
    for (auto* v : {&L.dinv32, &L.consts32, &L.b32, &L.y32, &L.xa32, &L.xb32, &L.d32, &L.t32, &L.A32v, &L.P32v, &L.R32v})
      v->reset();
    L.A16v.reset();
    L.A32 = L.P32 = L.R32 = SpOpLow<float>{};
    L.A16 = SpOpLow<__nv_bfloat16>{};
  }
  H->low_ready = false;
}

void release_batch_operators(tam_amg_s* H) {
  for (Level& L : H->levels) {
    for (auto* v : {&L.A32mv, &L.P32mv, &L.R32mv}) v->reset();
    L.A16mv.reset();
    L.A32m = L.P32m = L.R32m = SpOpLow<float>{};
    L.A16m = SpOpLow<__nv_bfloat16>{};
  }
  H->batch_ready = false;
}

}  // namespace tam
