// Learned CG initial guess: a node-wise multilayer perceptron, trained and
// evaluated with the kernels in this file.
//
// The paper has no learned component.  The network maps per-node features
// (coordinates, temperature, temperature gradient, distance to the clamped
// boundary) to a displacement guess that seeds AMG-PCG; the solver always
// iterates to the tolerance from it, and a guess whose preconditioned
// residual energy <r, M r> is not below that of the zero guess is replaced by
// zero (tam_learned_guess), so the network can cost iterations but never
// accuracy.
//
// Layers: tanh hidden layers, linear output.  Inputs are standardised,
// (x - shift) * scale, inside the first layer; outputs are multiplied by
// out_scale.  Training minimises the mean squared error with Adam.  All
// parameters are FP32 (master copy); inference can read a BF16 copy of the
// weights.  Each FP32 dense layer is one tiled kernel (dense_kernel), its
// weight gradient a split sum over row tiles (weight_grad_kernel).
#include <cmath>
#include <functional>
#include <type_traits>
#include <vector>

#include "handles.cuh"

struct tam_mlp_s {
  int n_in = 0, width = 0, depth = 0, n_out = 0;
  std::vector<std::pair<int, int>> shapes;  // (fan-in, fan-out) per layer
  std::vector<long long> offset;            // start of W_l in theta (bias follows)
  long long n_par = 0;
  tam::DBuf<float> theta, grad, m1, m2, shift, scale, out_scale;
  tam::DBuf<__nv_bfloat16> theta16;
  bool theta16_valid = false;
  int adam_t = 0;
  tam::DBuf<float> act;  // activations of the current batch, layer after layer
  size_t act_cap = 0;
  tam::DBuf<float> dbuf[2];
  size_t dcap = 0;
  tam::DBuf<float> part;  // the blocks' partial weight gradients of one layer
  tam::DBuf<double> red;  // loss reduction
  tam::DBuf<unsigned int> ticket;
};

namespace tam {
namespace {

constexpr int ROWS = 128;  // rows of the activation tile per block
constexpr int DENSE_THREADS = 512;
constexpr int THREADS = 256;

// Two FP32 multiply-adds in one instruction (each rounded as fmaf's): the FP32
// kernels below are bound by instruction issue, and the packed form halves
// their multiply-adds' share of it.
__device__ __forceinline__ void fma2(float2& acc, float2 a, float2 b) {
  unsigned long long& c = reinterpret_cast<unsigned long long&>(acc);
  asm("fma.rn.f32x2 %0, %1, %2, %0;"
      : "+l"(c)
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
}

// out[n x N] = epi(A[n x K] W + bias) with W [K x N] row-major (or W^T when
// TRANS: W stored [N x K]).  MODE: 0 linear, 1 tanh, 2 output (* out_scale),
// 3 backward through tanh: out = (A W^T) * (1 - H^2) with H = `aux`.
// STD: standardise A on load with (a - shift) * scale.
//
// Bound by the FP32 pipe and its operands' way out of shared memory (60% and
// 64% busy on 131,072 rows of a 128 x 128 layer, 16 warps an SM): a 128-row
// tile of the activations and the whole weight matrix (zero-padded to Kp x Np) sit in shared memory, and each of the
// 512 threads keeps a TM x TN tile of outputs in registers, so that four
// steps of k cost TM + TN 16-byte shared loads for 4 TM TN multiply-adds (the
// kernel before, one row by 8 outputs a thread with scalar loads and a bounds
// test per product, spent nine loads on eight products).  Threads: NG column
// groups x 512 / NG row groups, a warp 8 x 4 of them, so that its weight reads
// are 128 bytes; a thread's rows are its group's number plus multiples of the
// group count, which keeps a warp's row reads on different banks.  The next
// tile is copied while this one is multiplied, one barrier a tile (two blocks
// of 256 threads an SM, each loading and then multiplying 64 rows: 1.09 ms).
// Each output sums its products in increasing k.  The 8-128-128-128-3 network
// on 468,864 rows: 8.74 -> 1.03 ms (31 TFLOP/s of 76.8).
template <int MODE, bool TRANS, bool STD, int TM, int TN, int NG>
__global__ void __launch_bounds__(DENSE_THREADS, 1)
dense_kernel(const float* __restrict__ A, long long n, int K, int N, const float* __restrict__ W,
             const float* __restrict__ bias, const float* __restrict__ shift, const float* __restrict__ scale,
             const float* __restrict__ out_scale, const float* __restrict__ aux, float* __restrict__ out, bool a_vec,
             bool o_vec) {
  constexpr int RG = DENSE_THREADS / NG, Np = NG * TN;
  static_assert(RG * TM == ROWS && (TN == 1 || TN == 4 || TN == 8), "dense_kernel: tile");
  extern __shared__ __align__(16) float sm[];
  const int Kp = (K + 3) & ~3, lda = Kp + 4;
  float* Ws = sm;                     // [Kp][Np]
  float* As = sm + (size_t)Kp * Np;   // two buffers of [ROWS][lda]
  // the tile of rows r0 .. into buffer b (asynchronously where it is copied as it is)
  auto fetch = [&](long long r0, int b) {
    float* dst = As + (size_t)b * ROWS * lda;
    if (a_vec && !STD) {
      const int q = K >> 2;  // K = Kp: whole 16-byte groups
      for (int e = threadIdx.x; e < ROWS * q; e += DENSE_THREADS) {
        const int r = e / q, k = (e - r * q) * 4;
        const bool in = r0 + r < n;
        const unsigned to = (unsigned)__cvta_generic_to_shared(dst + r * lda + k);
        const float* from = A + (in ? (r0 + r) * K + k : 0);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(in ? 16 : 0));
      }
    } else {
      for (int e = threadIdx.x; e < ROWS * Kp; e += DENSE_THREADS) {
        const int r = e / Kp, k = e - r * Kp;
        float a = 0.f;
        if (r0 + r < n && k < K) {
          a = A[(r0 + r) * K + k];
          if (STD) a = (a - shift[k]) * scale[k];
        }
        dst[r * lda + k] = a;
      }
    }
  };
  long long r0 = (long long)blockIdx.x * ROWS;
  const long long stride = (long long)gridDim.x * ROWS;
  if (r0 < n) fetch(r0, 0);
  if (TRANS) {
    for (int e = threadIdx.x; e < Kp * Np; e += DENSE_THREADS) Ws[e] = 0.f;
    __syncthreads();
    // a warp transposes 8 rows x 4 groups of 4 columns: 8 lines per read, 4
    // lanes per bank and write
    const int kq = (K + 3) >> 2, jb = (N + 7) >> 3, kb = (kq + 3) >> 2;
    for (int t = threadIdx.x >> 5; t < jb * kb; t += DENSE_THREADS / 32) {
      const int j = (t % jb) * 8 + (threadIdx.x & 7), k = ((t / jb) * 4 + ((threadIdx.x & 31) >> 3)) * 4;
      if (j < N)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (k + q < K) Ws[(k + q) * Np + j] = W[(size_t)j * K + k + q];
    }
  } else {
    for (int e = threadIdx.x; e < Kp * Np; e += DENSE_THREADS) {
      const int k = e / Np, j = e - k * Np;
      Ws[e] = (k < K && j < N) ? W[(size_t)k * N + j] : 0.f;
    }
  }
  // a warp: CW column groups (128 bytes of a weight row) x 32 / CW row groups
  constexpr int CW = NG < 8 ? NG : 8, NW = NG / CW;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int cg = lane % CW + CW * (wid % NW), rg = lane / CW + (32 / CW) * (wid / NW);
  for (int b = 0; r0 < n; r0 += stride, b ^= 1) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // this tile is in place, and the other buffer's readers are done
    if (r0 + stride < n) fetch(r0 + stride, b ^ 1);
    const float* Ab = As + (size_t)b * ROWS * lda;
    constexpr int TP = (TN + 1) / 2;  // output pairs (TN = 1: the second half idle)
    float2 acc[TM][TP];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TP; ++j) acc[i][j] = make_float2(0.f, 0.f);
    // a warp without rows (a small batch fills a few) leaves the issue slots to
    // the others: one row of 128-128-128-128: 61.4 -> 37.6 us
    const int k_end = r0 + (32 / CW) * (wid / NW) < n ? Kp : 0;
    for (int k = 0; k < k_end; k += 4) {
      float av[TM][4];
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 a = *reinterpret_cast<const float4*>(Ab + (rg + i * RG) * lda + k);
        av[i][0] = a.x;
        av[i][1] = a.y;
        av[i][2] = a.z;
        av[i][3] = a.w;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float* wr = Ws + (k + kk) * Np;
        if constexpr (TN == 1) {
          const float w = wr[cg];
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][0].x = fmaf(av[i][kk], w, acc[i][0].x);
        } else {
          float2 w[TP];
#pragma unroll
          for (int h = 0; h < TN / 4; ++h) {
            const float4 v = *reinterpret_cast<const float4*>(wr + h * 4 * NG + cg * 4);
            w[2 * h] = make_float2(v.x, v.y);
            w[2 * h + 1] = make_float2(v.z, v.w);
          }
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float2 a = make_float2(av[i][kk], av[i][kk]);
#pragma unroll
            for (int j = 0; j < TP; ++j) fma2(acc[i][j], a, w[j]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const long long row = r0 + rg + i * RG;
      if (row >= n) continue;
#pragma unroll
      for (int h = 0; h < (TN + 3) / 4; ++h) {
        constexpr int V = TN < 4 ? TN : 4;
        const int c0 = h * 4 * NG + cg * V;
        float z[V];
#pragma unroll
        for (int q = 0; q < V; ++q) {
          const int c = c0 + q;
          z[q] = 0.f;
          if (c >= N) continue;
          const float2 p = acc[i][(h * 4 + q) / 2];
          z[q] = ((q & 1) ? p.y : p.x) + (bias ? bias[c] : 0.f);
          if (MODE == 1) z[q] = tanhf(z[q]);
          else if (MODE == 2) z[q] *= out_scale[c];
          else if (MODE == 3) {
            const float hh = aux[row * N + c];
            z[q] *= (1.f - hh * hh);
          }
        }
        if (V == 4 && o_vec && c0 < N) {  // N a multiple of 4: the group is whole
          *reinterpret_cast<float4*>(out + row * N + c0) = make_float4(z[0], z[V > 1 ? 1 : 0], z[V > 2 ? 2 : 0], z[V > 3 ? 3 : 0]);
        } else {
#pragma unroll
          for (int q = 0; q < V; ++q)
            if (c0 + q < N) out[row * N + c0 + q] = z[q];
        }
      }
    }
  }
}

// Weight gradients, part 1: block b sums grad_W = H^T D and grad_b =
// colsum(D) over its tiles of WG_ROWS rows and writes its partial sums to
// part[b][K * N + N].  Bound by the FP32 pipe and, on few rows, the trip to
// memory before each tile (pipe 48% busy on 32,768 rows of 128 x 128, load
// latency the most frequent stall): a thread keeps a TK x TN tile of grad_W in
// registers (8 x 8 for a 128 x 128 layer) and reads TK + TN
// values of a row for TK TN products; the kernel before held every 256th
// entry and read two values per product.
// Narrow layers (K, N <= 16: a product a thread and row) are bound by the trip
// to memory and the two barriers of a tile instead: four times the rows a
// tile, each quarter with a sum of its own (a gradient on 300,001 rows of 8-3-3:
// 240 -> 190 us).  Their partial sums, where at most WG_LAST blocks wrote some,
// are added by the last block to finish, not by a launch of its own (3,000 rows of
// 8-8-8-3: 110 -> 105 us).
constexpr int WG_ROWS = 32, WG_LAST = 32;
constexpr int wg_quarters(int TK, int TN) { return TK == 1 && TN == 1 ? 4 : 1; }

template <int TK, int TN>
__global__ void __launch_bounds__(THREADS, 2)
weight_grad_kernel(const float* __restrict__ H, const float* __restrict__ D, long long n, int K, int N,
                   const float* __restrict__ shift, const float* __restrict__ scale, float* __restrict__ part,
                   bool h_vec, bool d_vec, float* __restrict__ grad, unsigned int* __restrict__ ticket) {
  constexpr int Kp = 16 * TK, Np = 16 * TN;  // 16 x 16 threads
  constexpr int Q = wg_quarters(TK, TN), ROWS_T = Q * WG_ROWS;
  __shared__ __align__(16) float Hs[ROWS_T][Kp];
  __shared__ __align__(16) float Ds[ROWS_T][Np];
  // a warp: 4 x 8 threads, so that its reads of a row are 64 and 128 bytes
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int kg = (lane >> 3) + 4 * (wid >> 1), ng = (lane & 7) + 8 * (wid & 1);
  constexpr int TP = (TN + 1) / 2;  // pairs of outputs (TN = 1: the second half idle)
  float2 acc[TK][TP];
  float accb[TN];
#pragma unroll
  for (int j = 0; j < TN; ++j) accb[j] = 0.f;
#pragma unroll
  for (int j = 0; j < TP; ++j)
#pragma unroll
    for (int i = 0; i < TK; ++i) acc[i][j] = make_float2(0.f, 0.f);
  [[maybe_unused]] float accq[Q] = {}, accbq[Q] = {};  // Q > 1: the quarters' sums
  // rows of src [n x M] from r0 into dst [ROWS_T][Mp], zero-padded
  auto fill = [&](const float* __restrict__ src, int M, int Mp, float* dst, bool vec, bool std_, long long r0) {
    if (vec) {
      const int q = Mp >> 2;
      for (int e = threadIdx.x; e < ROWS_T * q; e += THREADS) {
        const int r = e / q, k = (e - r * q) * 4;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + r < n && k < M) {
          a = *reinterpret_cast<const float4*>(src + (r0 + r) * M + k);
          if (std_) {
            a.x = (a.x - shift[k]) * scale[k];
            a.y = (a.y - shift[k + 1]) * scale[k + 1];
            a.z = (a.z - shift[k + 2]) * scale[k + 2];
            a.w = (a.w - shift[k + 3]) * scale[k + 3];
          }
        }
        *reinterpret_cast<float4*>(dst + r * Mp + k) = a;
      }
    } else {
      for (int e = threadIdx.x; e < ROWS_T * Mp; e += THREADS) {
        const int r = e / Mp, k = e - r * Mp;
        float a = 0.f;
        if (r0 + r < n && k < M) {
          a = src[(r0 + r) * M + k];
          if (std_) a = (a - shift[k]) * scale[k];
        }
        dst[e] = a;
      }
    }
  };
  // T consecutive-by-4 values of a row: 4 at 4 g, the next 4 half a row on (no bank conflicts)
  auto take = [&](const float* row, int g, auto& v) {
    constexpr int T = sizeof(v) / sizeof(float);
    if constexpr (T == 1) {
      v[0] = row[g];
    } else {
#pragma unroll
      for (int h = 0; h < T / 4; ++h) {
        const float4 x = *reinterpret_cast<const float4*>(row + h * 64 + 4 * g);
        v[4 * h] = x.x;
        v[4 * h + 1] = x.y;
        v[4 * h + 2] = x.z;
        v[4 * h + 3] = x.w;
      }
    }
  };
  for (long long r0 = (long long)blockIdx.x * ROWS_T; r0 < n; r0 += (long long)gridDim.x * ROWS_T) {
    __syncthreads();
    fill(H, K, Kp, &Hs[0][0], h_vec, shift != nullptr, r0);
    fill(D, N, Np, &Ds[0][0], d_vec, false, r0);
    __syncthreads();
    if constexpr (Q > 1) {
#pragma unroll 4
      for (int r = 0; r < WG_ROWS; ++r)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const float d = Ds[q * WG_ROWS + r][ng];
          accbq[q] += d;
          accq[q] = fmaf(Hs[q * WG_ROWS + r][kg], d, accq[q]);
        }
      continue;
    }
#pragma unroll 4
    for (int r = 0; r < WG_ROWS; ++r) {
      float h[TK], d[TN];
      take(Hs[r], kg, h);
      take(Ds[r], ng, d);
      if (kg == 0)
#pragma unroll
        for (int j = 0; j < TN; ++j) accb[j] += d[j];
#pragma unroll
      for (int i = 0; i < TK; ++i) {
        if constexpr (TN == 1) {
          acc[i][0].x = fmaf(h[i], d[0], acc[i][0].x);
        } else {
          const float2 hh = make_float2(h[i], h[i]);
#pragma unroll
          for (int j = 0; j < TP; ++j) fma2(acc[i][j], hh, make_float2(d[2 * j], d[2 * j + 1]));
        }
      }
    }
  }
  if constexpr (Q > 1) {
    acc[0][0].x = (accq[0] + accq[1]) + (accq[2] + accq[3]);
    accb[0] = (accbq[0] + accbq[1]) + (accbq[2] + accbq[3]);
  }
  float* __restrict__ o = part + (size_t)blockIdx.x * ((size_t)K * N + N);
#pragma unroll
  for (int i = 0; i < TK; ++i) {
    const int k = TK == 1 ? kg : (i / 4) * 64 + 4 * kg + (i & 3);
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = TN == 1 ? ng : (j / 4) * 64 + 4 * ng + (j & 3);
      if (k < K && c < N) o[(size_t)k * N + c] = (j & 1) ? acc[i][j / 2].y : acc[i][j / 2].x;
      if (kg == 0 && i == 0 && c < N) o[(size_t)K * N + c] = accb[j];
    }
  }
  if constexpr (Q > 1) {
    if (gridDim.x > WG_LAST) return;  // weight_grad_reduce_kernel follows
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int M = K * N + N;
    for (int e = threadIdx.x; e < M; e += THREADS) {  // in weight_grad_reduce_kernel's order
      float s[8] = {};
      for (int b = 0; b < (int)gridDim.x; b += 8)
#pragma unroll
        for (int w = 0; w < 8; ++w)
          if (b + w < (int)gridDim.x) s[w] += __ldcg(part + (size_t)(b + w) * M + e);
#pragma unroll
      for (int w = 1; w < 8; ++w) s[0] += s[w];
      grad[e] = s[0];
    }
    if (threadIdx.x == 0) *ticket = 0u;
  }
}

// Part 2: the blocks' partial sums, in block order (8 lanes' worth of blocks
// at a time, combined in a fixed order): grad[e] for the layer's M entries.
__global__ void __launch_bounds__(256) weight_grad_reduce_kernel(const float* __restrict__ part, int blocks, int M,
                                                                 float* __restrict__ grad) {
  __shared__ float sh[8][33];
  const int e = blockIdx.x * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
  float s = 0.f;
  if (e < M)
    for (int b = w; b < blocks; b += 8) s += part[(size_t)b * M + e];
  sh[w][threadIdx.x & 31] = s;
  __syncthreads();
  if (w == 0 && e < M) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s += sh[q][threadIdx.x];
    grad[e] = s;
  }
}

// d = 2 (pred - Y) / (n m) * out_scale;  loss = mean (pred - Y)^2
__global__ void loss_grad_kernel(const float* __restrict__ pred, const float* __restrict__ Y, long long n, int m,
                                 const float* __restrict__ out_scale, float* __restrict__ d, GridReduce gr,
                                 double* __restrict__ loss) {
  __shared__ double sh[32];
  double acc[1] = {0.0};
  const double inv = 1.0 / ((double)n * m);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n * m; i += (long long)gridDim.x * blockDim.x) {
    const float diff = pred[i] - Y[i];
    acc[0] += (double)diff * diff;
    d[i] = (float)(2.0 * diff * inv) * out_scale[i % m];
  }
  double tot[1];
  if (grid_reduce<1>(gr, acc, tot, sh) && threadIdx.x == 0) *loss = tot[0] * inv;
}

// Adam (Kingma & Ba 2015): bias-corrected first/second moments
__global__ void adam_kernel(float* __restrict__ theta, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

__global__ void init_params_kernel(float* __restrict__ theta, long long off, int a, int b, unsigned long long seed) {
  const long long nw = (long long)a * b;
  const float lim = sqrtf(6.f / (float)(a + b));  // Glorot uniform
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nw + b; i += (long long)gridDim.x * blockDim.x) {
    if (i < nw) {
      const uint64_t z = splitmix64(seed ^ (uint64_t)(off + i) * 0x9E3779B97F4A7C15ull);
      const float u = (float)((z >> 40) * (1.0 / 16777216.0));
      theta[off + i] = (2.f * u - 1.f) * lim;
    } else {
      theta[off + i] = 0.f;
    }
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ in, __nv_bfloat16* __restrict__ out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = __float2bfloat16(in[i]);
}

// ---------------------------------------------------------------------------
// BF16 inference on the tensor cores: out = epi(A W + bias) with BF16 weights
// and BF16-rounded activations, FP32 accumulation (mma.sync m16n8k16).  A
// block of 4 warps takes 64 rows; warp w multiplies rows 16w..16w+15 of the
// tile by all of W.  W is kept transposed (n-major) in shared memory so that
// the two k-consecutive values of a B fragment are one 32-bit word; the A
// tile likewise.  K is padded to a multiple of 16 and N to a multiple of 8
// with zeros (K, N <= 128).
// ---------------------------------------------------------------------------
constexpr int MMA_ROWS = 64;
constexpr int MMA_THREADS = 128;
constexpr int MMA_KMAX = 128, MMA_NMAX = 128;
constexpr int MMA_LD = MMA_KMAX + 8;  // row stride in bf16 elements (staggers the banks)

__device__ __forceinline__ void mma_bf16_16x8x16(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                                 unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four 8 x 8 matrices of 16-bit values from shared memory; lane q supplies the
// (16-byte aligned) address of row q % 8 of matrix q / 8.
__device__ __forceinline__ void ldmatrix_x4(unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3, const void* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(a));
}

template <int MODE, bool STD>
__global__ void __launch_bounds__(MMA_THREADS)
dense_mma_kernel(const float* __restrict__ A, long long n, int K, int N, const __nv_bfloat16* __restrict__ W,
                 const float* __restrict__ bias, const float* __restrict__ shift, const float* __restrict__ scale,
                 const float* __restrict__ out_scale, float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __nv_bfloat16* Wt = reinterpret_cast<__nv_bfloat16*>(sm_raw);  // [Np][MMA_LD]
  const int Kp = (K + 15) & ~15, Np = (N + 7) & ~7;
  __nv_bfloat16* At = Wt + (size_t)Np * MMA_LD;                  // [MMA_ROWS][MMA_LD]
  for (int e = threadIdx.x; e < Np * Kp; e += MMA_THREADS) {
    const int nn = e / Kp, k = e % Kp;
    Wt[nn * MMA_LD + k] = (nn < N && k < K) ? W[(size_t)k * N + nn] : __float2bfloat16(0.f);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  for (long long r0 = (long long)blockIdx.x * MMA_ROWS; r0 < n; r0 += (long long)gridDim.x * MMA_ROWS) {
    __syncthreads();
    for (int e = threadIdx.x; e < MMA_ROWS * Kp; e += MMA_THREADS) {
      const int r = e / Kp, k = e % Kp;
      const long long row = r0 + r;
      float a = 0.f;
      if (row < n && k < K) {
        a = A[row * K + k];
        if (STD) a = (a - shift[k]) * scale[k];
      }
      At[r * MMA_LD + k] = __float2bfloat16(a);
    }
    __syncthreads();
    float acc[MMA_NMAX / 8][4];
#pragma unroll
    for (int j = 0; j < MMA_NMAX / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    const __nv_bfloat16* Aw = At + (warp * 16) * MMA_LD;
    for (int k0 = 0; k0 < Kp; k0 += 16) {
      // A fragment: (g, 2t..2t+1), (g+8, 2t..), (g, 2t+8..), (g+8, 2t+8..)
      const unsigned a0 = *reinterpret_cast<const unsigned*>(Aw + g * MMA_LD + k0 + 2 * t);
      const unsigned a1 = *reinterpret_cast<const unsigned*>(Aw + (g + 8) * MMA_LD + k0 + 2 * t);
      const unsigned a2 = *reinterpret_cast<const unsigned*>(Aw + g * MMA_LD + k0 + 2 * t + 8);
      const unsigned a3 = *reinterpret_cast<const unsigned*>(Aw + (g + 8) * MMA_LD + k0 + 2 * t + 8);
#pragma unroll
      for (int j = 0; j < MMA_NMAX / 8; ++j) {
        if (j * 8 >= Np) break;
        // B fragment (column n = 8j + g): k = 2t..2t+1 and 2t+8..2t+9
        const __nv_bfloat16* wb = Wt + (j * 8 + g) * MMA_LD + k0 + 2 * t;
        mma_bf16_16x8x16(acc[j], a0, a1, a2, a3, *reinterpret_cast<const unsigned*>(wb),
                         *reinterpret_cast<const unsigned*>(wb + 8));
      }
    }
    // C fragment: (g, 2t..2t+1) and (g+8, 2t..2t+1) of each 16x8 tile
#pragma unroll
    for (int j = 0; j < MMA_NMAX / 8; ++j) {
      if (j * 8 >= Np) break;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const long long row = r0 + warp * 16 + g + (h >= 2 ? 8 : 0);
        const int c = j * 8 + 2 * t + (h & 1);
        if (row >= n || c >= N) continue;
        float z = acc[j][h] + (bias ? bias[c] : 0.f);
        if (MODE == 1) z = tanhf(z);
        else if (MODE == 2) z *= out_scale[c];
        out[row * N + c] = z;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The whole network in one kernel (BF16 inference): every layer's transposed
// BF16 weights and FP32 biases sit in shared memory for the kernel's life;
// each warp takes 16 rows at a time through all layers with the activations
// in registers -- the FP32 accumulators of one layer's 16 x 8 output tiles,
// biased, passed through tanh and rounded to BF16, are exactly the A
// fragments of the next layer's m16n8k16 products (tiles 2m and 2m+1 form
// k-chunk m).  Per row only the n_in inputs are read and the n_out outputs
// written.  Same roundings, products and summation order as the layer-by-
// layer kernel above, so the results are bitwise the same.  No pipe
// is full (issue slots 61% busy, ALU 48, FMA 24, tensor 23, special functions
// 15): accumulators and fragments take 128 registers a thread, and with the 16
// warps an SM that leaves, their product and tanh phases (384 tanh a row) do
// not cover each other.  The weight fragments come four registers a request
// (11.6M rows of 8-128-128-128-3: 6.40 -> 6.25 ms).
// ---------------------------------------------------------------------------
constexpr int FUSED_WARPS = 8;
constexpr int FUSED_MAX_LAYERS = 8;
constexpr int FUSED_WMAX = 128;  // widest layer (inputs and outputs)

struct FusedNet {
  int L;
  int K[FUSED_MAX_LAYERS], N[FUSED_MAX_LAYERS];    // true fan-in / fan-out
  int Kp[FUSED_MAX_LAYERS], Np[FUSED_MAX_LAYERS];  // padded: K to 16, N to 16 (hidden) or 8 (last)
  int wsm[FUSED_MAX_LAYERS], bsm[FUSED_MAX_LAYERS];  // shared-memory offsets (bf16 / float elements)
  long long woff[FUSED_MAX_LAYERS];                // W_l in theta (bias follows)
  int w_elems, b_elems;
};

__device__ __forceinline__ unsigned pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}

__global__ void __launch_bounds__(FUSED_WARPS * 32, 2)
mlp_fused_kernel(const float* __restrict__ X, long long n, FusedNet net, const __nv_bfloat16* __restrict__ th16,
                 const float* __restrict__ th, const float* __restrict__ shift, const float* __restrict__ scale,
                 const float* __restrict__ out_scale, float* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __nv_bfloat16* Ws = reinterpret_cast<__nv_bfloat16*>(sm_raw);
  float* Bs = reinterpret_cast<float*>(sm_raw + (((size_t)net.w_elems * 2 + 15) & ~(size_t)15));
  // W_l^T [Np][Kp + 8] (zero-padded) and b_l [Np]
  for (int l = 0; l < net.L; ++l) {
    const int K = net.K[l], N = net.N[l], Kp = net.Kp[l], Np = net.Np[l], ld = Kp + 8;
    const __nv_bfloat16* W = th16 + net.woff[l];
    for (int e = threadIdx.x; e < Np * ld; e += blockDim.x) {
      const int nn = e / ld, k = e - nn * ld;
      Ws[net.wsm[l] + e] = (nn < N && k < K) ? W[(size_t)k * N + nn] : __float2bfloat16(0.f);
    }
    const float* b = th + net.woff[l] + (long long)K * N;
    for (int e = threadIdx.x; e < Np; e += blockDim.x) Bs[net.bsm[l] + e] = e < N ? b[e] : 0.f;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int n_in = net.K[0], n_out = net.N[net.L - 1];
  for (long long r0 = ((long long)blockIdx.x * FUSED_WARPS + warp) * 16; r0 < n;
       r0 += (long long)gridDim.x * FUSED_WARPS * 16) {
    unsigned af[FUSED_WMAX / 16][4];
    // layer 0's A fragments from the standardised inputs of rows r0+g, r0+g+8
    {
      const long long ra = r0 + g, rb = r0 + g + 8;
#pragma unroll
      for (int m = 0; m < FUSED_WMAX / 16; ++m) {
        if (m * 16 >= net.Kp[0]) break;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          // q: 0,1 (ra, 2t..), 2,3 (rb, 2t..), 4,5 (ra, 2t+8..), 6,7 (rb, 2t+8..)
          const long long row = (q & 2) ? rb : ra;
          const int k = m * 16 + 2 * t + (q & 1) + ((q & 4) ? 8 : 0);
          float a = 0.f;
          if (row < n && k < n_in) a = (X[row * n_in + k] - shift[k]) * scale[k];
          v[q] = a;
        }
        af[m][0] = pack_bf16x2(v[0], v[1]);
        af[m][1] = pack_bf16x2(v[2], v[3]);
        af[m][2] = pack_bf16x2(v[4], v[5]);
        af[m][3] = pack_bf16x2(v[6], v[7]);
      }
    }
    for (int l = 0; l < net.L; ++l) {
      const int Kp = net.Kp[l], Np = net.Np[l], ld = Kp + 8;
      const __nv_bfloat16* Wt = Ws + net.wsm[l];
      float acc[FUSED_WMAX / 8][4];
#pragma unroll
      for (int j = 0; j < FUSED_WMAX / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
      for (int m = 0; m < FUSED_WMAX / 16; ++m) {
        if (m * 16 >= Kp) break;
#pragma unroll
        for (int j = 0; j < FUSED_WMAX / 8; j += 2) {
          if (j * 8 >= Np) break;
          // B fragments of column tiles j and j + 1 (k 0..7 and 8..15 of the
          // chunk) in one request: lane q supplies row q % 8 of matrix q / 8;
          // tile j + 1 of an odd last pair repeats tile j, unused
          const int jj = (j + 1) * 8 < Np ? j + (lane >> 4) : j;
          unsigned b0, b1, b2, b3;
          ldmatrix_x4(b0, b1, b2, b3, Wt + (jj * 8 + (lane & 7)) * ld + m * 16 + ((lane >> 3) & 1) * 8);
          mma_bf16_16x8x16(acc[j], af[m][0], af[m][1], af[m][2], af[m][3], b0, b1);
          if ((j + 1) * 8 < Np) mma_bf16_16x8x16(acc[j + 1], af[m][0], af[m][1], af[m][2], af[m][3], b2, b3);
        }
      }
      const float* bl = Bs + net.bsm[l];
      if (l + 1 < net.L) {
        // hidden layer: tanh(acc + b), rounded to BF16, becomes the next A
#pragma unroll
        for (int m = 0; m < FUSED_WMAX / 16; ++m) {
          if (m * 16 >= Np) break;
          float z[2][4];
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int h = 0; h < 4; ++h) z[u][h] = tanhf(acc[2 * m + u][h] + bl[(2 * m + u) * 8 + 2 * t + (h & 1)]);
          af[m][0] = pack_bf16x2(z[0][0], z[0][1]);
          af[m][1] = pack_bf16x2(z[0][2], z[0][3]);
          af[m][2] = pack_bf16x2(z[1][0], z[1][1]);
          af[m][3] = pack_bf16x2(z[1][2], z[1][3]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < FUSED_WMAX / 8; ++j) {
          if (j * 8 >= Np) break;
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const long long row = r0 + g + (h >= 2 ? 8 : 0);
            const int c = j * 8 + 2 * t + (h & 1);
            if (row < n && c < n_out) Y[row * n_out + c] = (acc[j][h] + bl[c]) * out_scale[c];
          }
        }
      }
    }
  }
}

// Shapes the fused kernel takes: at most FUSED_MAX_LAYERS layers, every fan-in
// and fan-out at most FUSED_WMAX; false otherwise (layer-by-layer kernels).
bool fused_net(const tam_mlp_s* M, FusedNet& f, size_t& smem) {
  const int L = (int)M->shapes.size();
  if (L < 1 || L > FUSED_MAX_LAYERS) return false;
  f = FusedNet{};
  f.L = L;
  int w = 0, b = 0;
  for (int l = 0; l < L; ++l) {
    const int K = M->shapes[l].first, N = M->shapes[l].second;
    if (K > FUSED_WMAX || N > FUSED_WMAX) return false;
    f.K[l] = K;
    f.N[l] = N;
    f.Kp[l] = (K + 15) & ~15;
    f.Np[l] = l + 1 < L ? (N + 15) & ~15 : (N + 7) & ~7;
    if (l > 0 && f.Kp[l] != f.Np[l - 1]) return false;  // chained widths
    f.wsm[l] = w;
    f.bsm[l] = b;
    f.woff[l] = M->offset[l];
    w += f.Np[l] * (f.Kp[l] + 8);
    b += f.Np[l];
  }
  f.w_elems = w;
  f.b_elems = b;
  smem = (((size_t)w * 2 + 15) & ~(size_t)15) + (size_t)b * 4;
  return smem <= 200 * 1024;
}

size_t dense_mma_smem(int N) {
  return sizeof(__nv_bfloat16) * ((size_t)((N + 7) & ~7) * MMA_LD + (size_t)MMA_ROWS * MMA_LD);
}

unsigned ew_grid(long long n) { return stride_grid(n, 256, 8); }
unsigned row_grid(long long n, int rows) {
  return (unsigned)std::min<long long>((n + rows - 1) / rows, (long long)sm_count() * 2);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <int MODE, bool TRANS, bool STD, int TM, int TN, int NG>
void dense_launch(const float* A, long long n, int K, int N, const float* W, const float* bias, const tam_mlp_s* M,
                  const float* aux, float* out, cudaStream_t s) {
  const int Kp = (K + 3) & ~3;
  const size_t smem = sizeof(float) * ((size_t)Kp * NG * TN + 2 * (size_t)ROWS * (Kp + 4));
  auto kern = dense_kernel<MODE, TRANS, STD, TM, TN, NG>;
  TAM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const unsigned grid = (unsigned)std::min<long long>((n + ROWS - 1) / ROWS, sm_count());
  kern<<<grid, DENSE_THREADS, smem, s>>>(A, n, K, N, W, bias, M->shift.p, M->scale.p, M->out_scale.p, aux, out,
                                         K % 4 == 0 && aligned16(A), N % 4 == 0 && aligned16(out));
  TAM_LAUNCH_CHECK();
}

template <typename TW, int MODE, bool TRANS, bool STD>
void dense(const float* A, long long n, int K, int N, const TW* W, const float* bias, const tam_mlp_s* M,
           const float* aux, float* out, cudaStream_t s) {
  if constexpr (std::is_same<TW, __nv_bfloat16>::value) {  // BF16 inference: tensor cores
    const size_t smem = dense_mma_smem(N);
    TAM_CUDA(cudaFuncSetAttribute(dense_mma_kernel<MODE, STD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const unsigned grid = std::min<unsigned>((unsigned)((n + MMA_ROWS - 1) / MMA_ROWS), (unsigned)sm_count() * 8u);
    dense_mma_kernel<MODE, STD><<<std::max(1u, grid), MMA_THREADS, smem, s>>>(A, n, K, N, W, bias, M->shift.p,
                                                                              M->scale.p, M->out_scale.p, out);
    TAM_LAUNCH_CHECK();
  } else if (N <= 4) {  // the smallest tile that holds the N outputs (padded columns are multiplied too)
    dense_launch<MODE, TRANS, STD, 1, 1, 4>(A, n, K, N, W, bias, M, aux, out, s);
  } else if (N <= 32) {
    dense_launch<MODE, TRANS, STD, 2, 4, 8>(A, n, K, N, W, bias, M, aux, out, s);
  } else if (N <= 64) {
    dense_launch<MODE, TRANS, STD, 4, 4, 16>(A, n, K, N, W, bias, M, aux, out, s);
  } else {
    dense_launch<MODE, TRANS, STD, 4, 8, 16>(A, n, K, N, W, bias, M, aux, out, s);
  }
}

template <int TK>
void weight_grad_tn(tam_mlp_s* M, int N, unsigned blocks, const float* H, const float* D, long long n, int K,
                    const float* shift, const float* scale, float* grad, cudaStream_t s) {
  float* part = M->part.p;
  unsigned int* t = M->ticket.p;
  const bool hv = K % 4 == 0 && aligned16(H) && TK >= 4, dv = N % 4 == 0 && aligned16(D);
  if (N <= 16)
    weight_grad_kernel<TK, 1><<<blocks, THREADS, 0, s>>>(H, D, n, K, N, shift, scale, part, hv, dv, grad, t);
  else if (N <= 64)
    weight_grad_kernel<TK, 4><<<blocks, THREADS, 0, s>>>(H, D, n, K, N, shift, scale, part, hv, dv, grad, t);
  else
    weight_grad_kernel<TK, 8><<<blocks, THREADS, 0, s>>>(H, D, n, K, N, shift, scale, part, hv, dv, grad, t);
  TAM_LAUNCH_CHECK();
}

// grad[0 .. K N + N) = the layer's weight and bias gradients (row count n)
void weight_grad(tam_mlp_s* M, const float* H, const float* D, long long n, int K, int N, const float* shift,
                 const float* scale, float* grad, cudaStream_t s) {
  const bool narrow = K <= 16 && N <= 16;
  const unsigned blocks = row_grid(n, WG_ROWS * (narrow ? wg_quarters(1, 1) : 1));
  const int m = K * N + N;
  if (K <= 16) weight_grad_tn<1>(M, N, blocks, H, D, n, K, shift, scale, grad, s);
  else if (K <= 64) weight_grad_tn<4>(M, N, blocks, H, D, n, K, shift, scale, grad, s);
  else weight_grad_tn<8>(M, N, blocks, H, D, n, K, shift, scale, grad, s);
  if (narrow && blocks <= WG_LAST) return;  // added up by its last block
  weight_grad_reduce_kernel<<<(m + 31) / 32, 256, 0, s>>>(M->part.p, (int)blocks, m, grad);
  TAM_LAUNCH_CHECK();
}

// FP32 inference takes the rows in pieces whose activations (two buffers of
// 67 MB) stay in L2 between layers and bound the workspace: 2^17 rows at width
// 128, more where the layers are narrower (2^17 at any width: 4M rows of a
// network of width 1 took 509 us, 353 without pieces).
constexpr long long PIECE = (1LL << 17) * 128;  // values

// keep: every layer's activations stay in M->act, layer after layer (training
// needs them for the backward pass); otherwise the layers alternate between
// the two ping-pong buffers.
void ensure_workspace(tam_mlp_s* M, long long n, bool keep, cudaStream_t s) {
  size_t need = 0;
  for (auto& sh : M->shapes) need += (size_t)n * sh.second;
  if (keep && need > M->act_cap) {
    M->act = DBuf<float>(need, s);
    M->act_cap = need;
  }
  size_t dneed = (size_t)n * std::max(M->width, M->n_out);
  if (dneed > M->dcap) {
    M->dbuf[0] = DBuf<float>(dneed, s);
    M->dbuf[1] = DBuf<float>(dneed, s);
    M->dcap = dneed;
  }
}

// n rows through the network (workspace sized); Y: where the last layer
// writes (NULL: M->act, after the other layers' activations).  Returns the
// output pointer ([n x n_out]).
template <typename TW>
float* forward(tam_mlp_s* M, const float* X, long long n, const TW* theta, float* Y, cudaStream_t s) {
  const float* in = X;
  float* o = Y ? M->dbuf[0].p : M->act.p;
  const int L = (int)M->shapes.size();
  for (int l = 0; l < L; ++l) {
    const int a = M->shapes[l].first, b = M->shapes[l].second;
    const TW* W = theta + M->offset[l];
    // bias is FP32 in both precisions: read from the master copy
    const float* bias = M->theta.p + M->offset[l] + (long long)a * b;
    const bool last = l == L - 1;
    if (last && Y) o = Y;
    if (l == 0) {
      if (last) dense<TW, 2, false, true>(in, n, a, b, W, bias, M, nullptr, o, s);
      else dense<TW, 1, false, true>(in, n, a, b, W, bias, M, nullptr, o, s);
    } else {
      if (last) dense<TW, 2, false, false>(in, n, a, b, W, bias, M, nullptr, o, s);
      else dense<TW, 1, false, false>(in, n, a, b, W, bias, M, nullptr, o, s);
    }
    in = o;
    o = Y ? M->dbuf[(l + 1) & 1].p : o + (size_t)n * b;
  }
  return const_cast<float*>(in);
}

double loss_and_grad(tam_mlp_s* M, const float* X, const float* Y, long long n, cudaStream_t s) {
  ensure_workspace(M, n, true, s);
  float* pred = forward<float>(M, X, n, M->theta.p, nullptr, s);
  const int L = (int)M->shapes.size();
  if (!M->part.p) {
    size_t most = 0;
    for (auto& sh : M->shapes) most = std::max(most, (size_t)sh.first * sh.second + sh.second);
    M->part = DBuf<float>(most * sm_count() * 2, s);
  }
  GridReduce gr{reinterpret_cast<double*>(M->red.p), M->ticket.p};
  DBuf<double> loss(1, s);
  float* d = M->dbuf[0].p;
  float* d2 = M->dbuf[1].p;
  loss_grad_kernel<<<ew_grid(n * M->n_out), 256, 0, s>>>(pred, Y, n, M->n_out, M->out_scale.p, d, gr, loss.p);
  TAM_LAUNCH_CHECK();
  // activations of layer l are at act + sum_{l'<l} n * b_l'
  std::vector<float*> acts(L);
  {
    float* o = M->act.p;
    for (int l = 0; l < L; ++l) {
      acts[l] = o;
      o += (size_t)n * M->shapes[l].second;
    }
  }
  for (int l = L - 1; l >= 0; --l) {
    const int a = M->shapes[l].first, b = M->shapes[l].second;
    const float* Hin = l == 0 ? X : acts[l - 1];
    weight_grad(M, Hin, d, n, a, b, l == 0 ? M->shift.p : nullptr, l == 0 ? M->scale.p : nullptr,
                M->grad.p + M->offset[l], s);
    if (l > 0) {
      // d_prev = (d W^T) * (1 - H_{l-1}^2)
      dense<float, 3, true, false>(d, n, b, a, M->theta.p + M->offset[l], nullptr, M, acts[l - 1], d2, s);
      std::swap(d, d2);
    }
  }
  return read_back_double(loss.p, s);
}

void ensure_bf16(tam_mlp_s* M, cudaStream_t s) {
  if (!M->theta16_valid) {
    to_bf16_kernel<<<ew_grid(M->n_par), 256, 0, s>>>(M->theta.p, M->theta16.p, M->n_par);
    TAM_LAUNCH_CHECK();
    M->theta16_valid = true;
  }
}

}  // namespace

// bf16: 0 FP32 layer by layer; 1 BF16 tensor cores, the whole network in one
// kernel when its shapes allow (else layer by layer); 2 BF16 layer by layer.
void mlp_forward_device(tam_mlp_s* M, long long n, const float* X, float* Y, int bf16, cudaStream_t s) {
  NvtxRange nvtx("tam: network inference");
  FusedNet f;
  size_t smem = 0;
  if (bf16 == 1 && fused_net(M, f, smem)) {
    ensure_bf16(M, s);
    if (n > 0) {
      TAM_CUDA(cudaFuncSetAttribute(mlp_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      const long long tiles = (n + 15) / 16;
      const unsigned grid = (unsigned)std::min<long long>((tiles + FUSED_WARPS - 1) / FUSED_WARPS,
                                                          (long long)sm_count() * 2);
      mlp_fused_kernel<<<std::max(1u, grid), FUSED_WARPS * 32, smem, s>>>(
          X, n, f, M->theta16.p, M->theta.p, M->shift.p, M->scale.p, M->out_scale.p, Y);
      TAM_LAUNCH_CHECK();
    }
    return;
  }
  if (bf16) ensure_bf16(M, s);
  // The BF16 layers take all rows at once: a piece of 2^17 rows is 1.7 waves of
  // their tiles (1M rows of 8-128-128-128-3: 3.05 ms in pieces, 1.89 without).
  const long long piece = bf16 ? std::max(n, 1LL) : PIECE / M->width;
  ensure_workspace(M, std::min(n, piece), false, s);
  // a piece's outputs over the inputs of later ones (a caller's Y may overlap
  // its X): all outputs aside first
  DBuf<float> aside;
  float* out = Y;
  if (n > piece && std::less<const float*>()(X, Y + n * M->n_out) && std::less<const float*>()(Y, X + n * M->n_in)) {
    aside = DBuf<float>((size_t)n * M->n_out, s);
    out = aside.p;
  }
  for (long long r = 0; r < n; r += piece) {
    const long long m = std::min(piece, n - r);
    const float* Xr = X + r * M->n_in;
    float* Yr = out + r * M->n_out;
    if (bf16) forward<__nv_bfloat16>(M, Xr, m, M->theta16.p, Yr, s);
    else forward<float>(M, Xr, m, M->theta.p, Yr, s);
  }
  if (aside.p) TAM_CUDA(cudaMemcpyAsync(Y, aside.p, sizeof(float) * (size_t)n * M->n_out, cudaMemcpyDeviceToDevice, s));
}
int mlp_n_in(tam_mlp_s* M) { return M->n_in; }
int mlp_n_out(tam_mlp_s* M) { return M->n_out; }

}  // namespace tam

using namespace tam;

namespace {
template <class F>
int guarded_mlp(F&& f) {
  try {
    set_last_error("");
    return f();
  } catch (const Error& e) {
    set_last_error(e.what());
    return e.code;
  } catch (const std::exception& e) {
    set_last_error(e.what());
    return TAM_ERR_INTERNAL;
  }
}
}  // namespace

extern "C" {

int tam_mlp_create(int n_in, int width, int depth, int n_out, unsigned long long seed, tam_mlp* out) {
  return guarded_mlp([&] {
    TAM_CHECK(out && n_in >= 1 && n_in <= 128 && width >= 1 && width <= 128 && depth >= 1 && depth <= 16 &&
                  n_out >= 1 && n_out <= 128,
              TAM_ERR_INVALID_ARG, "tam_mlp_create: sizes out of range (1..128, depth 1..16)");
    auto M = new tam_mlp_s();
    cudaStream_t s = nullptr;
    M->n_in = n_in;
    M->width = width;
    M->depth = depth;
    M->n_out = n_out;
    std::vector<int> dims{n_in};
    for (int i = 0; i < depth; ++i) dims.push_back(width);
    dims.push_back(n_out);
    long long off = 0;
    for (size_t l = 0; l + 1 < dims.size(); ++l) {
      M->shapes.emplace_back(dims[l], dims[l + 1]);
      M->offset.push_back(off);
      off += (long long)dims[l] * dims[l + 1] + dims[l + 1];
    }
    M->n_par = off;
    M->theta = DBuf<float>(off, s);
    M->grad = DBuf<float>(off, s);
    M->m1 = DBuf<float>(off, s);
    M->m2 = DBuf<float>(off, s);
    M->theta16 = DBuf<__nv_bfloat16>(off, s);
    M->m1.zero();
    M->m2.zero();
    for (size_t l = 0; l < M->shapes.size(); ++l)
      init_params_kernel<<<64, 256, 0, s>>>(M->theta.p, M->offset[l], M->shapes[l].first, M->shapes[l].second,
                                            seed);
    TAM_LAUNCH_CHECK();
    M->shift = DBuf<float>(n_in, s);
    M->scale = DBuf<float>(n_in, s);
    M->out_scale = DBuf<float>(n_out, s);
    std::vector<float> zero(n_in, 0.f), one(std::max(n_in, n_out), 1.f);
    TAM_CUDA(cudaMemcpy(M->shift.p, zero.data(), 4 * n_in, cudaMemcpyHostToDevice));
    TAM_CUDA(cudaMemcpy(M->scale.p, one.data(), 4 * n_in, cudaMemcpyHostToDevice));
    TAM_CUDA(cudaMemcpy(M->out_scale.p, one.data(), 4 * n_out, cudaMemcpyHostToDevice));
    M->red = DBuf<double>((size_t)sm_count() * 8 * 2, s);
    M->ticket = DBuf<unsigned int>(1, s);
    M->ticket.zero();
    TAM_CUDA(cudaStreamSynchronize(s));
    *out = M;
    return TAM_OK;
  });
}

int tam_mlp_destroy(tam_mlp M) {
  return guarded_mlp([&] {
    delete M;
    return TAM_OK;
  });
}

int tam_mlp_info(tam_mlp M, long long* n_params, int* n_layers) {
  return guarded_mlp([&] {
    TAM_CHECK(M, TAM_ERR_INVALID_ARG, "tam_mlp_info: NULL handle");
    if (n_params) *n_params = M->n_par;
    if (n_layers) *n_layers = (int)M->shapes.size();
    return TAM_OK;
  });
}

int tam_mlp_set_normalization(tam_mlp M, const float* shift_host, const float* scale_host,
                              const float* out_scale_host) {
  return guarded_mlp([&] {
    TAM_CHECK(M && shift_host && scale_host && out_scale_host, TAM_ERR_INVALID_ARG, "tam_mlp_set_normalization: NULL");
    TAM_CUDA(cudaMemcpy(M->shift.p, shift_host, 4 * M->n_in, cudaMemcpyHostToDevice));
    TAM_CUDA(cudaMemcpy(M->scale.p, scale_host, 4 * M->n_in, cudaMemcpyHostToDevice));
    TAM_CUDA(cudaMemcpy(M->out_scale.p, out_scale_host, 4 * M->n_out, cudaMemcpyHostToDevice));
    return TAM_OK;
  });
}

int tam_mlp_get_params(tam_mlp M, float* theta_host) {
  return guarded_mlp([&] {
    TAM_CHECK(M && theta_host, TAM_ERR_INVALID_ARG, "tam_mlp_get_params: NULL");
    TAM_CUDA(cudaMemcpy(theta_host, M->theta.p, 4 * (size_t)M->n_par, cudaMemcpyDeviceToHost));
    return TAM_OK;
  });
}

int tam_mlp_set_params(tam_mlp M, const float* theta_host) {
  return guarded_mlp([&] {
    TAM_CHECK(M && theta_host, TAM_ERR_INVALID_ARG, "tam_mlp_set_params: NULL");
    TAM_CUDA(cudaMemcpy(M->theta.p, theta_host, 4 * (size_t)M->n_par, cudaMemcpyHostToDevice));
    M->theta16_valid = false;
    return TAM_OK;
  });
}

int tam_mlp_forward(tam_mlp M, long long n, const float* X, float* Y, int bf16, void* stream) {
  return guarded_mlp([&] {
    TAM_CHECK(M && X && Y && n >= 0, TAM_ERR_INVALID_ARG, "tam_mlp_forward: bad argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (n == 0) return TAM_OK;
    mlp_forward_device(M, n, X, Y, bf16, s);
    return TAM_OK;
  });
}

int tam_mlp_loss_grad(tam_mlp M, long long n, const float* X, const float* Yt, double* loss_host, float* grad_host,
                      void* stream) {
  return guarded_mlp([&] {
    TAM_CHECK(M && X && Yt && n > 0, TAM_ERR_INVALID_ARG, "tam_mlp_loss_grad: bad argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    double L = loss_and_grad(M, X, Yt, n, s);
    if (loss_host) *loss_host = L;
    if (grad_host) {
      TAM_CUDA(cudaMemcpyAsync(grad_host, M->grad.p, 4 * (size_t)M->n_par, cudaMemcpyDeviceToHost, s));
      TAM_CUDA(cudaStreamSynchronize(s));
    }
    return TAM_OK;
  });
}

int tam_mlp_train_step(tam_mlp M, long long n, const float* X, const float* Yt, float lr, double* loss_host,
                       void* stream) {
  return guarded_mlp([&] {
    TAM_CHECK(M && X && Yt && n > 0 && lr > 0.f, TAM_ERR_INVALID_ARG, "tam_mlp_train_step: bad argument");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    double L = loss_and_grad(M, X, Yt, n, s);
    M->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)M->adam_t), c2 = 1.f - powf(b2, (float)M->adam_t);
    adam_kernel<<<ew_grid(M->n_par), 256, 0, s>>>(M->theta.p, M->grad.p, M->m1.p, M->m2.p, M->n_par, lr, b1, b2,
                                                  1e-8f, c1, c2);
    TAM_LAUNCH_CHECK();
    M->theta16_valid = false;
    if (loss_host) *loss_host = L;
    return TAM_OK;
  });
}

}  // extern "C"
