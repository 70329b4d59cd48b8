// Assembly of the thermoelastic system (paper Sec. 3, Eq. wf_elastic, steady,
// traction free, with the Dirichlet condition of Eq. u-dbc).
//
//   K[(a,i),(b,j)] = int lambda d_i phi_a d_j phi_b + mu d_j phi_a d_i phi_b
//                        + mu delta_ij grad phi_a . grad phi_b
//   f[(a,i)]       = int (3 lambda + 2 mu) alpha (T_h - T_ref) d_i phi_a + int f_h,i phi_a
//
// (isotropic C, eps_T = alpha (T - T_ref) I, so C:eps_T = (3 lambda + 2 mu) alpha (T - T_ref) I).
//
// Pipeline: cell-node incidence (count, scan, fill) -> block-CSR pattern, one
// warp per node (gather, bitonic sort, unique) -> element kernels with FP64
// atomic scatter -> Dirichlet rows.  Dirichlet couplings never enter the
// pattern: an element block K_ab with a free row a and a Dirichlet column b
// is lifted straight into the load (f_a -= K_ab u_b) and rows of Dirichlet
// nodes become identity rows -- the symmetric elimination of Eq. u-dbc.
#include <cstdlib>

#include <atomic>

#include "handles.cuh"
#include "tet.cuh"

namespace tam {
namespace {

constexpr int PAT_WARPS = 4;
constexpr int PAT_CAP = 1024;  // candidate node ids per row (incident cells x nodes per cell + 1)

__global__ void validate_kernel(const int* __restrict__ cells, long long n_entries, int npc, int n_nodes,
                                const int* __restrict__ mat, int n_cells, int n_mat, int* __restrict__ bad) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n_entries) {
    int v = cells[t];
    if (v < 0 || v >= n_nodes) atomicExch(bad, 1);
  }
  if (mat && t < n_cells) {
    int m = mat[t];
    if (m < 0 || m >= n_mat) atomicExch(bad, 2);
  }
}

__global__ void incidence_count_kernel(const int* __restrict__ cells, long long n_entries, int* __restrict__ cnt) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n_entries) atomicAdd(&cnt[cells[t]], 1);
}

__global__ void incidence_fill_kernel(const int* __restrict__ cells, long long n_entries, int npc,
                                      const int* __restrict__ ptr, int* __restrict__ cursor,
                                      int* __restrict__ inc) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_entries) return;
  int v = cells[t];
  inc[ptr[v] + atomicAdd(&cursor[v], 1)] = (int)(t / npc);
}

// One warp per node: candidate columns = self + all nodes of incident cells,
// minus Dirichlet nodes (a Dirichlet row keeps only its diagonal).
// Open-addressing insert of node j into a table of hsz (a power of two)
// slots; true if j was new.  The table has room for every candidate.
__device__ __forceinline__ bool pat_insert(int* tab, int j, int hsz) {
  const unsigned mask = (unsigned)hsz - 1u;
  unsigned h = ((unsigned)j * 2654435761u) & mask;
  const int key = j + 1;
  for (int probe = 0; probe < hsz; ++probe) {
    const int prev = atomicCAS(&tab[h], 0, key);
    if (prev == 0) return true;
    if (prev == key) return false;
    h = (h + 1) & mask;
  }
  return false;
}

template <bool FILL>
__global__ void __launch_bounds__(PAT_WARPS * 32)
pattern_kernel(int n_nodes, int npc, const int* __restrict__ cells, const int* __restrict__ inc_ptr,
               const int* __restrict__ inc, const unsigned char* __restrict__ dmask,
               int* __restrict__ row_cnt, const int* __restrict__ row_ptr, int* __restrict__ col_idx,
               int* __restrict__ overflow, int* __restrict__ big_list = nullptr, int big_cap = 0) {
  __shared__ int buf_all[PAT_WARPS][PAT_CAP];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * PAT_WARPS + wid;
  if (i >= n_nodes) return;
  int* buf = buf_all[wid];
  const bool di = dmask[i] != 0;
  const int s = inc_ptr[i], e = inc_ptr[i + 1];
  const int n_cand = di ? 1 : 1 + (e - s) * npc;
  if (n_cand > PAT_CAP) {
    if (lane == 0) {
      // rows beyond the shared-memory capacity: to pattern_big_kernel when a
      // list is given (it writes the count), else reported
      const int k = big_list ? atomicAdd(overflow + 1, 1) : -1;
      if (k >= 0 && k < big_cap) big_list[k] = i;
      else atomicExch(overflow, 1);
      if (row_cnt) row_cnt[i] = FILL ? 0 : 1;
    }
    return;
  }
  // distinct candidates through a shared-memory hash set (open addressing,
  // keys stored + 1, 0 empty), so that only the row's distinct columns --
  // ~15 of ~97 candidates for a P1 row, ~60 of ~400 for P2 -- are sorted
  int hsz = 32;
  while (hsz < 2 * n_cand && hsz < PAT_CAP) hsz <<= 1;
  for (int t = lane; t < hsz; t += 32) buf[t] = 0;
  __syncwarp();
  int ins = lane == 0 ? (pat_insert(buf, i, hsz) ? 1 : 0) : 0;
  if (!di) {
    for (int t = lane; t < (e - s) * npc; t += 32) {
      const int c = inc[s + t / npc];
      const int j = cells[(size_t)c * npc + (t % npc)];
      if (!dmask[j]) ins += pat_insert(buf, j, hsz) ? 1 : 0;
    }
  }
  __syncwarp();
  const int cnt = warp_sum_i(ins);
  int base = 0;  // compact the occupied slots (decoded) to the front
  for (int t0 = 0; t0 < hsz; t0 += 32) {
    const int v = buf[t0 + lane];
    const unsigned m = __ballot_sync(0xffffffffu, v != 0);
    __syncwarp();
    if (v != 0) buf[base + __popc(m & ((1u << lane) - 1u))] = v - 1;
    base += __popc(m);
    __syncwarp();
  }
  const int n2 = next_pow2(cnt);
  for (int t = cnt + lane; t < n2; t += 32) buf[t] = 0x7fffffff;
  __syncwarp();
  warp_bitonic_sort<false>(buf, nullptr, n2);
  __syncwarp();
  if (!FILL) {
    if (lane == 0) row_cnt[i] = cnt;
  } else {
    const int r0 = row_ptr[i];
    for (int t = lane; t < cnt; t += 32) col_idx[r0 + t] = buf[t];
    if (lane == 0 && row_cnt) row_cnt[i] = cnt;
  }
}

// Candidate count of each row (upper bound of its pattern length): self plus
// the nodes of its incident cells; 1 for a Dirichlet row.  A row with more
// candidates than the warp builder's shared memory holds (PAT_CAP) gets three
// times that room: its candidates are sorted in global memory in the upper
// two thirds (padded to a power of two) and its columns written to the front.
__global__ void pattern_bound_kernel(int n_nodes, int npc, const int* __restrict__ inc_ptr,
                                     const unsigned char* __restrict__ dmask, int* __restrict__ bound) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  const int b = dmask[i] ? 1 : 1 + (inc_ptr[i + 1] - inc_ptr[i]) * npc;
  bound[i] = b > PAT_CAP ? 3 * b : b;
}

// One block per row whose candidates exceed PAT_CAP (the list built by
// pattern_kernel): candidates gathered into the row's scratch range, padded
// with INT_MAX to a power of two, bitonic-sorted by the block in global
// memory, then the distinct ones compacted to the front of the range
// (block-wide scan of the keep flags) and the count written to row_cnt.
constexpr int BIG_THREADS = 256;

__global__ void __launch_bounds__(BIG_THREADS)
pattern_big_kernel(const int* __restrict__ list, int npc, const int* __restrict__ cells,
                   const int* __restrict__ inc_ptr, const int* __restrict__ inc, const unsigned char* __restrict__ dmask,
                   const int* __restrict__ bptr, int* __restrict__ tmp, int* __restrict__ row_cnt) {
  __shared__ int wsum[BIG_THREADS / 32];
  __shared__ int carry;
  const int i = list[blockIdx.x];
  const int s = inc_ptr[i], e = inc_ptr[i + 1];
  const int n = 1 + (e - s) * npc;
  int n2 = 1;
  while (n2 < n) n2 <<= 1;
  int* cand = tmp + bptr[i] + n;  // [n, n + n2) of the 3n range
  int* outp = tmp + bptr[i];
  for (int t = threadIdx.x; t < n2; t += BIG_THREADS) {
    int v = 0x7fffffff;
    if (t == 0) v = i;
    else if (t < n) {
      const int j = cells[(size_t)inc[s + (t - 1) / npc] * npc + (t - 1) % npc];
      if (!dmask[j]) v = j;
    }
    cand[t] = v;
  }
  __syncthreads();
  for (int k = 2; k <= n2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < n2; t += BIG_THREADS) {
        const int x = t ^ j;
        if (x > t) {
          const int a = cand[t], b = cand[x];
          if ((a > b) == ((t & k) == 0)) {
            cand[t] = b;
            cand[x] = a;
          }
        }
      }
      __syncthreads();
    }
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int base = 0; base < n2; base += BIG_THREADS) {
    const int t = base + threadIdx.x;
    const int v = t < n2 ? cand[t] : 0x7fffffff;
    const int keep = (v != 0x7fffffff) && (t == 0 || cand[t - 1] != v);
    int x = keep;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    int off = carry;
    for (int w = 0; w < wid; ++w) off += wsum[w];
    if (keep) outp[off + x - 1] = v;
    __syncthreads();
    if (threadIdx.x == BIG_THREADS - 1) carry = off + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) row_cnt[i] = carry;
}

// Rows written at their bound offsets in tmp, packed into col_idx (warp per row).
__global__ void pattern_pack_kernel(int n_nodes, const int* __restrict__ bptr, const int* __restrict__ tmp,
                                    const int* __restrict__ row_ptr, int* __restrict__ col_idx) {
  const int i = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= n_nodes) return;
  const int src = bptr[i], dst = row_ptr[i], cnt = row_ptr[i + 1] - dst;
  for (int t = lane; t < cnt; t += 32) col_idx[dst + t] = tmp[src + t];
}

__device__ __forceinline__ void lame(double E, double nu, double& lam, double& mu) {
  mu = E / (2.0 * (1.0 + nu));
  lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu));
}

struct AsmArgs {
  const double* coords;
  const int* cells;
  const int* mat;
  const double* props;
  const double* T;
  double T_ref;
  const double* body;
  const unsigned char* dmask;
  const double* ud;
  const int* row_ptr;
  const int* col_idx;
  double* vals;
  double* rhs;
  int n_cells;
  int* bad_cell;
  int loads_only;  // 1: only the load vector (K of this mesh exists already)
  // deterministic mode (non-null): every element block and load goes to its
  // own slot, ck[((c npc + a) npc + b) 9 + e] and cf[(c npc + a) 3 + d], and
  // gather_kernel sums them per node in cell order (no atomics)
  double* ck = nullptr;
  double* cf = nullptr;
  int npc = 0;
};

// Whether the element blocks go into K's values: not in the deterministic
// mode (slots of its own) nor for the loads alone.
__device__ __forceinline__ bool fills_values(const AsmArgs& A) { return !A.ck && !A.loads_only; }

// Scatter one 3x3 block (row node na, col node nb; local a, b of cell c) or
// lift it into the load; in deterministic mode store it in its slot.
__device__ __forceinline__ void scatter_block(const AsmArgs& A, int c, int a, int b, int na, int nb,
                                              const double k[9]) {
  if (A.ck) {
    double* dst = A.ck + (((size_t)c * A.npc + a) * A.npc + b) * 9;
#pragma unroll
    for (int e = 0; e < 9; ++e) dst[e] = k[e];
    return;
  }
  if (A.dmask[nb]) {
    if (A.ud) {
      const double* u = A.ud + 3 * (size_t)nb;
      for (int r = 0; r < 3; ++r)
        atomicAdd(&A.rhs[3 * (size_t)na + r], -(k[3 * r] * u[0] + k[3 * r + 1] * u[1] + k[3 * r + 2] * u[2]));
    }
    return;
  }
  if (A.loads_only) return;
  int slot = bsearch_i32(A.col_idx, A.row_ptr[na], A.row_ptr[na + 1], nb);
  double* dst = A.vals + (size_t)slot * 9;
#pragma unroll
  for (int e = 0; e < 9; ++e) atomicAdd(dst + e, k[e]);
}

// Where the 3x3 block k (row na, column nb; local a, b of cell c) goes: its
// slot in K's values, or -1 when it went elsewhere (the deterministic mode's
// own slot, the load of a prescribed column) or nowhere.  fixed: nb is a
// Dirichlet node.
__device__ __forceinline__ int block_slot(const AsmArgs& A, int c, int a, int b, int na, int nb, bool fixed,
                                          const double (&k)[9]) {
  if (fixed || !fills_values(A)) {
    scatter_block(A, c, a, b, na, nb, k);
    return -1;
  }
  return bsearch_i32(A.col_idx, A.row_ptr[na], A.row_ptr[na + 1], nb);
}

// A warp's 32 blocks (lane l's: k, to slot[l] of K's values; slot < 0: none)
// added as one run of 32 x 9 values through the warp's shared memory, so that
// a request covers neighbouring values of a block.  Called by the whole warp.
__device__ __forceinline__ void scatter_run(double* __restrict__ vals, const double (&k)[9], int my_slot, double* out,
                                            int* slot, int lane) {
#pragma unroll
  for (int e = 0; e < 9; ++e) out[lane * 9 + e] = k[e];
  slot[lane] = my_slot;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const int idx = q * 32 + lane, cl = idx / 9;
    if (slot[cl] >= 0) atomicAdd(vals + (size_t)slot[cl] * 9 + (idx - cl * 9), out[idx]);
  }
  __syncwarp();
}

// P1: constant gradients, one thread per cell, a warp's blocks scattered as
// runs.  Bound by the FP64 pipe (about 270 operations a cell: K_ab is formed
// for a <= b only, with K_aa's symmetry and the trace term in one multiply-add
// per diagonal entry) and by the 144 atomic additions a cell.  6,291,456 cells:
// 5.7 -> 4.6 ms.
constexpr int P1_THREADS = 128;

__global__ void __launch_bounds__(P1_THREADS) assemble_p1_kernel(AsmArgs A) {
  __shared__ double s_out[P1_THREADS / 32][32 * 9];
  __shared__ int s_slot[P1_THREADS / 32][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long cl = (long long)blockIdx.x * P1_THREADS + threadIdx.x;
  const int c = (int)min(cl, (long long)A.n_cells - 1);  // idle lanes repeat the last cell, unscattered
  int v[4];
  if ((reinterpret_cast<size_t>(A.cells) & 15) == 0) {  // the caller's array need not be
    const int4 q = reinterpret_cast<const int4*>(A.cells)[c];
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  } else {
    for (int a = 0; a < 4; ++a) v[a] = A.cells[4 * (size_t)c + a];
  }
  double g[4][3], vol;
  bool ok = tet_geometry(A.coords, v, g, vol);
  if (!ok) {
    atomicExch(A.bad_cell, 1);
    vol = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int d = 0; d < 3; ++d) g[a][d] = 0.0;
  }
  ok = ok && cl < A.n_cells;
  const int m = A.mat[c];
  double lam, mu;
  lame(A.props[3 * m], A.props[3 * m + 1], lam, mu);
  bool fixed[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) fixed[a] = A.dmask[v[a]] != 0;
  // the loads alone need no stiffness unless a prescribed displacement is
  // lifted: a warp without Dirichlet nodes skips it, the others the pairs that
  // no lane needs (786,432 cells, one face of the box held: 677 -> 320 us; each
  // pair of every cell otherwise)
  const bool lifted = A.ud && (fixed[0] || fixed[1] || fixed[2] || fixed[3]);
  if (!A.loads_only || __any_sync(0xffffffffu, lifted)) {
    // K_ab[i][j] = lg_a[i] g_b[j] + mg_a[j] g_b[i] + delta_ij (mg_a . g_b),
    // lg = lam vol g, mg = mu vol g; K_ba = K_ab^T
    const double lv = lam * vol, mv = mu * vol;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      double lg[3], mg[3], sg[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        lg[i] = lv * g[a][i];
        mg[i] = mv * g[a][i];
        sg[i] = lg[i] + mg[i];
      }
#pragma unroll
      for (int b = a; b < 4; ++b) {
        const bool ab = ok && !fixed[a] && (!A.loads_only || (fixed[b] && A.ud));
        const bool ba = b != a && ok && !fixed[b] && (!A.loads_only || (fixed[a] && A.ud));
        if (A.loads_only && !__any_sync(0xffffffffu, ab || ba)) continue;
        const double mgg = fma(mg[0], g[b][0], fma(mg[1], g[b][1], mg[2] * g[b][2]));
        double k[9];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            if (i == j) k[3 * i + j] = fma(sg[i], g[b][i], mgg);
            else if (a != b) k[3 * i + j] = fma(lg[i], g[b][j], mg[j] * g[b][i]);
            else k[3 * i + j] = i < j ? sg[i] * g[a][j] : k[3 * j + i];
          }
        int s = -1;
        if (ab) s = block_slot(A, c, a, b, v[a], v[b], fixed[b], k);
        if (fills_values(A)) scatter_run(A.vals, k, s, s_out[wid], s_slot[wid], lane);
        if (b != a) {
          const double kt[9] = {k[0], k[3], k[6], k[1], k[4], k[7], k[2], k[5], k[8]};
          s = -1;
          if (ba) s = block_slot(A, c, b, a, v[b], v[a], fixed[a], kt);
          if (fills_values(A)) scatter_run(A.vals, kt, s, s_out[wid], s_slot[wid], lane);
        }
      }
    }
  }
  if (!ok) return;
  // thermal: int (T_h - T_ref) d_i phi_a = vol (mean vertex T - T_ref) g_a[i]
  const double alpha = A.props[3 * m + 2];
  double cT = 0.0;
  if (A.T) cT = (3.0 * lam + 2.0 * mu) * alpha * vol * (0.25 * (A.T[v[0]] + A.T[v[1]] + A.T[v[2]] + A.T[v[3]]) - A.T_ref);
  double fsum[3] = {0, 0, 0};
  if (A.body)
    for (int b = 0; b < 4; ++b)
      for (int d = 0; d < 3; ++d) fsum[d] += A.body[3 * (size_t)v[b] + d];
  for (int a = 0; a < 4; ++a) {
    const int na = v[a];
    if (fixed[a]) continue;
    // body: int f_h phi_a = vol/20 (sum_b f_b + f_a) (P1 mass matrix vol (1 + delta_ab)/20)
    for (int i = 0; i < 3; ++i) {
      double f = cT * g[a][i];
      if (A.body) f += vol / 20.0 * (fsum[i] + A.body[3 * (size_t)na + i]);
      if (A.cf) A.cf[((size_t)c * 4 + a) * 3 + i] = f;
      else atomicAdd(&A.rhs[3 * (size_t)na + i], f);
    }
  }
}

// P2 reference integrals / |K| (affine cells).  With grad phi_a =
// (4 lambda_a - 1) G_a on vertices and 4 (lambda_q G_p + lambda_p G_q) on the
// edge (p, q), a P2 stiffness block is a sum of at most four of the P1 blocks
// B_kl = vol (lam G_k G_l^T + mu G_l G_k^T + mu (G_k . G_l) I):
//   vertex a, vertex b:  0.6 B_aa, or -0.2 B_ab
//   vertex a, edge pq:   c_q B_ap + c_p B_aq, c_k = int (4 l_a - 1) 4 l_k = 0.6 (k = a) or -0.2
//   edge pq, edge rs:    d_qs B_pr + d_qr B_ps + d_ps B_qr + d_pr B_qs, d_kl = int 16 l_k l_l = 1.6 (k = l) or 0.8
// The loads contract nodal values with int phi_a phi_b (body) and
// int phi_c lambda_k (thermal).  All exact for the polynomial degrees involved.
__constant__ int c_edge[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};

// int phi_a phi_b / |K| of two P2 functions
__device__ __forceinline__ double p2_mass(int a, int b) {
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  if (hi < 4) return lo == hi ? 6.0 / 420.0 : 1.0 / 420.0;
  const int r = c_edge[hi - 4][0], s = c_edge[hi - 4][1];
  if (lo < 4) return (lo == r || lo == s) ? -4.0 / 420.0 : -6.0 / 420.0;
  if (lo == hi) return 32.0 / 420.0;
  const int p = c_edge[lo - 4][0], q = c_edge[lo - 4][1];
  return (p == r || p == s || q == r || q == s) ? 16.0 / 420.0 : 8.0 / 420.0;
}

// int phi_c lambda_k / |K|
__device__ __forceinline__ double p2_moment(int c, int k) {
  if (c < 4) return c == k ? 0.0 : -1.0 / 60.0;
  return (c_edge[c - 4][0] == k || c_edge[c - 4][1] == k) ? 4.0 / 60.0 : 2.0 / 60.0;
}

// P2: 32 cells per block, one per lane; the block's warps share out the 55
// node pairs a <= b.  The FP64 pipe (2 lanes per cycle and SM) and the atomic
// scatter bound this kernel: the contraction of the ten P1 blocks takes about
// 2,000 FP64 operations a cell where the 4-point (stiffness) and 11-point
// (loads) quadrature took 13,000, every lane works (one entry for 32 cells at a time,
// table indices warp-uniform, per-cell quantities in shared memory by
// [quantity][cell]), and a warp's 32 blocks are scattered as one run of
// 32 x 9 values, so that a request covers 9 neighbouring values of a block
// (3 sectors) instead of one value of 32 blocks (32 sectors).  15.3 -> 1.4 ms
// on 331,776 cells (the operations alone: 1.1 ms at the measured FP64 rate);
// the whole assembly 18.0 -> 3.8 ms.
constexpr int P2_WARPS = 8, P2_CELLS = 32;

struct P2Tile {
  double B[10][9][32];             // P1 blocks, k <= l, row-major
  double G[4][3][32];              // gradients of the barycentric coordinates
  double f[10][3][32];             // nodal body force
  double mu[5][32];                // int (T_h - T_ref) lambda_k / |K|, then int (T_h - T_ref) / |K|
  double vol[32];
  double out[P2_WARPS][32][9];     // a warp's 32 blocks on their way out
  int slot[P2_WARPS][32];
  int v[10][32];
  unsigned char dm[10][32], ok[32];
};

__global__ void __launch_bounds__(P2_WARPS * 32) assemble_p2_kernel(AsmArgs A) {
  extern __shared__ __align__(16) unsigned char p2_smem[];
  P2Tile& S = *reinterpret_cast<P2Tile*>(p2_smem);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long c0 = (long long)blockIdx.x * P2_CELLS;
  const int c = (int)min(c0 + lane, (long long)A.n_cells - 1);  // idle lanes repeat the last cell, unscattered
  for (int t = threadIdx.x; t < 320; t += P2_WARPS * 32) {
    const int cl = t / 10;
    S.v[t - cl * 10][cl] = A.cells[min(c0 + cl, (long long)A.n_cells - 1) * 10 + (t - cl * 10)];
  }
  __syncthreads();
  const int m = A.mat[c];
  double lam, mu;
  lame(A.props[3 * m], A.props[3 * m + 1], lam, mu);
  const double alpha = A.props[3 * m + 2];
  if (wid == 0) {
    int v[4];
    for (int a = 0; a < 4; ++a) v[a] = S.v[a][lane];
    double g[4][3], vol;
    const bool good = tet_geometry(A.coords, v, g, vol);
    if (!good) atomicExch(A.bad_cell, 1);
    S.ok[lane] = good && c0 + lane < A.n_cells;
    if (good) {
      S.vol[lane] = vol;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int d = 0; d < 3; ++d) S.G[k][d][lane] = g[k][d];
    }
  } else if (wid == 1) {
    double sum = 0.0, mk[4] = {0.0, 0.0, 0.0, 0.0};
    if (A.T)
#pragma unroll
      for (int a = 0; a < 10; ++a) {
        const double t = A.T[S.v[a][lane]] - A.T_ref;
        sum = fma(a < 4 ? -0.05 : 0.2, t, sum);
#pragma unroll
        for (int k = 0; k < 4; ++k) mk[k] = fma(p2_moment(a, k), t, mk[k]);
      }
#pragma unroll
    for (int k = 0; k < 4; ++k) S.mu[k][lane] = mk[k];
    S.mu[4][lane] = sum;
  } else {
    for (int a = wid - 2; a < 10; a += P2_WARPS - 2) {
      const int n = S.v[a][lane];
      S.dm[a][lane] = A.dmask[n];
      if (A.body)
        for (int d = 0; d < 3; ++d) S.f[a][d][lane] = A.body[3 * (size_t)n + d];
    }
  }
  __syncthreads();
  const double vol = S.vol[lane];
  const bool ok = S.ok[lane] != 0;
  // the loads alone need no stiffness unless a prescribed displacement is lifted
  const bool stiffness = !A.loads_only || A.ud != nullptr;
  if (stiffness) {
    for (int p = wid; p < 10; p += P2_WARPS) {
      const int k = p < 4 ? 0 : (p < 7 ? 1 : (p < 9 ? 2 : 3));
      const int l = p - (k * 4 - k * (k - 1) / 2) + k;
      double gk[3], gl[3], lg[3], mg[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        gk[d] = S.G[k][d][lane];
        gl[d] = S.G[l][d][lane];
        lg[d] = lam * vol * gk[d];
        mg[d] = mu * vol * gk[d];
      }
      const double mgg = mg[0] * gl[0] + mg[1] * gl[1] + mg[2] * gl[2];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
          S.B[p][3 * i + j][lane] = i == j ? fma(lg[i] + mg[i], gl[i], mgg) : fma(lg[i], gl[j], mg[j] * gl[i]);
    }
    __syncthreads();
  }
  if (stiffness)
    for (int pidx = wid; pidx < 55; pidx += P2_WARPS) {
      int a = 0, r = pidx;
      while (r >= 10 - a) {
        r -= 10 - a;
        ++a;
      }
      const int b = a + r;
      const int na = S.v[a][lane], nb = S.v[b][lane];
      const bool da = S.dm[a][lane] != 0, db = S.dm[b][lane] != 0;
      const bool ab = ok && !da && (!A.loads_only || (db && A.ud));
      const bool ba = ok && b != a && !db && (!A.loads_only || (da && A.ud));
      double k[9];
#pragma unroll
      for (int e = 0; e < 9; ++e) k[e] = 0.0;
      auto add = [&](double w, int p, int q) {  // k += w B_pq
        const int lo = p < q ? p : q, hi = p < q ? q : p;
        const double(*B)[32] = S.B[lo * 4 - lo * (lo - 1) / 2 + (hi - lo)];
        if (p <= q) {
#pragma unroll
          for (int e = 0; e < 9; ++e) k[e] = fma(w, B[e][lane], k[e]);
        } else {
#pragma unroll
          for (int e = 0; e < 9; ++e) k[e] = fma(w, B[(e % 3) * 3 + e / 3][lane], k[e]);
        }
      };
      if (b < 4) {
        add(a == b ? 0.6 : -0.2, a, b);
      } else {
        const int br = c_edge[b - 4][0], bs = c_edge[b - 4][1];
        if (a < 4) {
          add(a == bs ? 0.6 : -0.2, a, br);
          add(a == br ? 0.6 : -0.2, a, bs);
        } else {
          const int ap = c_edge[a - 4][0], aq = c_edge[a - 4][1];
          add(aq == bs ? 1.6 : 0.8, ap, br);
          add(aq == br ? 1.6 : 0.8, ap, bs);
          add(ap == bs ? 1.6 : 0.8, aq, br);
          add(ap == br ? 1.6 : 0.8, aq, bs);
        }
      }
      // the block to (a, b), then its transpose to (b, a)
      int slot = -1;
      if (ab) slot = block_slot(A, c, a, b, na, nb, db, k);
      if (fills_values(A)) scatter_run(A.vals, k, slot, S.out[wid][0], S.slot[wid], lane);
      if (a != b) {
        const double kt[9] = {k[0], k[3], k[6], k[1], k[4], k[7], k[2], k[5], k[8]};
        slot = -1;
        if (ba) slot = block_slot(A, c, b, a, nb, na, da, kt);
        if (fills_values(A)) scatter_run(A.vals, kt, slot, S.out[wid][0], S.slot[wid], lane);
      }
    }
  // loads: f_a = kT vol int (T_h - T_ref) grad phi_a + vol int f_h phi_a
  if (A.T || A.body) {
    const double kT = (3.0 * lam + 2.0 * mu) * alpha * vol;
    for (int a = wid; a < 10; a += P2_WARPS) {
      if (!ok || S.dm[a][lane]) continue;
      double f[3] = {0.0, 0.0, 0.0};
      if (A.T) {
        if (a < 4) {
          const double w = kT * (4.0 * S.mu[a][lane] - S.mu[4][lane]);
          for (int d = 0; d < 3; ++d) f[d] = w * S.G[a][d][lane];
        } else {
          const int p = c_edge[a - 4][0], q = c_edge[a - 4][1];
          const double wp = 4.0 * kT * S.mu[q][lane], wq = 4.0 * kT * S.mu[p][lane];
          for (int d = 0; d < 3; ++d) f[d] = fma(wp, S.G[p][d][lane], wq * S.G[q][d][lane]);
        }
      }
      if (A.body) {
        double s[3] = {0.0, 0.0, 0.0};
        for (int b = 0; b < 10; ++b) {
          const double w = p2_mass(a, b);
#pragma unroll
          for (int d = 0; d < 3; ++d) s[d] = fma(w, S.f[b][d][lane], s[d]);
        }
        for (int d = 0; d < 3; ++d) f[d] = fma(vol, s[d], f[d]);
      }
      for (int d = 0; d < 3; ++d) {
        if (A.cf) A.cf[((size_t)c * 10 + a) * 3 + d] = f[d];
        else atomicAdd(&A.rhs[3 * (size_t)S.v[a][lane] + d], f[d]);
      }
    }
  }
}

void launch_p2(const AsmArgs& args, cudaStream_t s) {
  TAM_CUDA(cudaFuncSetAttribute(assemble_p2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(P2Tile)));
  assemble_p2_kernel<<<grid_for(args.n_cells, P2_CELLS), P2_WARPS * 32, sizeof(P2Tile), s>>>(args);
}

// ---------------------------------------------------------------------------
// Deterministic assembly: the element kernels store every block and load in
// its own slot; per node, a warp sums its cells' slots in increasing cell id
// order into the node's row of K and its load (Dirichlet columns lifted) --
// the same sums as the atomic scatter, in an order fixed by the mesh, so two
// runs give bitwise equal K and f.
// ---------------------------------------------------------------------------
constexpr int DET_WARPS = 4;
constexpr int DET_CAP = 1024;  // cells per node the sorting pass handles

// each node's incident cells in increasing id (warp per node, shared-memory
// bitonic sort); a node in more than DET_CAP cells sets *bad
__global__ void __launch_bounds__(DET_WARPS * 32)
incidence_sort_kernel(int n_nodes, const int* __restrict__ ptr, int* __restrict__ inc, int* __restrict__ bad) {
  __shared__ int tab[DET_WARPS][DET_CAP];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int v = blockIdx.x * DET_WARPS + wid;
  if (v >= n_nodes) return;  // warp-uniform
  const int p0 = ptr[v], len = ptr[v + 1] - p0;
  if (len > DET_CAP) {
    if (lane == 0) atomicExch(bad, 1);
    return;
  }
  int* t = tab[wid];
  const int n2 = next_pow2(len);
  for (int i = lane; i < n2; i += 32) t[i] = i < len ? inc[p0 + i] : 0x7fffffff;
  __syncwarp();
  warp_bitonic_sort<false>(t, nullptr, n2);
  for (int i = lane; i < len; i += 32) inc[p0 + i] = t[i];
}

__global__ void __launch_bounds__(DET_WARPS * 32)
gather_kernel(int n_nodes, int npc, const int* __restrict__ cells, const int* __restrict__ ptr,
              const int* __restrict__ inc, const unsigned char* __restrict__ dmask, const double* __restrict__ ud,
              const int* __restrict__ rp, const int* __restrict__ ci, double* __restrict__ vals,
              double* __restrict__ rhs, const double* __restrict__ ck, const double* __restrict__ cf, int has_loads) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * DET_WARPS + wid;
  if (i >= n_nodes || dmask[i]) return;  // warp-uniform; Dirichlet rows: dirichlet_rows_kernel
  double f = 0.0;  // lane d < 3: component d of the node's load
  for (int p = ptr[i]; p < ptr[i + 1]; ++p) {
    const int c = inc[p];
    const int* cn = cells + (size_t)c * npc;
    const unsigned m = __ballot_sync(0xffffffffu, lane < npc && cn[lane] == i);
    const int a = __ffs(m) - 1;  // the node's local index in cell c
    const double* kc = ck + ((size_t)c * npc + a) * npc * 9;
    if (has_loads && lane < 3) f += cf[((size_t)c * npc + a) * 3 + lane];
    if (vals)
      for (int it = lane; it < npc * 9; it += 32) {
        const int b = it / 9, e = it - b * 9, j = cn[b];
        if (dmask[j]) continue;
        const int slot = bsearch_i32(ci, rp[i], rp[i + 1], j);
        vals[(size_t)slot * 9 + e] += kc[it];
      }
    if (ud && lane < 3)
      for (int b = 0; b < npc; ++b) {
        const int j = cn[b];
        if (!dmask[j]) continue;
        const double* kb = kc + b * 9;
        const double* u = ud + 3 * (size_t)j;
        f -= kb[3 * lane] * u[0] + kb[3 * lane + 1] * u[1] + kb[3 * lane + 2] * u[2];
      }
    __syncwarp();
  }
  if (lane < 3) rhs[3 * (size_t)i + lane] = f;
}

// Dirichlet (and cell-less) rows: identity diagonal block, load = u_D.
__global__ void dirichlet_rows_kernel(int n, const unsigned char* __restrict__ dmask,
                                      const int* __restrict__ inc_ptr, const double* __restrict__ ud,
                                      const int* __restrict__ row_ptr, const int* __restrict__ col_idx,
                                      double* __restrict__ vals, double* __restrict__ rhs) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bool orphan = inc_ptr && inc_ptr[i + 1] == inc_ptr[i];
  if (!dmask[i] && !orphan) return;
  if (vals) {  // loads-only assembly leaves the existing K alone
    int slot = bsearch_i32(col_idx, row_ptr[i], row_ptr[i + 1], i);
    double* d = vals + (size_t)slot * 9;
    for (int e = 0; e < 9; ++e) d[e] = (e % 4 == 0) ? 1.0 : 0.0;
  }
  for (int r = 0; r < 3; ++r) rhs[3 * (size_t)i + r] = (dmask[i] && ud) ? ud[3 * (size_t)i + r] : 0.0;
}

}  // namespace

// Node and material ids of a mesh in range (INVALID_ARG otherwise).  Synchronising.
void validate_mesh(int n_nodes, int n_cells, int npc, const int* cells, const int* mat, int n_mat, const char* who,
                   cudaStream_t s) {
  if (n_cells <= 0) return;
  const long long n_entries = (long long)n_cells * npc;
  DBuf<int> bad(1, s);
  bad.zero();
  validate_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, npc, n_nodes, mat, n_cells, n_mat,
                                                            bad.p);
  TAM_LAUNCH_CHECK();
  const int b = read_back_int(bad.p, s);
  TAM_CHECK(b == 0, TAM_ERR_INVALID_ARG,
            std::string(who) + (b == 1 ? ": cell node id out of range" : ": material id out of range"));
}

// Node-adjacency pattern of a mesh: block row i holds i and every node that
// shares a cell with it, sorted, without the Dirichlet nodes (dmask) -- whose
// own rows keep only the diagonal.  Fills A.n_rows/n_cols, row_ptr, col_idx
// and nnzb (block sizes are the caller's), and returns the cell-node
// incidence (inc_ptr[n_nodes + 1], inc) that the pattern came from.  flag[1]
// is set when a node has too many incident cells for the shared-memory
// builder.  Synchronising.
// 64-bit sum of per-row counts (overflow check before an int32 scan)
__global__ void count_sum_kernel(const int* __restrict__ cnt, int n, unsigned long long* __restrict__ out) {
  unsigned long long v = 0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    v += (unsigned long long)(unsigned)cnt[i];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(out, v);
}

void build_node_pattern(int n_nodes, int n_cells, int npc, const int* cells, const unsigned char* dmask, Bsr& A,
                        DBuf<int>& inc_ptr, DBuf<int>& inc, int* flag, cudaStream_t s) {
  const long long n_entries = (long long)n_cells * npc;
  // cell-node incidence
  inc_ptr = DBuf<int>((size_t)n_nodes + 1, s);
  inc = DBuf<int>((size_t)std::max(1LL, n_entries), s);
  DBuf<int> cursor((size_t)n_nodes, s);
  inc_ptr.zero();
  cursor.zero();
  if (n_cells > 0) {
    incidence_count_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, inc_ptr.p);
    TAM_LAUNCH_CHECK();
  }
  exclusive_scan_i32(inc_ptr.p, inc_ptr.p, n_nodes, s);
  if (n_cells > 0) {
    incidence_fill_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, npc, inc_ptr.p, cursor.p,
                                                                   inc.p);
    TAM_LAUNCH_CHECK();
  }
  // pattern
  A.n_rows = A.n_cols = n_nodes;
  A.row_ptr = DBuf<int>((size_t)n_nodes + 1, s);
  unsigned pg = grid_for(n_nodes, PAT_WARPS);
  if (3 * ((long long)n_nodes + (long long)npc * npc * n_cells) < (1LL << 31)) {
    // one sort pass: each row's sorted unique columns go to its candidate-
    // bound offset in a scratch array (the bounds' sum, at most
    // 3 (n_nodes + npc^2 n_cells), fits the int32 scan), the counts give
    // row_ptr, then pack
    DBuf<int> bptr((size_t)n_nodes + 1, s);
    pattern_bound_kernel<<<grid_for(n_nodes, 256), 256, 0, s>>>(n_nodes, npc, inc_ptr.p, dmask, bptr.p);
    TAM_LAUNCH_CHECK();
    exclusive_scan_i32(bptr.p, bptr.p, n_nodes, s);
    const long long total = read_back_int(bptr.p + n_nodes, s);
    DBuf<int> tmp((size_t)std::max(1LL, total), s);
    // flag[1]: overflow beyond the list; big[0]: rows listed for pattern_big_kernel
    const int big_cap = std::max(1, std::min(n_nodes, 1 << 20));
    DBuf<int> big_list((size_t)big_cap, s), big(2, s);
    big.zero();
    pattern_kernel<true><<<pg, PAT_WARPS * 32, 0, s>>>(n_nodes, npc, cells, inc_ptr.p, inc.p, dmask, A.row_ptr.p,
                                                      bptr.p, tmp.p, big.p, big_list.p, big_cap);
    TAM_LAUNCH_CHECK();
    int n_big = 0, big_over = 0;
    read_back_int2(big.p + 1, big.p, &n_big, &big_over, s);
    TAM_CHECK(big_over == 0, TAM_ERR_UNSUPPORTED, "fem_assemble: too many high-valence nodes for the pattern builder");
    if (n_big > 0) {
      pattern_big_kernel<<<n_big, BIG_THREADS, 0, s>>>(big_list.p, npc, cells, inc_ptr.p, inc.p, dmask, bptr.p, tmp.p,
                                                      A.row_ptr.p);
      TAM_LAUNCH_CHECK();
    }
    exclusive_scan_i32(A.row_ptr.p, A.row_ptr.p, n_nodes, s);
    A.nnzb = read_back_int(A.row_ptr.p + n_nodes, s);
    A.col_idx = DBuf<int>((size_t)std::max(1LL, A.nnzb), s);
    pattern_pack_kernel<<<grid_for((long long)n_nodes * 32, 256), 256, 0, s>>>(n_nodes, bptr.p, tmp.p,
                                                                               A.row_ptr.p, A.col_idx.p);
    TAM_LAUNCH_CHECK();
  } else {
    // very large meshes: count pass, then fill pass (no scratch)
    pattern_kernel<false><<<pg, PAT_WARPS * 32, 0, s>>>(n_nodes, npc, cells, inc_ptr.p, inc.p, dmask, A.row_ptr.p,
                                                       nullptr, nullptr, flag + 1);
    TAM_LAUNCH_CHECK();
    {
      // block counts are int32 (K's arrays): refuse a pattern of 2^31 blocks or more
      DBuf<unsigned long long> tot(1, s);
      tot.zero();
      count_sum_kernel<<<stride_grid(n_nodes, 256, 8), 256, 0, s>>>(A.row_ptr.p, n_nodes, tot.p);
      TAM_LAUNCH_CHECK();
      TAM_CHECK(read_back_ll(reinterpret_cast<const long long*>(tot.p), s) < (1LL << 31), TAM_ERR_UNSUPPORTED,
                "fem_assemble: K would have 2^31 or more 3x3 blocks (int32 indices)");
    }
    exclusive_scan_i32(A.row_ptr.p, A.row_ptr.p, n_nodes, s);
    A.nnzb = read_back_int(A.row_ptr.p + n_nodes, s);
    TAM_CHECK(read_back_int(flag + 1, s) == 0, TAM_ERR_UNSUPPORTED,
              "fem_assemble: a node has too many incident cells for the pattern builder");
    A.col_idx = DBuf<int>((size_t)A.nnzb, s);
    pattern_kernel<true><<<pg, PAT_WARPS * 32, 0, s>>>(n_nodes, npc, cells, inc_ptr.p, inc.p, dmask, nullptr,
                                                      A.row_ptr.p, A.col_idx.p, flag + 1);
    TAM_LAUNCH_CHECK();
  }
}

std::atomic<int> g_deterministic_assembly{0};

// Deterministic assembly's second pass: sort the incidence lists, sum the
// slots per node (vals may be null: loads only).
static void gather_assembly(const AsmArgs& args, int n_nodes, int npc, const int* cells, const int* inc_ptr,
                            int* inc, const unsigned char* dmask, double* vals, double* rhs, bool has_loads,
                            cudaStream_t s) {
  DBuf<int> bad(1, s);
  bad.zero();
  incidence_sort_kernel<<<grid_for(n_nodes, DET_WARPS), DET_WARPS * 32, 0, s>>>(n_nodes, inc_ptr, inc, bad.p);
  TAM_LAUNCH_CHECK();
  TAM_CHECK(read_back_int(bad.p, s) == 0, TAM_ERR_UNSUPPORTED,
            "fem_assemble: deterministic assembly handles nodes in at most 1024 cells");
  gather_kernel<<<grid_for(n_nodes, DET_WARPS), DET_WARPS * 32, 0, s>>>(
      n_nodes, npc, cells, inc_ptr, inc, dmask, args.ud, args.row_ptr, args.col_idx, vals, rhs, args.ck, args.cf,
      has_loads ? 1 : 0);
  TAM_LAUNCH_CHECK();
}

tam_matrix_s* assemble_elasticity(int n_nodes, const double* coords, int n_cells, int npc, const int* cells,
                                  const int* mat, int n_mat, const double* props, const double* T,
                                  double T_ref, const double* body, const unsigned char* dmask,
                                  const double* ud, double* rhs, cudaStream_t s) {
  NvtxRange nvtx("tam: assemble K and f");
  TAM_CHECK(n_nodes > 0 && n_cells >= 0 && n_mat > 0, TAM_ERR_INVALID_ARG, "fem_assemble: bad sizes");
  TAM_CHECK(npc == 4 || npc == 10, TAM_ERR_INVALID_ARG, "fem_assemble: nodes_per_cell must be 4 or 10");
  TAM_CHECK(coords && (cells || n_cells == 0) && (mat || n_cells == 0) && props && dmask && rhs,
            TAM_ERR_INVALID_ARG, "fem_assemble: null pointer");
  auto M = new tam_matrix_s();
  M->nodes_per_cell = npc;
  try {
    M->n_nodes = n_nodes;
    const long long n_entries = (long long)n_cells * npc;
    DBuf<int> flag(2, s);
    flag.zero();
    if (n_cells > 0) {
      validate_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, npc, n_nodes, mat, n_cells,
                                                                n_mat, flag.p);
      TAM_LAUNCH_CHECK();
      int bad = read_back_int(flag.p, s);
      TAM_CHECK(bad == 0, TAM_ERR_INVALID_ARG,
                bad == 1 ? "fem_assemble: cell node id out of range" : "fem_assemble: material id out of range");
    }
    // cell-node incidence and block pattern
    Bsr& A = M->A;
    A.br = A.bc = 3;
    DBuf<int> inc_ptr, inc;
    build_node_pattern(n_nodes, n_cells, npc, cells, dmask, A, inc_ptr, inc, flag.p, s);
    // numeric
    A.vals = DBuf<double>((size_t)A.nnzb * 9, s);
    A.vals.zero();
    TAM_CUDA(cudaMemsetAsync(rhs, 0, sizeof(double) * 3 * (size_t)n_nodes, s));
    AsmArgs args{coords, cells, mat, props, T, T_ref, body, dmask, ud, A.row_ptr.p, A.col_idx.p,
                 A.vals.p, rhs, n_cells, flag.p, 0};
    const bool det = g_deterministic_assembly.load() != 0 && n_cells > 0;
    DBuf<double> ck, cf;
    if (det) {
      ck = DBuf<double>((size_t)n_cells * npc * npc * 9, s);
      cf = DBuf<double>((size_t)n_cells * npc * 3, s);
      args.ck = ck.p;
      args.cf = cf.p;
      args.npc = npc;
    }
    if (n_cells > 0) {
      if (npc == 4)
        assemble_p1_kernel<<<grid_for(n_cells, P1_THREADS), P1_THREADS, 0, s>>>(args);
      else
        launch_p2(args, s);
      TAM_LAUNCH_CHECK();
    }
    if (det) gather_assembly(args, n_nodes, npc, cells, inc_ptr.p, inc.p, dmask, A.vals.p, rhs, T || body, s);
    dirichlet_rows_kernel<<<grid_for(n_nodes, 256), 256, 0, s>>>(n_nodes, dmask, inc_ptr.p, ud, A.row_ptr.p,
                                                                 A.col_idx.p, A.vals.p, rhs);
    TAM_LAUNCH_CHECK();
    TAM_CHECK(read_back_int(flag.p, s) == 0, TAM_ERR_DEGENERATE_CELL,
              "fem_assemble: a cell has non-positive or non-finite volume");
    M->dmask = DBuf<unsigned char>((size_t)n_nodes, s);
    TAM_CUDA(cudaMemcpyAsync(M->dmask.p, dmask, n_nodes, cudaMemcpyDeviceToDevice, s));
    // split copies for the double-float SpMV: SELL always (the CG's own SpMVs
    // with K use it; written by the SELL fill), the block-CSR only where K's
    // operator runs on it
    // (none when K is outside the double-float range: every product is FP64)
    ExponentRange range;
    bsr_to_sell(A, M->S, s, true, &range);
    M->vmax_exp = range.max_exp;
    M->finite = range.finite;
    M->df_ok = M->finite && std::abs(M->vmax_exp) <= kDfExpLimit;
    if (!M->df_ok) {
      M->S.vals_df.reset();
    } else if (!M->S.vals_df.p) {  // memory was short: out of memory for good, or not
      alloc_split(M->S, s);
      sell_refresh_values(A, M->S, s);
    }
    if (M->df_ok && choose_lpr(A) != 0) build_df_values(A, s);
    TAM_CUDA(cudaStreamSynchronize(s));
  } catch (...) {
    delete M;
    throw;
  }
  return M;
}

// Load vector of another load case on the mesh of an existing K: thermal and
// body loads (and the lifting of prescribed displacements), Dirichlet rows
// set to u_D; K itself is not touched.
void assemble_loads(tam_matrix_s* K, const double* coords, int n_cells, int npc, const int* cells, const int* mat,
                    int n_mat, const double* props, const double* T, double T_ref, const double* body,
                    const double* ud, double* rhs, cudaStream_t s) {
  NvtxRange nvtx("tam: assemble f");
  TAM_CHECK(K && coords && props && rhs && n_mat > 0 && n_cells >= 0 && (npc == 4 || npc == 10) &&
                (cells || n_cells == 0) && (mat || n_cells == 0),
            TAM_ERR_INVALID_ARG, "fem_assemble_load: bad argument");
  const int n_nodes = K->n_nodes;
  DBuf<int> flag(2, s);
  flag.zero();
  const long long n_entries = (long long)n_cells * npc;
  if (n_cells > 0) {
    validate_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, npc, n_nodes, mat, n_cells, n_mat,
                                                              flag.p);
    TAM_LAUNCH_CHECK();
    TAM_CHECK(read_back_int(flag.p, s) == 0, TAM_ERR_INVALID_ARG, "fem_assemble_load: cell or material id out of range");
  }
  TAM_CUDA(cudaMemsetAsync(rhs, 0, sizeof(double) * 3 * (size_t)n_nodes, s));
  AsmArgs args{coords, cells, mat, props, T, T_ref, body, K->dmask.p, ud, K->A.row_ptr.p, K->A.col_idx.p,
               nullptr, rhs, n_cells, flag.p + 1, 1};
  const bool det = g_deterministic_assembly.load() != 0 && n_cells > 0;
  DBuf<double> ck, cf;
  DBuf<int> inc_ptr, inc;
  if (det) {
    ck = DBuf<double>((size_t)n_cells * npc * npc * 9, s);
    cf = DBuf<double>((size_t)n_cells * npc * 3, s);
    args.ck = ck.p;
    args.cf = cf.p;
    args.npc = npc;
    inc_ptr = DBuf<int>((size_t)n_nodes + 1, s);
    inc = DBuf<int>((size_t)n_entries, s);
    DBuf<int> cursor((size_t)n_nodes, s);
    inc_ptr.zero();
    cursor.zero();
    incidence_count_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, inc_ptr.p);
    TAM_LAUNCH_CHECK();
    exclusive_scan_i32(inc_ptr.p, inc_ptr.p, n_nodes, s);
    incidence_fill_kernel<<<grid_for(n_entries, 256), 256, 0, s>>>(cells, n_entries, npc, inc_ptr.p, cursor.p,
                                                                   inc.p);
    TAM_LAUNCH_CHECK();
  }
  if (n_cells > 0) {
    if (npc == 4)
      assemble_p1_kernel<<<grid_for(n_cells, P1_THREADS), P1_THREADS, 0, s>>>(args);
    else
      launch_p2(args, s);
    TAM_LAUNCH_CHECK();
  }
  if (det) gather_assembly(args, n_nodes, npc, cells, inc_ptr.p, inc.p, K->dmask.p, nullptr, rhs, T || body, s);
  dirichlet_rows_kernel<<<grid_for(n_nodes, 256), 256, 0, s>>>(n_nodes, K->dmask.p, nullptr, ud, nullptr, nullptr,
                                                               nullptr, rhs);
  TAM_LAUNCH_CHECK();
  TAM_CHECK(read_back_int(flag.p + 1, s) == 0, TAM_ERR_DEGENERATE_CELL,
            "fem_assemble_load: a cell has non-positive or non-finite volume");
}

}  // namespace tam
