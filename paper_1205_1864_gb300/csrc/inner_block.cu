// K3 + K4 on small grids: the batched inner PCG on A_0, one launch per solve,
// every column solved by its own thread block (or cluster of blocks).
//
// Same method, stopping rule, status bits and iteration counts as the
// stand-alone kernels of inner.cu. There an iteration is four to six launches
// inside a graph WHILE node, about 45 us whatever the grid; on the paper's
// own meshes (5 to 30 elements a side, FP64, some 50 iterations of the
// diagonal M_0 per solve) that was all of the time. Here the loop is inside
// the kernel and the column's vectors stay on chip:
//
//   k_block_diag    M_0 = diag(A_0), any grid of the Q1 stencil. A column is
//                   split by rows over the C blocks of a cluster; each thread
//                   keeps its nodes' stencil, r, p, x in registers, p with its
//                   ghost rows in shared memory. Two cluster barriers per
//                   iteration (p.q, then r.r with r.z): the neighbours' rows of
//                   q travel with the first one, and each block carries r and
//                   p of its ghost rows along itself.
//   k_block_vcycle  M_0 = one V-cycle, finest grid of at most 1024 nodes: one
//                   block per column, all grids in shared memory with zero
//                   borders (no boundary tests in the stencils).
//   k_block_vcycle63  the same on 63 x 63 nodes in FP32, the finest grid's
//                   stencils in registers.
//   k_vcycle_coarse  not a solver: the V-cycle's coarse grids for the
//                   stand-alone kernels, through the same code.
//
// What bounds them: the FP64 unit of each SM quarter takes a warp instruction
// every 69 clocks (measured; one at a time, whatever the number of active
// lanes or independent operands), so an iteration costs 69 clocks for every
// FP64 instruction in the longest chain of one warp: the node's own sixteen,
// then one for each step of a sum, and about eight for a division; a cluster
// barrier adds 370 clocks. The blocks therefore use four warps where they can
// (one per quarter), C is the largest split for which the batch still finds
// an SM for every block, and every addition saved counts.
//
// Measured against the stand-alone kernels, sg_inner_solve with its copies
// and synchronisation, 20 steps of the diagonal M_0 or 2 of the V-cycle:
// 29 x 29 nodes, FP64, 20 columns 1284 -> 154 us, 1000 columns 4724 -> 1021;
// 63 x 63, FP64, 300 columns 2824 -> 1502; 9 x 9, 20 columns 1288 -> 127;
// V-cycle 15 x 15, FP64, 20 columns 218 -> 91, 31 x 31, FP64, 20 columns 256 ->
// 128, FP32, 300 columns 199 -> 105, 63 x 63, FP32, 300 columns 286 -> 146. No
// size it can hold was slower (1 to 1000 columns, both types), so every batch
// that fits takes it before the stand-alone kernels. Whole FP64 solves: 16 x 16
// elements, M = 3, p = 3, 6.64 -> 1.30 ms; 30 x 30, diagonal M_0, M = 4, p = 4,
// 274 -> 15.4 ms; lognormal 10 x 10, M = 3, p = 3, 1034 -> 77.6 ms.
#include <cooperative_groups.h>

#include <algorithm>

#include "sghsc_internal.cuh"
#include "vec.cuh"

namespace cg = cooperative_groups;

namespace sghsc {

namespace blk {
constexpr int NT = 256;          // threads of k_block_diag at most
constexpr int NW = NT / 32;
constexpr int MAX_ITEMS = 4;     // nodes per thread of k_block_diag
constexpr int MAX_C = 8;         // blocks per cluster
constexpr int VNT = 256;         // threads of k_block_vcycle at most
constexpr int CNT = 512;         // threads of k_vcycle_coarse at most
constexpr int MAX_GRIDS = 16;    // grids of a hierarchy (a finest side of 2^16 - 1)
}  // namespace blk

struct BlockArgs {
  int n, nx, ny, w;
  int R, C;            // k_block_diag: rows per block, blocks per column
  double tol2;
  int maxit, fixed;
  int* status;
  long long* iacc;
  int* iters;          // per-column iteration counts, or null
};

// CG scalars of the block's column; every block of a cluster holds the same.
template <typename T>
struct BlockScalars {
  double rho, stop;   // r.z of the last step; the r.r at which the column is done
  T alpha, beta;
  int it, done;
};

// The scalar updates of the stand-alone finaliser (col_update in inner.cu),
// by one thread; report: this block writes status bits and counts.
__device__ __forceinline__ bool is_nan_bits(long long b) {
  return (b & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}
// x > 0 (false for NaN) and x <= y for non-negative y (false for a NaN x),
// from the bit patterns: a comparison on the FP64 unit costs as much as a
// multiply-add
__device__ __forceinline__ bool positive(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool at_most(double x, double y) {
  const long long b = __double_as_longlong(x), c = __double_as_longlong(y);
  return b <= c && !is_nan_bits(b) && c <= 0x7ff0000000000000LL;
}
template <typename T>
__device__ __forceinline__ void scal_init(BlockScalars<T>& S, double bb, const BlockArgs& a) {
  S.stop = a.tol2 * bb;
  S.done = !positive(bb);
  S.it = 0;
}
template <typename T>
__device__ __forceinline__ void scal_rho(BlockScalars<T>& S, double s) {
  S.beta = (T)(S.it == 0 ? 0.0 : s / S.rho);
  S.rho = s;
}
template <typename T>
__device__ __forceinline__ void scal_alpha(BlockScalars<T>& S, double s, const BlockArgs& a, bool report) {
  if (!positive(s)) {
    if (report) atomicOr(a.status, ST_INNER_NOT_SPD);
    S.alpha = T(0);
    S.done = 1;
  } else {
    S.alpha = (T)(S.rho / s);
  }
}
template <typename T>
__device__ __forceinline__ void scal_conv(BlockScalars<T>& S, double s, const BlockArgs& a, bool report) {
  const int it = ++S.it;
  bool fin;
  if (a.fixed > 0) {
    fin = it >= a.fixed;
  } else {
    fin = at_most(s, S.stop);
    if (!fin && it >= a.maxit) {
      fin = true;
      if (report) atomicOr(a.status, ST_INNER_MAXIT);
    }
  }
  if (is_nan_bits(__double_as_longlong(s))) {   // non-finite residual: stop the column and flag it
    fin = true;
    if (report) atomicOr(a.status, ST_INNER_NOT_SPD);
  }
  S.done = fin;
  if (fin && report) {
    atomicAdd((unsigned long long*)&a.iacc[0], (unsigned long long)it);
    atomicMax(&a.iacc[1], (long long)it);
  }
}

// Butterfly sum over the warp (every lane gets it).
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The sums of v0 and v1 over the warp for the additions of one: lanes below
// 16 end with the sum of v0, the others with that of v1.
template <typename T>
__device__ __forceinline__ T half_sums(T v0, T v1, int lane) {
  const bool lo = lane < 16;
  T v = lo ? v0 : v1;
  v += __shfl_xor_sync(0xffffffffu, lo ? v1 : v0, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------- diagonal M_0 ---

// Dynamic shared memory: p with ghost rows and columns [(R + 2)(nx + 2)],
// then per ghost row side (above, below) q as received, r, dinv [2][nx] each.
template <typename T>
static size_t diag_smem(int R, int nx) {
  return ((size_t)(R + 2) * (nx + 2) + 6 * (size_t)nx) * sizeof(T);
}

template <typename TS, typename T, typename TD, int ITEMS>
__global__ void __launch_bounds__(blk::NT) k_block_diag(BlockArgs a, const T* __restrict__ st,
                                                        const T* __restrict__ dinv, const TS* __restrict__ src,
                                                        int lds, TD* __restrict__ dst, int ldd) {
  using namespace blk;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T red[3][MAX_C * NW];   // warp sums of every block of the cluster: r.r, r.z, p.q
  __shared__ BlockScalars<T> S;
  cg::cluster_group cl = cg::this_cluster();
  const int C = a.C, rank = C > 1 ? (int)cl.block_rank() : 0;
  const int col = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = a.nx, W = nx + 2;
  const int r0 = rank * a.R, nr = max(0, min(a.ny - r0, a.R)), own = nr * nx;
  T* ps = reinterpret_cast<T*>(smem_raw);
  T* qg = ps + (size_t)(a.R + 2) * W;
  T* rg = qg + 2 * nx;
  T* dg = rg + 2 * nx;
  const bool above = C > 1 && nr > 0 && r0 > 0, below = C > 1 && nr > 0 && r0 + nr < a.ny;
  const int nt = blockDim.x, nw = nt / 32;
  auto barrier = [&]() {
    if (C > 1) cl.sync();
    else __syncthreads();
  };
  auto put = [&](int k, int to, T v) {   // this warp's sum into slot k of block `to` of the cluster
    T* s = &red[k][rank * nw + warp];
    if (C > 1) *cl.map_shared_rank(s, to) = v;
    else *s = v;
  };
  // warp sums into every block of the cluster: one sum, or two at the price
  // of one (half a warp each; FP64 additions are what the sums cost)
  auto push = [&](int k, T v) {
    v = warp_sum(v);
    if (lane < C) put(k, lane, v);
  };
  auto push2 = [&](T v0, T v1) {
    const T s = half_sums(v0, v1, lane);
    if ((lane & 15) < C) put(lane >> 4, lane & 15, s);
  };
  // totals, by one warp in a fixed order
  const int ns = C * nw;   // warp sums per slot
  auto total = [&](int k) {
    T v = lane < ns ? red[k][lane] : T(0);
    if (ns > 32) v += lane + 32 < ns ? red[k][lane + 32] : T(0);
    for (int o = 16; o > 0; o >>= 1)
      if (o < ns) v += __shfl_xor_sync(0xffffffffu, v, o);
    return (double)v;
  };
  auto total2 = [&](double& s0, double& s1) {
    const int l16 = lane & 15;
    T v = l16 < ns ? red[lane >> 4][l16] : T(0);
    for (int i = l16 + 16; i - l16 < ns; i += 16) v += i < ns ? red[lane >> 4][i] : T(0);
    for (int o = 8; o > 0; o >>= 1)
      if (o < ns) v += __shfl_xor_sync(0xffffffffu, v, o);
    s0 = (double)__shfl_sync(0xffffffffu, v, 0);
    s1 = (double)__shfl_sync(0xffffffffu, v, 16);
  };
  for (int i = tid; i < (a.R + 2) * W; i += nt) ps[i] = T(0);
  T s9[ITEMS][9], r[ITEMS], x[ITEMS], z[ITEMS], d[ITEMS], q[ITEMS], p[ITEMS];
  int pc[ITEMS];   // padded index
  bool up[ITEMS], dn[ITEMS];   // node of the first / last own row, which a neighbour keeps as a ghost
#pragma unroll
  for (int u = 0; u < ITEMS; ++u) {
    const int i = tid + u * nt;
    const bool in = i < own;
    const int ly = in ? i / nx : 0, lx = in ? i - ly * nx : 0, g = (r0 + ly) * nx + lx;
    pc[u] = (ly + 1) * W + lx + 1;
    up[u] = in && ly == 0 && above;
    dn[u] = in && ly == nr - 1 && below;
#pragma unroll
    for (int e = 0; e < 9; ++e) s9[u][e] = in ? st[(size_t)g * 9 + e] : T(0);
    d[u] = in ? dinv[g] : T(0);
    r[u] = in ? widen<T>(src[(size_t)g * lds + col]) : T(0);
    x[u] = p[u] = q[u] = T(0);
  }
  for (int i = tid; i < 2 * nx; i += nt) {
    const int side = i / nx, lx = i - side * nx, g = (side ? r0 + nr : r0 - 1) * nx + lx;
    const bool in = side ? below : above;
    rg[i] = in ? widen<T>(src[(size_t)g * lds + col]) : T(0);
    dg[i] = in ? dinv[g] : T(0);
  }
  {
    T rr = T(0), rz = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      z[u] = d[u] * r[u];
      rr += r[u] * r[u];
      rz += r[u] * z[u];
    }
    if (C > 1) cl.sync();   // every block of the cluster has started
    push2(rr, rz);
  }
  barrier();
  if (warp == 0) {
    double bb, rz;
    total2(bb, rz);
    if (lane == 0) {
      scal_init(S, bb, a);
      if (!S.done) scal_rho(S, rz);
    }
  }
  __syncthreads();
  while (!S.done) {
    const T beta = S.beta;
    const bool first = S.it == 0;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      if (tid + u * nt < own) {
        p[u] = first ? z[u] : fma(beta, p[u], z[u]);
        ps[pc[u]] = p[u];
      }
    }
    if (C > 1)
      for (int i = tid; i < 2 * nx; i += nt) {
        const int side = i >= nx, lx = i - side * nx;
        if (side ? below : above) {
          T* pg = ps + (side ? nr + 1 : 0) * W + lx + 1;
          const T zv = dg[i] * rg[i];
          *pg = first ? zv : fma(beta, *pg, zv);
        }
      }
    __syncthreads();
    T pq = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      if (tid + u * nt < own) {
        T acc = T(0);
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx) acc = fma(s9[u][(dy + 1) * 3 + dx + 1], ps[pc[u] + dy * W + dx], acc);
        q[u] = acc;
        pq = fma(p[u], acc, pq);
        if (up[u]) cl.map_shared_rank(qg, rank - 1)[nx + pc[u] - W - 1] = acc;
        if (dn[u]) cl.map_shared_rank(qg, rank + 1)[pc[u] - nr * W - 1] = acc;
      }
    }
    push(2, pq);
    barrier();
    if (warp == 0) {
      const double s = total(2);
      if (lane == 0) scal_alpha(S, s, a, rank == 0);
    }
    __syncthreads();
    if (S.done) break;   // the same in every block of the cluster
    const T al = S.alpha;
    T rr = T(0), rz = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      if (tid + u * nt < own) {
        x[u] = fma(al, p[u], x[u]);
        r[u] = fma(-al, q[u], r[u]);
        z[u] = d[u] * r[u];
        rr = fma(r[u], r[u], rr);
        rz = fma(r[u], z[u], rz);
      }
    }
    if (C > 1)
      for (int i = tid; i < 2 * nx; i += nt) rg[i] = fma(-al, qg[i], rg[i]);
    push2(rr, rz);
    barrier();
    if (warp == 0) {
      double s, rzs;
      total2(s, rzs);
      if (lane == 0) {
        scal_conv(S, s, a, rank == 0);
        if (!S.done) scal_rho(S, rzs);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < ITEMS; ++u) {
    const int i = tid + u * nt;
    if (i < own) {
      const int ly = i / nx, lx = i - ly * nx;
      dst[(size_t)((r0 + ly) * nx + lx) * ldd + col] = (TD)x[u];
    }
  }
  if (a.iters && rank == 0 && tid == 0) a.iters[col] = S.it;
  if (C > 1) cl.sync();   // no block leaves while another may still store into it
}

// ---------------------------------------------------------- V-cycle M_0 ---

// The hierarchy in shared memory: per grid (nx = ny = 2^k - 1, row stride
// W = nx + 2) the vectors b, x, y with zero borders, the stencils [n][9] and
// the inverse diagonal [n]; on the finest grid also p (with borders).
//
// With the default smoothing everything from the 7 x 7 grid down is one dense
// matrix on that grid's right-hand side (grid gm; -1: none): 13 phases of one
// to two warps, each a chain of a stencil's multiply-adds, are one phase of
// 49 / LP of them: 16 x 16 elements, M = 3, p = 3, FP64, whole solve 1.75 ->
// 1.40 ms; a step on 63 x 63 nodes, FP32, 17 -> 12.5 us.
struct BlockGrids {
  int G, gm;
  int k[blk::MAX_GRIDS];                       // nx + 1 = 2^k
  int vec[blk::MAX_GRIDS], coef[blk::MAX_GRIDS];   // element offsets of b (x, y follow) and of the stencils
  int p, total;                                // offset of p, elements in all
  const void* st[blk::MAX_GRIDS];   // (of grid gm: its matrix)
  const void* dinv[blk::MAX_GRIDS];
};

// The matrix of grid gm: LP threads per row, each every LP-th column; rows are
// padded with zeros to whole turns (odd multiples of LP in banks: no two lanes
// of a warp in one bank). The right-hand side lies compact before the padded
// solution.
namespace cmx {
constexpr int N = 49, W = 9;
__host__ __device__ constexpr int lp(int threads) { return threads / 64; }
__host__ __device__ constexpr int stride(int lp) { return (N + lp - 1) / lp * lp; }
constexpr int B = 56;                     // the longest row
constexpr int VECS = B + W * W;
constexpr int COEFS = N * B;
}  // namespace cmx

// f(padded index, node) over the nodes of a grid of nx + 1 = 2^k, by the
// threads t, t + nt, ... (columns of 2^k: the last of each row is skipped)
template <typename F>
__device__ __forceinline__ void each_node(int k, int t, int nt, F f) {
  const int m = 1 << k, nx = m - 1;
  for (int i = t; i < nx * m; i += nt) {
    const int x = i & nx, y = i >> k;
    if (x < nx) f((y + 1) * (m + 1) + x + 1, y * nx + x, x, y);
  }
}

// acc + sign * (A v) at the node of padded index c
template <int SIGN, typename T>
__device__ __forceinline__ T dot9(T acc, const T* __restrict__ s9, const T* v, int c, int W) {
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      const T a = s9[(dy + 1) * 3 + dx + 1];
      acc = fma(SIGN < 0 ? -a : a, v[c + dy * W + dx], acc);
    }
  return acc;
}

// Block barrier, or warp barrier while only warp 0 works (grids of at most 9
// nodes).
__device__ __forceinline__ void phase_sync(bool wm) {
  if (wm) __syncwarp();
  else __syncthreads();
}

// Zero vectors and the coefficients of the grids from g0 on, not yet visible
// to the other threads of the block; om: the damping. The stencils and the
// matrix are asynchronous copies, all in flight together: the caller waits for
// them (cp_async_wait_all) before a block barrier. Loaded and stored in a loop
// they were a chain of L2 latencies: 16 x 16 elements, FP64, whole solve 1.39 ->
// 1.30 ms, gradient on 64 x 64 elements 4.44 -> 4.25 ms.
template <typename T>
__device__ __forceinline__ void stage_grids(const BlockGrids& L, T* sm, T om, int g0 = 0) {
  const int tid = threadIdx.x, NT = blockDim.x;
  for (int g = g0; g < L.G; ++g) {
    const T* gs = (const T*)L.st[g];
    if (g == L.gm) {
      const int S = cmx::stride(cmx::lp(NT));
      for (int i = tid; i < cmx::VECS; i += NT) sm[L.vec[g] + i] = T(0);
      for (int i = tid; i < cmx::N * S; i += NT) {
        const int r = i / S, c = i - r * S;
        if (c < cmx::N) cp_async_elem(sm + L.coef[g] + i, gs + r * cmx::N + c);
        else sm[L.coef[g] + i] = T(0);
      }
      return;
    }
    const int Wg = (1 << L.k[g]) + 1, ng = (Wg - 2) * (Wg - 2);
    for (int i = tid; i < 3 * Wg * Wg; i += NT) sm[L.vec[g] + i] = T(0);
    const T* gd = (const T*)L.dinv[g];
    for (int i = tid; i < 9 * ng; i += NT) cp_async_elem(sm + L.coef[g] + i, gs + i);
    // the damped inverse diagonal (the plain one on the one-node grid, solved exactly)
    for (int i = tid; i < ng; i += NT) sm[L.coef[g] + 9 * ng + i] = g == L.G - 1 ? gd[i] : om * gd[i];
  }
}

// x = M b on grid gm
template <typename T, int LP>
__device__ __forceinline__ void apply_cmat(const T* M, const T* b, T* x) {
  constexpr int S = cmx::stride(LP);
  const int r = threadIdx.x / LP, l = threadIdx.x % LP;
  if (threadIdx.x / 32 > (cmx::N - 1) * LP / 32) return;   // whole warps
  const T* m = M + min(r, cmx::N - 1) * S + l;
  T acc = T(0);
#pragma unroll
  for (int j = 0; j < S / LP; ++j) acc = fma(m[j * LP], b[j * LP + l], acc);
#pragma unroll
  for (int o = LP / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (l == 0 && r < cmx::N) x[(r / 7 + 1) * cmx::W + r % 7 + 1] = acc;
}

// One V-cycle from grid g0's b; returns the buffer that holds the result.
// Every thread of the block calls it.
template <typename T>
__device__ T* block_vcycle(const BlockGrids& L, T* sm, int nu, int g0 = 0) {
  const int tid = threadIdx.x;
  const int G = L.gm < 0 ? L.G : L.gm + 1;
  auto wmode = [&](int g) { return L.k[g] <= 2 && g > 0; };
  auto vsize = [&](int g) { const int W = (1 << L.k[g]) + 1; return W * W; };
  auto odd = [&](int s) { return (s & 1) != 0; };
  // the iterate of grid g sits in x or y; pre-smoothing makes nu - 1 exchanges
  for (int g = g0; g < G; ++g) {
    const int W = (1 << L.k[g]) + 1, V = vsize(g), k = L.k[g], n = (W - 2) * (W - 2);
    const bool wm = wmode(g);
    const int nt = wm ? 32 : (int)blockDim.x;
    const T* st = sm + L.coef[g];
    const T* di = st + 9 * n;
    const T* b = sm + L.vec[g];
    T* c = sm + L.vec[g] + V;
    T* o = c + V;
    if (g == L.gm) {
      T* x = sm + L.vec[g] + cmx::B;
      if (blockDim.x == 128) apply_cmat<T, 2>(st, b, x);
      else if (blockDim.x == 256) apply_cmat<T, 4>(st, b, x);
      else apply_cmat<T, 8>(st, b, x);
      __syncthreads();
      break;
    }
    if (!wm || tid < 32) {
      if (g == G - 1) {   // one node: exact
        each_node(k, tid, nt, [&](int i, int node, int, int) { c[i] = di[node] * b[i]; });
        phase_sync(wm);
      } else {
        each_node(k, tid, nt, [&](int i, int node, int, int) { c[i] = di[node] * b[i]; });
        phase_sync(wm);
        for (int s = 1; s < nu; ++s) {
          each_node(k, tid, nt, [&](int i, int node, int, int) {
            o[i] = fma(di[node], dot9<-1>(b[i], st + 9 * node, c, i, W), c[i]);
          });
          phase_sync(wm);
          T* t = c; c = o; o = t;
        }
        each_node(k, tid, nt, [&](int i, int node, int, int) { o[i] = dot9<-1>(b[i], st + 9 * node, c, i, W); });
        phase_sync(wm);
        T* bc = sm + L.vec[g + 1];
        const bool compact = g + 1 == L.gm;
        each_node(L.k[g + 1], tid, nt, [&](int i, int node, int X, int Y) {
          const T* f = o + (2 * Y + 2) * W + 2 * X + 2;   // fine node (2X + 1, 2Y + 1)
          T acc = T(0);
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx)
              acc += ((dx == 0 ? T(1) : T(0.5)) * (dy == 0 ? T(1) : T(0.5))) * f[dy * W + dx];
          bc[compact ? node : i] = acc;
        });
        phase_sync(wm);
      }
    }
  }
  T* res = sm + L.vec[G - 1] + (L.gm < 0 ? vsize(G - 1) : cmx::B);
  for (int g = G - 2; g >= g0; --g) {
    const int W = (1 << L.k[g]) + 1, V = vsize(g), k = L.k[g], n = (W - 2) * (W - 2);
    const int Wc = (1 << L.k[g + 1]) + 1;
    const bool wm = wmode(g);
    const int nt = wm ? 32 : (int)blockDim.x;
    const T* st = sm + L.coef[g];
    const T* di = st + 9 * n;
    const T* b = sm + L.vec[g];
    T* c = sm + L.vec[g] + V;
    T* o = c + V;
    if (odd(nu - 1)) { T* t = c; c = o; o = t; }
    if (!wm && wmode(g + 1)) __syncthreads();   // results of warp 0
    if (!wm || tid < 32) {
      // bilinear interpolation: coarse node (X, Y) sits on fine (2X + 1, 2Y + 1);
      // the zero border stands for the coarse nodes outside
      const T* xc = res;
      each_node(k, tid, nt, [&](int i, int, int x, int y) {
        const int Xp = (x + 1) >> 1, Yp = (y + 1) >> 1;   // padded coarse index of the lower neighbour
        const T* q = xc + Yp * Wc + Xp;
        // weights 1 and 0 on odd coordinates, 1/2 and 1/2 on even ones: one
        // chain for every parity (the lanes of a warp hold both)
        const bool ox = x & 1, oy = y & 1;
        const T w1 = ox ? T(0) : (oy ? T(0.5) : T(0.25)), w2 = oy ? T(0) : (ox ? T(0.5) : T(0.25));
        const T w0 = ox ? (oy ? T(1) : T(0.5)) : (oy ? T(0.5) : T(0.25)), w3 = ox || oy ? T(0) : T(0.25);
        // a zero weight reads the lower neighbour (the upper one may hold anything)
        T v = fma(w0, q[0], c[i]);
        v = fma(w1, q[ox ? 0 : 1], v);
        v = fma(w2, q[oy ? 0 : Wc], v);
        v = fma(w3, q[ox || oy ? 0 : Wc + 1], v);
        c[i] = v;
      });
      phase_sync(wm);
      for (int s = 0; s < nu; ++s) {
        each_node(k, tid, nt, [&](int i, int node, int, int) {
          o[i] = fma(di[node], dot9<-1>(b[i], st + 9 * node, c, i, W), c[i]);
        });
        phase_sync(wm);
        T* t = c; c = o; o = t;
      }
    }
    else if (odd(nu)) c = o;
    res = c;
  }
  return res;
}

// Sum of v over the block, handed to f by one thread; ends with a barrier.
template <typename T, typename F>
__device__ __forceinline__ void block_sum(T* red, T v, F f) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    const T s = warp_sum(lane < (int)(blockDim.x >> 5) ? red[lane] : T(0));
    if (lane == 0) f((double)s);
  }
  __syncthreads();
}

template <typename TS, typename T, typename TD, int ITEMS>
__global__ void __launch_bounds__(blk::VNT) k_block_vcycle(BlockArgs a, BlockGrids L, T om, int nu,
                                                           const TS* __restrict__ src, int lds,
                                                           TD* __restrict__ dst, int ldd) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T red[blk::VNT / 32];
  __shared__ BlockScalars<T> S;
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int tid = threadIdx.x, NT = blockDim.x, col = blockIdx.x;
  const int k = L.k[0], m = 1 << k, nx = m - 1, W = m + 1, V = W * W;
  T* b = sm + L.vec[0];   // the residual is the V-cycle's right-hand side
  T* ps = sm + L.p;
  const T* st = sm + L.coef[0];
  T x[ITEMS], q[ITEMS], p[ITEMS];
  int pc[ITEMS], nd[ITEMS];
#pragma unroll
  for (int u = 0; u < ITEMS; ++u) {
    const int i = tid + u * NT, xx = i & nx, y = i >> k;
    const bool in = i < nx * m && xx < nx;
    nd[u] = in ? y * nx + xx : -1;
    pc[u] = in ? (y + 1) * W + xx + 1 : W + 1;
    x[u] = p[u] = q[u] = T(0);
  }
  stage_grids<T>(L, sm, om);
  for (int i = tid; i < V; i += NT) ps[i] = T(0);
  __syncthreads();
  {
    T rr = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u)
      if (nd[u] >= 0) {
        const T v = widen<T>(src[(size_t)nd[u] * lds + col]);
        b[pc[u]] = v;
        rr += v * v;
      }
    cp_async_wait_all();   // (published by the barriers of the sum)
    block_sum(red, rr, [&](double s) { scal_init(S, s, a); });
  }
  while (!S.done) {
    const T* z = block_vcycle<T>(L, sm, nu);   // ends with a block barrier
    T rz = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u)
      if (nd[u] >= 0) rz += b[pc[u]] * z[pc[u]];
    block_sum(red, rz, [&](double s) { scal_rho(S, s); });
    const T beta = S.beta;
    const bool first = S.it == 0;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u)
      if (nd[u] >= 0) {
        const T zv = z[pc[u]];
        p[u] = first ? zv : zv + beta * p[u];
        ps[pc[u]] = p[u];
      }
    __syncthreads();
    T pq = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u)
      if (nd[u] >= 0) {
        q[u] = dot9<1>(T(0), st + 9 * nd[u], ps, pc[u], W);
        pq = fma(p[u], q[u], pq);
      }
    block_sum(red, pq, [&](double s) { scal_alpha(S, s, a, true); });
    if (S.done) break;
    const T al = S.alpha;
    T rr = T(0);
#pragma unroll
    for (int u = 0; u < ITEMS; ++u)
      if (nd[u] >= 0) {
        x[u] += al * p[u];
        const T v = b[pc[u]] - al * q[u];
        b[pc[u]] = v;
        rr += v * v;
      }
    block_sum(red, rr, [&](double s) { scal_conv(S, s, a, true); });
  }
#pragma unroll
  for (int u = 0; u < ITEMS; ++u)
    if (nd[u] >= 0) dst[(size_t)nd[u] * ldd + col] = (TD)x[u];
  if (a.iters && tid == 0) a.iters[col] = S.it;
}

// The coarse end of the stand-alone V-cycle: everything from grid g0 down, one
// column at a time per block, the blocks striding over the columns (the grids'
// coefficients are staged once). Bounded by its chain of phases; 512 threads in
// FP32 (256 in FP64, where each phase waits for the FP64 units anyhow). From 31 x
// 31 nodes down, 20, 286 and 715 columns: 11, 17 and 37 us; the kernel before, of
// 1024 threads with boundary tests in its stencils, 17, 26 and 63.
template <typename T>
__global__ void __launch_bounds__(blk::CNT) k_vcycle_coarse(BlockGrids L, int g0, T om, int nu, int wp,
                                                            const T* __restrict__ bg, T* __restrict__ xg,
                                                            const int* __restrict__ done) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  T* b = sm + L.vec[g0];
  const int tid = threadIdx.x, NT = blockDim.x;
  bool staged = false;
  for (int col = blockIdx.x; col < wp; col += gridDim.x) {
    if (done[col]) continue;   // the same for every thread of the block
    if (!staged) {
      stage_grids<T>(L, sm, om, g0);
      __syncthreads();
      staged = true;
    }
    each_node(L.k[g0], tid, NT, [&](int i, int node, int, int) { b[i] = bg[(size_t)node * wp + col]; });
    cp_async_wait_all();
    __syncthreads();
    const T* z = block_vcycle<T>(L, sm, nu, g0);   // ends with a block barrier
    each_node(L.k[g0], tid, NT, [&](int i, int node, int, int) { xg[(size_t)node * wp + col] = z[i]; });
  }
}

// ------------------------------------------ V-cycle M_0 on 63 x 63, FP32 ---

// One block of 512 threads per column, as k_block_vcycle, but the finest
// grid's stencils live in registers (72 a thread: they are what a sweep from
// shared memory would read most of). Thread (y, s) owns the nodes 4 s .. 4 s + 3
// and 32 + 4 s .. of row y: a row is read as two 16-byte pieces per thread, the
// neighbours beside them come from the lanes beside it. The coarse grids run
// in shared memory through block_vcycle. What bounds it: the barriers and the
// chains between them (a step is 12.5 us, half of it on the coarse grids; 35% of
// the issue slots used, a warp waiting 2.6 clocks for shared memory and 2.0 at
// barriers of 11.2 between two instructions). Read node by node, the stencils
// took 4 us of a solve of two steps; from planes with rows of 64 they are whole
// lines.
namespace blk63 {
constexpr int NT = 512, NX = 63;
constexpr int W = 72;                 // row stride: node x at 4 + x, zeros around
constexpr int VEC = (NX + 2) * W;     // a vector with zero rows above and below
constexpr int OWN = 64 * 64;          // a vector read by its owners only
constexpr int FLOATS = 3 * VEC + 3 * OWN;
}  // namespace blk63

struct Own8 {   // a thread's eight nodes
  float v[8];
};

__device__ __forceinline__ Own8 own_ld(const float* p) {   // the second piece 32 nodes on
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 32);
  return Own8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
__device__ __forceinline__ void own_st(float* p, const Own8& o) {
  *reinterpret_cast<float4*>(p) = make_float4(o.v[0], o.v[1], o.v[2], o.v[3]);
  *reinterpret_cast<float4*>(p + 32) = make_float4(o.v[4], o.v[5], o.v[6], o.v[7]);
}

// acc + SIGN A v at the thread's nodes; v: its place in the padded vector
template <int SIGN>
__device__ __forceinline__ Own8 own_apply(Own8 acc, const float (&c)[8][9], const float* v, int s) {
#pragma unroll
  for (int dy = 0; dy < 3; ++dy) {
    const Own8 q = own_ld(v + (dy - 1) * blk63::W);
    // the nodes beside the two pieces, from the neighbouring lanes of the row
    // (0 beyond its ends: the coefficients there are zero)
    const float l0 = __shfl_sync(0xffffffffu, q.v[3], (s + 7) & 7, 8);
    const float l1 = __shfl_sync(0xffffffffu, s == 7 ? q.v[3] : q.v[7], (s + 7) & 7, 8);
    const float r0 = __shfl_sync(0xffffffffu, s == 0 ? q.v[4] : q.v[0], (s + 1) & 7, 8);
    const float r1 = __shfl_sync(0xffffffffu, q.v[4], (s + 1) & 7, 8);
    const float w0[6] = {s == 0 ? 0.f : l0, q.v[0], q.v[1], q.v[2], q.v[3], r0};
    const float w1[6] = {l1, q.v[4], q.v[5], q.v[6], q.v[7], s == 7 ? 0.f : r1};
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc.v[i] = fmaf(SIGN < 0 ? -c[i][dy * 3 + dx] : c[i][dy * 3 + dx], w0[i + dx], acc.v[i]);
        acc.v[4 + i] = fmaf(SIGN < 0 ? -c[4 + i][dy * 3 + dx] : c[4 + i][dy * 3 + dx], w1[i + dx], acc.v[4 + i]);
      }
  }
  return acc;
}

__device__ __forceinline__ float own_dot(const Own8& a, const Own8& b) {
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) s = fmaf(a.v[i], b.v[i], s);
  return s;
}

template <typename TS, typename TD>
__global__ void __launch_bounds__(blk63::NT, 1)
    k_block_vcycle63(BlockArgs a, BlockGrids L, float om, int nu, const float* __restrict__ planes,
                     const TS* __restrict__ src, int lds, TD* __restrict__ dst, int ldd) {
  using namespace blk63;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float red[NT / 32];
  __shared__ BlockScalars<float> S;
  float* const X = reinterpret_cast<float*>(smem_raw);   // X, Y, P: [VEC]; B, D, U: [OWN]
  float* const Y = X + VEC;
  float* const P = Y + VEC;
  float* const sm = X + FLOATS;                           // the coarse grids
  const int tid = threadIdx.x, col = blockIdx.x, s = tid & 7, y = tid >> 3;
  const bool act = y < NX;
  const int at = (min(y, NX - 1) + 1) * W + 4 + 4 * s;    // the thread's place in a padded vector
  float* const B = P + VEC + y * 64 + 4 * s;              // residual, damped inverse diagonal, solution
  float* const D = B + OWN;
  float* const U = D + OWN;
  for (int i = tid; i < 3 * VEC; i += NT) X[i] = 0.f;
  stage_grids<float>(L, sm, om, 1);
  float c[8][9];
  {
    Own8 b;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int x = 4 * s + (i & 3) + (i >= 4 ? 32 : 0);
      b.v[i] = act && x < NX ? widen<float>(src[(size_t)(y * NX + x) * lds + col]) : 0.f;
    }
    // the planes' rows are padded with zeros to 64 columns; the last thread row
    // takes the last grid row's and never publishes what it makes of them
    const float* pl = planes + min(y, NX - 1) * 64 + 4 * s;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const Own8 q = own_ld(pl + e * NX * 64);
#pragma unroll
      for (int i = 0; i < 8; ++i) c[i][e] = act ? q.v[i] : 0.f;
    }
    Own8 d = own_ld(pl + 9 * NX * 64);
#pragma unroll
    for (int i = 0; i < 8; ++i) d.v[i] = act ? om * d.v[i] : 0.f;
    own_st(D, d);
    own_st(B, b);
    own_st(U, Own8{{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}});
    cp_async_wait_all();   // (published by the barriers of the sum)
    block_sum(red, own_dot(b, b), [&](double v) { scal_init(S, v, a); });
  }
  while (!S.done) {
    Own8 cur;
    {
      const Own8 b = own_ld(B), d = own_ld(D);
#pragma unroll
      for (int i = 0; i < 8; ++i) cur.v[i] = d.v[i] * b.v[i];
    }
    float *v = X, *o = Y;
    if (act) own_st(v + at, cur);
    __syncthreads();
    // one more sweep of the iterate in v, its new values in cur
    auto sweep = [&]() {
      const Own8 r = own_apply<-1>(own_ld(B), c, v + at, s), d = own_ld(D);
#pragma unroll
      for (int i = 0; i < 8; ++i) cur.v[i] = fmaf(d.v[i], r.v[i], cur.v[i]);
    };
    auto publish = [&]() {
      if (act) own_st(o + at, cur);
      __syncthreads();
      float* t = v; v = o; o = t;
    };
    for (int it = 1; it < nu; ++it) {
      sweep();
      publish();
    }
    {
      const Own8 r = own_apply<-1>(own_ld(B), c, v + at, s);
      if (act) own_st(o + at, r);
    }
    __syncthreads();
    {
      float* bc = sm + L.vec[1];
      each_node(5, tid, NT, [&](int i, int, int Xc, int Yc) {
        const float* q = o + (2 * Yc + 2) * W + 4 + 2 * Xc + 1;   // fine node (2 Xc + 1, 2 Yc + 1)
        float acc = 0.f;
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx)
            acc += ((dx == 0 ? 1.f : 0.5f) * (dy == 0 ? 1.f : 0.5f)) * q[dy * W + dx];
        bc[i] = acc;
      });
    }
    __syncthreads();
    const float* xc = block_vcycle<float>(L, sm, nu, 1);   // ends with a block barrier
    {
      // coarse nodes 2 s' - 1 .. 2 s' + 1 beside each piece (s' = s, s + 8)
      const int Yl = (min(y, NX - 1) + 1) >> 1;
      const bool oy = y & 1;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        const float* q = xc + Yl * 33 + 2 * (s + 8 * g);
        float c0 = q[0], c1 = q[1], c2 = q[2];
        if (!oy) {
          c0 = 0.5f * (c0 + q[33]);
          c1 = 0.5f * (c1 + q[34]);
          c2 = 0.5f * (c2 + q[35]);
        }
        cur.v[4 * g] += 0.5f * (c0 + c1);
        cur.v[4 * g + 1] += c1;
        cur.v[4 * g + 2] += 0.5f * (c1 + c2);
        cur.v[4 * g + 3] += c2;
      }
      if (!act) cur = Own8{{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}};
    }
    publish();
    for (int it = 0; it < nu; ++it) {
      sweep();
      if (it + 1 < nu) publish();
    }
    block_sum(red, own_dot(own_ld(B), cur), [&](double t) { scal_rho(S, t); });
    {
      const float beta = S.beta;
      if (S.it > 0) {
        const Own8 p = own_ld(P + at);
#pragma unroll
        for (int i = 0; i < 8; ++i) cur.v[i] = fmaf(beta, p.v[i], cur.v[i]);
      }
      if (act) own_st(P + at, cur);
    }
    __syncthreads();
    Own8 q = own_apply<1>(Own8{{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}}, c, P + at, s);
    block_sum(red, act ? own_dot(cur, q) : 0.f, [&](double t) { scal_alpha(S, t, a, true); });
    if (S.done) break;
    {
      const float al = S.alpha;
      Own8 u = own_ld(U), b = own_ld(B);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        u.v[i] = fmaf(al, cur.v[i], u.v[i]);
        b.v[i] = fmaf(-al, q.v[i], b.v[i]);
      }
      own_st(U, u);
      own_st(B, b);
      block_sum(red, own_dot(b, b), [&](double t) { scal_conv(S, t, a, true); });
    }
  }
  if (act) {
    const Own8 u = own_ld(U);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int x = 4 * s + (i & 3) + (i >= 4 ? 32 : 0);
      if (x < NX) dst[(size_t)(y * NX + x) * ldd + col] = (TD)u.v[i];
    }
  }
  if (a.iters && tid == 0) a.iters[col] = S.it;
}

// ------------------------------------------------------------ host side ---

// Blocks per column of k_block_diag: as many (up to MAX_C) as leave an SM to
// every block of the batch and at least two warps of nodes to each block, and
// no fewer than hold the grid at MAX_ITEMS nodes a thread; 0 when that many
// do not fit in a cluster.
static int diag_split(const sg_problem* h, const GridLevel& G, int w) {
  using namespace blk;
  int C = 1;
  while (C < MAX_C && (w * 2 * C <= h->num_sms) && G.n / (2 * C) >= 64 && G.ny >= 4 * C) C *= 2;
  while (C <= MAX_C && ceil_div(G.ny, C) * G.nx > NT * MAX_ITEMS) C *= 2;
  return C <= MAX_C && C <= G.ny ? C : 0;
}

// Shared-memory layout of the grids from g0 on (0; 1 for k_block_vcycle63,
// which keeps the finest one elsewhere, in `before` bytes).
static bool vcycle_layout(const sg_problem* h, size_t es, const sg_prec_opts& o, BlockGrids& L, int g0 = 0,
                          size_t before = 0) {
  L = BlockGrids{};
  L.G = (int)h->grids.size();
  L.gm = h->cmat_base && o.nu == 2 && o.omega == 0.8 ? L.G - 3 : -1;   // (7 x 7, 3 x 3 and one node)

  if (!h->mg_full || L.G <= g0 || L.G > blk::MAX_GRIDS || h->grids[g0].n > 1024) return false;
  int off = 0;
  for (int g = g0; g < L.G; ++g) {
    const GridLevel& G = h->grids[g];
    int k = 0;
    while ((1 << k) < G.nx + 1) ++k;
    if (G.nx != G.ny || (1 << k) != G.nx + 1) return false;
    L.k[g] = k;
    L.vec[g] = off;
    if (g == L.gm) {
      off += cmx::VECS;
      L.coef[g] = off;
      off += cmx::COEFS;
      L.st[g] = es == 8 ? (const void*)h->cmat64 : (const void*)h->cmat32;
      break;
    }
    off += 3 * (G.nx + 2) * (G.nx + 2);
    L.coef[g] = off;
    off += 10 * G.n;
    L.st[g] = es == 8 ? (const void*)G.st64 : (const void*)G.st32;
    L.dinv[g] = es == 8 ? (const void*)G.dinv64 : (const void*)G.dinv32;
  }
  L.p = off;
  if (g0 == 0) off += (h->grids[0].nx + 2) * (h->grids[0].nx + 2);
  L.total = off;
  return before + (size_t)off * es <= (size_t)std::max(h->smem_optin, 48 * 1024) - 2048;
}

static bool layout63(const sg_problem* h, const sg_prec_opts& o, BlockGrids& L) {
  return !h->grids.empty() && h->grids[0].planes &&
         vcycle_layout(h, 4, o, L, 1, blk63::FLOATS * sizeof(float));
}

// FP32 V-cycle solves for which the block solvers are the faster ones: every
// grid up to 63 x 63. sg_inner_solve with two steps, clusters and blocks: 15 x
// 15 nodes 89 and 75 us (20 columns), 100 and 73 (100); 31 x 31 100 and 87, 121
// and 90; 63 x 63 112 and 100, 154 and 107. Which batches take them:
// cluster_path in inner_cluster.cu.
bool block_preferred(const sg_problem* h) {
  if (h->block_off || h->grids.empty()) return false;
  sg_prec_opts o;   // the default smoothing: the larger layout
  sg_default_prec_opts(&o);
  BlockGrids L;
  return vcycle_layout(h, 4, o, L) || layout63(h, o, L);
}

bool block_usable(const sg_problem* h, int dtype, int w, const sg_prec_opts& o) {
  if (h->block_off || h->grids.empty() || w <= 0) return false;
  const GridLevel& G = h->grids[0];
  if (o.m0 == SG_M0_DIAG) {
    const int C = diag_split(h, G, w);
    const size_t es = dtype == SG_F64 ? 8 : 4;
    return C > 0 && ((size_t)(ceil_div(G.ny, C) + 2) * (G.nx + 2) + 6 * (size_t)G.nx) * es <= 40 * 1024;
  }
  BlockGrids L;
  return vcycle_layout(h, dtype == SG_F64 ? 8 : 4, o, L) || (dtype == SG_F32 && layout63(h, o, L));
}

template <typename TS, typename T, typename TD>
static int solve_block_t(sg_problem* h, const TS* src, int lds, TD* dst, int ldd, int w, const sg_prec_opts& o,
                         cudaStream_t s) {
  using namespace blk;
  const GridLevel& G = h->grids[0];
  const InnerWork& iw = sizeof(T) == 8 ? h->iw64 : h->iw32;
  BlockArgs a;
  a.n = G.n;
  a.nx = G.nx;
  a.ny = G.ny;
  a.w = w;
  a.C = a.R = 1;
  a.tol2 = o.inner_tol * o.inner_tol;
  a.maxit = o.inner_maxit;
  a.fixed = o.inner_fixed_iters;
  a.status = h->status;
  a.iacc = h->iacc;
  a.iters = iw.iters && iw.wcap >= w ? iw.iters : nullptr;
  const T* st = sizeof(T) == 8 ? (const T*)G.st64 : (const T*)G.st32;
  const T* dinv = sizeof(T) == 8 ? (const T*)G.dinv64 : (const T*)G.dinv32;
  if (o.m0 == SG_M0_DIAG) {
    a.C = diag_split(h, G, w);
    a.R = ceil_div(G.ny, a.C);
    // one warp per SM quarter (each has its own FP64 unit), more nodes a thread
    // beyond that: a second warp would repeat the warp sums, not speed them up
    const int nodes = a.R * G.nx;
    const int threads = nodes > 128 * MAX_ITEMS ? NT : std::min(128, ceil_div(nodes, 32) * 32);
    const int items = ceil_div(nodes, threads);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(w * a.C));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = diag_smem<T>(a.R, G.nx);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = a.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (items <= 1)
      SG_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_block_diag<TS, T, TD, 1>, a, st, dinv, src, lds, dst, ldd));
    else if (items <= 2)
      SG_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_block_diag<TS, T, TD, 2>, a, st, dinv, src, lds, dst, ldd));
    else
      SG_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_block_diag<TS, T, TD, 4>, a, st, dinv, src, lds, dst, ldd));
    note_launch();
    return SG_OK;
  }
  BlockGrids L;
  if constexpr (sizeof(T) == 4) {
    if (layout63(h, o, L)) {
      const size_t smem = (blk63::FLOATS + (size_t)L.total) * sizeof(float);
      auto kern = k_block_vcycle63<TS, TD>;
      SG_TRY(allow_smem(h, kern));
      { kern<<<w, blk63::NT, smem, s>>>(a, L, (float)o.omega, o.nu, G.planes, src, lds, dst, ldd); note_launch(); }
      SG_CHECK_LAUNCH();
      return SG_OK;
    }
  }
  if (!vcycle_layout(h, sizeof(T), o, L)) {
    set_error("block inner solve: the hierarchy does not fit");
    return SG_ERR_UNSUPPORTED;
  }
  const size_t smem = (size_t)L.total * sizeof(T);
  auto go = [&](auto kern, int threads) -> int {
    SG_TRY(allow_smem(h, kern));
    { kern<<<w, threads, smem, s>>>(a, L, (T)o.omega, o.nu, src, lds, dst, ldd); note_launch(); }
    SG_CHECK_LAUNCH();
    return SG_OK;
  };
  if (G.nx <= 15) return go(k_block_vcycle<TS, T, TD, 2>, 128);
  return go(k_block_vcycle<TS, T, TD, 4>, 256);
}

template <typename T>
static int launch_coarse_t(sg_problem* h, int g0, const T* b, T* x, int wp, const sg_prec_opts& o, const int* done,
                           cudaStream_t s) {
  BlockGrids L;
  if (!vcycle_layout(h, sizeof(T), o, L, g0)) {
    set_error("V-cycle: the coarse grids do not fit");
    return SG_ERR_UNSUPPORTED;
  }
  const size_t smem = (size_t)L.total * sizeof(T);
  const int threads = h->grids[g0].nx <= 15 ? 128 : sizeof(T) == 8 ? blk::VNT : blk::CNT;
  // as many blocks as are resident: beyond that each column would stage the grids anew
  const int per_sm = std::max(1, (int)((h->smem_optin + 1024) / (smem + 1024)));
  SG_TRY(allow_smem(h, k_vcycle_coarse<T>));
  { k_vcycle_coarse<T><<<std::min(wp, h->num_sms * std::min(per_sm, 4)), threads, smem, s>>>(L, g0, (T)o.omega, o.nu, wp, b, x, done); note_launch(); }
  SG_CHECK_LAUNCH();
  return SG_OK;
}

int launch_coarse(sg_problem* h, int dtype, int g0, const void* b, void* x, int wp, const sg_prec_opts& o,
                  const int* done, cudaStream_t s) {
  if (dtype == SG_F64) return launch_coarse_t<double>(h, g0, (const double*)b, (double*)x, wp, o, done, s);
  return launch_coarse_t<float>(h, g0, (const float*)b, (float*)x, wp, o, done, s);
}

int inner_solve_block(sg_problem* h, int dtype, const void* src, int lds, int src_t, void* dst, int ldd, int dst_t,
                      int w, const sg_prec_opts& o, cudaStream_t s) {
  const bool s64 = src_t == SG_F64, d64 = dst_t == SG_F64;
  if (dtype == SG_F64) {
    if (s64 && d64) return solve_block_t<double, double, double>(h, (const double*)src, lds, (double*)dst, ldd, w, o, s);
    set_error("block inner solve: FP64 solves take FP64 blocks");
    return SG_ERR_UNSUPPORTED;
  }
  if (s64 && d64) return solve_block_t<double, float, double>(h, (const double*)src, lds, (double*)dst, ldd, w, o, s);
  if (s64) return solve_block_t<double, float, float>(h, (const double*)src, lds, (float*)dst, ldd, w, o, s);
  if (d64) return solve_block_t<float, float, double>(h, (const float*)src, lds, (double*)dst, ldd, w, o, s);
  return solve_block_t<float, float, float>(h, (const float*)src, lds, (float*)dst, ldd, w, o, s);
}

}  // namespace sghsc
