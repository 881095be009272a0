// Problem setup: validation of the inputs, the chaos tables and the sparse G_k
// couplings (Sec. 2, eq. (gPC-u), (global-system); Sec. 3), and the Galerkin
// multigrid hierarchy of the mean-value matrix A_0 used by the inner solves.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <atomic>
#include <map>

#include "df64.cuh"
#include "graph.cuh"
#include "sghsc_internal.cuh"

namespace sghsc {

static thread_local char g_err[1024] = "";
static std::atomic<long long> g_launches{0};

void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
}

// Graded multi-indices; inside one degree, descending lexicographic order.
static void emit_degree(int M, int pos, int remaining, std::vector<int>& cur, std::vector<int>& out) {
  if (pos == M - 1) {
    cur[pos] = remaining;
    out.insert(out.end(), cur.begin(), cur.end());
    return;
  }
  for (int a = remaining; a >= 0; --a) {
    cur[pos] = a;
    emit_degree(M, pos + 1, remaining - a, cur, out);
  }
}

// E[xi psi_m psi_{m+1}] for the orthonormal 1-D family. Legendre with
// xi ~ U(-sqrt3, sqrt3): sqrt3 (m+1) / sqrt((2m+1)(2m+3)); Hermite with
// xi ~ N(0,1): sqrt(m+1).
static double xi_coupling(int m, int family) {
  if (family == SG_HERMITE) return std::sqrt((double)m + 1.0);
  return std::sqrt(3.0) * (m + 1.0) / std::sqrt((2.0 * m + 1.0) * (2.0 * m + 3.0));
}

template <typename T>
static int upload(T** dst, const T* src, size_t count) {
  if (count == 0) {
    *dst = nullptr;
    return SG_OK;
  }
  SG_TRY_CUDA(cudaMalloc((void**)dst, count * sizeof(T)));
  SG_TRY_CUDA(cudaMemcpy(*dst, src, count * sizeof(T), cudaMemcpyHostToDevice));
  return SG_OK;
}

// FP32 stencils [n][9] and inverse diagonals into 48-byte records and planes
// (GridLevel::st12, planes)
__global__ void k_pack_stencil(int nx, int ny, const float* __restrict__ st, const float* __restrict__ dinv,
                               float* __restrict__ st12, float* __restrict__ planes) {
  const int n = nx * ny;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * 12; i += gridDim.x * blockDim.x) {
    const int node = i / 12, e = i - node * 12, c = e & 3;
    const float v = c < 3 ? st[node * 9 + e / 4 * 3 + c] : (e == 11 ? dinv[node] : 0.f);
    st12[i] = v;
    const int plane = c < 3 ? e / 4 * 3 + c : (e == 11 ? 9 : -1);
    if (planes && plane >= 0) planes[(plane * ny + node / nx) * (nx + 1) + node % nx] = v;
  }
}

static int pack_stencils(GridLevel& g) {
  { k_pack_stencil<<<std::min((g.n * 12 + 255) / 256, 4096), 256>>>(g.nx, g.ny, g.st32, g.dinv32, g.st12, g.planes); ::sghsc::note_launch(); }
  SG_CHECK_LAUNCH();
  return SG_OK;
}

struct HostEdges {
  std::vector<int> ptr{0}, k, j;
  std::vector<double> c;
};

// The order in which the 32 output slots of a warp take their couplings, so
// that the words a warp reads together lie in different shared-memory banks
// (in list order a step's reads met up to eight deep in one bank). addr[s]:
// word address of each coupling of slot s; entry c * 32 + s of the result is
// the coupling that slot s takes at step c, or -1 (padding). As many steps as
// the longest list. Greedy: at each step the slots with most left choose
// first, the address that shares its bank with the fewest others; a slot with
// steps to spare waits rather than collide.
static std::vector<int> schedule_warp(const std::vector<int>* addr, int n) {
  int rows = 0;
  std::vector<int> left[32];
  int demand[32] = {0}, order[32];
  for (int s = 0; s < n; ++s) {
    rows = std::max(rows, (int)addr[s].size());
    order[s] = s;
    for (int i = 0; i < (int)addr[s].size(); ++i) {
      left[s].push_back(i);
      ++demand[addr[s][i] & 31];
    }
  }
  std::vector<int> take((size_t)rows * 32, -1);
  if (rows > 64) {   // the dense couplings of a gPC coefficient: list order (the search is quadratic)
    for (int s = 0; s < n; ++s)
      for (int r = 0; r < (int)addr[s].size(); ++r) take[(size_t)r * 32 + s] = r;
    return take;
  }
  for (int r = 0; r < rows; ++r) {
    int cnt[32] = {0}, seen[32][32];   // distinct addresses read so far, by bank
    auto in = [&](int a) {
      for (int i = 0; i < cnt[a & 31]; ++i)
        if (seen[a & 31][i] == a) return true;
      return false;
    };
    std::stable_sort(order, order + n, [&](int a, int b) { return left[a].size() > left[b].size(); });
    for (int o = 0; o < n; ++o) {
      const int s = order[o];
      int best = -1, cost = 0;
      for (int q = 0; q < (int)left[s].size(); ++q) {
        const int a = addr[s][left[s][q]], c = in(a) ? 0 : cnt[a & 31];
        if (best < 0 || c < cost || (c == cost && demand[a & 31] > demand[addr[s][left[s][best]] & 31])) {
          best = q;
          cost = c;
        }
      }
      if (best < 0 || (cost > 0 && (int)left[s].size() < rows - r)) continue;
      const int a = addr[s][left[s][best]];
      if (!in(a)) seen[a & 31][cnt[a & 31]++] = a;
      --demand[a & 31];
      take[(size_t)r * 32 + s] = left[s][best];
      left[s].erase(left[s].begin() + best);
    }
  }
  return take;
}

static int upload_edges(const HostEdges& he, EdgeList& E, int out0, int in0, int nin, int terms) {
  E.out0 = out0;
  E.in0 = in0;
  E.nin = nin;
  E.nout = (int)he.ptr.size() - 1;
  E.nedges = (int)he.k.size();
  std::vector<float> c32(he.c.begin(), he.c.end());
  // Outputs ordered by their number of couplings, so the lanes of a warp run
  // coupling loops of equal length (equal counts keep column order).
  std::vector<int> perm(E.nout);
  for (int l = 0; l < E.nout; ++l) perm[l] = l;
  std::stable_sort(perm.begin(), perm.end(), [&](int a, int b) {
    return he.ptr[a + 1] - he.ptr[a] > he.ptr[b + 1] - he.ptr[b];
  });
  SG_TRY(upload(&E.perm, perm.data(), perm.size()));
  SG_TRY(upload(&E.ptr, he.ptr.data(), he.ptr.size()));
  SG_TRY(upload(&E.k, he.k.data(), he.k.size()));
  SG_TRY(upload(&E.j, he.j.data(), he.j.size()));
  SG_TRY(upload(&E.c64, he.c.data(), he.c.size()));
  SG_TRY(upload(&E.c32, c32.data(), c32.size()));
  {
    std::vector<df64> cdf(he.c.size());
    for (size_t t = 0; t < he.c.size(); ++t) cdf[t] = df_split_host(he.c[t]);
    df64* d = nullptr;
    SG_TRY(upload(&d, cdf.data(), cdf.size()));
    E.cdf = d;
  }
  std::map<std::pair<int, int>, int> pairs;
  for (int t = 0; t < E.nedges; ++t) pairs.emplace(std::make_pair(he.k[t], he.j[t]), 0);
  std::vector<int> pk, pj, pair(E.nedges);
  for (auto& kv : pairs) {
    kv.second = (int)pk.size();
    pk.push_back(kv.first.first);
    pj.push_back(kv.first.second);
  }
  for (int t = 0; t < E.nedges; ++t) pair[t] = pairs.at(std::make_pair(he.k[t], he.j[t]));
  E.npair = (int)pk.size();
  {
    std::vector<unsigned> w(pk.size());
    bool fits = true;
    for (size_t q = 0; q < pk.size(); ++q) {
      fits = fits && pk[q] * DF_VS < 65536 && pj[q] * DF_XS < 65536;
      w[q] = ((unsigned)(pk[q] * DF_VS) << 16) | (unsigned)(pj[q] * DF_XS);
    }
    if (fits && pk.size() < (1u << 20)) SG_TRY(upload(&E.pkj, w.data(), w.size()));
  }
  {
    // coefficient classes; class 0 is the coefficient 0, which pads the shorter
    // slots of a warp to the warp's longest
    std::map<double, int> cls;
    for (double c : he.c) cls.emplace(c, 0);
    if (cls.size() + (cls.count(0.0) ? 0 : 1) <= 256 && E.npair < (1 << 24)) {
      std::vector<df64> tab{df64(0.f, 0.f)};
      std::vector<float> tab32{0.f};
      for (auto& kv : cls) {
        if (kv.first == 0.0) continue;
        kv.second = (int)tab.size();
        tab.push_back(df_split_host(kv.first));
        tab32.push_back((float)kv.first);
      }
      SG_TRY(upload(&E.ctab32, tab32.data(), tab32.size()));
      // slot-transposed packing: warp w (slots 32w .. 32w+31, counts sorted
      // descending) takes 32 words per coupling of its first slot, and 32 more
      // for an even number
      auto steps = [&](int sl) { return (he.ptr[perm[sl & ~31] + 1] - he.ptr[perm[sl & ~31]] + 1) & ~1; };
      std::vector<int> tb(E.nout);
      size_t total = 0;
      for (int w0 = 0; w0 < E.nout; w0 += 32) {
        const int cmax = steps(w0);
        for (int sl = w0; sl < std::min(w0 + 32, E.nout); ++sl) tb[sl] = (int)total + (sl - w0);
        total += (size_t)32 * cmax;
      }
      if (total >= (size_t)1 << 31) return SG_ERR_UNSUPPORTED;
      std::vector<unsigned> packed(std::max<size_t>(total, 1), 0u), pkj;
      E.rows32 = rows32_rows(nin, E.nout, nin == E.nout && in0 == out0, terms);
      const int wts = rows32_stride(nin, E.rows32);   // the row stride of the FP32 row kernel's term sums
      const bool kj_ok = (long long)terms * wts < (1 << 24);
      if (kj_ok) pkj.assign(packed.size(), (unsigned)(terms * wts));
      std::vector<unsigned> cof(E.nedges);
      for (int t = 0; t < E.nedges; ++t) cof[t] = (unsigned)cls.at(he.c[t]);
      for (int w0 = 0; w0 < E.nout; w0 += 32) {
        const int ws = std::min(32, E.nout - w0);
        std::vector<int> as[32];   // words of the double-float products' sums
        for (int i = 0; i < ws; ++i) {
          const int l = perm[w0 + i];
          for (int t = he.ptr[l]; t < he.ptr[l + 1]; ++t) {
            as[i].push_back(pair[t]);
            // the FP32 row kernel adds in list order (the bits of the gather form)
            if (kj_ok)
              pkj[(size_t)tb[w0 + i] + 32 * (t - he.ptr[l])] = cof[t] << 24 | (unsigned)(he.k[t] * wts + he.j[t]);
          }
        }
        const std::vector<int> ss = schedule_warp(as, ws);
        for (int c = 0; c < steps(w0); ++c)
          for (int i = 0; i < ws; ++i) {
            const int qs = (size_t)c * 32 < ss.size() ? ss[c * 32 + i] : -1, own = as[i].empty() ? 0 : as[i][0];
            packed[(size_t)tb[w0 + i] + 32 * c] =
                qs < 0 ? (unsigned)own << 12 : (unsigned)as[i][qs] << 12 | cof[he.ptr[perm[w0 + i]] + qs] << 2;
          }
      }
      if (E.nout < 65536) {
        // per slot: its first word and (output << 16 | steps of its warp), so the
        // lanes of a warp run the same coupling loop
        std::vector<int2> sd(E.nout);
        bool ok = true;
        for (int sl = 0; sl < E.nout; ++sl) {
          const int l = perm[sl], cnt = steps(sl);
          ok = ok && cnt < 65536;
          sd[sl] = make_int2(tb[sl], (int)(((unsigned)l << 16) | (unsigned)cnt));
        }
        if (ok) {
          SG_TRY(upload(&E.sdesc, sd.data(), sd.size()));
          if (kj_ok) SG_TRY(upload(&E.ckj, pkj.data(), pkj.size()));
        }
      }
      df64* dt = nullptr;
      SG_TRY(upload(&E.ctr, packed.data(), packed.size()));
      SG_TRY(upload(&dt, tab.data(), tab.size()));
      E.ctab = dt;
      E.ncls = (int)tab.size();
    }
  }
  SG_TRY(upload(&E.pk, pk.data(), pk.size()));
  SG_TRY(upload(&E.pj, pj.data(), pj.size()));
  SG_TRY(upload(&E.pair, pair.data(), pair.size()));
  return SG_OK;
}

static void free_edges(EdgeList& E) {
  cudaFree(E.perm);
  cudaFree(E.ptr);
  cudaFree(E.k);
  cudaFree(E.j);
  cudaFree(E.c64);
  cudaFree(E.c32);
  cudaFree(E.cdf);
  cudaFree(E.ctr);
  cudaFree(E.ckj);
  cudaFree(E.sdesc);
  cudaFree(E.ctab);
  cudaFree(E.ctab32);
  cudaFree(E.pkj);
  cudaFree(E.pk);
  cudaFree(E.pj);
  cudaFree(E.pair);
  E = EdgeList();
}

// E[psi_a psi_b psi_c] of normalised 1-D Hermite polynomials: with s = (a+b+c)/2,
// sqrt(a! b! c!) / ((s-a)! (s-b)! (s-c)!) when s is an integer >= a, b, c, else 0.
static double hermite_triple(int a, int b, int c) {
  const int t = a + b + c;
  if (t & 1) return 0.0;
  const int s = t / 2;
  if (s < a || s < b || s < c) return 0.0;
  return std::exp(0.5 * (std::lgamma(a + 1.0) + std::lgamma(b + 1.0) + std::lgamma(c + 1.0)) -
                  std::lgamma(s - a + 1.0) - std::lgamma(s - b + 1.0) - std::lgamma(s - c + 1.0));
}

// Couplings of a gPC-expanded coefficient (Remark K-L): for every output l of
// [lo_out, hi_out) and input j of [lo_in, hi_in), every coefficient term
// i >= 1 with c = E[psi_i psi_j psi_l] != 0 (the product of the 1-D Hermite
// triple products over the coordinates). The term i = 0 is the identity
// (E[psi_j psi_l] = delta_jl): the diagonal part of the product kernels.
static HostEdges build_edges_gpc(const sg_problem* h, int lo_out, int hi_out, int lo_in, int hi_in) {
  HostEdges he;
  const int M = h->M;
  for (int l = lo_out; l < hi_out; ++l) {
    const int* al = h->alpha.data() + (size_t)l * M;
    for (int j = lo_in; j < hi_in; ++j) {
      const int* aj = h->alpha.data() + (size_t)j * M;
      for (int i = 1; i < h->nterm; ++i) {
        const int* gi = h->gamma.data() + (size_t)i * M;
        double c = 1.0;
        for (int k = 0; k < M && c != 0.0; ++k) c *= hermite_triple(gi[k], aj[k], al[k]);
        if (c == 0.0) continue;
        he.k.push_back(i);
        he.j.push_back(j - lo_in);
        he.c.push_back(c);
      }
    }
    he.ptr.push_back((int)he.k.size());
  }
  return he;
}

// Build the gather-form couplings. For every output column l of [lo_out, hi_out)
// and every KL index k, the neighbours alpha_l +- e_k inside [lo_in, hi_in).
static HostEdges build_edges(const sg_problem* h, const std::map<std::vector<int>, int>& index, int lo_out,
                             int hi_out, int lo_in, int hi_in) {
  HostEdges he;
  const int M = h->M;
  std::vector<int> b(M);
  for (int l = lo_out; l < hi_out; ++l) {
    const int* a = h->alpha.data() + (size_t)l * M;
    for (int k = 0; k < M; ++k) {
      for (int step = -1; step <= 1; step += 2) {
        for (int i = 0; i < M; ++i) b[i] = a[i];
        b[k] += step;
        if (b[k] < 0) continue;
        auto it = index.find(b);
        if (it == index.end()) continue;
        int j = it->second;
        if (j < lo_in || j >= hi_in) continue;
        he.k.push_back(k + 1);
        he.j.push_back(j - lo_in);
        he.c.push_back(xi_coupling(std::min(a[k], b[k]), h->family));
      }
    }
    he.ptr.push_back((int)he.k.size());
  }
  return he;
}

// Bilinear prolongation weight of coarse node X (fine position 2X+1) at fine node x.
static inline double w1(int d) { return d == 0 ? 1.0 : ((d == 1 || d == -1) ? 0.5 : 0.0); }

// Galerkin coarse stencil P^T A P for full coarsening with bilinear P.
static void galerkin_coarsen(int nx, int ny, const std::vector<double>& st, int nxc, int nyc,
                             std::vector<double>& stc) {
  stc.assign((size_t)nxc * nyc * 9, 0.0);
  for (int Y = 0; Y < nyc; ++Y) {
    for (int X = 0; X < nxc; ++X) {
      const size_t C = (size_t)Y * nxc + X;
      const int cxf = 2 * X + 1, cyf = 2 * Y + 1;
      for (int fy = cyf - 1; fy <= cyf + 1; ++fy) {
        for (int fx = cxf - 1; fx <= cxf + 1; ++fx) {
          const double wf = w1(fx - cxf) * w1(fy - cyf);
          const size_t f = (size_t)fy * nx + fx;
          for (int s = 0; s < 9; ++s) {
            const double a = st[f * 9 + s];
            if (a == 0.0) continue;
            const int gx = fx + (s % 3 - 1), gy = fy + (s / 3 - 1);
            int Xs[2], Ys[2];
            double wx[2], wy[2];
            int nxs = 0, nys = 0;
            if (gx & 1) { Xs[nxs] = (gx - 1) / 2; wx[nxs++] = 1.0; }
            else { Xs[nxs] = gx / 2 - 1; wx[nxs++] = 0.5; Xs[nxs] = gx / 2; wx[nxs++] = 0.5; }
            if (gy & 1) { Ys[nys] = (gy - 1) / 2; wy[nys++] = 1.0; }
            else { Ys[nys] = gy / 2 - 1; wy[nys++] = 0.5; Ys[nys] = gy / 2; wy[nys++] = 0.5; }
            for (int iy = 0; iy < nys; ++iy) {
              if (Ys[iy] < 0 || Ys[iy] >= nyc) continue;
              for (int ix = 0; ix < nxs; ++ix) {
                if (Xs[ix] < 0 || Xs[ix] >= nxc) continue;
                const int dX = Xs[ix] - X, dY = Ys[iy] - Y;
                stc[C * 9 + (dY + 1) * 3 + (dX + 1)] += wf * a * wx[ix] * wy[iy];
              }
            }
          }
        }
      }
    }
  }
}

// The matrix of one V-cycle (two damped Jacobi sweeps, omega 0.8, before and
// after; the one-node grid exactly) on a grid of m x m nodes; st: the stencils
// of this grid and of those below it. In FP64, for all unit right-hand sides at
// once: vectors are [m m][N] with N columns.
static std::vector<double> vcycle_columns(const std::vector<double>* st, int m, int N, const std::vector<double>& b) {
  const int n = m * m;
  const std::vector<double>& s9 = *st;
  std::vector<double> x((size_t)n * N, 0.0), r(b);
  auto add = [N](double* to, double a, const double* from) {
    for (int j = 0; j < N; ++j) to[j] += a * from[j];
  };
  if (m == 1) {
    add(x.data(), 1.0 / s9[4], b.data());
    return x;
  }
  auto residual = [&]() {
    r = b;
    for (int i = 0; i < n; ++i)
      for (int e = 0; e < 9; ++e) {
        const int X = i % m + e % 3 - 1, Y = i / m + e / 3 - 1;
        if (X >= 0 && Y >= 0 && X < m && Y < m) add(&r[(size_t)i * N], -s9[i * 9 + e], &x[(size_t)(Y * m + X) * N]);
      }
  };
  auto sweep = [&]() {   // r is the residual of x on entry
    for (int i = 0; i < n; ++i) add(&x[(size_t)i * N], 0.8 / s9[i * 9 + 4], &r[(size_t)i * N]);
    residual();
  };
  sweep();
  sweep();
  const int mc = (m - 1) / 2;
  auto transfer = [&](auto f) {   // f(coarse node, fine node, weight)
    for (int c = 0; c < mc * mc; ++c)
      for (int e = 0; e < 9; ++e)
        f(c, (2 * (c / mc) + e / 3) * m + 2 * (c % mc) + e % 3, (e % 3 == 1 ? 1.0 : 0.5) * (e / 3 == 1 ? 1.0 : 0.5));
  };
  std::vector<double> bc((size_t)mc * mc * N, 0.0);
  transfer([&](int c, int i, double w) { add(&bc[(size_t)c * N], w, &r[(size_t)i * N]); });
  const std::vector<double> xc = vcycle_columns(st + 1, mc, N, bc);
  transfer([&](int c, int i, double w) { add(&x[(size_t)i * N], w, &xc[(size_t)c * N]); });
  residual();
  sweep();
  sweep();
  return x;
}

static std::vector<double> vcycle_matrix(int m, const std::vector<std::vector<double>>& st) {
  const int n = m * m;
  std::vector<double> unit((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i) unit[(size_t)i * n + i] = 1.0;
  return vcycle_columns(st.data(), m, n, unit);
}

static int upload_grid(GridLevel& g, const std::vector<double>& st, bool finest) {
  SG_TRY(upload(&g.st_base, st.data(), st.size()));
  std::vector<float> st32(st.begin(), st.end());
  std::vector<double> dinv(g.n);
  for (int i = 0; i < g.n; ++i) dinv[i] = 1.0 / st[(size_t)i * 9 + 4];
  std::vector<float> dinv32(dinv.begin(), dinv.end());
  SG_TRY(upload(&g.st64, st.data(), st.size()));
  SG_TRY(upload(&g.st32, st32.data(), st32.size()));
  SG_TRY(upload(&g.dinv64, dinv.data(), dinv.size()));
  SG_TRY(upload(&g.dinv32, dinv32.data(), dinv32.size()));
  SG_TRY_CUDA(cudaMalloc((void**)&g.st12, dinv32.size() * 12 * sizeof(float)));
  if (finest && g.nx == 63 && g.ny == 63) {
    SG_TRY_CUDA(cudaMalloc((void**)&g.planes, 10 * 63 * 64 * sizeof(float)));
    SG_TRY_CUDA(cudaMemset(g.planes, 0, 10 * 63 * 64 * sizeof(float)));
  }
  SG_TRY(pack_stencils(g));
  return SG_OK;
}

static int setup_impl(const sg_mesh* mesh, int M, int p, int family, int n, int nnz, const int* rowptr,
                      const int* colidx, const double* vals, const double* mass_vals, sg_problem* h, int q) {
  if (q >= 0 && (family != SG_HERMITE || M < 1 || q > 16)) {
    set_error("sg_setup_gpc: the gPC coefficient needs Hermite chaos, M >= 1 and a degree q <= 16");
    return q >= 0 && family != SG_HERMITE ? SG_ERR_UNSUPPORTED : SG_ERR_INVALID_ARG;
  }
  if (M < 0 || p < 0 || n <= 0 || nnz <= 0 || !rowptr || !colidx || !vals) {
    set_error("sg_setup: invalid sizes or null pointers (M=%d p=%d n=%d nnz=%d)", M, p, n, nnz);
    return SG_ERR_INVALID_ARG;
  }
  if (family != SG_LEGENDRE && family != SG_HERMITE) {
    set_error("sg_setup: unknown chaos family %d", family);
    return SG_ERR_INVALID_ARG;
  }
  if (rowptr[0] != 0 || rowptr[n] != nnz) {
    set_error("sg_setup: rowptr[0] must be 0 and rowptr[n] == nnz");
    return SG_ERR_INVALID_ARG;
  }
  int max_row = 0;
  for (int r = 0; r < n; ++r) {
    if (rowptr[r + 1] < rowptr[r]) {
      set_error("sg_setup: rowptr not monotone at row %d", r);
      return SG_ERR_INVALID_ARG;
    }
    max_row = std::max(max_row, rowptr[r + 1] - rowptr[r]);
    for (int e = rowptr[r]; e < rowptr[r + 1]; ++e) {
      if (colidx[e] < 0 || colidx[e] >= n || (e > rowptr[r] && colidx[e] <= colidx[e - 1])) {
        set_error("sg_setup: column index out of range or unsorted in row %d", r);
        return SG_ERR_INVALID_ARG;
      }
    }
  }
  // value terms per nonzero: the linear KL expansion has M + 1, the gPC one C(M + q, M)
  long long nterm = M + 1;
  if (q >= 0) {
    nterm = 1;
    for (int i = 1; i <= M; ++i) nterm = nterm * (q + i) / i;
    if (nterm > 4096) {
      set_error("sg_setup_gpc: %lld coefficient terms exceed the supported 4096", nterm);
      return SG_ERR_UNSUPPORTED;
    }
  }
  h->q = q;
  h->nterm = (int)nterm;
  const size_t nv = (size_t)nnz * nterm;
  for (size_t i = 0; i < nv; ++i) {
    if (!std::isfinite(vals[i])) {
      set_error("sg_setup: non-finite matrix value at %zu", i);
      return SG_ERR_INVALID_ARG;
    }
  }
  h->n = n;
  h->nnz = nnz;
  h->M = M;
  h->p = p;
  h->family = family;
  h->max_row_nnz = max_row;
  SG_TRY_CUDA(cudaGetDevice(&h->device));
  SG_TRY_CUDA(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device));
  SG_TRY_CUDA(cudaDeviceGetAttribute(&h->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device));

  // chaos table
  h->off.assign(1, 0);
  std::vector<int> cur(std::max(M, 1));
  for (int d = 0; d <= p; ++d) {
    if (M == 0) {  // the constant polynomial only
      h->off.push_back(1);
      continue;
    }
    emit_degree(M, 0, d, cur, h->alpha);
    h->off.push_back((int)(h->alpha.size() / M));
  }
  h->P = h->off.back();
  if (M == 0) h->alpha.clear();
  h->wmax = 0;
  for (int d = 0; d <= p; ++d) h->wmax = std::max(h->wmax, h->off[d + 1] - h->off[d]);
  if (h->P > 2048) {
    set_error("sg_setup: P = %d chaos polynomials exceeds the supported 2048", h->P);
    return SG_ERR_UNSUPPORTED;
  }

  std::map<std::vector<int>, int> index;
  for (int l = 0; l < h->P; ++l)
    index[std::vector<int>(h->alpha.begin() + (size_t)l * M, h->alpha.begin() + (size_t)(l + 1) * M)] = l;
  const std::vector<int>& off = h->off;
  h->pre.resize(p + 1);
  h->post.resize(p + 1);
  if (q < 0) {
    SG_TRY(upload_edges(build_edges(h, index, 0, h->P, 0, h->P), h->all, 0, 0, h->P, h->nterm));
    for (int l = 1; l <= p; ++l) {
      SG_TRY(upload_edges(build_edges(h, index, off[l - 1], off[l], off[l], off[l + 1]), h->pre[l], off[l - 1],
                          off[l], off[l + 1] - off[l], h->nterm));
      SG_TRY(upload_edges(build_edges(h, index, off[l], off[l + 1], off[l - 1], off[l]), h->post[l], off[l],
                          off[l - 1], off[l] - off[l - 1], h->nterm));
    }
    if (p >= 1) SG_TRY(upload_edges(build_edges(h, index, 0, off[p], 0, off[p]), h->sub, 0, 0, off[p], h->nterm));
  } else {
    // the coefficient terms in the same graded order
    std::vector<int> cur(M);
    for (int d = 0; d <= q; ++d) emit_degree(M, 0, d, cur, h->gamma);
    SG_TRY(upload_edges(build_edges_gpc(h, 0, h->P, 0, h->P), h->all, 0, 0, h->P, h->nterm));
    h->dlev.resize(p + 1);
    for (int l = 1; l <= p; ++l) {
      // B_l: every lower level from level l; C_l: level l from every lower level; D_l: level l with itself
      SG_TRY(upload_edges(build_edges_gpc(h, 0, off[l], off[l], off[l + 1]), h->pre[l], 0, off[l],
                          off[l + 1] - off[l], h->nterm));
      SG_TRY(upload_edges(build_edges_gpc(h, off[l], off[l + 1], 0, off[l]), h->post[l], off[l], 0, off[l], h->nterm));
      SG_TRY(upload_edges(build_edges_gpc(h, off[l], off[l + 1], off[l], off[l + 1]), h->dlev[l], off[l], off[l],
                          off[l + 1] - off[l], h->nterm));
    }
    // the pair form keeps one sum per distinct (term, input) in shared memory:
    // too many with a dense coupling, so the gPC products use the gather form
    h->k1_pairs[0] = h->k1_pairs[1] = h->outer_pairs = 0;
  }

  // matrices
  SG_TRY(upload(&h->rowptr, rowptr, (size_t)n + 1));
  SG_TRY(upload(&h->colidx, colidx, (size_t)nnz));
  SG_TRY(upload(&h->vals64, vals, nv));
  SG_TRY(upload(&h->vals_base, vals, nv));
  h->scales.assign(h->nterm, 1.0);
  SG_TRY(upload(&h->scales_dev, h->scales.data(), h->scales.size()));
  {
    std::vector<float> v32(vals, vals + nv);
    SG_TRY(upload(&h->vals32, v32.data(), nv));
    std::vector<df64> vdf(nv);
    for (size_t i = 0; i < nv; ++i) vdf[i] = df_split_host(vals[i]);
    df64* d = nullptr;
    SG_TRY(upload(&d, vdf.data(), nv));
    h->vals_df = d;
  }
  if (mass_vals) SG_TRY(upload(&h->mass64, mass_vals, (size_t)nnz));

  // multigrid hierarchy of A_0 on the structured grid
  if (mesh && mesh->ne_x > 1 && mesh->ne_y > 1) {
    const int nx = mesh->ne_x - 1, ny = mesh->ne_y - 1;
    if ((long long)nx * ny != n) {
      set_error("sg_setup: mesh %dx%d has %d interior nodes, n = %d", mesh->ne_x, mesh->ne_y, nx * ny, n);
      return SG_ERR_INVALID_ARG;
    }
    const int ne = mesh->ne_x;
    // the inner solves need the 9-point stencil of A_0 on the grid; the
    // multigrid hierarchy also a power-of-two square mesh
    const bool pow2 = mesh->ne_x == mesh->ne_y && (ne & (ne - 1)) == 0;
    bool ok = true;
    std::vector<double> st((size_t)n * 9, 0.0);
    for (int r = 0; r < n && ok; ++r) {
      const int x = r % nx, y = r / nx;
      for (int e = rowptr[r]; e < rowptr[r + 1]; ++e) {
        const int c = colidx[e], cx = c % nx, cy = c / nx;
        const int dx = cx - x, dy = cy - y;
        if (dx < -1 || dx > 1 || dy < -1 || dy > 1) { ok = false; break; }
        st[(size_t)r * 9 + (dy + 1) * 3 + (dx + 1)] += vals[(size_t)e * h->nterm];
      }
      if (ok && !(st[(size_t)r * 9 + 4] > 0.0)) ok = false;
    }
    if (ok) {
      h->nx = nx;
      h->ny = ny;
      int gx = nx, gy = ny;
      std::vector<std::vector<double>> small;   // stencils from the 7 x 7 grid on
      while (true) {
        if (pow2 && gx <= 7 && nx > 7) small.push_back(st);
        GridLevel g;
        g.nx = gx; g.ny = gy; g.n = gx * gy;
        SG_TRY(upload_grid(g, st, h->grids.empty()));
        h->grids.push_back(g);
        if (!pow2) break;            // the finest grid alone: diagonal M_0 only
        if (gx <= 1) {
          h->mg_full = true;
          if (!small.empty()) {
            const std::vector<double> M = vcycle_matrix(7, small);
            const std::vector<float> M32(M.begin(), M.end());
            SG_TRY(upload(&h->cmat_base, M.data(), M.size()));
            SG_TRY(upload(&h->cmat64, M.data(), M.size()));
            SG_TRY(upload(&h->cmat32, M32.data(), M32.size()));
          }
          break;
        }
        const int nxc = (gx - 1) / 2, nyc = (gy - 1) / 2;
        std::vector<double> stc;
        galerkin_coarsen(gx, gy, st, nxc, nyc, stc);
        st.swap(stc);
        gx = nxc; gy = nyc;
      }
    }
  }
  // the in-block coarse V-cycle takes over at the first grid with <= 1024 nodes
  h->cb_level = (int)h->grids.size();
  for (int g = 0; g < (int)h->grids.size(); ++g)
    if (h->grids[g].n <= 1024) { h->cb_level = g; break; }
  if (h->mg_full) SG_TRY(cluster_setup(h));
  for (auto& cs : h->cap) SG_TRY_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  {
    const char* ev = getenv("SGHSC_EAGER");
    h->eager = ev && ev[0] == '1';
  }
  {
    const char* ev = getenv("SGHSC_NO_PIPE");
    h->pipe_off = ev && ev[0] == '1';
    const char* eb = getenv("SGHSC_NO_BLOCK");
    h->block_off = eb && eb[0] == '1';
  }
  {
    const char* ev = getenv("SGHSC_GATHER_FORM");   // start from the gather form of the full product
    if (ev && ev[0] == '1') h->k1_pairs[0] = h->k1_pairs[1] = h->outer_pairs = h->outer_pairs_df = 0;
    const char* eg = getenv("SGHSC_GENERIC_PRODUCTS");   // the one-row-at-a-time kernels only
    if ((ev && ev[0] == '1') || (eg && eg[0] == '1')) h->staged_pairs = 0;
  }
  SG_TRY_CUDA(cudaMalloc((void**)&h->loopflags, 8 * sizeof(int)));
  SG_TRY_CUDA(cudaMemset(h->loopflags, 0, 8 * sizeof(int)));
  SG_TRY_CUDA(cudaMallocHost((void**)&h->loopflag_host, sizeof(int)));
  SG_TRY_CUDA(cudaMalloc((void**)&h->status, sizeof(int)));
  SG_TRY_CUDA(cudaMemset(h->status, 0, sizeof(int)));
  SG_TRY_CUDA(cudaMallocHost((void**)&h->status_host, sizeof(int)));
  SG_TRY_CUDA(cudaMalloc((void**)&h->iacc, 2 * sizeof(long long)));
  SG_TRY_CUDA(cudaMemset(h->iacc, 0, 2 * sizeof(long long)));
  return SG_OK;
}

// vals = base * scale[k] for every nonzero (FP64 and FP32 copies)
__global__ void k_scale_vals(long long count, int M1, const double* __restrict__ base, const double* __restrict__ scale,
                             double* __restrict__ v64, float* __restrict__ v32, df64* __restrict__ vdf) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    const double v = base[i] * scale[i % M1];
    v64[i] = v;
    v32[i] = (float)v;
    const float h = __double2float_rn(v);
    vdf[i] = df64(h, __double2float_rn(v - (double)h));
  }
}

// multigrid stencils of s * A_0: st = s * base, dinv = 1 / (s * base_centre),
// and their FP32 copies (GridLevel::st12, planes; the padding stays as packed at
// set-up). On the 7 x 7 grid also the V-cycle matrix, that of A_0 divided by s
// (cbase: null elsewhere). One launch a grid: with the copies and the matrix in
// launches of their own sg_set_scales took 52, 69 and 80 us on 15, 63 and 127
// nodes a side, so 34, 42 and 50 (32, 40 and 48 without either).
__global__ void k_scale_grid(GridLevel g, double s, const double* __restrict__ cbase, double* __restrict__ c64,
                             float* __restrict__ c32) {
  const int first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  for (int i = first; i < g.n * 9; i += step) {
    const int node = i / 9, e = i - node * 9, x = node % g.nx, y = node / g.nx;
    const double v = s * g.st_base[i];
    g.st64[i] = v;
    g.st32[i] = (float)v;
    g.st12[node * 12 + e / 3 * 4 + e % 3] = (float)v;
    if (g.planes) g.planes[(e * g.ny + y) * (g.nx + 1) + x] = (float)v;
    if (e == 4) {
      const double d = 1.0 / v;
      g.dinv64[node] = d;
      g.dinv32[node] = (float)d;
      g.st12[node * 12 + 11] = (float)d;
      if (g.planes) g.planes[(9 * g.ny + y) * (g.nx + 1) + x] = (float)d;
    }
  }
  if (cbase)
    for (int i = first; i < 49 * 49; i += step) {
      const double v = cbase[i] / s;
      c64[i] = v;
      c32[i] = (float)v;
    }
}

}  // namespace sghsc

using namespace sghsc;

extern "C" {

int sg_set_scales(sg_problem* h, const double* scale) {
  set_error("");
  if (!h || !scale) {
    set_error("sg_set_scales: invalid arguments");
    return SG_ERR_INVALID_ARG;
  }
  for (int k = 0; k < h->nterm; ++k)
    if (!std::isfinite(scale[k])) {
      set_error("sg_set_scales: non-finite scale %d", k);
      return SG_ERR_INVALID_ARG;
    }
  if (!(scale[0] > 0.0) && !h->grids.empty()) {
    set_error("sg_set_scales: the mean matrix needs a positive scale");
    return SG_ERR_INVALID_ARG;
  }
  SG_TRY_CUDA(cudaDeviceSynchronize());   // no solve may be reading the values
  h->scales.assign(scale, scale + h->nterm);
  SG_TRY_CUDA(cudaMemcpy(h->scales_dev, scale, h->nterm * sizeof(double), cudaMemcpyHostToDevice));
  const long long count = (long long)h->nnz * h->nterm;
  { k_scale_vals<<<(int)std::min<long long>((count + 255) / 256, 4096), 256>>>(count, h->nterm, h->vals_base, h->scales_dev, h->vals64, h->vals32, (df64*)h->vals_df); ::sghsc::note_launch(); }
  for (auto& g : h->grids) {
    const double* cbase = h->cmat_base && &g == &h->grids[h->grids.size() - 3] ? h->cmat_base : nullptr;
    { k_scale_grid<<<std::min((g.n * 9 + 255) / 256, 4096), 256>>>(g, scale[0], cbase, h->cmat64, h->cmat32); ::sghsc::note_launch(); }
  }
  SG_TRY_CUDA(cudaGetLastError());
  SG_TRY_CUDA(cudaDeviceSynchronize());
  return SG_OK;
}


const char* sg_last_error(void) { return sghsc::g_err; }

long long sg_kernel_launches(void) { return sghsc::g_launches.load(); }

void sg_default_prec_opts(sg_prec_opts* o) {
  if (!o) return;
  o->precision = SG_F32;
  o->top_level_f64 = 1;
  o->inner_tol = 1e-2;
  o->inner_maxit = 200;
  o->inner_fixed_iters = 0;
  o->nu = 2;
  o->omega = 0.8;
  o->m0 = SG_M0_VCYCLE;
  o->level_tol = 1e-8;
  o->level_maxit = 500;
  o->md_m0 = 0;
  o->df64 = 0;
}

void sg_default_solve_opts(sg_solve_opts* o) {
  if (!o) return;
  o->precond = SG_PREC_HSC;
  sg_default_prec_opts(&o->prec);
  o->tol = 1e-8;
  o->maxit = 500;
  o->flexible = 1;
  o->use_x0 = 0;
  o->check_true_residual = 1;
  o->schur_reduced = 0;
  o->schur_inner_tol = 1e-11;
}

int sg_setup(const sg_mesh* mesh, int M, int p, int family, int n, int nnz, const int* rowptr,
             const int* colidx, const double* vals, const double* mass_vals, sg_problem** out) {
  set_error("");
  if (!out) {
    set_error("sg_setup: out is null");
    return SG_ERR_INVALID_ARG;
  }
  *out = nullptr;
  sg_problem* h = new sg_problem();
  int st = setup_impl(mesh, M, p, family, n, nnz, rowptr, colidx, vals, mass_vals, h, -1);
  if (st != SG_OK) {
    sg_destroy(h);
    return st;
  }
  *out = h;
  return SG_OK;
}

int sg_setup_gpc(const sg_mesh* mesh, int M, int p, int q, int family, int n, int nnz, const int* rowptr,
                 const int* colidx, const double* vals, const double* mass_vals, sg_problem** out) {
  set_error("");
  if (!out) {
    set_error("sg_setup_gpc: out is null");
    return SG_ERR_INVALID_ARG;
  }
  *out = nullptr;
  if (q < 0) {
    set_error("sg_setup_gpc: q < 0");
    return SG_ERR_INVALID_ARG;
  }
  sg_problem* h = new sg_problem();
  int st = setup_impl(mesh, M, p, family, n, nnz, rowptr, colidx, vals, mass_vals, h, q);
  if (st != SG_OK) {
    sg_destroy(h);
    return st;
  }
  *out = h;
  return SG_OK;
}

int sg_problem_terms(const sg_problem* h, int* nterm, int* q) {
  if (!h) {
    set_error("sg_problem_terms: null handle");
    return SG_ERR_INVALID_ARG;
  }
  if (nterm) *nterm = h->nterm;
  if (q) *q = h->q;
  return SG_OK;
}

void sg_destroy(sg_problem* h) {
  if (!h) return;
  free_edges(h->all);
  for (auto& e : h->pre) free_edges(e);
  for (auto& e : h->post) free_edges(e);
  free_edges(h->sub);
  for (auto& e : h->dlev) free_edges(e);
  cudaFree(h->cmat_base); cudaFree(h->cmat64); cudaFree(h->cmat32);
  for (auto& g : h->grids) {
    cudaFree(g.st_base); cudaFree(g.st64); cudaFree(g.st32); cudaFree(g.dinv64); cudaFree(g.dinv32); cudaFree(g.st12); cudaFree(g.planes);
  }
  if (h->cap[0]) cudaDeviceSynchronize();
  clear_graphs(h);
  free_inner_work(h);
  cluster_free(h);
  void* bufs[] = {h->rowptr, h->colidx, h->vals64, h->vals32, h->mass64, h->R32, h->Z32, h->T32, h->R64w,
                  h->T64, h->fF, h->fx, h->fr, h->fz, h->fpA, h->fpB, h->fq, h->opart, h->osc, h->octl,
                  h->hist_alpha, h->hist_beta, h->hist_res, h->io_in, h->io_out, h->status, h->iacc, h->wdev, h->loopflags, h->vals_base, h->scales_dev, h->fG, h->vals_df,
                  h->lx, h->lr, h->lz, h->lp, h->lq, h->lb, h->lctl, h->lsc, h->lhist_alpha, h->lhist_beta,
                  h->lhist_res};
  for (void* b : bufs) cudaFree(b);
  for (auto& cs : h->cap)
    if (cs) cudaStreamDestroy(cs);
  if (h->osc_host) cudaFreeHost(h->osc_host);
  if (h->status_host) cudaFreeHost(h->status_host);
  if (h->loopflag_host) cudaFreeHost(h->loopflag_host);
  delete h;
}

int sg_problem_dims(const sg_problem* h, int* n, int* P, int* M, int* p, int* nnz) {
  if (!h) {
    set_error("sg_problem_dims: null handle");
    return SG_ERR_INVALID_ARG;
  }
  if (n) *n = h->n;
  if (P) *P = h->P;
  if (M) *M = h->M;
  if (p) *p = h->p;
  if (nnz) *nnz = h->nnz;
  return SG_OK;
}

int sg_chaos_table(const sg_problem* h, int* alpha, int* level_offsets) {
  if (!h) {
    set_error("sg_chaos_table: null handle");
    return SG_ERR_INVALID_ARG;
  }
  if (alpha && !h->alpha.empty()) std::memcpy(alpha, h->alpha.data(), h->alpha.size() * sizeof(int));
  if (level_offsets) std::memcpy(level_offsets, h->off.data(), h->off.size() * sizeof(int));
  return SG_OK;
}

}  // extern "C"
