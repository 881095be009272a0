// The V-cycle's work on one grid in two passes over the batch (FP32, two
// sweeps before and after the coarse correction), included by inner.cu.
//
//   k_mg_down  b -> bc = P^T (b - A x), x the two sweeps from zero
//   k_mg_up    b, xc -> z: x again, x + P xc, two sweeps; r . z for the CG
//
// x is not stored: forming it again from b costs one stencil of arithmetic and
// saves a write and two reads of the batch. One kernel per sweep read or wrote
// the n x w block ten and a half times per V-cycle on a grid; these two read b
// twice and write z and a quarter-size bc: three and a half times.
//
// A block owns strips of 64 nodes by 4 PG columns and walks a strip row by row.
// Thread (lx, grp) stays on node x0 - 2 + lx and column group grp for every
// stencil of the pass. A stencil is summed as its rows arrive: the three values
// of the new row (left, own, right, from shared memory) complete the sum of the
// row above, continue the present one and start the one below, so each value is
// read three times and not nine, two partial sums stay in registers, and only
// the newest row of each intermediate vector is in shared memory (two
// buffers). The stencils of one step work on rows written in earlier steps
// (row t of b, row t - 2 of x + P xc, row t - 4 of the first sweep's result),
// so a step has one barrier. Rows of b, of the stencils and of xc arrive by
// cp.async two steps ahead; everything outside the grid or the batch is
// zero-filled, the diagonal included, so no value needs a test: outside nodes
// stay zero.
//
// What bounds it: instruction issue. At 255 x 255 x 716 columns 62% of the issue
// slots are used by the 17 warps that an SM holds (the rings take its shared
// memory); a warp's wait between two instructions, 6.8 clocks, is shared-memory
// latency (1.8), another warp chosen (1.2) and the block's barrier per row
// (1.0). 290 and 440 instructions a thread and row on the way down and up, a
// quarter of them the stencils' multiply-adds; DRAM moves 35% of its rate. The
// four kernels this replaces took 135 + 180 + 234 + 163 us, these two 157 + 256;
// a V-cycle 1245 -> 830 us, at 511 x 511 4433 -> 2761 us. Tried: b's own values
// of five rows in registers (spills at 96 registers a thread doubled the time of
// the way up), rows of b on whole 128-byte lines (46% and 31% fewer bytes from
// DRAM, the same time, and the padding cost every other kernel: inner.cu).
//
// Nodes x0 - 2 .. x0 + 65 (68 lanes) carry the two nodes a side that the last
// sweep's neighbours need. A run of rows starts three rows early and ends five
// steps late; the rows formed in between are not complete and nothing reads
// them.
namespace mg {
constexpr int OUT = 64;              // output nodes of a strip
constexpr int LX = OUT + 4;          // nodes carried
constexpr int BX = LX + 2;           // nodes of a b row
constexpr int SR = 16, CR = 8;       // ring slots: stencils, coarse rows
constexpr int BRD = 4, BRU = 8;      // and b, on the way down and up (rows t - 5 .. t + 2)
constexpr int CN = OUT / 2 + 4;      // coarse nodes of a strip (x0 / 2 - 2 ..)
constexpr int SF = 12;               // floats per staged stencil: three rows of three, dinv in the last slot
}  // namespace mg

template <int PG, bool UP>
static constexpr size_t mg_smem_bytes() {
  using namespace mg;
  return (size_t)16 * PG * ((UP ? BRU : BRD) * BX + 4 * BX + (UP ? CR * CN : 0)) + (size_t)4 * SR * BX * SF;
}

__device__ __forceinline__ void mg_fma3(float4& s, const float4& c, const float4& v0, const float4& v1,
                                        const float4& v2) {
  s.x = fmaf(c.x, v0.x, s.x); s.y = fmaf(c.x, v0.y, s.y); s.z = fmaf(c.x, v0.z, s.z); s.w = fmaf(c.x, v0.w, s.w);
  s.x = fmaf(c.y, v1.x, s.x); s.y = fmaf(c.y, v1.y, s.y); s.z = fmaf(c.y, v1.z, s.z); s.w = fmaf(c.y, v1.w, s.w);
  s.x = fmaf(c.z, v2.x, s.x); s.y = fmaf(c.z, v2.y, s.y); s.z = fmaf(c.z, v2.z, s.z); s.w = fmaf(c.z, v2.w, s.w);
}
__device__ __forceinline__ float4 mg_scale(float a, const float4& v) {
  return make_float4(a * v.x, a * v.y, a * v.z, a * v.w);
}
// x + d (b - s)
__device__ __forceinline__ float4 mg_relax(const float4& x, float d, const float4& b, const float4& s) {
  return make_float4(x.x + d * (b.x - s.x), x.y + d * (b.y - s.y), x.z + d * (b.z - s.z), x.w + d * (b.w - s.w));
}

// A stencil summed row by row: the sums of the row above (two rows in), of the
// present row (one row in).
struct MgSum {
  float4 a1, a0;
  __device__ __forceinline__ void clear() { a1 = a0 = make_float4(0.f, 0.f, 0.f, 0.f); }
  // row r has arrived: returns the sum of row r - 1. dn, mid, up: the last
  // stencil row of r - 1, the middle one of r, the first one of r + 1.
  __device__ __forceinline__ float4 step(const float4& dn, const float4& mid, const float4& up, const float4& v0,
                                         const float4& v1, const float4& v2) {
    float4 done = a1;
    mg_fma3(done, dn, v0, v1, v2);
    a1 = a0;
    mg_fma3(a1, mid, v0, v1, v2);
    a0 = make_float4(0.f, 0.f, 0.f, 0.f);
    mg_fma3(a0, up, v0, v1, v2);
    return done;
  }
};

// What both passes share: the rings and their copies, and the first stencil
// (b -> the two sweeps from zero). What a thread copies of a row is the same
// place in every row of a strip: the places are worked out once per strip.
template <int PG, int BR>
struct MgRows {
  static constexpr int NT = mg::LX * PG;
  static constexpr int NS = (mg::BX * 3 + NT - 1) / NT;   // 16-byte pieces of a stencil row per thread
  const float *st, *B;   // st: [n][SF]
  int nx, ny, wp, x0, c0;
  float4* br;   // [BR][BX][PG]
  float* sr;    // [SR][BX][SF]
  int bo, bo2;          // element offsets within a row of b (the threads' first and second piece), -1: none
  int so[NS];           // within a row of the stencils

  __device__ __forceinline__ void place(int x0_, int c0_) {
    using namespace mg;
    x0 = x0_;
    c0 = c0_;
    auto at = [&](int i) {
      const int x = x0 - 3 + i / PG, c = c0 + 4 * (i % PG);
      return i < BX * PG && x >= 0 && x < nx && c < wp ? x * wp + c : -1;
    };
    bo = at(threadIdx.x);
    bo2 = at(threadIdx.x + NT);
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      const int i = threadIdx.x + q * NT, x = x0 - 3 + i / 3;
      so[q] = i < BX * 3 && x >= 0 && x < nx ? (x0 - 3) * SF + 4 * i : -1;
    }
  }
  __device__ __forceinline__ void issue_b(int r) const {
    using namespace mg;
    const bool row = r >= 0 && r < ny;
    const float* src = B + (row ? (size_t)r * nx * wp : 0);
    float4* d = br + (r & (BR - 1)) * BX * PG + threadIdx.x;
    const bool ok = row && bo >= 0;
    cp_async16_z(d, src + (ok ? bo : 0), ok);
    if (threadIdx.x < BX * PG - NT) {
      const bool ok2 = row && bo2 >= 0;
      cp_async16_z(d + NT, src + (ok2 ? bo2 : 0), ok2);
    }
  }
  __device__ __forceinline__ void issue_s(int r) const {
    using namespace mg;
    const bool row = r >= 0 && r < ny;
    const float* src = st + (row ? (size_t)r * nx * SF : 0);
    float* d = sr + (r & (SR - 1)) * BX * SF + 4 * threadIdx.x;
#pragma unroll
    for (int q = 0; q < NS; ++q)
      if ((int)threadIdx.x + q * NT < BX * 3) {
        const bool ok = row && so[q] >= 0;
        cp_async16_z(d + 4 * q * NT, src + (ok ? so[q] : 0), ok);
      }
  }
  // stencil row k (0 above, 1 own, 2 below; its fourth entry: of row 2 the
  // inverse diagonal) of node j in grid row r
  __device__ __forceinline__ float4 coef(int r, int j, int k) const {
    using namespace mg;
    return *reinterpret_cast<const float4*>(sr + ((r & (SR - 1)) * BX + j) * SF + 4 * k);
  }
  __device__ __forceinline__ float diag(int r, int j) const {
    using namespace mg;
    return sr[((r & (SR - 1)) * BX + j) * SF + 11];
  }
  __device__ __forceinline__ const float4* row(int r, int j, int grp) const {   // b, staged node j
    using namespace mg;
    return br + ((r & (BR - 1)) * BX + j) * PG + grp;
  }
  // row t of b has arrived: the two sweeps from zero on row t - 1 at staged
  // node j (row t - 1 of b is still in its slot)
  __device__ __forceinline__ float4 sweeps(MgSum& s, int t, int j, int grp, float om) const {
    using namespace mg;
    const float4* b = row(t, j, grp);
    const float4 dn = coef(t - 1, j, 2);
    const float4 ax = s.step(dn, coef(t, j, 1), coef(t + 1, j, 0), mg_scale(diag(t, j - 1), b[-PG]),
                             mg_scale(diag(t, j), b[0]), mg_scale(diag(t, j + 1), b[PG]));
    const float di = om * dn.w;
    const float4 bc = *row(t - 1, j, grp);
    return make_float4(di * bc.x + di * (bc.x - om * ax.x), di * bc.y + di * (bc.y - om * ax.y),
                       di * bc.z + di * (bc.z - om * ax.z), di * bc.w + di * (bc.w - om * ax.w));
  }
};

// Whether the chunk of 4 PG columns from c0 has a column still iterating (the
// whole block calls it).
template <int PG>
__device__ __forceinline__ bool mg_chunk_active(const int* __restrict__ done, int c0, int wp) {
  const int c = c0 + (int)threadIdx.x;
  return __syncthreads_or(threadIdx.x < 4 * PG && c < wp && !done[c]);
}

template <int PG>
__global__ void __launch_bounds__(mg::LX * PG, 1)
    k_mg_down(int nx, int ny, int nxc, int nyc, int wp, const float* __restrict__ st, const float* B,
              float* bc, float om, const int* __restrict__ done) {
  using namespace mg;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MgRows<PG, BRD> R;
  R.st = st;
  R.B = B;
  R.nx = nx;
  R.ny = ny;
  R.wp = wp;
  R.br = reinterpret_cast<float4*>(smem_raw);
  float4* xr = R.br + BRD * BX * PG;   // [2][BX][PG] newest rows of x
  float4* rr = xr + 2 * BX * PG;      // [2][BX][PG] newest rows of b - A x
  R.sr = reinterpret_cast<float*>(rr + 2 * BX * PG);
  const int grp = threadIdx.x % PG, j = threadIdx.x / PG + 1;   // staged node, x = x0 - 3 + j
  const int nseg = (nxc + OUT / 2 - 1) / (OUT / 2), nch = (wp + 4 * PG - 1) / (4 * PG);
  const long long tot = (long long)nch * nseg * nyc;
  long long u = tot * blockIdx.x / gridDim.x;
  const long long u1 = tot * (blockIdx.x + 1) / gridDim.x;
  for (int i = threadIdx.x; i < 4 * BX * PG; i += MgRows<PG, BRD>::NT) xr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  while (u < u1) {
    const int strip = (int)(u / nyc);
    const int Ya = (int)(u - (long long)strip * nyc);
    const int Yb = (int)min((long long)nyc, (long long)Ya + (u1 - u));
    const int ch = strip / nseg, sg = strip - ch * nseg;
    u += Yb - Ya;
    R.place(sg * OUT, ch * 4 * PG);
    if (!mg_chunk_active<PG>(done, R.c0, wp)) continue;
    const int x = R.x0 - 3 + j, c = R.c0 + 4 * grp;
    // residual rows 2 Ya .. 2 Yb; b from two rows before to two after
    const int t0 = 2 * Ya - 2, t1 = 2 * Yb + 2;
    for (int r = t0 - 1; r <= t0 + 1; ++r) R.issue_s(r);
    R.issue_b(t0);
    cp_async_commit();
    R.issue_b(t0 + 1);
    R.issue_s(t0 + 2);
    cp_async_commit();
    MgSum sx, sa;
    sx.clear();
    sa.clear();
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 bn = zero, b1 = zero, b2 = zero, b3 = zero, acc = zero;
    // step t: x on row t - 1, the residual on row t - 3, its restriction on row t - 4
    for (int t = t0; t <= 2 * Yb + 4; ++t) {
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncthreads();
      if (t + 2 <= t1) R.issue_b(t + 2);
      if (t + 3 <= t1 + 1) R.issue_s(t + 3);
      cp_async_commit();
      if (t <= t1) {
        xr[((t - 1) & 1) * BX * PG + j * PG + grp] = R.sweeps(sx, t, j, grp, om);
        bn = *R.row(t, j, grp);
      }
      {
        const float4* v = xr + ((t - 2) & 1) * BX * PG + j * PG + grp;
        const float4 ax = sa.step(R.coef(t - 3, j, 2), R.coef(t - 2, j, 1), R.coef(t - 1, j, 0), v[-PG], v[0], v[PG]);
        rr[((t - 3) & 1) * BX * PG + j * PG + grp] =
            make_float4(b3.x - ax.x, b3.y - ax.y, b3.z - ax.z, b3.w - ax.w);
      }
      if (x & 1) {   // coarse node (x - 1) / 2
        const float4* v = rr + ((t - 4) & 1) * BX * PG + j * PG + grp;
        const float4 l = v[-PG], m = v[0], r = v[PG];
        const float4 h = make_float4(0.5f * l.x + m.x + 0.5f * r.x, 0.5f * l.y + m.y + 0.5f * r.y,
                                     0.5f * l.z + m.z + 0.5f * r.z, 0.5f * l.w + m.w + 0.5f * r.w);
        const int row = t - 4;
        if (row & 1) {
          acc = make_float4(acc.x + h.x, acc.y + h.y, acc.z + h.z, acc.w + h.w);
        } else {
          const int Y = row / 2 - 1, X = (x - 1) >> 1;
          acc = make_float4(acc.x + 0.5f * h.x, acc.y + 0.5f * h.y, acc.z + 0.5f * h.z, acc.w + 0.5f * h.w);
          if (row >= 2 * Ya + 2 && X >= R.x0 / 2 && X < R.x0 / 2 + OUT / 2 && X < nxc && c < wp)
            *reinterpret_cast<float4*>(bc + ((size_t)Y * nxc + X) * wp + c) = acc;
          acc = mg_scale(0.5f, h);
        }
      }
      b3 = b2;
      b2 = b1;
      b1 = bn;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // the rings are free
  }
}

template <int PG, bool DOT>
__global__ void __launch_bounds__(mg::LX * PG, 1)
    k_mg_up(int nx, int ny, int nxc, int nyc, int wp, const float* __restrict__ st, const float* B,
            const float* XC, float* out, float om, FinArgs f) {
  using namespace mg;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float colacc[DOT ? 1024 : 1];
  MgRows<PG, BRU> R;
  R.st = st;
  R.B = B;
  R.nx = nx;
  R.ny = ny;
  R.wp = wp;
  R.br = reinterpret_cast<float4*>(smem_raw);
  float4* xr = R.br + BRU * BX * PG;   // [2][BX][PG] newest rows of x + P xc
  float4* yr = xr + 2 * BX * PG;      // [2][BX][PG] newest rows of the first sweep after it
  float4* cr = yr + 2 * BX * PG;      // [CR][CN][PG] coarse rows
  R.sr = reinterpret_cast<float*>(cr + CR * CN * PG);
  constexpr int NT = MgRows<PG, BRU>::NT;
  const int grp = threadIdx.x % PG, lx = threadIdx.x / PG, j = lx + 1;   // staged node, x = x0 - 3 + j
  const int nseg = (nx + OUT - 1) / OUT, nch = (wp + 4 * PG - 1) / (4 * PG);
  const long long tot = (long long)nch * nseg * ny;
  long long u = tot * blockIdx.x / gridDim.x;
  const long long u1 = tot * (blockIdx.x + 1) / gridDim.x;
  if (DOT)
    for (int i = threadIdx.x; i < wp; i += NT) colacc[i] = 0.f;
  for (int i = threadIdx.x; i < 4 * BX * PG; i += NT) xr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  while (u < u1) {
    const int strip = (int)(u / ny);
    const int ya = (int)(u - (long long)strip * ny);
    const int yb = (int)min((long long)ny, (long long)ya + (u1 - u));
    const int ch = strip / nseg, sg = strip - ch * nseg;
    u += yb - ya;
    R.place(sg * OUT, ch * 4 * PG);
    if (!mg_chunk_active<PG>(f.done, R.c0, wp)) continue;
    const int x = R.x0 - 3 + j, c = R.c0 + 4 * grp, X0 = R.x0 / 2 - 2;
    // (node lx of the coarse row, column group grp: CN <= LX)
    const int co = lx < CN && X0 + lx >= 0 && X0 + lx < nxc && c < wp ? (X0 + lx) * wp + c : -1;
    auto issue_c = [&](int Y) {
      const bool ok = Y >= 0 && Y < nyc && co >= 0;
      if (lx < CN)
        cp_async16_z(&cr[((Y & (CR - 1)) * CN + lx) * PG + grp], XC + (ok ? (size_t)Y * nxc * wp + co : 0), ok);
    };
    const int t0 = ya - 3, t1 = yb + 2;          // rows of b
    int cnext = (t0 >> 1) - 1;                   // coarse rows: fine row y takes ((y + 1) >> 1) - 1 and y >> 1
    auto issue_cs = [&](int y) {
      for (; cnext <= (min(y, yb + 1) >> 1); ++cnext) issue_c(cnext);
    };
    for (int r = t0 - 1; r <= t0 + 1; ++r) R.issue_s(r);
    R.issue_b(t0);
    issue_cs(t0 - 1);
    cp_async_commit();
    R.issue_b(t0 + 1);
    R.issue_s(t0 + 2);
    issue_cs(t0);
    cp_async_commit();
    MgSum sx, s1, s2;
    sx.clear();
    s1.clear();
    s2.clear();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    // weights of the two coarse columns beside x (odd x: its own, even x: half of each)
    const bool ox = x & 1;
    const float wx0 = ox ? 1.f : 0.5f, wx1 = ox ? 0.f : 0.5f;
    const int ck = ((x + 1) >> 1) - 1 - X0, ck1 = ox ? ck : ck + 1;
    // step t: x and x + P xc on row t - 1, the sweeps on rows t - 3 and t - 5
    for (int t = t0; t <= yb + 4; ++t) {
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncthreads();
      if (t + 2 <= t1) R.issue_b(t + 2);
      if (t + 3 <= t1 + 1) R.issue_s(t + 3);
      issue_cs(t + 1);
      cp_async_commit();
      // this thread's own values of rows t - 3 and t - 5, from the slots that
      // rows t - 1 and t - 3 take in this step
      float4* const xw = xr + (((t - 1) & 1) * BX + j) * PG + grp;
      float4* const yw = yr + (((t - 3) & 1) * BX + j) * PG + grp;
      const float4 xp = *xw, yp = *yw;
      if (t <= t1) {
        float4 v = R.sweeps(sx, t, j, grp, om);
        const int y = t - 1, Yl = ((y + 1) >> 1) - 1;
        const bool oy = y & 1;
        const float4* q = cr + (Yl & (CR - 1)) * CN * PG + grp;
        const float4 q0 = q[ck * PG], q1 = q[ck1 * PG];
        const float w0 = oy ? wx0 : 0.5f * wx0, w1 = oy ? wx1 : 0.5f * wx1;
        v.x += w0 * q0.x + w1 * q1.x;
        v.y += w0 * q0.y + w1 * q1.y;
        v.z += w0 * q0.z + w1 * q1.z;
        v.w += w0 * q0.w + w1 * q1.w;
        if (!oy) {
          const float4* p = cr + ((Yl + 1) & (CR - 1)) * CN * PG + grp;
          const float4 p0 = p[ck * PG], p1 = p[ck1 * PG];
          v.x += w0 * p0.x + w1 * p1.x;
          v.y += w0 * p0.y + w1 * p1.y;
          v.z += w0 * p0.z + w1 * p1.z;
          v.w += w0 * p0.w + w1 * p1.w;
        }
        *xw = v;
      }
      {
        const float4* v = xr + ((t - 2) & 1) * BX * PG + j * PG + grp;
        const float4 dn = R.coef(t - 3, j, 2);
        const float4 ax = s1.step(dn, R.coef(t - 2, j, 1), R.coef(t - 1, j, 0), v[-PG], v[0], v[PG]);
        *yw = mg_relax(xp, om * dn.w, *R.row(t - 3, j, grp), ax);
      }
      {
        const float4* v = yr + ((t - 4) & 1) * BX * PG + j * PG + grp;
        const float4 dn = R.coef(t - 5, j, 2);
        const float4 ax = s2.step(dn, R.coef(t - 4, j, 1), R.coef(t - 3, j, 0), v[-PG], v[0], v[PG]);
        const int y = t - 5;
        if (y >= ya && lx >= 2 && lx < LX - 2 && x < nx && c < wp) {
          const float4 b5 = *R.row(t - 5, j, grp);
          const float4 z = mg_relax(yp, om * dn.w, b5, ax);
          *reinterpret_cast<float4*>(out + ((size_t)y * nx + x) * wp + c) = z;
          if (DOT) {
            acc.x += b5.x * z.x;
            acc.y += b5.y * z.y;
            acc.z += b5.z * z.z;
            acc.w += b5.w * z.w;
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // the rings are free
    if (DOT) {
      // the strip's sums per column, nodes in order. They overwrite rows of b:
      // the next strip's copies fill every row that it reads of those. (What the
      // buffers of x and y still hold goes only into the rows formed before the
      // run's own, which nothing reads.)
      float* red = reinterpret_cast<float*>(R.br);   // [LX][4 PG]
      reinterpret_cast<float4*>(red)[lx * PG + grp] = acc;
      __syncthreads();
      if ((int)threadIdx.x < 4 * PG && R.c0 + (int)threadIdx.x < wp) {
        float sum = 0.f;
        for (int i = 2; i < LX - 2; ++i) sum += red[i * 4 * PG + threadIdx.x];
        colacc[R.c0 + threadIdx.x] += sum;
      }
      __syncthreads();
    }
  }
  if (DOT) {
    __syncthreads();
    float* part = (float*)f.part;
    for (int i = threadIdx.x; i < wp; i += NT) part[(size_t)blockIdx.x * f.ldp + i] = colacc[i];
    __threadfence();
    if (last_block(&f.ctl->ticket)) fin_columns<float>(f, FIN_RHO, wp, gridDim.x);
  }
}
