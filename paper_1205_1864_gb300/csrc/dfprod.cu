// Double-float SG products whose input block holds FP32 values (the output
// of the mixed-precision preconditioner): the outer solver's fused product
// q = A p (eq. (global-system) in MAT-VEC form, with the CG update) and the
// level-p products B_p, C_p of Algorithm 1. The arithmetic is double-float
// (df64.cuh) on the FP32 units; this file lays the work out for those units.
//
// Pair form, one spatial row at a time per block (grid-stride over rows):
//   stage   the row's values a_k(r, c) as [k][e] and the input rows X(c, :)
//           as [j][e] (e the nonzero, CH = 9 slots, zero-filled), so the
//           inner loop over the 9 nonzeros uses constant offsets only and the
//           lanes of a warp (consecutive pairs: the same k, consecutive j)
//           read one broadcast value and 32 distinct banks (stride 9 words);
//   pairs   every distinct (k, j) of the couplings: S_q = sum_e a_k(e) X(e, j)
//           into shared memory, a thread reading its pairs' offsets one turn
//           ahead; with DIAG also the k = 0 term of its own outputs;
//   couple  Y(r, l) = diag + sum_t c_t S_pair(t) over the couplings of l.
// Rows longer than CH are done in chunks of CH (the first chunk stores, later
// ones add).
#include <algorithm>
#include <type_traits>

#include "df64.cuh"
#include "sghsc_internal.cuh"
#include "vec.cuh"

namespace sghsc {

constexpr int DF_CH = 9;       // nonzeros per staged chunk (the Q1 stencil row)
constexpr int DF_MAXQ = 12;    // pairs per thread and row at most (what was measured: the sums are in shared memory)

// FP32 value of an input element that is FP32-exact: a float as it is, a
// double (the FP64 widening of an FP32 number) re-packed with integer
// operations (truncating the fraction, which is exact for such values).
__device__ __forceinline__ float exact_float(float v) { return v; }
__device__ __forceinline__ float exact_float(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((b >> 52) & 0x7ff);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  if (E == 0) return __uint_as_float(sign);
  const int ef = E - 1023 + 127;
  if (ef < 1 || ef > 254) return __double2float_rn(v);   // outside the normal FP32 range (not expected)
  return __uint_as_float(sign | ((unsigned)ef << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}

// an input element as FP64: a float widened with integer operations, a double as it is
__device__ __forceinline__ double widen_exact(float v) { return f2d_bits(v); }
__device__ __forceinline__ double widen_exact(double v) { return v; }

// a (double-float) times x (FP32): exact product of a.hi and x plus a.lo x
__device__ __forceinline__ df64 df_mul_f(const df64& a, float x) {
  const float p = a.hi * x;
  float e = fmaf(a.hi, x, -p);
  e = fmaf(a.lo, x, e);
  return df64(p, e);
}

// Packed FP32 operations (f32x2): two per instruction. The FP32 lanes are no
// faster (38 T operations/s packed or not), but the arithmetic takes half the
// issue slots, which the addresses, loads and integer work share. Measured with
// the packed sums and couplings (and the order of the couplings chosen against
// bank conflicts in setup.cu) against the scalar form: full product 255^2,
// M = 10, p = 4 2.54 -> 2.43 ms, 200^2, M = 8, p = 4 0.711 -> 0.691; level
// products 255^2, M = 10, 715 -> 220 columns 1.04 -> 0.99, M = 4, 20 <-> 35
// columns 0.247 -> 0.200, 10 <- 55 columns 0.290 -> 0.236; the even and odd
// partial sums halve the error against 64 bits (9.8e-15 -> 4.9e-15). Also
// tried: two sums per lane sharing the term's values, the next row prefetched
// into registers, half of a block's warps coupling while the others sum (2.6 to
// 2.8 ms each at M = 10, p = 4): the sums alone, in registers, run at 0.75 of
// the lanes' rate, and staging, couplings and conversions each need issue slots
// that a second role on the same SM does not find free.
struct df64x2 {   // two double-float values
  float2 hi, lo;
};
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }   // folds into the operand

// the products of a.hi and x exactly, plus lo (a.lo x)
__device__ __forceinline__ df64x2 df_mul_f2(float2 hi, float2 lo, float2 x) {
  df64x2 r;
  r.hi = __fmul2_rn(hi, x);
  r.lo = __ffma2_rn(lo, x, __ffma2_rn(hi, x, neg2(r.hi)));
  return r;
}
// s += v: two-sum of the hi parts, the lo parts in FP32
__device__ __forceinline__ void df_add2(df64x2& s, const df64x2& v) {
  const float2 t = __fadd2_rn(s.hi, v.hi);
  const float2 bb = __fadd2_rn(t, neg2(s.hi));
  const float2 e = __fadd2_rn(__fadd2_rn(s.hi, neg2(__fadd2_rn(t, neg2(bb)))), __fadd2_rn(v.hi, neg2(bb)));
  s.hi = t;
  s.lo = __fadd2_rn(__fadd2_rn(s.lo, v.lo), e);
}

// Layout of the staged chunk (DF_VS, DF_XS: sghsc_internal.cuh, the setup packs
// the pairs' offsets). A term's nine double-float values: eight hi parts,
// eight lo parts (neighbouring nonzeros side by side for the packed
// operations), then the ninth pair. An input column's nine values, padded to
// 12 floats: the eight lanes of a 16-byte load phase of consecutive columns
// then hit distinct banks.

// Stage chunk cs..cs+nzc-1 (nzc <= DF_CH), slots e >= nzc zero. The input rows
// go column position by column position (no integer division), the loads of
// all slots of a position in flight before their 16-byte stores.
template <typename TX>
__device__ __forceinline__ void df_stage(int cs, int nzc, int M1, const int* __restrict__ colidx,
                                         const df64* __restrict__ vals, const TX* __restrict__ X, int ldx, int wx,
                                         float* Vt, float* Xt) {
  for (int k = threadIdx.x; k < M1; k += blockDim.x) {
#pragma unroll
    for (int e = 0; e < DF_CH; ++e) {
      const df64 v = e < nzc ? vals[(size_t)(cs + e) * M1 + k] : df64(0.f, 0.f);
      Vt[k * DF_VS + (e < 8 ? e : 16)] = v.hi;
      Vt[k * DF_VS + (e < 8 ? 8 + e : 17)] = v.lo;
    }
  }
  int col[DF_CH];
#pragma unroll
  for (int e = 0; e < DF_CH; ++e) col[e] = e < nzc ? colidx[cs + e] : -1;
  for (int j = threadIdx.x; j < wx; j += blockDim.x) {
    float v[DF_CH];
#pragma unroll
    for (int e = 0; e < DF_CH; ++e) v[e] = col[e] >= 0 ? exact_float(X[(size_t)col[e] * ldx + j]) : 0.f;
    float4* xr = reinterpret_cast<float4*>(Xt + j * DF_XS);
    xr[0] = make_float4(v[0], v[1], v[2], v[3]);
    xr[1] = make_float4(v[4], v[5], v[6], v[7]);
    xr[2] = make_float4(v[8], 0.f, 0.f, 0.f);
  }
}

// sum_e a[e] x[e] over the DF_CH slots of one staged term row and one staged
// input column: the even and odd slots in packed sums, then the two halves
// added and the ninth slot.
__device__ __forceinline__ df64 df_dot9(const float* __restrict__ a, const float* __restrict__ x) {
  const float4* av = reinterpret_cast<const float4*>(a);
  const float4* xv = reinterpret_cast<const float4*>(x);
  auto lo2 = [](const float4& v) { return make_float2(v.x, v.y); };
  auto hi2 = [](const float4& v) { return make_float2(v.z, v.w); };
  const float4 x0 = xv[0], x1 = xv[1], h0 = av[0], h1 = av[1], l0 = av[2], l1 = av[3];
  const float2 t8 = *reinterpret_cast<const float2*>(a + 16);
  const float x8 = x[8];
  df64x2 s = df_mul_f2(lo2(h0), lo2(l0), lo2(x0));
  df_add2(s, df_mul_f2(hi2(h0), hi2(l0), hi2(x0)));
  df_add2(s, df_mul_f2(lo2(h1), lo2(l1), lo2(x1)));
  df_add2(s, df_mul_f2(hi2(h1), hi2(l1), hi2(x1)));
  df64 r(s.hi.x, s.lo.x);
  r += df64(s.hi.y, s.lo.y);
  r += df_mul_f(df64(t8.x, t8.y), x8);
  return r;
}

// an FP32 number as FP64 (f2d_bits), the common case first: a normal number's
// exponent rebiased and its fraction moved, five operations
__device__ __forceinline__ double f2d_fast(float f) {
  const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
  if (e - 1u < 254u)
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
  return f2d_bits(f);
}

enum { DF_SUB = 0, DF_PLAIN = 1, DF_OUTER = 2 };

// MODE DF_SUB: a level product, Y = Yin - sum (Yin FP64, Y FP32), the
// difference in double-float, rounded once to FP32. DF_PLAIN: the full
// product, Y = sum (FP64, one add of the pair per output). DF_OUTER: the
// outer CG step (as k_outer_matvec): p_new = z + beta p_old, q = A z + beta
// q_old, p_new . q and alpha, with X = z (FP32, or FP64 storage of FP32
// values).
// Shared memory (16-byte aligned parts): pair sums Ss[npair], diagonal terms
// Ds[wy] (DIAG, by output column in natural order, so the lanes of a warp
// read consecutive inputs), the coefficient classes Ctab[ncls] (loaded once
// per block), then the staged chunk Vt, Xt. The packed couplings stay in
// global memory, read coalesced through L1 (in shared memory they held a
// block to one per SM at P = 1001); each output slot's first word and count
// come from a descriptor, so a thread takes any number of outputs.
template <bool DIAG, int MODE, typename TX, typename TY, int LB>
__global__ void __launch_bounds__(LB, LB <= 256 ? 4 : 2) k_df_pairs(
    int n, const int* __restrict__ rowptr, const int* __restrict__ colidx, const df64* __restrict__ vals, int M1,
    const TX* __restrict__ X, int ldx, int wx, int npair, const unsigned* __restrict__ pkj,
    const unsigned* __restrict__ ctr, const int2* __restrict__ sdesc, const df64* __restrict__ ctab, int ncls, int wy,
    const double* __restrict__ Yin, int ldyin, TY* __restrict__ Y, int ldy, double* pA, double* pB,
    double* __restrict__ q, OuterArgs a) {
  constexpr bool OUTER = MODE == DF_OUTER;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // pairs and diagonal outputs padded to whole passes of the block, so every
  // warp runs the same loops (the padding pairs read staged slot 0 and write
  // sums nothing reads)
  const int nq = (npair + LB - 1) / LB, nd = DIAG ? (wy + LB - 1) / LB : 0;
  // hi and lo parts apart: the packed coupling sums read them as they are
  float* Sh = reinterpret_cast<float*>(smem_raw);
  float* Sl = Sh + (size_t)nq * LB;
  float* Dh = Sl + (size_t)nq * LB;
  float* Dl = Dh + (size_t)nd * LB;
  float* Vt = Dl + (size_t)nd * LB;
  float* Xt = Vt + (size_t)M1 * DF_VS;
  __shared__ float Ch[256], Cl[256];
  for (int t = threadIdx.x; t < ncls; t += blockDim.x) {
    Ch[t] = ctab[t].hi;
    Cl[t] = ctab[t].lo;
  }
  int it = 0;
  double beta = 0.0, dot = 0.0;
  const double* pold = nullptr;
  double* pnew = nullptr;
  if constexpr (OUTER) {
    it = a.ctl->it;
    beta = it == 0 ? 0.0 : a.sc[SC_BETA];
    pold = (it & 1) ? pB : pA;
    pnew = (it & 1) ? pA : pB;
  }
  for (int r = blockIdx.x; r < n; r += gridDim.x) {
    const int rb = rowptr[r], re = rowptr[r + 1];
    for (int cs = rb; cs < re; cs += DF_CH) {
      const int nzc = min(DF_CH, re - cs);
      __syncthreads();
      df_stage<TX>(cs, nzc, M1, colidx, vals, X, ldx, wx, Vt, Xt);
      __syncthreads();
      const bool first = cs == rb;
      if (DIAG) {
        for (int i = 0; i < nd; ++i) {
          const int l = threadIdx.x + i * LB;
          df64 d = df_dot9(Vt, Xt + min(l, wx - 1) * DF_XS);
          if (!first) d += df64(Dh[l], Dl[l]);
          Dh[l] = d.hi;
          Dl[l] = d.lo;
        }
      }
      // consecutive threads: consecutive pairs, each as its staged offsets
      const unsigned* pp = pkj + threadIdx.x;
      unsigned next = threadIdx.x < npair ? __ldg(pp) : 0u;
#pragma unroll 2
      for (int qi = threadIdx.x; qi < nq * LB; qi += LB) {
        const unsigned o = next;
        pp += LB;
        next = qi + LB < npair ? __ldg(pp) : 0u;
        df64 s = df_dot9(Vt + (o >> 16), Xt + (o & 0xffffu));
        if (!first) s += df64(Sh[qi], Sl[qi]);
        Sh[qi] = s.hi;
        Sl[qi] = s.lo;
      }
    }
    __syncthreads();
    for (int slot = threadIdx.x; slot < wy; slot += LB) {
      const int2 d = __ldg(sdesc + slot);
      const int l = (int)((unsigned)d.y >> 16), ncl = d.y & 0xffff;   // ncl: the warp's count
      double zv = 0.0, po = 0.0, qo = 0.0, yin = 0.0;   // loaded before the sums that they meet
      if constexpr (OUTER) {
        const size_t g = (size_t)r * wx + l;
        zv = widen_exact(X[g]);
        if (it != 0) {
          po = pold[g];
          qo = q[g];
        }
      }
      if constexpr (MODE == DF_SUB) yin = Yin[(size_t)r * ldyin + l];
      df64 acc(0.f, 0.f);
      if (re > rb) {
        if (DIAG) acc = df64(Dh[l], Dl[l]);
        // two couplings at a time, side by side in packed sums (the counts are even)
        auto at = [](const float* p, unsigned byte) {
          return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(p) + byte);
        };
        auto couple = [&](unsigned w0, unsigned w1, df64x2& s) {
          const unsigned k0 = w0 & 0x3ffu, k1 = w1 & 0x3ffu, q0 = w0 >> 10, q1 = w1 >> 10;
          const float2 ch = make_float2(at(Ch, k0), at(Ch, k1)), cl = make_float2(at(Cl, k0), at(Cl, k1));
          const float2 sh = make_float2(at(Sh, q0), at(Sh, q1)), sl = make_float2(at(Sl, q0), at(Sl, q1));
          df64x2 v;
          v.hi = __fmul2_rn(ch, sh);
          v.lo = __ffma2_rn(cl, sh, __ffma2_rn(ch, sl, __ffma2_rn(ch, sh, neg2(v.hi))));
          df_add2(s, v);
        };
        const unsigned* cw = ctr + d.x;
        df64x2 s;
        s.hi = s.lo = make_float2(0.f, 0.f);
        int c = 0;
        for (; c + 4 <= ncl; c += 4, cw += 128) {
          const unsigned w0 = __ldg(cw), w1 = __ldg(cw + 32), w2 = __ldg(cw + 64), w3 = __ldg(cw + 96);
          couple(w0, w1, s);
          couple(w2, w3, s);
        }
        for (; c < ncl; c += 2, cw += 64) couple(__ldg(cw), __ldg(cw + 32), s);
        acc += df64(s.hi.x, s.lo.x);
        acc += df64(s.hi.y, s.lo.y);
      }
      acc = df_norm(acc);
      if constexpr (OUTER) {
        const size_t g = (size_t)r * wx + l;
        const double av = f2d_fast(acc.hi) + f2d_fast(acc.lo);
        const double pv = it == 0 ? zv : zv + beta * po;
        const double qv = it == 0 ? av : av + beta * qo;
        pnew[g] = pv;
        q[g] = qv;
        dot += pv * qv;
      } else if constexpr (MODE == DF_PLAIN) {
        Y[(size_t)r * ldy + l] = f2d_fast(acc.hi) + f2d_fast(acc.lo);
      } else {
        // Yin - sum in double-float, rounded once to FP32
        df64 v = df_from_double(yin);
        v += df64(-acc.hi, -acc.lo);
        Y[(size_t)r * ldy + l] = v.hi + v.lo;
      }
    }
  }
  if constexpr (OUTER) {
    double pq, unused;
    // (the sums' shared memory is free after the last row)
    __syncthreads();
    double* red = reinterpret_cast<double*>(smem_raw);
    if (outer_reduce_last(dot, 0.0, a, pq, unused, red, red + LB) && threadIdx.x == 0) {
      a.sc[SC_PQ] = pq;
      if (!(pq > 0.0)) {
        atomicOr(a.status, ST_OUTER_BREAKDOWN);
        a.sc[SC_ALPHA] = 0.0;
      } else {
        a.sc[SC_ALPHA] = a.sc[SC_RHO] / pq;
      }
      a.hist_alpha[it] = a.sc[SC_ALPHA];
    }
  }
}

// Block size: 256 threads up to DF_MAXQ pairs a thread, else 512 (more, smaller
// blocks hide the row barriers better).
static int df_threads(const EdgeList& E) { return E.npair <= DF_MAXQ * 256 ? 256 : 512; }

// (at least the outer step's final sums of two doubles per thread)
static size_t df_smem(const EdgeList& E, int M1, int wx, bool diag) {
  const size_t t = (size_t)df_threads(E);
  auto pad = [t](size_t v) { return (v + t - 1) / t * t; };
  return std::max((2 * (pad(E.npair) + (diag ? pad(E.nout) : 0)) + (size_t)M1 * DF_VS + (size_t)wx * DF_XS) *
                      sizeof(float),
                  t * 2 * sizeof(double));
}

// Usable up to DF_MAXQ pairs for each of 512 threads (beyond, the general
// kernel), when the couplings have a compact table with slot descriptors, the
// pairs' offsets fit 16 bits and sums and staging fit a block's shared memory.
bool df_pairs_usable(const sg_problem* h, const EdgeList& E, int wx) {
  return h->staged_pairs && E.npair <= DF_MAXQ * 512 && (E.pkj || E.npair == 0) && E.ncls > 0 && E.sdesc && h->nterm * DF_VS < 65536 &&
         wx * DF_XS < 65536 && df_smem(E, h->nterm, wx, true) + 4 * 1024 <= (size_t)std::max(h->smem_optin, 48 * 1024);
}

template <bool DIAG, int MODE, typename TX, typename TY>
static int launch_df(sg_problem* h, const EdgeList& E, const TX* X, int ldx, int wx, const double* Yin, int ldyin,
                     TY* Y, int ldy, const OuterArgs* oa, cudaStream_t s) {
  const int wy = E.nout;
  if (wy == 0) return SG_OK;
  const int threads = df_threads(E);
  const size_t smem = df_smem(E, h->nterm, wx, DIAG);
  OuterArgs a = oa ? *oa : OuterArgs{};
  auto go = [&](auto kern) -> int {
    SG_TRY(allow_smem(h, kern));
    int per_sm = 0;
    SG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    int grid = std::min(h->n, h->num_sms * std::max(per_sm, 1));
    if (MODE == DF_OUTER) grid = std::min(grid, h->opart_blocks);
    { kern<<<grid, threads, smem, s>>>(h->n, h->rowptr, h->colidx, (const df64*)h->vals_df, h->nterm, X, ldx, wx,
                                       E.npair, E.pkj, E.ctr, E.sdesc, (const df64*)E.ctab, E.ncls, wy, Yin,
                                       ldyin, Y, ldy, h->fpA, h->fpB, h->fq, a); ::sghsc::note_launch(); }
    SG_CHECK_LAUNCH();
    return SG_OK;
  };
  if (threads == 256) return go(k_df_pairs<DIAG, MODE, TX, TY, 256>);
  return go(k_df_pairs<DIAG, MODE, TX, TY, 512>);
}

int launch_df_level(sg_problem* h, const EdgeList& E, const float* X, int ldx, int wx, const double* Yin, int ldyin,
                    float* Y, int ldy, cudaStream_t s) {
  return launch_df<false, DF_SUB, float, float>(h, E, X, ldx, wx, Yin, ldyin, Y, ldy, nullptr, s);
}

int launch_df_outer(sg_problem* h, const OuterArgs& a, cudaStream_t s, const float* z32) {
  // z itself in FP32 when the preconditioner leaves it there (half the staging reads, no conversion)
  float* none = nullptr;
  if (z32) return launch_df<true, DF_OUTER, float, float>(h, h->all, z32, h->P, h->P, nullptr, 0, none, 0, &a, s);
  return launch_df<true, DF_OUTER, double, float>(h, h->all, h->fz, h->P, h->P, nullptr, 0, none, 0, &a, s);
}

int launch_df_apply(sg_problem* h, const float* U, double* Y, cudaStream_t s) {
  return launch_df<true, DF_PLAIN, float, double>(h, h->all, U, h->P, h->P, nullptr, 0, Y, h->P, nullptr, s);
}

}  // namespace sghsc
