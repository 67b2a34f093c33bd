#pragma once
// KS: summation with the permuted block on chip, for layouts whose d permuted
// indices form one dense block of O^d elements per spectator position (a
// torch-contiguous tensor: permuted indices fastest, spectators outside, at
// any strides).
//
// There the members of an orbit are scattered inside a block of O^d elements
// (14 KB for O = 12, d = 3), so a CTA copies the blocks of NS spectator
// positions into shared memory with unit-stride asynchronous copies, runs
// every element orbit in shared memory and stores the blocks back with
// unit-stride stores: each element crosses HBM once each way. The general
// kernel KG reads and writes the same elements as scattered 8-byte accesses,
// unranks a tuple per thread and sums with FP64 instructions: 2480 us on
// A[32^3, 12^3], factorized Table II row 1 (0.37 TB/s), against 396 us here (507 with one
// buffer per CTA, 470 with the multiplication by alpha predicated into the common path).
//
// - Canonical tuples come from a table in shared memory, grouped by equality
//   pattern and built once per CTA, so warps run one pattern's code and no
//   thread searches for its tuple.
// - For even O every row, plane and volume of the block is followed by one
//   unused element: all index strides in shared memory are odd, so lanes that
//   step along any permuted index fall on different banks.
// - KG's FP64 arithmetic is native FP64 in the reference order; GB300's FP64
//   pipe (2 operations per SM per clock) limits that to 57 G elements/s on the
//   three-factor-term chains. Here the sums run in 64-bit integers on a grid
//   fine enough that the result is as accurate as the FP64 sum (fixed_sum
//   below); groups outside its range, groups of an operator with zero
//   coefficients whose magnitudes are too far apart, and SPINSUM_STRICT take
//   the FP64 order.
#include <algorithm>
#include <array>
#include <cmath>

#include "ss_devcache.h"
#include "ss_k2.cuh"

namespace ss {

// kernel-template choices of this file: FP64 through fixed_sum; the same with an alpha that is
// no power of two (one kernel for both would issue the multiplication, predicated off, on the
// FP64 pipe, the busiest one); and with fixed_sum's guard, for operators with zero coefficients,
// any alpha (compiled into the first, unused: A[32^3,12^3] 404 us against 396)
constexpr int AR_FIXED = 4, AR_FIXED_MUL = 5, AR_FIXED_GUARD = 6;

struct KsArgs {
  int ns;             // spectator positions per round
  int T, Tp;          // elements of a permuted block, and with its padding
  int nbuf;           // buffers of ns blocks (2: the next round is copied under the sums)
  unsigned mT, mO;    // ceil(2^32 / T), ceil(2^32 / O)
  unsigned mO2, mO3;  // ceil(2^32 / O^2), ceil(2^32 / O^3)
  unsigned mN[8];     // ceil(2^32 / orbits of pattern p)
  int pad;            // 1: padded rows, planes, volumes (even O)
  int pst[4];         // shared-memory stride of permuted index k
  int ntot;           // canonical tuples
  int otab;           // offset of the tables in shared memory (bytes)
  int bits;           // AR_FIXED: an input's magnitude stays below 2^bits
  int sh0;            // AR_FIXED: result exponent offset (see fixed_sum)
  unsigned emin, emax;
  int supp[8];        // AR_FIXED: fewest inputs of an output of pattern p; 0: all of them
  int guard;          // AR_FIXED: some of supp are not 0
  unsigned below;     // AR_FIXED: an input this far (exponent field) below the largest is small
};

// quotient by a constant n > 1 with its precomputed reciprocal (numerators below 2^16)
__device__ __forceinline__ int ks_div(int n, unsigned m) { return (int)__umulhi((unsigned)n, m); }

// A fixed-point value lo + hi 2^32 with a SIGNED low word, so that a product
// with a 32-bit coefficient is one 32 x 32 -> 64-bit multiply-add and one
// 32-bit one.
struct Fix64 {
  int lo, hi;
};
__device__ __forceinline__ Fix64 fix64(long long X) {
  const int lo = (int)(unsigned)X;
  return Fix64{lo, (int)(X >> 32) + (int)((unsigned)lo >> 31)};
}
// (sums modulo 2^64: where the total fits, partial sums may pass 2^63)
__device__ __forceinline__ long long wrap_add(long long a, long long b) {
  return (long long)((unsigned long long)a + (unsigned long long)b);
}
__device__ __forceinline__ long long wrap_sub(long long a, long long b) {
  return (long long)((unsigned long long)a - (unsigned long long)b);
}
__device__ __forceinline__ void fix64_mac(long long& acc, int c, const Fix64& x) {
  acc = wrap_add(acc, (long long)c * (long long)x.lo);
  acc = wrap_add(acc, (long long)((unsigned long long)((unsigned)c * (unsigned)x.hi) << 32));
}

// The orbit operator of pattern P in 64-bit integers. Inputs are rounded to
// the grid 2^(E + 1 - bits) (2^E the leading power of the group's largest
// input), bits = 62 - log2 sum|a| (d = 4: the largest for which four times the
// result stays below 2^63), so that every sum is exact in 64 bits; the only other
// rounding is the final one to FP64. Error: at most sum|a| 2^(E - bits) + half a unit
// in the last place.
// That is below the FP64 sum's (a rounding of every product and partial sum) where
// an output takes the largest input of its group. An operator with zero coefficients
// has outputs that take only some: where all of an output's inputs may lie far below
// the largest (ka.below), the group is summed in FP64. Relative to sum |a x| of each
// output, largest over 4000 random groups with magnitudes over 0 / 4 / 8 decades
// (without that guard / with it / FP64 order): Table II row 2 1.1e-16, 3.2e-15, 8.1e-12 /
// 1.1e-16, 1.4e-16, 2.1e-16 / 2.2e-16, 2.1e-16, 2.2e-16; row 5, whose outputs take all
// inputs, 9e-17, 3e-16, 5e-16 / FP64 2.2e-16, 3.3e-16, 4.7e-16.
// Returns false for such groups and for those whose exponents leave [emin, emax]
// (infinities and NaNs among them).
template <int D, int P, bool GUARD, class Sink>
__device__ __forceinline__ bool fixed_sum(const KParams& kp, const KsArgs& ka, const double (&x)[Pat<D, P>::M],
                                          Sink&& sink) {
  constexpr int M = Pat<D, P>::M;
  unsigned mx = 0;
#pragma unroll
  for (int v = 0; v < M; v++) mx = max(mx, (unsigned)__double2hiint(x[v]) & 0x7FFFFFFFu);
  unsigned E = mx & 0x7FF00000u;
  if (E < ka.emin || E > ka.emax) {
    unsigned any = mx;
#pragma unroll
    for (int v = 0; v < M; v++) any |= (unsigned)__double2loint(x[v]);
    if (any != 0) return false;
    E = ka.emin;  // a group of zeros is exact on any grid
  }
  if (GUARD && ka.supp[P] != 0) {
    const unsigned small = E > ka.below ? E - ka.below : 0;
    int n = 0, z = 0;  // small inputs, and zeros (exact on any grid)
#pragma unroll
    for (int v = 0; v < M; v++) {
      const unsigned a = (unsigned)__double2hiint(x[v]) & 0x7FFFFFFFu;
      n += a < small;
      z += (a | (unsigned)__double2loint(x[v])) == 0;
    }
    if (n > z && n >= ka.supp[P]) return false;
  }
  // (E | 0xFFFFF) - |x|'s high word borrows nothing from the exponent field
  const unsigned base = (E | 0xFFFFFu) + ((unsigned)(62 - ka.bits) << 20);
  long long X[M];
#pragma unroll
  for (int v = 0; v < M; v++) {
    const unsigned hi = (unsigned)__double2hiint(x[v]), lo = (unsigned)__double2loint(x[v]);
    const unsigned k = (base - (hi & 0x7FFFFFFFu)) >> 20;
    const unsigned long long mant =
        (((unsigned long long)((hi & 0x000FFFFFu) | 0x00100000u) << 32) | lo) << 10;  // below 2^63
    const long long q = (long long)((shr64(mant, k) + 1) >> 1);                       // rounded to the grid
    X[v] = (int)hi < 0 ? -q : q;
  }
  const int sh = (int)(E >> 20) + ka.sh0;
  if constexpr (D == 4 && wht_ok<P>()) {
    constexpr int NB = M / 4, WOFF = wh_offset(P);
    Fix64 t[M];
#pragma unroll
    for (int o = 0; o < NB; o++) {
      const long long x0 = X[kWht<P>.orb[o][0]], x1 = X[kWht<P>.orb[o][1]], x2 = X[kWht<P>.orb[o][2]],
                      x3 = X[kWht<P>.orb[o][3]];
      const long long a0 = x0 + x1, a1 = x0 - x1, a2 = x2 + x3, a3 = x2 - x3;  // below 2^62
      t[4 * o] = fix64(wrap_add(a0, a2));  // characters 0..3
      t[4 * o + 1] = fix64(wrap_add(a1, a3));
      t[4 * o + 2] = fix64(wrap_sub(a0, a2));
      t[4 * o + 3] = fix64(wrap_sub(a1, a3));
    }
#pragma unroll
    for (int o = 0; o < NB; o++) {
      long long yh[4] = {0, 0, 0, 0};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int i = 4 * o + k;
#pragma unroll
        for (int q = 0; q < 6; q++)
          if (q < kWht<P>.nnz[i]) fix64_mac(yh[k], kp.wh[WOFF + kWht<P>.woff[i] + q], t[kWht<P>.col[i][q]]);
      }
      const long long b0 = wrap_add(yh[0], yh[1]), b1 = wrap_sub(yh[0], yh[1]);
      const long long b2 = wrap_add(yh[2], yh[3]), b3 = wrap_sub(yh[2], yh[3]);
      const long long y4[4] = {wrap_add(b0, b2), wrap_add(b1, b3), wrap_sub(b0, b2), wrap_sub(b1, b3)};  // 4 Y
#pragma unroll
      for (int vi = 0; vi < 4; vi++) sink(kWht<P>.orb[o][vi], fixed_rn(y4[vi], sh - 2));
    }
  } else {
    Fix64 t[M];
    long long acc[M];
#pragma unroll
    for (int v = 0; v < M; v++) t[v] = fix64(X[v]);
    if constexpr (P == 0) {
#pragma unroll
      for (int st = 0; st < MAXSTAGE_EXACT; st++) {
        if (st >= kp.nci) break;
        if (st > 0) {
#pragma unroll
          for (int u = 0; u < M; u++) t[u] = fix64(acc[u]);
        }
#pragma unroll
        for (int u = 0; u < M; u++) acc[u] = 0;
#pragma unroll
        for (int s = 0; s < fact(D); s++) {
          const int c = kp.ci[st][s];
          if (c != 0) {
#pragma unroll
            for (int u = 0; u < M; u++) fix64_mac(acc[u], c, t[Pat<D, P>::idx(u, s)]);
          }
        }
      }
    } else {
      const int* mp = kp.mp + mp_offset<D>(P);
#pragma unroll
      for (int u = 0; u < M; u++) {
        acc[u] = 0;
#pragma unroll
        for (int v = 0; v < M; v++) fix64_mac(acc[u], mp[u * M + v], t[v]);
      }
    }
#pragma unroll
    for (int u = 0; u < M; u++) sink(u, fixed_rn(acc[u], sh));
  }
  return true;
}

// shared-memory place of member u of the orbit with values val
template <int D, int P>
__device__ __forceinline__ int ks_slot(const KsArgs& ka, int u, const int (&val)[4]) {
  int a = 0;
#pragma unroll
  for (int k = 0; k < D; k++) a += val[Pat<D, P>::lab(u, k)] * ka.pst[k];
  return a;
}

// the FP64 reference order for one group, out of line: rare in AR_FIXED, and
// inlined its FP64 instructions may be predicated into the common path
template <int D, int P>
static __device__ __noinline__ void ks_strict_group(const KParams& kp, const KsArgs& ka, unsigned tup, double* sm) {
  constexpr int M = Pat<D, P>::M;
  const int val[4] = {(int)(tup & 255), (int)(tup >> 8 & 255), (int)(tup >> 16 & 255), (int)(tup >> 24)};
  double x[M];
#pragma unroll
  for (int u = 0; u < M; u++) x[u] = sm[ks_slot<D, P>(ka, u, val)];
  strict_core<D, P>(kp, x);
#pragma unroll
  for (int u = 0; u < M; u++) sm[ks_slot<D, P>(ka, u, val)] = __dmul_rn(kp.alpha, x[u]);
}

template <int D, int P, int AR, typename T>
__device__ __forceinline__ void ks_group(const KParams& kp, const KsArgs& ka, unsigned tup, T* sm) {
  constexpr int M = Pat<D, P>::M;
  const int val[4] = {(int)(tup & 255), (int)(tup >> 8 & 255), (int)(tup >> 16 & 255), (int)(tup >> 24)};
  if constexpr (AR == AR_STRICT) {
    ks_strict_group<D, P>(kp, ka, tup, sm);
  } else {
    T x[M];
#pragma unroll
    for (int u = 0; u < M; u++) x[u] = sm[ks_slot<D, P>(ka, u, val)];
    if constexpr (AR == AR_FIXED || AR == AR_FIXED_MUL || AR == AR_FIXED_GUARD) {
      auto sink = [&](int u, double y) {
        if (AR == AR_FIXED_MUL || (AR == AR_FIXED_GUARD && D < 4 && (kp.flags & KF_ALPHA_MUL))) y = __dmul_rn(kp.alpha, y);
        sm[ks_slot<D, P>(ka, u, val)] = y;
      };
      if (!fixed_sum<D, P, AR == AR_FIXED_GUARD>(kp, ka, x, sink)) ks_strict_group<D, P>(kp, ka, tup, sm);
    } else {
      T y[M];
      apply_group<D, P, AR, T>(kp, x, y);
#pragma unroll
      for (int u = 0; u < M; u++) sm[ks_slot<D, P>(ka, u, val)] = y[u];
    }
  }
}

// every orbit of pattern P of the round's ns blocks; `first` is the table index
// of the pattern's first tuple, `rot` spreads short patterns over the warps
template <int D, int P, int AR, typename T>
__device__ __forceinline__ void ks_pattern(const KParams& kp, const KsArgs& ka, const unsigned* tab, int ns, T* sm,
                                           int& first, int& rot) {
  const int n = (int)kp.norb[P];
  const int total = n * ns;
  int q = (int)threadIdx.x - rot;
  if (q < 0) q += (int)blockDim.x;
  for (; q < total; q += (int)blockDim.x) {
    const int s = n == 1 ? q : ks_div(q, ka.mN[P]);
    ks_group<D, P, AR, T>(kp, ka, tab[first + q - s * n], sm + s * ka.Tp);
  }
  first += n;
  rot = (rot + total) % (int)blockDim.x & ~31;
}

template <int D, int P>
__device__ __forceinline__ void ks_table(const KParams& kp, unsigned* tab, int& first) {
  const int n = (int)kp.norb[P];
  for (int g = threadIdx.x; g < n; g += blockDim.x) {
    int v[4] = {0, 0, 0, 0};
    unrank<Pat<D, P>::ND>(g, kp.O, v);
    tab[first + g] = (unsigned)v[0] | (unsigned)v[1] << 8 | (unsigned)v[2] << 16 | (unsigned)v[3] << 24;
  }
  first += n;
}

template <int D, int AR, int NT, int MINB, typename T>
__global__ void __launch_bounds__(NT, MINB) ks_kernel(const __grid_constant__ KParams kp, const __grid_constant__ KsArgs ka) {
  extern __shared__ __align__(16) unsigned char ks_smem[];
  T* const buf = reinterpret_cast<T*>(ks_smem);
  // tables: spectator offsets of A and B [3][2][ns] (the round that is stored, the
  // one that is summed and the one that is copied), canonical tuples, padded places
  int64_t* const soff = reinterpret_cast<int64_t*>(ks_smem + ka.otab);
  unsigned* const tab = reinterpret_cast<unsigned*>(soff + 6 * ka.ns);
  unsigned short* const place = reinterpret_cast<unsigned short*>(tab + ka.ntot);
  {
    int first = 0;
    ks_table<D, 0>(kp, tab, first);
    ks_table<D, 1>(kp, tab, first);
    if constexpr (D >= 3) {
      ks_table<D, 2>(kp, tab, first);
      ks_table<D, 3>(kp, tab, first);
    }
    if constexpr (D == 4) {
      ks_table<D, 4>(kp, tab, first);
      ks_table<D, 5>(kp, tab, first);
      ks_table<D, 6>(kp, tab, first);
      ks_table<D, 7>(kp, tab, first);
    }
  }
  // padded place of block element t
  for (int t = threadIdx.x; t < ka.T; t += NT) {
    int f = t;
    if (ka.pad) {
      f += ks_div(t, ka.mO);
      if constexpr (D >= 3) f += ks_div(t, ka.mO2);
      if constexpr (D == 4) f += ks_div(t, ka.mO3);
    }
    place[t] = (unsigned short)f;
  }
  const T* const A = static_cast<const T*>(kp.A);
  T* const B = static_cast<T*>(kp.B);
  const int64_t step = (int64_t)gridDim.x * ka.ns;
  auto offsets = [&](int64_t s0, int64_t* so) {
    for (int i = threadIdx.x; i < ka.ns && s0 + i < kp.S; i += NT) {
      int64_t s = s0 + i, a = 0, b = 0;
#pragma unroll
      for (int k = 0; k < D; k++) {
        const int64_t q = s / kp.sext[k], r = s - q * kp.sext[k];
        a += r * kp.slda[k];
        b += r * kp.sldb[k];
        s = q;
      }
      so[i] = a;
      so[ka.ns + i] = b;
    }
  };
  auto count = [&](int64_t s0) { return (int)min((int64_t)ka.ns, kp.S - s0); };
  // f(block of the round, element of the block): by whole blocks where they fill the CTA
  auto each = [&](int ns, auto&& f) {
    if (ka.T >= 4 * NT) {
      for (int i = 0; i < ns; i++)
        for (int t = threadIdx.x; t < ka.T; t += NT) f(i, t);
    } else {
      const int ne = ns * ka.T;
      for (int e = threadIdx.x; e < ne; e += NT) {
        const int i = ka.ns == 1 ? 0 : ks_div(e, ka.mT);
        f(i, e - i * ka.T);
      }
    }
  };
  auto load = [&](int ns, T* sm, const int64_t* so) {
    each(ns, [&](int i, int t) { cp_async<sizeof(T)>(sm + i * ka.Tp + place[t], A + so[i] + t); });
  };
  const bool beta = kp.flags & KF_BETA;
  const T bt = beta_of<T>(kp);
  int64_t s0 = (int64_t)blockIdx.x * ka.ns;
  offsets(s0, soff);
  __syncthreads();
  if (ka.nbuf == 2) {
    load(count(s0), buf, soff);
    cp_async_commit();
  }
  for (int k = 0; s0 < kp.S; s0 += step, k++) {
    const int ns = count(s0);
    T* const sm = buf + (ka.nbuf == 2 && (k & 1) ? ka.ns * ka.Tp : 0);
    int64_t* const so = soff + k % 3 * 2 * ka.ns;
    int64_t* const son = soff + (k + 1) % 3 * 2 * ka.ns;
    offsets(s0 + step, son);
    if (ka.nbuf == 2) {
      __syncthreads();  // the next offsets are there; the previous round's stores have read the other buffer
      if (s0 + step < kp.S) load(count(s0 + step), buf + ((k & 1) ? 0 : ka.ns * ka.Tp), son);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      load(ns, sm, so);
      cp_async_commit();
      cp_async_wait<0>();
    }
    __syncthreads();
    int first = 0, rot = 0;
    ks_pattern<D, 0, AR, T>(kp, ka, tab, ns, sm, first, rot);
    ks_pattern<D, 1, AR, T>(kp, ka, tab, ns, sm, first, rot);
    if constexpr (D >= 3) {
      ks_pattern<D, 2, AR, T>(kp, ka, tab, ns, sm, first, rot);
      ks_pattern<D, 3, AR, T>(kp, ka, tab, ns, sm, first, rot);
    }
    if constexpr (D == 4) {
      ks_pattern<D, 4, AR, T>(kp, ka, tab, ns, sm, first, rot);
      ks_pattern<D, 5, AR, T>(kp, ka, tab, ns, sm, first, rot);
      ks_pattern<D, 6, AR, T>(kp, ka, tab, ns, sm, first, rot);
      ks_pattern<D, 7, AR, T>(kp, ka, tab, ns, sm, first, rot);
    }
    __syncthreads();
    if (beta)
      each(ns, [&](int i, int t) {
        T* g = B + so[ka.ns + i] + t;
        *g = add_beta(sm[i * ka.Tp + place[t]], *g, bt);
      });
    else
      each(ns, [&](int i, int t) { B[so[ka.ns + i] + t] = sm[i * ka.Tp + place[t]]; });
    if (ka.nbuf == 1) __syncthreads();  // the buffer is free again
  }
}

// most shared memory of a CTA
constexpr int KS_SMEM_MAX = 227 * 1024 - 1024;
// shared memory a round's blocks aim at: three CTAs per SM with two buffers each;
// larger blocks take one position per round, and one buffer where two do not fit
// (A[32^3,12^3] FP64: 396 us; CTAs of 128 threads, six or eight per SM, 400 and 413; four CTAs of
// 256 threads at 64 registers 455)
constexpr int KS_SMEM_AIM = 32 * 1024;

// Whether the problem has KS's layout (permuted strides 1, O, .., O^(d-1) in
// some order, the same in A and B) and its block fits on chip; fills ka and
// the CTA's shared-memory bytes. Below O^d = 64 the rows are too short to be
// worth staging. *fixed: the problem has an AR_FIXED form (FP64 with d = 4 needs the
// transform's weights, KF_WHT, for it).
inline bool ks_plan(int d, const KParams& kp, int es, KsArgs* ka, int* smem, bool* fixed) {
  const int64_t O = kp.O;
  int64_t T = 1;
  for (int k = 0; k < d; k++) T *= O;
  if (O < 2 || O > 255 || T < 64 || T > 40000) return false;
  int rank[4] = {0, 0, 0, 0};
  unsigned seen = 0;
  for (int k = 0; k < d; k++) {
    if (kp.lda[k] != kp.ldb[k]) return false;
    int r = -1;
    int64_t p = 1;
    for (int q = 0; q < d; q++, p *= O)
      if (kp.lda[k] == p) r = q;
    if (r < 0 || (seen >> r & 1)) return false;
    seen |= 1u << r;
    rank[k] = r;
  }
  ka->pad = O % 2 == 0;
  int64_t P[5] = {1, O + ka->pad, 0, 0, 0};
  for (int q = 2; q <= d; q++) P[q] = O * P[q - 1] + ka->pad;
  for (int k = 0; k < 4; k++) ka->pst[k] = k < d ? (int)P[rank[k]] : 0;
  ka->T = (int)T;
  ka->Tp = (int)P[d];
  int64_t ntot = 0;
  for (int p = 0; p < npatterns(d); p++) ntot += kp.norb[p];
  ka->ntot = (int)ntot;
  int64_t ns = KS_SMEM_AIM / (P[d] * es);
  if (ns < 1) ns = 1;
  if (ns > 64) ns = 64;
  if (ns > 65535 / T) ns = 65535 / T > 0 ? 65535 / T : 1;  // ks_div's numerators
  if (ns > kp.S) ns = kp.S;
  ka->ns = (int)ns;
  if (P[d] > 65535) return false;  // 16-bit places
  const int64_t tables = 48 * ns + 4 * ntot + (2 * T + 15) / 16 * 16;
  for (ka->nbuf = 2; ka->nbuf >= 1; ka->nbuf--) {
    ka->otab = (int)((ka->nbuf * ns * P[d] * es + 15) / 16 * 16);
    *smem = (int)(ka->otab + tables);
    if (*smem <= KS_SMEM_MAX) break;
  }
  if (ka->nbuf == 0) return false;
  for (int p = 0; p < 8; p++) ka->mN[p] = 0;
  for (int p = 0; p < npatterns(d); p++)
    if (kp.norb[p] > 0) ka->mN[p] = (unsigned)(((1ull << 32) + kp.norb[p] - 1) / kp.norb[p]);
  auto recip = [](int64_t n) { return (unsigned)(((1ull << 32) + n - 1) / n); };
  ka->mT = recip(T);
  ka->mO = recip(O);
  ka->mO2 = recip(O * O);
  ka->mO3 = d == 4 ? recip(O * O * O) : 0;
  // AR_FIXED: the grid from the operator's 1-norm (chain: product of the factors')
  *fixed = d <= 3 || (kp.flags & KF_WHT);
  double L = 1;
  for (int st = 0; st < kp.nci; st++) {
    double n = 0;
    for (int s = 0; s < (d == 2 ? 2 : (d == 3 ? 6 : 24)); s++) n += kp.ci[st][s] < 0 ? -kp.ci[st][s] : kp.ci[st][s];
    L *= n;
  }
  int lg = 0;
  while ((double)(1 << lg) < L) lg++;
  // (d = 4: 4 L 2^bits < 2^63)
  ka->bits = d == 4 ? ((double)(1 << lg) > L ? 61 - lg : 60 - lg) : 62 - lg;
  if (ka->bits > 60) ka->bits = 60;
  // kp.cexp = (53 - 2 W + kdrop + aexp) << 20 + 0x80000, aexp = alpha's and the coefficients' scale
  const int aexp = ((kp.cexp - 0x80000) >> 20) - 53 + 2 * kp.W - kp.kdrop;
  ka->sh0 = -1023 - (ka->bits - 1) + aexp;
  // the conversion's offsets 2^(1075 + sh - 2) .. 2^(1107 + sh) stay normal numbers
  int lo = 3 - 1075 - ka->sh0, hi = 2040 - 1107 - ka->sh0;
  if (lo < 72) lo = 72;  // subnormal inputs shift out entirely
  if (hi > 2046) hi = 2046;
  if (lo > hi) *fixed = false;
  ka->emin = (unsigned)lo << 20;
  ka->emax = (unsigned)hi << 20;
  return true;
}

// The inputs that the outputs of each pattern take, for fixed_sum's guard; *fixed is
// cleared for operators whose outputs take so few that the guard would send groups
// of like magnitudes to FP64 (of M uniform inputs, s or more lie 2^k below the largest
// with a probability of about C(M, s) 2^(-(k + 1) s)).
template <int D>
void ks_support(const KParams& kp, KsArgs* ka, bool* fixed) {
  static const Pattern<D> pt = make_pattern<D>(0);
  static const std::array<int, 8> moff = [] {
    std::array<int, 8> a{};
    for (int p = 1; p < npatterns(D); p++) a[p] = mp_offset<D>(p);
    return a;
  }();
  static const std::array<int, 8> mem = [] {
    std::array<int, 8> a{};
    for (int p = 0; p < npatterns(D); p++) a[p] = make_pattern<D>(p).m;
    return a;
  }();
  constexpr int M = fact(D);
  // the generic orbit: the chain's row of output 0, last stage first
  double w[M] = {};
  for (int s = 0; s < M; s++) w[pt.idx[0][s]] += kp.ci[kp.nci - 1][s];
  for (int st = kp.nci - 2; st >= 0; st--) {
    double t[M] = {};
    for (int v = 0; v < M; v++)
      for (int s = 0; s < M; s++) t[pt.idx[v][s]] += w[v] * kp.ci[st][s];
    for (int v = 0; v < M; v++) w[v] = t[v];
  }
  int n = 0;
  double sq = 0, least = 1e30;
  for (double c : w)
    if (c != 0) {
      n++;
      sq += c * c;
      least = std::min(least, std::fabs(c));
    }
  for (int& v : ka->supp) v = 0;
  ka->supp[0] = n < M ? n : 0;
  bool any = ka->supp[0] != 0;
  for (int p = 1; p < npatterns(D); p++) {
    const int m = mem[p];
    int few = m;
    for (int u = 0; u < m; u++) {
      int k = 0;
      for (int v = 0; v < m; v++) k += kp.mp[moff[p] + u * m + v] != 0;
      if (k > 0) few = std::min(few, k);
    }
    ka->supp[p] = few < m ? few : 0;
    any = any || ka->supp[p] != 0;
  }
  if (!any || n == 0) return;
  // an output's inputs reach 2^(E - k): the grid's share, about sqrt(sum a^2) 2^(E - bits), is
  // then a few half units of the output's own sum
  int k = (int)std::floor(ka->bits - 53 - std::log2(std::sqrt(sq) / least) + 2);
  k = std::max(3, std::min(6, k));
  ka->below = (unsigned)k << 20;
  ka->guard = 1;
  double few = 1;
  for (int i = 0; i < ka->supp[0]; i++) few *= (double)(M - i) / (i + 1) / (2 << k);
  if (ka->supp[0] != 0 && few > 0.002) *fixed = false;
}

// Whether KS is faster than KG, which takes a thread per orbit and position: a CTA of KS
// builds its tables (O^d places, the tuples) and takes whole blocks, so a call of few
// positions leaves SMs idle behind CTAs that mostly prepare. Measured over S = 1 .. 98304,
// inputs not in L2 where larger (KS / KG, us):
//   d = 2, fixed or FP32: O = 16, S = 1024 8.6 / 6.8, 2048 9.3 / 11.0; O = 64, S = 256 30 / 24,
//     512 38 / 42; O = 128, S = 1 140 / 8.5, 256 164 / 124, 512 205 / 242; FP32 alike;
//     strict (FP64 pipe in both): O = 32, S = 4096 67 / 64, 16384 237 / 324.
//   d = 3, fixed: O = 8, S = 64 10.8 / 10.1, 512 11.1 / 16.2; O = 20, S = 64 26 / 24, 128
//     27 / 38; O = 27, S = 64 64 / 42, 128 66 / 78. FP32: O = 8, S = 1024 9.2 / 8.8, 2048
//     10.0 / 13.6; O = 24, S = 256 39 / 39, 512 54 / 75. Strict: O = 12, S = 4096 400 / 235.
//   d = 4, fixed: O = 3, S = 16 16 / 48, 4096 16 / 43; O = 12, S = 1 42 / 68, 1024 270 / 1240.
//     FP32 (KG holds its own while the tensors stay in L2): O = 8, S = 2048 170 / 131, 8192
//     638 / 829; O = 12, S = 256 71 / 70, 1024 223 / 409. Strict: O = 8, S = 1024 573 / 262.
inline bool ks_faster(int d, bool f32, bool fixed, int64_t S, int64_t O, int64_t T) {
  const int64_t N = S * T;
  if (d == 2) {
    if (!f32 && !fixed) return N >= 9000000;
    return N >= 520000 && S >= (O < 80 ? 520 : 340);
  }
  if (f32) return d == 3 ? N >= 650000 && S >= 250 : N >= 11000000;
  if (!fixed) return false;
  return d == 4 || T < 3000 || S >= 96;
}

template <int D, int AR, int NT, int MINB, typename T>
cudaError_t launch_ks_impl(const KParams& kp, const KsArgs& ka, int smem, cudaStream_t st) {
  auto fn = ks_kernel<D, AR, NT, MINB, T>;
  static DeviceCache cache;  // SMs, after raising the kernel's shared-memory limit
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  long long sms = 0;
  const int rc = cache.get(dev, &sms, [&](long long* val) {
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, KS_SMEM_MAX);
    if (err != cudaSuccess) return (int)err;
    int n = 0;
    err = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    *val = n;
    return (int)err;
  });
  if (rc != 0) return rc < 0 ? cudaErrorInvalidDevice : (cudaError_t)rc;
  const int64_t rounds = (kp.S + ka.ns - 1) / ka.ns;
  int per = (KS_SMEM_MAX + 1024) / (smem + 1024);
  if (per > MINB) per = MINB;
  const int64_t grid = rounds < sms * per ? rounds : sms * per;
  fn<<<(unsigned)grid, NT, smem, st>>>(kp, ka);
  return cudaGetLastError();
}

// true (and *e the launch status) when KS takes the problem
template <int D>
bool launch_ks(const KParams& kp, int ar, cudaStream_t st, cudaError_t* e) {
  KsArgs ka{};
  int smem = 0;
  bool fixed = false;
  if (!ks_plan(D, kp, ar == AR_F32 ? 4 : 8, &ka, &smem, &fixed)) return false;
  fixed = fixed && ar == AR_EXACT;
  if (fixed) ks_support<D>(kp, &ka, &fixed);
  if (!ks_faster(D, ar == AR_F32, fixed, kp.S, kp.O, ka.T)) return false;
  if constexpr (D == 4) {
    // 24-member groups take 128 registers: two CTAs of 256 threads, or, where a
    // block leaves room for one CTA only, one of 512
    if (ar == AR_F32) *e = launch_ks_impl<4, AR_F32, 256, 2, float>(kp, ka, smem, st);
    else if (smem > KS_SMEM_MAX / 2)
      *e = ka.guard ? launch_ks_impl<4, AR_FIXED_GUARD, 512, 1, double>(kp, ka, smem, st)
                    : launch_ks_impl<4, AR_FIXED, 512, 1, double>(kp, ka, smem, st);
    else if (ka.guard) *e = launch_ks_impl<4, AR_FIXED_GUARD, 256, 2, double>(kp, ka, smem, st);
    else *e = launch_ks_impl<4, AR_FIXED, 256, 2, double>(kp, ka, smem, st);
  } else {
    if (ar == AR_F32) *e = launch_ks_impl<D, AR_F32, 256, 5, float>(kp, ka, smem, st);
    else if (fixed && ka.guard) *e = launch_ks_impl<D, AR_FIXED_GUARD, 256, 3, double>(kp, ka, smem, st);
    else if (fixed && (kp.flags & KF_ALPHA_MUL)) *e = launch_ks_impl<D, AR_FIXED_MUL, 256, 3, double>(kp, ka, smem, st);
    else if (fixed) *e = launch_ks_impl<D, AR_FIXED, 256, 3, double>(kp, ka, smem, st);
    else if constexpr (D == 2) *e = launch_ks_impl<D, AR_STRICT, 256, 3, double>(kp, ka, smem, st);
  }
  return true;
}

}  // namespace ss
