#pragma once
// K2T: the tiled kernel for the paper's layout (see ss_k2.cuh for the method),
// fed and drained by TMA.
//
// K2's CTA copies a block orbit's tiles with its own threads, meets at a
// barrier, sums, meets again, and copies the tiles back: 59 % (3D) and 40 % (4D)
// issue with the barriers as the top stall, and a third of the instructions
// spent on the copies. Here
// - one warp finds the block orbits and loads their m_b <= d! tiles by TMA (one
//   box per lane) into a ring of NST stages, another stores finished stages back by
//   TMA (clipped at the upper edge by the hardware), and eight warps only sum; every
//   hand-over is an mbarrier, so loads, sums and stores of different block orbits
//   overlap within a CTA;
// - a CTA takes its next id from the hardware's launch queue (cluster launch
//   control) instead of a fixed share: ids are worked on in launch order by
//   whichever CTA is free, so the rows of neighbouring tiles meet in L2 (A[544]^3 /
//   A[112]^4 with runs of 4 / 8 ids per CTA: 497 / 1278 us, with four requests in
//   flight 424 / 919, against 416 / 707);
// - tiles lie in shared memory as TMA writes them, without a swizzle: the lanes
//   of a half warp take canonical offsets on a linear code over GF(2) (elem below)
//   chosen so that all d! permuted reads fall on 16 different bank pairs
//   (tests/test_k2t_cpu.py checks every permutation).
//
// FP64, factorized Table II rows 1 and 5: A[544]^3 590 -> 412 us (6.2 TB/s, 0.92 of the
// copy; bound by DRAM and, next, FP64 and issue), A[112]^4 1084 -> 563 us (4.5 TB/s; 48 KB
// block orbits leave room for four in flight per SM: the sums wait for loads).
//
// TMA needs 16-byte strides (even extents for FP64); other tensors, the beta
// term, strict order, dense d = 4 operators, tensors in host memory and d = 2 (two
// 8 KB tiles per block orbit: 271 us against K2's 217 at N = 8192) stay with K2.
#include <cuda.h>

#include "ss_k2.cuh"
#include "ss_tma.cuh"

namespace ss {

template <int D>
struct K2TShape;
template <>
struct K2TShape<3> {
  static constexpr int BL = 8, NT = 512;
  __host__ __device__ static constexpr void elem(int e, int (&w)[4]) {
    const int a = e & 1, b = (e >> 1) & 1, c = (e >> 2) & 1, d = (e >> 3) & 1;
    w[0] = (b ^ c) | c << 1 | d << 2;
    w[1] = (a ^ c ^ ((e >> 4) & 1)) | a << 1 | (d ^ ((e >> 5) & 1)) << 2;
    w[2] = ((a ^ b) | a << 1 | d << 2) ^ ((e >> 6) & 7);
    w[3] = 0;
  }
};
template <>
struct K2TShape<4> {
  static constexpr int BL = 4, NT = 256;
  // w0 = x, w1 = y, w2 = x + y + z, w3 = x + g y + t over GF(4) (g its generator):
  // any two of the four determine (x, y)
  __host__ __device__ static constexpr void elem(int e, int (&w)[4]) {
    const int x = e & 3, y = (e >> 2) & 3, z = (e >> 4) & 3, t = (e >> 6) & 3;
    const int gy = (y >> 1) | (((y ^ (y >> 1)) & 1) << 1);
    w[0] = x;
    w[1] = y;
    w[2] = x ^ y ^ z;
    w[3] = x ^ gy ^ t;
  }
};

// block patterns as run-time tables: members, their labels, and the member that
// permutation n (lexicographic) of the sorted block tuple gives
template <int D>
struct K2TTab {
  signed char m[8] = {};
  signed char lab[8][24][4] = {};
  signed char mem[8][24] = {};
};
template <int D>
constexpr K2TTab<D> make_k2ttab() {
  K2TTab<D> r{};
  const Sym<D> S = make_sym<D>();
  for (int p = 0; p < npatterns(D); p++) {
    const Pattern<D> pb = make_pattern<D>(p);
    r.m[p] = (signed char)pb.m;
    for (int u = 0; u < pb.m; u++)
      for (int k = 0; k < D; k++) r.lab[p][u][k] = (signed char)pb.lab[u][k];
    for (int n = 0; n < fact(D); n++)
      for (int u = 0; u < pb.m; u++) {
        bool same = true;
        for (int k = 0; k < D; k++) same = same && pb.lab[0][S.p[n][k]] == pb.lab[u][k];
        if (same) r.mem[p][n] = (signed char)u;
      }
  }
  return r;
}
template <int D>
__device__ constexpr K2TTab<D> kK2TTab = make_k2ttab<D>();

// member u of an element orbit: permutation u (lexicographic)
template <int D>
__device__ constexpr Sym<D> kK2TSym = make_sym<D>();

// the canonical offsets of a degenerate block orbit (some block coordinates equal:
// sorted within them), packed one byte per index
template <int D, int BP>
constexpr K2List<D> make_k2tlist() {
  using K = K2TShape<D>;
  K2List<D> r{};
  const Pattern<D> pb = make_pattern<D>(BP);
  for (int e0 = 0; e0 < K::NT; e0++) {
    int w[4] = {0, 0, 0, 0};
    K::elem(e0, w);
    bool ok = true;
    for (int k = 0; k + 1 < D; k++)
      if (pb.lab[0][k] == pb.lab[0][k + 1]) ok = ok && w[k] <= w[k + 1];
    if (ok) r.e[r.n++] = (unsigned)w[0] | (unsigned)w[1] << 8 | (unsigned)w[2] << 16 | (unsigned)w[3] << 24;
  }
  return r;
}
template <int D, int BP>
__device__ constexpr K2List<D> kK2TList = make_k2tlist<D, BP>();

struct K2TStage {
  int bp;        // block pattern; -1: no more block orbits
  int lim;       // elements left in the largest coordinate's tile
  int val[4];    // distinct block coordinates
  int tb[24];    // shared-memory offset (elements) of the tile of permutation n
};

// binomial table's columns: coarse blocks + d - 1 <= 259 for extents up to 4096
constexpr int K2T_BIN = 264;

template <int D, int NST>
struct K2TShared {
  K2TStage st[NST];
  uint64_t full[NST], done[NST], empty[NST];
  alignas(16) uint4 next;      // cluster launch control's answer
  uint64_t next_bar;
  unsigned bin[D][K2T_BIN];         // C(c, k + 1)
};

// in-tile place of offset w o (permutation u)
template <int D>
__device__ __forceinline__ int k2t_lin(int u, const int (&w)[4]) {
  constexpr int SH = D == 3 ? 3 : 2;
  int a = 0;
#pragma unroll
  for (int k = 0; k < D; k++) a += w[kK2TSym<D>.p[u][k]] << (SH * k);
  return a;
}

// the strict core for a group outside the fixed-point range, out of line
template <int D>
static __device__ __noinline__ void k2t_strict_group(const KParams& kp, unsigned pk, const int* tb, double* sm) {
  constexpr int M = fact(D);
  const int w[4] = {(int)(pk & 255), (int)(pk >> 8 & 255), (int)(pk >> 16 & 255), (int)(pk >> 24)};
  double x[M];
#pragma unroll
  for (int u = 0; u < M; u++) x[u] = sm[tb[u] + k2t_lin<D>(u, w)];
  strict_core<D, 0>(kp, x);
#pragma unroll
  for (int u = 0; u < M; u++) sm[tb[u] + k2t_lin<D>(u, w)] = __dmul_rn(kp.alpha, x[u]);
}

// One element orbit, always through the operator on all d! permutations: where
// indices are equal, members coincide, each is read and written by this thread as
// often as permutations give it, and every copy gets the same value (the sums over the
// permutations are the pattern's own, term by term). A body per equality pattern, as
// in K2, made 75 KB of code for d = 4: "no instruction" was the second largest stall
// (A[112]^4 687 us; one body for all 24-member orbits 584; one for everything 563).
// GEN: of a generic block orbit, whose tile n is permutation n's.
template <int D, int AR, bool GEN, typename T>
__device__ __forceinline__ void k2t_group(const KParams& kp, unsigned pk, const int (&w)[4], const int* tb, T* sm) {
  constexpr int M = fact(D);
  auto slot = [&](int u) { return (GEN ? u * K2TShape<D>::NT : tb[u]) + k2t_lin<D>(u, w); };
  T x[M];
#pragma unroll
  for (int u = 0; u < M; u++) x[u] = sm[slot(u)];
  if constexpr (AR == AR_F32) {
    T y[M];
    apply_group<D, 0, AR_F32, T>(kp, x, y);
#pragma unroll
    for (int u = 0; u < M; u++) sm[slot(u)] = y[u];
  } else if constexpr (D == 4) {
    auto sink = [&](int u, double v, int) { sm[slot(u)] = v; };
    if (!exact_core_wht4<0>(kp, x, sink)) k2t_strict_group<D>(kp, pk, tb, sm);
  } else {
    T y[M];
    if (exact_core<D, 0>(kp, x, y)) {
      if (kp.flags & KF_ALPHA_MUL) {
#pragma unroll
        for (int u = 0; u < M; u++) y[u] = __dmul_rn(kp.alpha, y[u]);
      }
#pragma unroll
      for (int u = 0; u < M; u++) sm[slot(u)] = y[u];
    } else {
      k2t_strict_group<D>(kp, pk, tb, sm);
    }
  }
}

// the element orbits at offsets list[0..n), or (no list) at the thread's own offset pk0
template <int D, int AR, typename T>
__device__ __forceinline__ void k2t_listed(const KParams& kp, const K2TStage& st, const unsigned* list, int n, unsigned pk0,
                                           T* sm) {
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += 256) {
    const unsigned pk = list ? list[i] : pk0;
    const int w[4] = {(int)(pk & 255), (int)(pk >> 8 & 255), (int)(pk >> 16 & 255), (int)(pk >> 24)};
    if (w[D - 1] >= st.lim) continue;
    k2t_group<D, AR, false, T>(kp, pk, w, st.tb, sm);
  }
}

// the block tuple of work id `id` (see k2_next), given its group's coarse multiset v:
// distinct values val and pattern bp; false if the tuple is not sorted
template <int D>
__device__ __forceinline__ bool k2t_decode(const KParams& kp, const int (&v)[4], int64_t id, int (&val)[4], int& bp) {
  const int lf = kp.k2lf;
  const int nb = (kp.O + K2TShape<D>::BL - 1) / K2TShape<D>::BL;
  const unsigned dl = (unsigned)id & ((1u << (D * lf)) - 1u);
  int b[4] = {0, 0, 0, 0};
  bool ok = true;
#pragma unroll
  for (int k = 0; k < D; k++) {
    b[k] = ((v[k] - k) << lf) + (int)((dl >> (k * lf)) & ((1u << lf) - 1u));
    ok = ok && b[k] < nb;
  }
  unsigned eq = 0;
  int j = 0;
  val[0] = b[0];
  val[1] = val[2] = val[3] = 0;
#pragma unroll
  for (int k = 0; k + 1 < D; k++) {
    ok = ok && b[k] <= b[k + 1];
    if (b[k] == b[k + 1]) {
      eq |= 1u << k;
    } else {
      j++;
      if (j == 1) val[1] = b[k + 1];
      if (j == 2) val[2] = b[k + 1];
      if (j == 3) val[3] = b[k + 1];
    }
  }
  bp = k2_elem_pattern<D>(eq);
  return ok;
}

template <int D>
__device__ __forceinline__ void k2t_load(void* dst, const CUtensorMap* map, const int (&c)[4], uint64_t* bar) {
  if constexpr (D == 3)
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
                     smem_u32(dst)), "l"(map), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(smem_u32(bar)) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
                     smem_u32(dst)), "l"(map), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]), "r"(smem_u32(bar)) : "memory");
}
template <int D>
__device__ __forceinline__ void k2t_store(const void* src, const CUtensorMap* map, const int (&c)[4]) {
  if constexpr (D == 3)
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map), "r"(c[0]),
                 "r"(c[1]), "r"(c[2]), "r"(smem_u32(src)) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(map),
                 "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]), "r"(smem_u32(src)) : "memory");
}

// corner of tile u of a block orbit of pattern bp
template <int D>
__device__ __forceinline__ void k2t_corner(int bp, int u, const int (&val)[4], int (&c)[4]) {
#pragma unroll
  for (int k = 0; k < D; k++) {
    const int l = kK2TTab<D>.lab[bp][u][k];
    c[k] = (l == 0 ? val[0] : (l == 1 ? val[1] : (l == 2 ? val[2] : val[3]))) * K2TShape<D>::BL;
  }
}

constexpr int K2T_THREADS = 256 + 64;

template <int D, int AR, int NST, int MINB, typename T>
__global__ void __launch_bounds__(K2T_THREADS, MINB)
    k2t_kernel(const __grid_constant__ KParams kp, const __grid_constant__ CUtensorMap mapA,
               const __grid_constant__ CUtensorMap mapB) {
  using K = K2TShape<D>;
  constexpr int SE = fact(D) * K::NT;  // elements of a stage
  extern __shared__ __align__(128) unsigned char k2t_smem[];
  __shared__ K2TShared<D, NST> sh;
  T* const buf = reinterpret_cast<T*>(k2t_smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; s++) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.done[s], 8);
      mbar_init(&sh.empty[s], 1);
    }
    mbar_init(&sh.next_bar, 1);
    fence_mbar_init();
  }
  // binomials of the unranking: all of them fit 32 bits, since the grid does
  const int nc = (((kp.O + K::BL - 1) / K::BL - 1) >> kp.k2lf) + 1;
  for (int i = threadIdx.x; i < D * K2T_BIN; i += K2T_THREADS) {
    const int k = i / K2T_BIN, c = i % K2T_BIN;
    const int64_t v = k == 0 ? binom(c, 1) : (k == 1 ? binom(c, 2) : (k == 2 ? binom(c, 3) : binom(c, 4)));
    sh.bin[k][c] = v > 0xFFFFFFFFLL ? 0xFFFFFFFFu : (unsigned)v;
  }
  __syncthreads();
  const long long lim = kp.wait_limit;
  bool ok = true;  // every wait is bounded: a role whose wait runs out reports and leaves its loop
  if (warp < 8) {
    // ---- sums ----
    int w0[4];
    K::elem(threadIdx.x, w0);
    for (int k = 0;; k++) {
      const int s = k % NST;
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[s], (k / NST) & 1, lim));
      if (!ok) break;
      const K2TStage& st = sh.st[s];
      const int bp = st.bp;
      T* const sm = buf + s * SE;
      if (D == 3 && bp == 0) {
        // the generic block orbit's tile offsets as constants: a second copy of the six
        // members' code, which is small
#pragma unroll 1
        for (int e = 0; e < K::NT; e += 256) {
          const int w[4] = {w0[0], w0[1], w0[2] ^ (e >> 8) << 2, 0};  // bit 8 of the element index
          if (w[2] < st.lim)
            k2t_group<D, AR, D == 3, T>(kp, (unsigned)(w[0] | w[1] << 8 | w[2] << 16), w, st.tb, sm);
        }
      } else if (bp >= 0) {
        const unsigned* list = nullptr;
        int n = K::NT;
        if (bp == 1) { list = kK2TList<D, 1>.e; n = kK2TList<D, 1>.n; }
        if (bp == 2) { list = kK2TList<D, 2>.e; n = kK2TList<D, 2>.n; }
        if (bp == 3) { list = kK2TList<D, 3>.e; n = kK2TList<D, 3>.n; }
        if constexpr (D == 4) {
          if (bp == 4) { list = kK2TList<D, 4>.e; n = kK2TList<D, 4>.n; }
          if (bp == 5) { list = kK2TList<D, 5>.e; n = kK2TList<D, 5>.n; }
          if (bp == 6) { list = kK2TList<D, 6>.e; n = kK2TList<D, 6>.n; }
          if (bp == 7) { list = kK2TList<D, 7>.e; n = kK2TList<D, 7>.n; }
        }
        k2t_listed<D, AR, T>(kp, st, list, n, (unsigned)(w0[0] | w0[1] << 8 | w0[2] << 16 | w0[3] << 24), sm);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the TMA store reads the stage
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.done[s]);
      if (bp < 0) break;
    }
  } else if (warp == 8) {
    // ---- block orbits and loads ----
    auto ask = [&] {
      if (lane == 0) {
        mbar_arrive_expect_tx(&sh.next_bar, 16);
        asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(
                         smem_u32(&sh.next)), "r"(smem_u32(&sh.next_bar)) : "memory");
      }
    };
    int64_t id = blockIdx.x;
    int k = 0;
    unsigned ph = 0;
    for (;;) {
      ask();  // the next id, while this one is worked on
      // colex unranking by the warp: 32 candidates at a time (see unrank_warp)
      int v[4] = {0, 0, 0, 0};
      unsigned r = (unsigned)(id >> (D * kp.k2lf));
#pragma unroll
      for (int i = D - 1; i >= 0; i--) {
        int cnt = 0;
        for (int c0 = i; c0 < nc + D - 1; c0 += 32) {
          const int c = c0 + lane;
          const unsigned m = __ballot_sync(0xffffffffu, c < nc + D - 1 && sh.bin[i][c] <= r);
          cnt += __popc(m);
          if (m != 0xffffffffu) break;
        }
        v[i] = i + cnt - 1;
        r -= sh.bin[i][v[i]];
      }
      int val[4], bp;
      if (k2t_decode<D>(kp, v, id, val, bp)) {
        const int s = k % NST;
        ok = __all_sync(0xffffffffu, k < NST || mbar_wait(&sh.empty[s], (k / NST - 1) & 1, lim));
        if (ok) {
          const int m = kK2TTab<D>.m[bp];
          K2TStage& st = sh.st[s];
          if (lane < fact(D)) st.tb[lane] = kK2TTab<D>.mem[bp][lane] * K::NT;
          if (lane < 4) st.val[lane] = lane == 0 ? val[0] : (lane == 1 ? val[1] : (lane == 2 ? val[2] : val[3]));
          if (lane == 0) {
            const int l = kK2TTab<D>.lab[bp][0][D - 1];
            st.bp = bp;
            st.lim = kp.O - (l == 0 ? val[0] : (l == 1 ? val[1] : (l == 2 ? val[2] : val[3]))) * K::BL;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive_expect_tx(&sh.full[s], (uint32_t)(m * K::NT * sizeof(T)));
          __syncwarp();
          if (lane < m) {
            int c[4] = {0, 0, 0, 0};
            k2t_corner<D>(bp, lane, val, c);
            k2t_load<D>(buf + s * SE + lane * K::NT, &mapA, c, &sh.full[s]);
          }
            k++;
        }
      }
      // the answer is always waited for, so that none is in flight at the end, also where the
      // wait ran out (the block it may have taken over is then lost, and the call reported)
      if (!__all_sync(0xffffffffu, mbar_wait(&sh.next_bar, ph, lim))) {
        mbar_wait(&sh.next_bar, ph, kDrainLimit);
        ok = false;
        break;
      }
      ph ^= 1;
      unsigned got = 0, x = 0;
      asm volatile(
          "{\n\t.reg .b128 r;\n\t.reg .pred p;\n\t"
          "ld.shared.b128 r, [%2];\n\t"
          "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t"
          "mov.u32 %1, 0;\n\t"
          "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, r;\n\t}"
          : "=r"(got), "=r"(x)
          : "r"(smem_u32(&sh.next))
          : "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the next answer overwrites this one
      __syncwarp();
      if (!got || !ok) break;
      id = x;
    }
    if (ok) {  // the end mark
      const int s = k % NST;
      ok = __all_sync(0xffffffffu, k < NST || mbar_wait(&sh.empty[s], (k / NST - 1) & 1, lim));
      if (ok && lane == 0) {
        sh.st[s].bp = -1;
        mbar_arrive(&sh.full[s]);
      }
    }
    if (!ok) {
      // loads in flight land before the CTA's shared memory is given up
      for (int j = k > NST ? k - NST : 0; j < k; j++) mbar_wait(&sh.full[j % NST], (j / NST) & 1, kDrainLimit);
    }
  } else {
    // ---- stores ----
    for (int k = 0;; k++) {
      const int s = k % NST;
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.done[s], (k / NST) & 1, lim));
      if (!ok) break;
      const K2TStage& st = sh.st[s];
      const int bp = st.bp;
      if (bp < 0) break;
      if (lane < kK2TTab<D>.m[bp]) {
        const int val[4] = {st.val[0], st.val[1], st.val[2], st.val[3]};
        int c[4] = {0, 0, 0, 0};
        k2t_corner<D>(bp, lane, val, c);
        k2t_store<D>(buf + s * SE + lane * K::NT, &mapB, c);
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the stage has been read
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.empty[s]);
    }
  }
  if (!ok) report_timeout(kp);
}

// cuTensorMapEncodeTiled, from the driver at run time (the library links the CUDA runtime only)
typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiled encode_tiled() {
  static const EncodeTiled f = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return (EncodeTiled) nullptr;
    }
    return (EncodeTiled)p;
  }();
  return f;
}

// tile boxes of the N^D tensor at p with element strides ld (ld[0] = 1)
template <int D, typename T>
bool k2t_map(CUtensorMap* map, const void* p, const int64_t* ld, int64_t N) {
  const EncodeTiled f = encode_tiled();
  if (!f || (uintptr_t)p % 16 != 0) return false;
  cuuint64_t dims[4], strides[4];
  cuuint32_t box[4], one[4];
  for (int k = 0; k < D; k++) {
    dims[k] = (cuuint64_t)N;
    box[k] = K2TShape<D>::BL;
    one[k] = 1;
    if (k > 0) {
      const int64_t b = ld[k] * (int64_t)sizeof(T);
      // TMA's rules; and rows that do not overlap (a broadcast input stays with K2)
      if (b % 16 != 0 || b >= (1LL << 40) || ld[k] < N) return false;
      strides[k - 1] = (cuuint64_t)b;
    }
  }
  return f(map, sizeof(T) == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, D, const_cast<void*>(p),
           dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// true (and *e the launch status) when K2T takes the problem
template <int D, int AR, int NST, int MINB, typename T>
bool launch_k2t(const KParams& kp, cudaStream_t st, cudaError_t* e) {
  if (kp.flags & (KF_BETA | KF_HOST)) return false;
  CUtensorMap ma, mb;
  if (!k2t_map<D, T>(&ma, kp.A, kp.lda, kp.O) || !k2t_map<D, T>(&mb, kp.B, kp.ldb, kp.O)) return false;
  auto fn = k2t_kernel<D, AR, NST, MINB, T>;
  constexpr int smem = NST * fact(D) * K2TShape<D>::NT * (int)sizeof(T);
  static DeviceCache cache;  // 1 once the kernel's attributes are set on a device
  int dev = 0;
  *e = cudaGetDevice(&dev);
  if (*e != cudaSuccess) return true;
  long long v = 0;
  const int rc = cache.get(dev, &v, [&](long long* val) {
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err == cudaSuccess) err = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    *val = 1;
    return (int)err;
  });
  if (rc != 0) {
    *e = rc < 0 ? cudaErrorInvalidDevice : (cudaError_t)rc;
    return true;
  }
  fn<<<(unsigned)kp.pre[npatterns(D)], K2T_THREADS, smem, st>>>(kp, ma, mb);
  *e = cudaGetLastError();
  return true;
}

}  // namespace ss
