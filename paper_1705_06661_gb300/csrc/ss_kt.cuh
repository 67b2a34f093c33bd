#pragma once
// KT: the summation fused into a contraction, on the tensor cores.
//
//   C[s, y] = sum_t S(A)[s, t] * W[y, t]       (ss_contract.cuh's SUM = true)
//
// The FP64 form (KC) is bound by the FP64 pipe: 2 multiply-adds per SM and
// clock, 25.7 ms for A[48^3,16^3] and 32 columns, 48 times the time of reading
// A. Here both factors are split into 8-bit digits and the products run as
// FP16 matrix instructions (tcgen05), whose FP32 sums of small integers are
// exact: the splitting of Ozaki, Ogita, Oishi and Rump ("Error-free
// transformations of matrix multiplication", Numer. Algorithms 59, 2012).
//
// - The tuples t are taken in chunks of 144. Per chunk, a row s of S(A) and a
//   column y of W each get one power-of-two scale (from the largest |A| resp. |W|
//   of the chunk) and become 55-bit signed integers v = sum_i d_i 256^(6-i),
//   i = 0..6, -128 <= d_i <= 127. The orbit operator runs on the integers of A
//   (two limbs of 24 and up to 26 bits, 32-bit multiply-adds): S(A) is exact on
//   the grid 2^(E + 1 - bits), bits = 54 - log2 sum|a|.
// - D_d = sum over t and i + j = d of d_i(A) d_j(W), d = 0..6: at most
//   7 * 144 products of magnitude at most 2^14, below 2^24, so exact in FP32.
//   Digit pairs with i + j > 6 lie below 2^-56 of the largest product and are left
//   out, as FP64 would round them off.
// - Per chunk the D_d are joined in 64-bit integers (sum d <= 5 of
//   D_d 256^(5-d), and D_6 rounded to D_5's unit), scaled, rounded once to FP64 and
//   added to the FP64 sum of the chunks.
// - A tile whose chunk scales leave a safe exponent range (infinities, NaN,
//   magnitudes beyond 2^+-440) is recomputed in FP64 by its epilogue warps.
//
// A CTA owns 128 rows x 32 columns. Warps 0-7 find the scales (a first read of
// the chunk's A, which also brings it into L2), sum the orbits and write the digits;
// one thread issues the matrix instructions; warps 8-11 join the sums; one warp
// finds the chunks' tuples. Digit i of A meets digits 0..6-i of W, which lie
// side by side as one N = 32 (7 - i) operand, so each digit of A is read once from
// shared memory per step and its products land in the accumulators i..6: 7
// instructions per 16 tuples instead of 28.
#include "ss_contract.cuh"
#include "ss_devcache.h"
#include "ss_tma.cuh"

#include <cuda_fp16.h>

namespace ss {

constexpr int KT_ROWS = 128, KT_COLS = 32, KT_ND = 7;
constexpr int KT_UNIT = 24;                       // tuples of a unit: 24 / m orbits of one pattern
constexpr int KT_UPC = 6;                         // units of a chunk
constexpr int KT_CHUNK = KT_UNIT * KT_UPC;        // 144 tuples
constexpr int KT_PROD = 256;                      // producer threads: two per row
constexpr int KT_THREADS = KT_PROD + 128 + 64;    // + epilogue + (matrix, table) warps
// operand layout (K-major, no swizzle): 8 tuples x 8 rows as 128 contiguous bytes
constexpr int KT_AKG = KT_ROWS * 16;              // bytes of 8 tuples of one digit of A
constexpr int KT_AD = 6 * KT_AKG;                 // bytes of one digit of A: a stage's two units
constexpr int KT_WKG = KT_ND * KT_COLS * 16;      // bytes of 8 tuples of all digits of W
constexpr int KT_STAGE = KT_ND * KT_AD + 6 * KT_WKG;
constexpr unsigned KT_ELO = (1023u - 440u) << 20, KT_EHI = (1023u + 440u) << 20;

struct KtArgs {
  const double* W;
  double* C;
  int64_t Y, ldw, ldc;
  int64_t tiles;       // row tiles x column tiles
  int ytiles;
  int nchunk;
  int upre[9];         // unit prefix per pattern
  int bits;            // |A| < 2^bits on its grid
  int sh0;             // exponent of a joined sum's unit, less the two scales' exponents
  int opow[4];
};

struct KtShared {
  unsigned rowmax[2][KT_ROWS];
  // chunk scales by chunk mod 8: producers run at most two chunks ahead of the
  // matrix warp, and that at most two ahead of the epilogue
  unsigned rowexp[8][KT_ROWS];   // exponent fields
  unsigned colmax[8][KT_COLS];   // high words of the largest |W|
  int tix[2][KT_CHUNK];          // tuple indices of a chunk, -1: none
  int pat[2][KT_UPC];            // pattern of each unit, -1: none
  int bad[8];                    // by tile mod 8: a scale is out of range
  uint64_t tab_full[2], tab_empty[2], st_full[2], st_empty[2], acc_full[2], acc_empty[2], drain;
  uint32_t tmem;
};

__device__ __forceinline__ void kt_proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void kt_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint64_t kt_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)(lbo >> 4) << 16 | (uint64_t)(sbo >> 4) << 32 | 1ull << 46;
}
__device__ __forceinline__ void kt_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"((unsigned)acc)
      : "memory");
}
__device__ __forceinline__ void kt_ld8(uint32_t addr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
}
// barrier `id` over n threads; true if `ok` holds in all of them (threads whose
// bounded wait ran out leave together with the others)
template <int ID, int N>
__device__ __forceinline__ bool kt_sync(bool ok) {
  unsigned r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((unsigned)ok), "n"(ID), "n"(N)
      : "memory");
  return r != 0;
}

// |x| on the grid of the scale: 2^(bits) mantissa positions below the scale's
// next power of two, truncated; signed
__device__ __forceinline__ long long kt_fixed(double x, unsigned base, int up) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned k = (base - (hi & 0x7FFFFFFFu)) >> 20;
  const unsigned long long mant = (((unsigned long long)((hi & 0x000FFFFFu) | 0x00100000u) << 32) | lo) << up;
  const long long q = (long long)shr64(mant, k);
  return (int)hi < 0 ? -q : q;
}

// limbs y1 2^24 + y0 -> the biased digits: byte 3..0 of z1, then byte 2..0 of z0, each digit + 128
__device__ __forceinline__ void kt_digits(int y0, int y1, unsigned& z0, unsigned& z1) {
  const int t = y0 + 0x808080;
  z0 = (unsigned)t;
  z1 = (unsigned)y1 + (unsigned)(t >> 24) + 0x80808080u;
}

// one digit of two tuples as FP16: the byte behind the exponent of 1024, less 1024 + 128
template <int B>
__device__ __forceinline__ unsigned kt_pair(unsigned a, unsigned b) {
  const unsigned w = (__byte_perm(a, b, B | B << 4 | (4 + B) << 8 | (4 + B) << 12) & 0x00FF00FFu) | 0x64006400u;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<const unsigned*>(&h);
}
template <int B>
__device__ __forceinline__ uint4 kt_pack(const unsigned* z) {
  return make_uint4(kt_pair<B>(z[0], z[1]), kt_pair<B>(z[2], z[3]), kt_pair<B>(z[4], z[5]), kt_pair<B>(z[6], z[7]));
}
// the seven digits of 8 tuples of one row: dst + digit * stride
__device__ __forceinline__ void kt_store8(unsigned char* dst, int stride, const unsigned* z0, const unsigned* z1) {
  *reinterpret_cast<uint4*>(dst) = kt_pack<3>(z1);
  *reinterpret_cast<uint4*>(dst + stride) = kt_pack<2>(z1);
  *reinterpret_cast<uint4*>(dst + 2 * stride) = kt_pack<1>(z1);
  *reinterpret_cast<uint4*>(dst + 3 * stride) = kt_pack<0>(z1);
  *reinterpret_cast<uint4*>(dst + 4 * stride) = kt_pack<2>(z0);
  *reinterpret_cast<uint4*>(dst + 5 * stride) = kt_pack<1>(z0);
  *reinterpret_cast<uint4*>(dst + 6 * stride) = kt_pack<0>(z0);
}

// one unit (24 tuples of pattern P) of one row: loads, orbit operator, digits
template <int D, int P>
__device__ __forceinline__ void kt_unit(const KParams& kp, const KtArgs& ka, const double* As, bool act, const int* tix,
                                        unsigned base, unsigned char* dst) {
  constexpr int M = Pat<D, P>::M, NO = KT_UNIT / M;
  double x[KT_UNIT];
#pragma unroll
  for (int e = 0; e < KT_UNIT; e++) {
    const int t = tix[e];
    x[e] = act && t >= 0 ? As[(int64_t)t * kp.S] : 0.0;
  }
  unsigned z0[KT_UNIT], z1[KT_UNIT];
#pragma unroll
  for (int o = 0; o < NO; o++) {
    int l0[M], l1[M], y0[M], y1[M];
#pragma unroll
    for (int v = 0; v < M; v++) {
      const long long X = kt_fixed(x[o * M + v], base, 0);
      l0[v] = (int)((unsigned)X & 0xFFFFFFu);
      l1[v] = (int)(X >> 24);
    }
    if constexpr (P == 0) {
#pragma unroll
      for (int st = 0; st < (D == 4 ? 1 : MAXSTAGE_EXACT); st++) {
        if (D < 4 && st >= kp.nci) break;
#pragma unroll
        for (int u = 0; u < M; u++) { y0[u] = 0; y1[u] = 0; }
#pragma unroll
        for (int s = 0; s < fact(D); s++) {
          const int c = kp.ci[st][s];
          if (c != 0) {
#pragma unroll
            for (int u = 0; u < M; u++) {
              y0[u] += c * l0[Pat<D, P>::idx(u, s)];
              y1[u] += c * l1[Pat<D, P>::idx(u, s)];
            }
          }
        }
        if (D < 4) {
#pragma unroll
          for (int u = 0; u < M; u++) { l0[u] = y0[u]; l1[u] = y1[u]; }
        }
      }
      if constexpr (D < 4) {
#pragma unroll
        for (int u = 0; u < M; u++) { y0[u] = l0[u]; y1[u] = l1[u]; }
      }
    } else {
      const int* mp = kp.mp + mp_offset<D>(P);
#pragma unroll
      for (int u = 0; u < M; u++) {
        y0[u] = 0;
        y1[u] = 0;
#pragma unroll
        for (int v = 0; v < M; v++) {
          y0[u] += mp[u * M + v] * l0[v];
          y1[u] += mp[u * M + v] * l1[v];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < M; u++) kt_digits(y0[u], y1[u], z0[o * M + u], z1[o * M + u]);
  }
#pragma unroll
  for (int g = 0; g < 3; g++) kt_store8(dst + g * KT_AKG, KT_AD, z0 + 8 * g, z1 + 8 * g);
}

template <int D>
__device__ __forceinline__ void kt_unit_any(const KParams& kp, const KtArgs& ka, int p, const double* As, bool act,
                                            const int* tix, unsigned base, unsigned char* dst) {
  switch (p) {
    case 0: kt_unit<D, 0>(kp, ka, As, act, tix, base, dst); break;
    case 1: kt_unit<D, 1>(kp, ka, As, act, tix, base, dst); break;
    case 2: if constexpr (npatterns(D) > 2) kt_unit<D, 2>(kp, ka, As, act, tix, base, dst); break;
    case 3: if constexpr (npatterns(D) > 3) kt_unit<D, 3>(kp, ka, As, act, tix, base, dst); break;
    case 4: if constexpr (npatterns(D) > 4) kt_unit<D, 4>(kp, ka, As, act, tix, base, dst); break;
    case 5: if constexpr (npatterns(D) > 4) kt_unit<D, 5>(kp, ka, As, act, tix, base, dst); break;
    case 6: if constexpr (npatterns(D) > 4) kt_unit<D, 6>(kp, ka, As, act, tix, base, dst); break;
    case 7: if constexpr (npatterns(D) > 4) kt_unit<D, 7>(kp, ka, As, act, tix, base, dst); break;
    default:  // no tuples left: digits of zero
      const unsigned z[8] = {0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u};
      for (int g = 0; g < 3; g++) kt_store8(dst + g * KT_AKG, KT_AD, z, z);
  }
}

// the orbit `rank` of pattern P into its unit's entries tix[0..m)
template <int D, int P>
__device__ __forceinline__ void kt_orbit(const KParams& kp, const KtArgs& ka, int64_t rank, int* tix) {
  constexpr int M = Pat<D, P>::M;
  int v[4] = {0, 0, 0, 0};
  const bool ok = rank < kp.norb[P];
  if (ok) unrank<Pat<D, P>::ND>(rank, kp.O, v);
#pragma unroll
  for (int u = 0; u < M; u++) {
    int t = 0;
#pragma unroll
    for (int k = 0; k < D; k++) t += v[Pat<D, P>::lab(u, k)] * ka.opow[k];
    tix[u] = ok ? t : -1;
  }
}

// members of pattern p (0 < p < npatterns), for the unit geometry
template <int D>
__device__ __forceinline__ int kt_members(int p) {
  if constexpr (D == 2) return p == 0 ? 2 : 1;
  else if constexpr (D == 3) return p == 0 ? 6 : (p == 3 ? 1 : 3);
  else return p == 0 ? 24 : (p <= 3 ? 12 : (p == 4 ? 6 : (p == 7 ? 1 : 4)));
}

// FP64 form of one tile (rare): a thread per row, KC's loop over the orbits
template <int D>
static __device__ __noinline__ void kt_tile_fp64(const KParams& kp, const KtArgs& ka, int64_t s, int64_t y0, int ny) {
  const bool act = s < kp.S;
  for (int yb = 0; yb < ny; yb += 4) {
    const int n = min(4, ny - yb);
    const double* Wt = ka.W + y0 + yb;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    kc_pattern<D, 0, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
    kc_pattern<D, 1, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
    if constexpr (D >= 3) {
      kc_pattern<D, 2, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
      kc_pattern<D, 3, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
    }
    if constexpr (D == 4) {
      kc_pattern<D, 4, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
      kc_pattern<D, 5, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
      kc_pattern<D, 6, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
      kc_pattern<D, 7, AR_EXACT, 4, true>(kp, Wt, ka.ldw, n, s, act, acc);
    }
    if (act)
      for (int j = 0; j < n; j++) ka.C[s + ka.ldc * (y0 + yb + j)] = acc[j];
  }
}

// FP64 value of Y * 2^sh, rounded once to nearest: the two 32-bit halves as
// FP64 numbers with offsets 2^84 and 2^52 (times 2^sh)
__device__ __forceinline__ double kt_to_double(long long Y, int sh) {
  const int s = (int)((unsigned)sh << 20);
  const double h = __hiloint2double(0x45300000 + s, (int)((unsigned)(Y >> 32) ^ 0x80000000u));
  const double c = __hiloint2double(0x45300000 + s, (int)0x80100000u);  // 2^84 + 2^63 + 2^52
  const double l = __hiloint2double(0x43300000 + s, (int)(unsigned)Y);
  return __dadd_rn(__dsub_rn(h, c), l);
}

template <int D>
__global__ void __launch_bounds__(KT_THREADS, 1) kt_kernel(const __grid_constant__ KParams kp, const __grid_constant__ KtArgs ka) {
  extern __shared__ __align__(128) unsigned char kt_smem[];
  __shared__ KtShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < 2; i++) {
      mbar_init(&sh.tab_full[i], 32);
      mbar_init(&sh.tab_empty[i], KT_PROD);
      mbar_init(&sh.st_full[i], KT_PROD);
      mbar_init(&sh.st_empty[i], 1);
      mbar_init(&sh.acc_full[i], 1);
      mbar_init(&sh.acc_empty[i], 128);
    }
    mbar_init(&sh.drain, 1);
    fence_mbar_init();
  }
  if (tid < KT_COLS)
    for (int i = 0; i < 8; i++) sh.colmax[i][tid] = 0;
  if (tid < 8) sh.bad[tid] = 0;
  if (warp == 12) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sh.tmem)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh.tmem;
  const int nunit = ka.upre[npatterns(D)];
  auto stages_of = [&](int ch) { return (min(KT_UPC, nunit - ch * KT_UPC) + 1) / 2; };
  const long long lim = kp.wait_limit;
  bool ok = true;  // every wait is bounded: a role whose wait runs out reports and leaves its loop

  if (warp < 8) {
    // ---- producers: scales, orbit sums, digits ----
    const int row = tid & (KT_ROWS - 1), half = tid >> 7;
    int c = 0, n = 0, it = 0;  // chunks, stages and tiles so far
    for (int64_t tile = blockIdx.x; tile < ka.tiles; tile += gridDim.x, it++) {
      const int64_t s = tile / ka.ytiles * KT_ROWS + row, y0 = tile % ka.ytiles * KT_COLS;
      const int ny = (int)min((int64_t)KT_COLS, ka.Y - y0);
      const bool act = s < kp.S;
      const double* As = static_cast<const double*>(kp.A) + s;
      const double* Wy = ka.W + y0 + (tid & 31);
      const bool wact = (tid & 31) < ny;
      for (int ch = 0; ch < ka.nchunk; ch++, c++) {
        const int* tix = sh.tix[c & 1];
        ok = kt_sync<1, KT_PROD>(ok && mbar_wait(&sh.tab_full[c & 1], (c >> 1) & 1, lim));
        if (!ok) break;
        // scales: the largest |A| of the row and |W| of the column in this chunk
        unsigned mx = 0, low = 0, wmx = 0, wlow = 0;
#pragma unroll 1
        for (int j = 0; j < 3; j++) {
          const int* te = tix + (2 * j + half) * KT_UNIT;
          double v[KT_UNIT];
#pragma unroll
          for (int e = 0; e < KT_UNIT; e++) {
            const int t = te[e];
            v[e] = act && t >= 0 ? As[(int64_t)t * kp.S] : 0.0;
          }
#pragma unroll
          for (int e = 0; e < KT_UNIT; e++) {
            mx = max(mx, (unsigned)__double2hiint(v[e]) & 0x7FFFFFFFu);
            low |= (unsigned)__double2loint(v[e]);
          }
        }
#pragma unroll
        for (int j = 0; j < KT_CHUNK / 8; j++) {
          const int t = tix[(tid >> 5) + 8 * j];
          const double v = wact && t >= 0 ? Wy[(int64_t)t * ka.ldw] : 0.0;
          wmx = max(wmx, (unsigned)__double2hiint(v) & 0x7FFFFFFFu);
          wlow |= (unsigned)__double2loint(v);
        }
        if (wmx == 0 && wlow != 0) wmx = 1;  // subnormal only: out of range below
        if (mx == 0 && low != 0) mx = 1;
        sh.rowmax[half][row] = mx;
        atomicMax(&sh.colmax[c & 7][tid & 31], wmx);
        kt_sync<1, KT_PROD>(true);
        mx = max(sh.rowmax[0][row], sh.rowmax[1][row]);
        wmx = sh.colmax[c & 7][tid & 31];
        auto scale = [&](unsigned m) {
          unsigned E = m & 0x7FF00000u;
          if (E < KT_ELO || E > KT_EHI) {
            if (m != 0) sh.bad[it & 7] = 1;
            E = KT_ELO;
          }
          return E;
        };
        const unsigned E = scale(mx), Ew = scale(wmx);
        if (half == 0) sh.rowexp[c & 7][row] = E;
        if (tid < 32) sh.colmax[(c + 2) & 7][tid] = 0;  // of chunk c - 6
        // largest |A| below 2^bits, largest |W| below 2^54
        const unsigned base = (E | 0xFFFFFu) + ((unsigned)(53 - ka.bits) << 20);
        const unsigned wbase = Ew | 0xFFFFFu;
        const int ns = stages_of(ch);
        for (int j = 0; ok && j < ns; j++, n++) {
          unsigned char* st = kt_smem + (n & 1) * KT_STAGE;
          ok = mbar_wait(&sh.st_empty[n & 1], ((n >> 1) & 1) ^ 1, lim);
          if (!ok) break;  // all leave at the next chunk's barrier
          const int u = 2 * j + half;
          kt_unit_any<D>(kp, ka, sh.pat[c & 1][u], As, act, tix + u * KT_UNIT, base,
                         st + half * 3 * KT_AKG + row * 16);
          if (tid < 6 * 32) {
            const int kg = tid >> 5;
            unsigned z0[8], z1[8];
            double w[8];
#pragma unroll
            for (int e = 0; e < 8; e++) {
              const int t = tix[2 * j * KT_UNIT + kg * 8 + e];
              w[e] = wact && t >= 0 ? Wy[(int64_t)t * ka.ldw] : 0.0;
            }
#pragma unroll
            for (int e = 0; e < 8; e++) {
              const long long X = kt_fixed(w[e], wbase, 1);
              kt_digits((int)((unsigned)X & 0xFFFFFFu), (int)(X >> 24), z0[e], z1[e]);
            }
            kt_store8(st + KT_ND * KT_AD + kg * KT_WKG + (tid & 31) * 16, KT_COLS * 16, z0, z1);
          }
          kt_proxy_fence();
          mbar_arrive(&sh.st_full[n & 1]);
        }
        mbar_arrive(&sh.tab_empty[c & 1]);
      }
      if (!kt_sync<1, KT_PROD>(ok)) { ok = false; break; }
    }
  } else if (warp < 12) {
    // ---- epilogue: join the digit sums of a chunk, add up the chunks ----
    const int row = tid - KT_PROD;
    const uint32_t lanes = (uint32_t)(warp & 3) << 21;  // TMEM lane 32 (warp mod 4)
    int c = 0, it = 0;
    for (int64_t tile = blockIdx.x; ok && tile < ka.tiles; tile += gridDim.x, it++) {
      const int64_t s = tile / ka.ytiles * KT_ROWS + row, y0 = tile % ka.ytiles * KT_COLS;
      const int ny = (int)min((int64_t)KT_COLS, ka.Y - y0);
      double acc[KT_COLS];
#pragma unroll
      for (int y = 0; y < KT_COLS; y++) acc[y] = 0.0;
      for (int ch = 0; ch < ka.nchunk; ch++, c++) {
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc_full[c & 1], (c >> 1) & 1, lim));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int er = (int)(sh.rowexp[c & 7][row] >> 20) + ka.sh0;
        const uint32_t t0 = tmem + (uint32_t)(c & 1) * 256 + lanes;
#pragma unroll
        for (int yb = 0; yb < KT_COLS; yb += 8) {
          uint32_t d[KT_ND][8];
#pragma unroll
          for (int i = 0; i < KT_ND; i++) kt_ld8(t0 + i * KT_COLS + yb, d[i]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int y = 0; y < 8; y++) {
            int v[KT_ND];
#pragma unroll
            for (int i = 0; i < KT_ND; i++) v[i] = __float2int_rn(__uint_as_float(d[i][y]));
            // |D_0| <= 2^20.2, |D_1| <= 2^22.2, |D_d| < 2^24: the joined sum stays below 2^61
            long long V = (long long)((unsigned long long)(unsigned)(v[0] * 256 + v[1]) << 32);
            V += (long long)v[2] * (1 << 24) + (long long)v[3] * (1 << 16);
            V += (long long)v[4] * 256 + (long long)(v[5] + ((v[6] + 128) >> 8));
            acc[yb + y] += kt_to_double(V, er + (int)(max(sh.colmax[c & 7][yb + y], KT_ELO) >> 20));
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(&sh.acc_empty[c & 1]);
      }
      ok = kt_sync<2, 128>(ok);
      if (!ok) break;
      const int bad = sh.bad[it & 7];
      kt_sync<2, 128>(true);
      if (bad) {
        if (row == 0) sh.bad[it & 7] = 0;
        kt_tile_fp64<D>(kp, ka, s, y0, ny);
      } else if (s < kp.S) {
#pragma unroll
        for (int y = 0; y < KT_COLS; y++)
          if (y < ny) ka.C[s + ka.ldc * (y0 + y)] = acc[y];
      }
    }
  } else if (warp == 12) {
    // ---- matrix instructions, by one thread ----
    if (lane == 0) {
      const uint32_t sbase = smem_u32(kt_smem);
      int c = 0, n = 0;
      for (int64_t tile = blockIdx.x; ok && tile < ka.tiles; tile += gridDim.x)
        for (int ch = 0; ok && ch < ka.nchunk; ch++, c++) {
          if (!mbar_wait(&sh.acc_empty[c & 1], ((c >> 1) & 1) ^ 1, lim)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t acc = tmem + (uint32_t)(c & 1) * 256;
          const int ns = stages_of(ch);
          for (int j = 0; j < ns; j++, n++) {
            if (!mbar_wait(&sh.st_full[n & 1], (n >> 1) & 1, lim)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sa = sbase + (n & 1) * KT_STAGE, sw = sa + KT_ND * KT_AD;
            for (int ks = 0; ks < 3; ks++)
#pragma unroll
              for (int i = 0; i < KT_ND; i++) {
                // FP16 x FP16 -> FP32, K-major operands, M = 128, N = 32 (7 - i)
                const uint32_t idesc = 1u << 4 | (uint32_t)(KT_COLS * (KT_ND - i) / 8) << 17 | (uint32_t)(KT_ROWS / 16) << 24;
                kt_mma(acc + i * KT_COLS, kt_desc(sa + i * KT_AD + ks * 2 * KT_AKG, KT_AKG, 128),
                       kt_desc(sw + ks * 2 * KT_WKG, KT_WKG, 128), idesc, j + ks + i > 0);
              }
            kt_commit(&sh.st_empty[n & 1]);
          }
          if (ok) kt_commit(&sh.acc_full[c & 1]);
        }
      // no matrix instruction is in flight when the accumulators are given back
      kt_commit(&sh.drain);
      ok = mbar_wait(&sh.drain, 0, lim) && ok;
    }
    __syncwarp();
  } else {
    // ---- the chunks' tuples ----
    int c = 0;
    for (int64_t tile = blockIdx.x; ok && tile < ka.tiles; tile += gridDim.x)
      for (int ch = 0; ok && ch < ka.nchunk; ch++, c++) {
        if (!mbar_wait(&sh.tab_empty[c & 1], ((c >> 1) & 1) ^ 1, lim)) { ok = false; break; }
        int p[KT_UPC], mo = 1;
#pragma unroll
        for (int u = 0; u < KT_UPC; u++) {
          const int g = ch * KT_UPC + u;
          p[u] = -1;
          if (g < nunit) {
            p[u] = 0;
#pragma unroll
            for (int q = 1; q < npatterns(D); q++)
              if (g >= ka.upre[q]) p[u] = q;
            mo = max(mo, KT_UNIT / kt_members<D>(p[u]));
          }
          if (lane == 0) sh.pat[c & 1][u] = p[u];
        }
        for (int q = lane; q < KT_UPC * mo; q += 32) {
          const int u = q % KT_UPC, o = q / KT_UPC, g = ch * KT_UPC + u;
          if (g >= nunit) {
            if (o == 0)
              for (int e = 0; e < KT_UNIT; e++) sh.tix[c & 1][u * KT_UNIT + e] = -1;
            continue;
          }
          int pp = 0;
#pragma unroll
          for (int r = 1; r < npatterns(D); r++)
            if (g >= ka.upre[r]) pp = r;
          const int m = kt_members<D>(pp), no = KT_UNIT / m;
          if (o >= no) continue;
          const int64_t rank = (int64_t)(g - ka.upre[pp]) * no + o;
          int* dst = sh.tix[c & 1] + u * KT_UNIT + o * m;
          switch (pp) {
            case 0: kt_orbit<D, 0>(kp, ka, rank, dst); break;
            case 1: kt_orbit<D, 1>(kp, ka, rank, dst); break;
            case 2: if constexpr (npatterns(D) > 2) kt_orbit<D, 2>(kp, ka, rank, dst); break;
            case 3: if constexpr (npatterns(D) > 3) kt_orbit<D, 3>(kp, ka, rank, dst); break;
            case 4: if constexpr (npatterns(D) > 4) kt_orbit<D, 4>(kp, ka, rank, dst); break;
            case 5: if constexpr (npatterns(D) > 4) kt_orbit<D, 5>(kp, ka, rank, dst); break;
            case 6: if constexpr (npatterns(D) > 4) kt_orbit<D, 6>(kp, ka, rank, dst); break;
            case 7: if constexpr (npatterns(D) > 4) kt_orbit<D, 7>(kp, ka, rank, dst); break;
          }
        }
        mbar_arrive(&sh.tab_full[c & 1]);
      }
  }
  if (!ok) report_timeout(kp);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 12) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// Whether KT takes the contraction: exact arithmetic with integer coefficients
// (the operator's 1-norm is then at most 127, so the limb sums stay below 2^31),
// and at least four row tiles. Smaller calls stay with KC, whose FP64 sums equal
// those of the summation followed by the contraction alone bit for bit.
template <int D>
bool launch_kt(const KParams& kp, const double* W, int64_t Y, int64_t ldw, double* C, int64_t ldc, cudaStream_t st,
               cudaError_t* e) {
  double L = 1;
  for (int q = 0; q < kp.nci; q++) {
    double n = 0;
    for (int s = 0; s < fact(D); s++) n += kp.ci[q][s] < 0 ? -kp.ci[q][s] : kp.ci[q][s];
    L *= n;
  }
  int64_t T = 1;
  for (int k = 0; k < D; k++) T *= kp.O;
  if (T < 1 || T > 0x7FFFFFFF || kp.S < 4 * KT_ROWS || (kp.flags & KF_ALPHA_MUL) || L > 127) return false;
  int lg = 0;
  while ((double)(1 << lg) < L) lg++;
  KtArgs ka{};
  ka.W = W;
  ka.C = C;
  ka.Y = Y;
  ka.ldw = ldw;
  ka.ldc = ldc;
  ka.ytiles = (int)((Y + KT_COLS - 1) / KT_COLS);
  ka.tiles = (kp.S + KT_ROWS - 1) / KT_ROWS * ka.ytiles;
  ka.bits = lg > 0 ? 54 - lg : 53;  // the 53 bits of an FP64 mantissa are enough
  // kp.cexp = (53 - 2 W + kdrop + aexp) << 20 + 0x80000, aexp = the coefficients' scale;
  // a joined sum counts 2^56 of the products' units 2^(E_A + 1 - bits + aexp) 2^(E_W - 53)
  const int aexp = ((kp.cexp - 0x80000) >> 20) - 53 + 2 * kp.W - kp.kdrop;
  ka.sh0 = 56 + 1 - ka.bits + aexp - 53 - 2 * 1023;
  if (aexp < -50 || aexp > 50) return false;
  int64_t units = 0;
  const int m3[4] = {6, 3, 3, 1}, m4[8] = {24, 12, 12, 12, 6, 4, 4, 1}, m2[2] = {2, 1};
  for (int p = 0; p < npatterns(D); p++) {
    const int per = KT_UNIT / (D == 2 ? m2[p] : (D == 3 ? m3[p] : m4[p]));
    ka.upre[p] = (int)units;
    units += (kp.norb[p] + per - 1) / per;
  }
  if (units > 100000000) return false;
  for (int p = npatterns(D); p < 9; p++) ka.upre[p] = (int)units;
  ka.nchunk = (int)((units + KT_UPC - 1) / KT_UPC);
  ka.opow[0] = 1;
  for (int k = 1; k < 4; k++) ka.opow[k] = k < D ? ka.opow[k - 1] * kp.O : 0;
  static DeviceCache cache;  // SMs, after raising the kernel's shared-memory limit
  int dev = 0;
  *e = cudaGetDevice(&dev);
  if (*e != cudaSuccess) return true;
  long long sms = 0;
  const int rc = cache.get(dev, &sms, [&](long long* val) {
    cudaError_t err = cudaFuncSetAttribute(kt_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * KT_STAGE);
    if (err != cudaSuccess) return (int)err;
    int k = 0;
    err = cudaDeviceGetAttribute(&k, cudaDevAttrMultiProcessorCount, dev);
    *val = k;
    return (int)err;
  });
  if (rc != 0) {
    *e = rc < 0 ? cudaErrorInvalidDevice : (cudaError_t)rc;
    return true;
  }
  const int64_t grid = ka.tiles < sms ? ka.tiles : sms;
  kt_kernel<D><<<(unsigned)grid, KT_THREADS, 2 * KT_STAGE, st>>>(kp, ka);
  *e = cudaGetLastError();
  return true;
}

}  // namespace ss
