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
// - The tuples t are taken in chunks of 192. Per chunk, a row s of S(A) and a
//   column y of W each get one power-of-two scale (from the largest |A| resp. |W|
//   of the chunk) and become 55-bit signed integers v = sum_i d_i 256^(6-i),
//   i = 0..6, -128 <= d_i <= 127. The orbit operator runs on the integers of A
//   (two limbs of 24 and up to 28 bits, 32-bit multiply-adds), rounded to the grid
//   2^(E + 1 - bits), bits = 54 - log2 sum|a| and at most 52; S(A) is exact on it.
// - D_d = sum over t and i + j = d of d_i(A) d_j(W), d = 0..6. Leading digits are at
//   most 64, so |D_d| <= 192 d 2^14: below 2^24, hence exact in FP32, for d <= 5; D_6
//   may round above 2^24, by a unit 2^-8 of the smallest that is kept.
//   Digit pairs with i + j > 6 lie below 2^-56 of the largest product and are left
//   out, as FP64 would round them off.
// - Per chunk the D_d are joined in 64-bit integers (sum d <= 5 of
//   D_d 256^(5-d), and D_6 rounded to D_5's unit), scaled, rounded once to FP64 and
//   added to the FP64 sum of the chunks.
// - A tile whose chunk scales leave a safe exponent range (infinities, NaN,
//   magnitudes beyond 2^+-440), or whose magnitudes are too far apart for one
//   scale (below), is left to KC, which follows and takes those tiles only.
//
// One scale per row and chunk costs the elements far below it their low bits. The
// error, relative to sum_t |S(A) W| as that of FP64 sums is, is about 2^(q - bits) over
// the square root of the number of tuples, where 2^-q is the mean of |A W| against the
// product of the two largest. By the inequality of the means q is at most
// the mean of log2(max|A| / |A|) plus that of log2(max|W| / |W|), which take one sum of
// exponents each; the limit for it is bits - 43, where the error meets that of KC's
// FP64 sums of a few hundred tuples, and a fluctuation, 6 / sqrt(tuples). Row 1 of Table
// II, 512 tuples, largest error relative to sum |S W| (KT / KC, and q): uniform 1e-16 /
// 4e-16, 3.0; Gaussian 2e-16 / 6e-16, 5.1; A and W over one decade each, W large where A
// is small, 4e-16 / 6e-16, 5.9; over two 2e-15 / 4e-16, 8.9; over four 1e-13, 15. (A zero
// counts as an element at the limit: it is exact on any grid.) The sums of exponents and
// KC's launch over no tiles cost 3 %: 2148 -> 2225 us on A[48^3,16^3] with 32 columns (with a
// shift and an addition in place of the dot product 2430).
//
// A CTA owns 128 rows x 32 columns. Warps 0-15 find the scales (a first read of
// the chunk's A, which also brings it into L2), sum the orbits and write the digits;
// one thread issues the matrix instructions; warps 16-19 join the sums; one warp
// finds the chunks' tuples. Digit i of A meets digits 0..6-i of W, which lie
// side by side as one N = 32 (7 - i) operand, so each digit of A is read once from
// shared memory per step and its products land in the accumulators i..6: 7
// instructions per 16 tuples instead of 28.
#include "ss_contract.cuh"
#include "ss_devcache.h"
#include "ss_tma.cuh"

#include <algorithm>
#include <atomic>
#include <new>

#include <cuda_fp16.h>

namespace ss {

void count_launches(int n);

constexpr int KT_ROWS = 128, KT_COLS = 32, KT_ND = 7;
constexpr int KT_UNIT = 24;                       // tuples of a unit: 24 / m orbits of one pattern
constexpr int KT_UPC = 8;                         // units of a chunk: four stages of two
constexpr int KT_CHUNK = KT_UNIT * KT_UPC;        // 192 tuples
constexpr int KT_PROD = 512;                      // producer threads: four per row, two groups taking stages in turn
constexpr int KT_THREADS = KT_PROD + 128 + 64;    // + epilogue + (matrix, table) warps
// operand layout (K-major, no swizzle): 8 tuples x 8 rows as 128 contiguous bytes
constexpr int KT_AKG = KT_ROWS * 16;              // bytes of 8 tuples of one digit of A
constexpr int KT_AD = 6 * KT_AKG;                 // bytes of one digit of A: a stage's two units
constexpr int KT_WKG = KT_ND * KT_COLS * 16;      // bytes of 8 tuples of all digits of W
constexpr int KT_WST = 6 * KT_WKG;                // bytes of a stage of W
constexpr int KT_STAGE = KT_ND * KT_AD + KT_WST;
constexpr unsigned KT_ELO = (1023u - 440u) << 20, KT_EHI = (1023u + 440u) << 20;
constexpr int KT_VOTE = 4096;                     // most column tiles of a call that may be left to KC as a whole
constexpr int KT_ZERO = (1023 - 440) * 16;        // a zero beside an element in that range, in 16ths

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
  int kappa;           // limit of the mean logarithms' sum, in 16ths
  // prepared by kt_prep_kernel in the call's workspace
  unsigned char* wdig;  // digits of W by column tile, chunk and stage
  unsigned* wexp;       // [column tile][chunk][32] scales
  int* room;            // [column tile][chunk] what is left of the limit for A; -1: a scale is out of range
  unsigned* vote;       // [column tile][chunk] which of eight sampled rows would be left to KC
  int* tix;             // [chunk][192] tuple indices
  int* pat;             // [chunk][8] unit patterns, -1: none
  // written by kt_kernel
  unsigned char* flag;  // [tile] 1: left to KC
};

struct KtShared {
  // by chunk mod 4 and quarter: exponent of the largest |A| and the next four bits; sum of
  // log2(largest / |A|) over the quarter's 48 tuples, in 16ths
  unsigned short rowmax[4][4][KT_ROWS], rowlog[4][4][KT_ROWS];
  // chunk scales by chunk mod 8: producers run at most two chunks ahead of the
  // matrix warp, and that at most two ahead of the epilogue
  unsigned rowexp[8][KT_ROWS];   // exponent fields
  unsigned colexp[16][KT_COLS];  // W's, by chunk mod 16 (the table warp runs ahead of the producers)
  alignas(16) int tix[3][KT_CHUNK];  // tuple indices of a chunk (no tuple left: another of the chunk's, and W's digits are 0)
  int pat[3][KT_UPC];            // pattern of each unit, -1: none
  int room[3];                   // of the limit
  int bad[8];                    // by tile mod 8: left to KC
  uint64_t tab_full[3], tab_empty[3], mx_full[2], st_full[2], w_full[2], st_empty[2], acc_full[2], acc_empty[2], drain;
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
__device__ __forceinline__ void kt_st8(uint32_t addr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
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

// x rounded to the grid of a scale, as two limbs l1 2^24 + l0 of x's sign: the mantissa,
// shifted up by UP, is shifted right to half grid units by (base - |x|'s high word) >> 20
// places (base: the scale's exponent field, plus the places that the grid drops less
// one, with 20 ones below it), and half of it plus one is the nearest integer, ties away
// from zero. (Truncated instead, inputs of one sign lose half a unit each. The signs come
// last, on the limbs: 2143 us on A[48^3,16^3] with 32 columns, as much as without
// rounding; on the 64-bit integer before its rounding 2230. One FP64 addition of
// 1.5 * 2^52 grid units does the same in five instructions, but at two FP64 operations
// per SM and clock: 2509 against 2275 us there.)
template <int UP>
__device__ __forceinline__ void kt_limbs(double x, unsigned base, int& l0, int& l1) {
  const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
  const unsigned k = (base - (xh & 0x7FFFFFFFu)) >> 20;
  const unsigned long long mant = (((unsigned long long)((xh & 0x000FFFFFu) | 0x00100000u) << 32) | xl) << UP;
  const long long q = (long long)shr64(mant, k);
  const unsigned long long r = (unsigned long long)q + 1;
  const int sg = (int)xh >> 31;
  l0 = (((int)((unsigned)(r >> 1) & 0xFFFFFFu)) ^ sg) - sg;
  l1 = (((int)(r >> 25)) ^ sg) - sg;
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

// N tuples' elements of one row (rows past the end read the last one: As)
template <int N>
__device__ __forceinline__ void kt_load(const double* As, int64_t S, const int* tix, double* x) {
  static_assert(N % 4 == 0, "whole int4");
#pragma unroll
  for (int e = 0; e < N; e += 4) {
    const int4 t = *reinterpret_cast<const int4*>(tix + e);
    x[e] = As[(int64_t)t.x * S];
    x[e + 1] = As[(int64_t)t.y * S];
    x[e + 2] = As[(int64_t)t.z * S];
    x[e + 3] = As[(int64_t)t.w * S];
  }
}

// one unit (24 tuples of pattern P) of one row: loads, orbit operator, digits. The first
// twelve values are in flight already (x0: loaded before the wait for the stage, so that
// the wait and the choice of the pattern hide their latency: 2222 -> 2119 us on
// A[48^3,16^3] with 32 columns; all 24 of them do not fit into 80 registers)
template <int D, int P>
__device__ __forceinline__ void kt_unit(const KParams& kp, const double* As, const int* tix,
                                        unsigned base, unsigned char* dst, double (&x0)[12]) {
  constexpr int M = Pat<D, P>::M, NO = KT_UNIT / M;
  if constexpr (M == 24) {
    // one 24-member orbit, by eights of outputs (registers)
    double x[KT_UNIT];
#pragma unroll
    for (int e = 0; e < 12; e++) x[e] = x0[e];
    kt_load<12>(As, kp.S, tix + 12, x + 12);
    int l0[M], l1[M];
#pragma unroll
    for (int v = 0; v < M; v++) {
      kt_limbs<0>(x[v], base, l0[v], l1[v]);
    }
#pragma unroll
    for (int g = 0; g < 3; g++) {
      int y0[8], y1[8];
      unsigned z0[8], z1[8];
#pragma unroll
      for (int j = 0; j < 8; j++) { y0[j] = 0; y1[j] = 0; }
#pragma unroll
      for (int s = 0; s < fact(D); s++) {
        const int c = kp.ci[0][s];
        if (c != 0) {
#pragma unroll
          for (int j = 0; j < 8; j++) {
            y0[j] += c * l0[Pat<D, P>::idx(8 * g + j, s)];
            y1[j] += c * l1[Pat<D, P>::idx(8 * g + j, s)];
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 8; j++) kt_digits(y0[j], y1[j], z0[j], z1[j]);
      kt_store8(dst + g * KT_AKG, KT_AD, z0, z1);
    }
    return;
  }
  // two batches of twelve tuples (registers)
  constexpr int NB = 12;
  double (&x)[NB] = x0;
  unsigned z0[KT_UNIT], z1[KT_UNIT];
#pragma unroll
  for (int o = 0; o < NO; o++) {
    if (o * M == NB) kt_load<NB>(As, kp.S, tix + NB, x);
    int l0[M], l1[M], y0[M], y1[M];
#pragma unroll
    for (int v = 0; v < M; v++) {
      kt_limbs<0>(x[o * M % NB + v], base, l0[v], l1[v]);
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
#pragma unroll
    for (int g = 0; g < 3; g++)  // eights that this orbit completed
      if (o * M < 8 * g + 8 && (o + 1) * M >= 8 * g + 8) kt_store8(dst + g * KT_AKG, KT_AD, z0 + 8 * g, z1 + 8 * g);
  }
}

template <int D>
__device__ __forceinline__ void kt_unit_any(const KParams& kp, int p, const double* As,
                                            const int* tix, unsigned base, unsigned char* dst, double (&x0)[12]) {
  switch (p) {
    case 0: kt_unit<D, 0>(kp, As, tix, base, dst, x0); break;
    case 1: kt_unit<D, 1>(kp, As, tix, base, dst, x0); break;
    case 2: if constexpr (npatterns(D) > 2) kt_unit<D, 2>(kp, As, tix, base, dst, x0); break;
    case 3: if constexpr (npatterns(D) > 3) kt_unit<D, 3>(kp, As, tix, base, dst, x0); break;
    case 4: if constexpr (npatterns(D) > 4) kt_unit<D, 4>(kp, As, tix, base, dst, x0); break;
    case 5: if constexpr (npatterns(D) > 4) kt_unit<D, 5>(kp, As, tix, base, dst, x0); break;
    case 6: if constexpr (npatterns(D) > 4) kt_unit<D, 6>(kp, As, tix, base, dst, x0); break;
    case 7: if constexpr (npatterns(D) > 4) kt_unit<D, 7>(kp, As, tix, base, dst, x0); break;
    default:  // no tuples left: digits of zero
      const unsigned z[8] = {0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u};
      for (int g = 0; g < 3; g++) kt_store8(dst + g * KT_AKG, KT_AD, z, z);
  }
}

// the orbit `rank` of pattern P into its unit's entries tix[0..m)
template <int D, int P>
__device__ __forceinline__ void kt_orbit(const KParams& kp, const KtArgs& ka, int64_t rank, int* tix, signed char* none) {
  constexpr int M = Pat<D, P>::M;
  int v[4] = {0, 0, 0, 0};
  const bool ok = rank < kp.norb[P];
  if (ok) unrank<Pat<D, P>::ND>(rank, kp.O, v);
#pragma unroll
  for (int u = 0; u < M; u++) {
    int t = 0;
#pragma unroll
    for (int k = 0; k < D; k++) t += v[Pat<D, P>::lab(u, k)] * ka.opow[k];
    tix[u] = t;
    none[u] = ok ? 0 : -1;
  }
}

// members of pattern p (0 < p < npatterns), for the unit geometry
template <int D>
__device__ __forceinline__ int kt_members(int p) {
  if constexpr (D == 2) return p == 0 ? 2 : 1;
  else if constexpr (D == 3) return p == 0 ? 6 : (p == 3 ? 1 : 3);
  else return p == 0 ? 24 : (p <= 3 ? 12 : (p == 4 ? 6 : (p == 7 ? 1 : 4)));
}

// W once per call: a CTA takes a chunk and 32 columns, finds the chunk's tuples (kept for
// the main kernel), the columns' scales and the digits, in the layout of a stage.
// (Digitised by every row tile's CTA instead, W cost 0.16 of 0.56 ms on A[48^3,8^3].)
template <int D>
__global__ void __launch_bounds__(256) kt_prep_kernel(const __grid_constant__ KParams kp, const __grid_constant__ KtArgs ka) {
  __shared__ int tix[KT_CHUNK], tuples[KT_CHUNK];
  __shared__ int wcount[KT_CHUNK / 32];
  __shared__ signed char none[KT_CHUNK];
  __shared__ unsigned colmax[KT_COLS];
  __shared__ int collog[KT_COLS], colzero[KT_COLS];
  __shared__ int left;
  __shared__ unsigned votes;
  const int tid = threadIdx.x, ch = blockIdx.x, yt = blockIdx.y;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // kt_kernel, which waits for this grid
  const int nunit = ka.upre[npatterns(D)];
  if (tid < KT_COLS) colmax[tid] = collog[tid] = colzero[tid] = 0;
  if (tid < KT_CHUNK) {
    tix[tid] = 0;
    none[tid] = -1;
  }
  __syncthreads();
  if (tid < KT_CHUNK) {
    // thread o + 24 u: orbit o of unit u
    const int u = tid / KT_UNIT, o = tid % KT_UNIT, g = ch * KT_UPC + u;
    int p = -1;
    if (g < nunit) {
      p = 0;
#pragma unroll
      for (int r = 1; r < npatterns(D); r++)
        if (g >= ka.upre[r]) p = r;
      const int m = kt_members<D>(p), no = KT_UNIT / m;
      if (o < no) {
        const int64_t rank = (int64_t)(g - ka.upre[p]) * no + o;
        int* dst = tix + u * KT_UNIT + o * m;
        signed char* dn = none + u * KT_UNIT + o * m;
        switch (p) {
          case 0: kt_orbit<D, 0>(kp, ka, rank, dst, dn); break;
          case 1: kt_orbit<D, 1>(kp, ka, rank, dst, dn); break;
          case 2: if constexpr (npatterns(D) > 2) kt_orbit<D, 2>(kp, ka, rank, dst, dn); break;
          case 3: if constexpr (npatterns(D) > 3) kt_orbit<D, 3>(kp, ka, rank, dst, dn); break;
          case 4: if constexpr (npatterns(D) > 4) kt_orbit<D, 4>(kp, ka, rank, dst, dn); break;
          case 5: if constexpr (npatterns(D) > 4) kt_orbit<D, 5>(kp, ka, rank, dst, dn); break;
          case 6: if constexpr (npatterns(D) > 4) kt_orbit<D, 6>(kp, ka, rank, dst, dn); break;
          case 7: if constexpr (npatterns(D) > 4) kt_orbit<D, 7>(kp, ka, rank, dst, dn); break;
        }
      }
    }
    if (yt == 0 && o == 0) ka.pat[ch * KT_UPC + u] = p;
  }
  __syncthreads();
  // Slots without a tuple (their W is 0) repeat the chunk's own tuples in turn: the main
  // kernel takes the chunk's row scales over all slots.
  unsigned has = 0;
  if (tid < KT_CHUNK) {
    has = __ballot_sync(0xffffffffu, none[tid] == 0);
    if ((tid & 31) == 0) wcount[tid >> 5] = __popc(has);
  }
  __syncthreads();
  int ntup = 0, before = 0;  // tuples of the chunk, and of the slots before this one
#pragma unroll
  for (int w = 0; w < KT_CHUNK / 32; w++) {
    if (w < tid >> 5) before += wcount[w];
    ntup += wcount[w];
  }
  before += __popc(has & ((1u << (tid & 31)) - 1u));
  if (tid < KT_CHUNK && none[tid] == 0) tuples[before] = tix[tid];
  __syncthreads();
  if (tid < KT_CHUNK && none[tid] != 0) tix[tid] = tuples[(tid - before) % ntup];
  __syncthreads();
  if (yt == 0 && tid < KT_CHUNK) ka.tix[ch * KT_CHUNK + tid] = tix[tid];
  const int y = tid & 31, q = tid >> 5;
  const bool act = (int64_t)yt * KT_COLS + y < ka.Y;
  const double* Wy = ka.W + (int64_t)yt * KT_COLS + y;
  auto load = [&](int e) { return act && none[e] == 0 ? Wy[(int64_t)tix[e] * ka.ldw] : 0.0; };
  // this warp's sampled row of A, for the votes below (loaded under the work on W)
  double sample[KT_CHUNK / 32];
#pragma unroll
  for (int e = 0; e < KT_CHUNK / 32; e++)
    sample[e] = static_cast<const double*>(kp.A)[(2 * q + 1) * kp.S / 16 + (int64_t)tix[e * 32 + y] * kp.S];
  unsigned m = 0;
  int logs = 0, zeros = 0;
#pragma unroll 8
  for (int e = q; e < KT_CHUNK; e += 8) {
    if (none[e] != 0) continue;
    const double v = load(e);
    const unsigned h = (unsigned)__double2hiint(v) & 0x7FFFFFFFu;
    m = max(m, h | ((unsigned)__double2loint(v) != 0));
    logs += h >> 16;
    zeros += h == 0;
  }
  atomicMax(&colmax[y], m);
  atomicAdd(&collog[y], logs);
  atomicAdd(&colzero[y], zeros);
  __syncthreads();
  m = colmax[y];
  unsigned E = m & 0x7FF00000u;
  bool bad = false;
  if (E < KT_ELO || E > KT_EHI) {
    bad = m != 0;
    E = KT_ELO;
  }
  if (q == 0) {
    ka.wexp[((int64_t)yt * ka.nchunk + ch) * KT_COLS + y] = E;
    // per tuple, over the 192 slots of the rows' sums (a column of zeros contributes exact zeros)
    const int far = m == 0 ? 0 : (ntup - colzero[y]) * (int)(m >> 16) - collog[y] + ka.kappa * colzero[y];
    const int worst = __reduce_max_sync(0xffffffffu, far);
    const int lim = (int)(KT_CHUNK * ((float)ka.kappa + 96.0f * rsqrtf((float)ntup)));
    const bool out = __any_sync(0xffffffffu, bad), any = __any_sync(0xffffffffu, m != 0);
    if (y == 0) {
      left = out ? -1 : (any ? max(0, lim - (int)((int64_t)worst * KT_CHUNK / ntup)) : 0x7FFFFFFF);
      votes = 0;
      ka.room[yt * ka.nchunk + ch] = left;
    }
  }
  __syncthreads();
  // a warp per sampled row: the main kernel's rule
  {
    unsigned h[KT_CHUNK / 32], top = 0;
    bool tiny = false;
#pragma unroll
    for (int e = 0; e < KT_CHUNK / 32; e++) {
      h[e] = (unsigned)__double2hiint(sample[e]) & 0x7FFFFFFFu;
      tiny |= h[e] == 0 && __double2loint(sample[e]) != 0;
      top = max(top, h[e]);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    int far = 0;
#pragma unroll
    for (int e = 0; e < KT_CHUNK / 32; e++) far += h[e] != 0 ? (int)(top >> 16) - (int)(h[e] >> 16) : ka.kappa;
    far = __reduce_add_sync(0xffffffffu, far);
    const bool out = top == 0 ? __any_sync(0xffffffffu, tiny) : (top & 0x7FF00000u) < KT_ELO || (top & 0x7FF00000u) > KT_EHI;
    if (y == 0 && (left < 0 || out || (top != 0 && far > left))) atomicOr(&votes, 1u << q);
  }
  __syncthreads();
  if (tid == 0) ka.vote[yt * ka.nchunk + ch] = votes;
  // largest |W| at most 2^54
  const unsigned base = E | 0xFFFFFu;
  for (int kg = q; kg < KT_CHUNK / 8; kg += 8) {
    unsigned z0[8], z1[8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
      int l0, l1;
      kt_limbs<2>(load(kg * 8 + e), base, l0, l1);
      kt_digits(l0, l1, z0[e], z1[e]);
    }
    unsigned char* dst = ka.wdig + (((int64_t)yt * ka.nchunk + ch) * 4 + kg / 6) * KT_WST + kg % 6 * KT_WKG + y * 16;
    kt_store8(dst, KT_COLS * 16, z0, z1);
  }
}

// sum of top - log2|A| in 16ths over N tuples with zeros among them (or magnitudes far out
// of range), kappa for a zero; out of line, rare
template <int N>
static __device__ __noinline__ int kt_logs_zeros(const unsigned* hw, const int* te, int64_t S, int top, int kappa) {
  int logs = 0;
#pragma unroll 1
  for (int e = 0; e < N; e++) {
    const unsigned h = hw[2 * (int64_t)te[e] * S] & 0x7FFFFFFFu;
    logs += h != 0 ? top - (int)(h >> 16) : kappa;
  }
  return logs;
}

// Where half the sampled rows of every column tile would be left to KC, the call is left to
// it as a whole: inputs of spread magnitudes, or an infinity in W, would take both kernels'
// time otherwise (25.7 against 27.9 ms on A[48^3,16^3] with 32 columns, 3.5 against 5.7 with
// 4). Out of line, where it leaves the main kernel's code as it was (2231 us on ordinary
// inputs; inlined 2480, and with the column tiles left out skipped one by one 2375).
static __device__ __noinline__ bool kt_all_left(const KtArgs& ka, unsigned* votes) {
  const int tid = threadIdx.x;
  for (int i = tid; i < ka.ytiles; i += KT_THREADS) votes[i] = 0;
  __syncthreads();
  for (int i = tid; i < ka.ytiles * ka.nchunk; i += KT_THREADS)
    if (const unsigned v = ka.vote[i]) atomicOr(&votes[i / ka.nchunk], v);
  __syncthreads();
  bool all = true;
  for (int i = tid; i < ka.ytiles; i += KT_THREADS) all = all && __popc(votes[i]) >= 4;
  all = __syncthreads_and(all);
  if (all)
    for (int64_t tile = blockIdx.x + (int64_t)tid * gridDim.x; tile < ka.tiles; tile += (int64_t)KT_THREADS * gridDim.x)
      ka.flag[tile] = 1;
  return all;
}

template <int D>
__global__ void __launch_bounds__(KT_THREADS, 1) kt_kernel(const __grid_constant__ KParams kp, const __grid_constant__ KtArgs ka) {
  extern __shared__ __align__(128) unsigned char kt_smem[];
  __shared__ KtShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // launched under the end of kt_prep_kernel
  if (ka.ytiles <= KT_VOTE && kt_all_left(ka, reinterpret_cast<unsigned*>(kt_smem))) return;
  if (tid == 0) {
    for (int i = 0; i < 3; i++) {
      mbar_init(&sh.tab_full[i], 32);
      mbar_init(&sh.tab_empty[i], KT_PROD);
    }
    for (int i = 0; i < 2; i++) {
      mbar_init(&sh.mx_full[i], KT_PROD);
      mbar_init(&sh.st_full[i], KT_PROD / 2);  // a group
      mbar_init(&sh.w_full[i], 1);             // W's copy
      mbar_init(&sh.st_empty[i], 1);
      mbar_init(&sh.acc_full[i], 1);
      mbar_init(&sh.acc_empty[i], 128);
    }
    mbar_init(&sh.drain, 1);
    fence_mbar_init();
  }
  if (tid < 8) sh.bad[tid] = 0;
  constexpr int MMA_WARP = KT_PROD / 32 + 4;
  if (warp == MMA_WARP) {
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

  if (warp < KT_PROD / 32) {
    // ---- producers: scales, orbit sums, digits ----
    const int row = tid & (KT_ROWS - 1), quarter = tid >> 7, half = quarter & 1, group = tid >> 8;
    const int64_t step = gridDim.x;
    auto row_of = [&](int64_t tile) {
      const int64_t s = tile / ka.ytiles * KT_ROWS + row;
      return static_cast<const double*>(kp.A) + (s < kp.S ? s : kp.S - 1);
    };
    // the largest |A| of the row in chunk c of a tile (a quarter of the tuples per
    // thread); run one chunk ahead, so that its loads and the meeting of all producers
    // hide under the chunk before
    auto maxima = [&](int64_t tile, int c) {
      if (!mbar_wait(&sh.tab_full[c % 3], (c / 3) & 1, lim)) return false;
      const int* tix = sh.tix[c % 3];
      const double* As = row_of(tile);
      unsigned mx = 0;
      int far = 0, n = 0;  // sum of log2(mx / |A|) in 16ths, tuples in it
      // high words only (half the registers: 24 loads in flight)
      const unsigned* hw = reinterpret_cast<const unsigned*>(As) + 1;
#pragma unroll 1
      for (int j = 0; j < 2; j++) {
        constexpr int N = KT_CHUNK / 8;
        const int* te = tix + quarter * (KT_CHUNK / 4) + j * N;
        unsigned v[N];
#pragma unroll
        for (int e = 0; e < N; e += 4) {
          const int4 t = *reinterpret_cast<const int4*>(te + e);
          v[e] = hw[2 * (int64_t)t.x * kp.S];
          v[e + 1] = hw[2 * (int64_t)t.y * kp.S];
          v[e + 2] = hw[2 * (int64_t)t.z * kp.S];
          v[e + 3] = hw[2 * (int64_t)t.w * kp.S];
        }
        unsigned m = 0;
        int logs = 0;
#pragma unroll
        for (int e = 0; e < N; e++) {
          const unsigned h = v[e] & 0x7FFFFFFFu;
          m = max(m, h);
          logs = (int)__dp2a_lo(h, 0x0100u, (unsigned)logs);  // + (h >> 16), in one instruction
        }
        if (m == 0) {  // zeros, or magnitudes below 2^-1042: the latter are out of range
          for (int e = 0; e < N; e++) m |= hw[2 * (int64_t)te[e] * kp.S - 1] != 0;
          far += N * ka.kappa;
        } else {
          const int top = (int)(m >> 16), was = (int)(mx >> 16);
          logs = N * top - logs;
          if (logs >= KT_ZERO) logs = kt_logs_zeros<N>(hw, te, kp.S, top, ka.kappa);
          far += logs + (top > was ? n * (top - was) : N * (was - top));
          n += N;
        }
        mx = max(mx, m);
      }
      // exponent 1 (out of range) for subnormal maxima
      sh.rowmax[c & 3][quarter][row] = (unsigned short)(mx >> 20 == 0 && mx != 0 ? 16 : mx >> 16);
      sh.rowlog[c & 3][quarter][row] = (unsigned short)min(far, 65535);
      mbar_arrive(&sh.mx_full[c & 1]);
      return true;
    };
    int c = 0, n = 0, it = 0;  // chunks, stages and tiles so far
    int copies = 0;            // of W, by this thread
    if (blockIdx.x < ka.tiles) ok = maxima(blockIdx.x, 0);
    for (int64_t tile = blockIdx.x; ok && tile < ka.tiles; tile += step, it++) {
      const double* As = row_of(tile);
      const unsigned char* wd = ka.wdig + tile % ka.ytiles * ka.nchunk * 4 * KT_WST;
      for (int ch = 0; ok && ch < ka.nchunk; ch++, c++) {
        const int64_t nt = ch + 1 < ka.nchunk ? tile : tile + step;
        if (nt < ka.tiles) ok = maxima(nt, c + 1);
        ok = ok && mbar_wait(&sh.mx_full[c & 1], (c >> 1) & 1, lim);
        if (!ok) break;
        const int* tix = sh.tix[c % 3];
        const unsigned short* rm = &sh.rowmax[c & 3][0][row];
        const int top = max(max(rm[0], rm[KT_ROWS]), max(rm[2 * KT_ROWS], rm[3 * KT_ROWS]));
        unsigned E = (unsigned)(top >> 4) << 20;
        bool bad = false;
        if (E < KT_ELO || E > KT_EHI) {
          bad = E != 0;
          E = KT_ELO;
        }
        if (half == 0) {
          const unsigned short* rl = &sh.rowlog[c & 3][0][row];
          int far = 0;
#pragma unroll
          for (int k = 0; k < 4; k++)
            far += rl[k * KT_ROWS] + (rm[k * KT_ROWS] != 0 ? KT_CHUNK / 4 * (top - rm[k * KT_ROWS]) : 0);
          const int room = sh.room[c % 3];
          bad |= room < 0 || (top != 0 && far > room);
        }
        // largest |A| at most 2^bits
        const unsigned base = (E + ((unsigned)(52 - ka.bits) << 20)) | 0xFFFFFu;
        const int ns = stages_of(ch);
        for (int j = 0; ok && j < ns; j++, n++) {
          if ((n & 1) != group) continue;  // the other group's stage
          // The epilogue reads the scales and the flag behind acc_full, which follows the
          // arrivals of the groups that filled the chunk's stages, and of no other: a chunk of
          // one stage orders one group's writes only. So the group that fills a stage
          // publishes them, ahead of its arrival. (A stage's buffer was free two stages ago, so
          // the epilogue is at most five chunks behind, within the rings of eight.)
          if (half == 0) {
            sh.rowexp[c & 7][row] = E;
            if (bad) sh.bad[it & 7] = 1;
          }
          unsigned char* st = kt_smem + (n & 1) * KT_STAGE;
          const int u = 2 * j + half;
          double x0[12];
          kt_load<12>(As, kp.S, tix + u * KT_UNIT, x0);
          ok = mbar_wait(&sh.st_empty[n & 1], ((n >> 1) & 1) ^ 1, lim);
          if (!ok) break;
          if ((tid & 255) == 0) {
            mbar_arrive_expect_tx(&sh.w_full[group], KT_WST);
            bulk_g2s(st + KT_ND * KT_AD, wd + ((int64_t)ch * 4 + j) * KT_WST, KT_WST, &sh.w_full[group]);
            copies++;
          }
          kt_unit_any<D>(kp, sh.pat[c % 3][u], As, tix + u * KT_UNIT, base, st + half * 3 * KT_AKG + row * 16, x0);
          kt_proxy_fence();
          mbar_arrive(&sh.st_full[n & 1]);
        }
        mbar_arrive(&sh.tab_empty[c % 3]);
      }
    }
    // no copy is in flight when the CTA's shared memory is given up, also where a wait ran
    // out (the copy before the last has landed: its stage was used and freed)
    if (copies > 0) ok = mbar_wait(&sh.w_full[group], (copies - 1) & 1, kDrainLimit) && ok;
  } else if (warp < MMA_WARP) {
    // ---- epilogue: join the digit sums of a chunk, add up the chunks ----
    const int row = tid - KT_PROD;
    const uint32_t lanes = (uint32_t)(warp & 3) << 21;  // TMEM lane 32 (warp mod 4)
    int c = 0, it = 0;
    for (int64_t tile = blockIdx.x; ok && tile < ka.tiles; tile += gridDim.x, it++) {
      const int64_t s = tile / ka.ytiles * KT_ROWS + row, y0 = tile % ka.ytiles * KT_COLS;
      const int ny = (int)min((int64_t)KT_COLS, ka.Y - y0);
      bool bad = false;
      for (int ch = 0; ch < ka.nchunk; ch++, c++) {
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc_full[c & 1], (c >> 1) & 1, lim));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const bool last = ch == ka.nchunk - 1;
        if (last) bad = sh.bad[it & 7] != 0;  // every scale of the tile is known
        const int er = (int)(sh.rowexp[c & 7][row] >> 20) + ka.sh0;
        const uint32_t t0 = tmem + (uint32_t)(c & 1) * 256 + lanes;
        // the FP64 sums of the 32 columns live in the 2 x 32 accumulator columns that the
        // digit sums leave free (in registers they would cap the producers' share)
        const uint32_t tlo = tmem + lanes + KT_ND * KT_COLS, thi = tlo + 256;
#pragma unroll 1
        for (int yb = 0; yb < KT_COLS; yb += 8) {
          uint32_t d[KT_ND][8], lo[8] = {}, hi[8] = {};
#pragma unroll
          for (int i = 0; i < KT_ND; i++) kt_ld8(t0 + i * KT_COLS + yb, d[i]);
          if (ch > 0) {
            kt_ld8(tlo + yb, lo);
            kt_ld8(thi + yb, hi);
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int y = 0; y < 8; y++) {
            int v[KT_ND];
#pragma unroll
            for (int i = 0; i < KT_ND; i++) v[i] = __float2int_rn(__uint_as_float(d[i][y]));
            // |D_0| <= 2^19.6, |D_d| <= 192 d 2^14: the joined sum stays below 2^61
            long long V = (long long)((unsigned long long)(unsigned)(v[0] * 256 + v[1]) << 32);
            V += (long long)v[2] * (1 << 24) + (long long)v[3] * (1 << 16);
            V += (long long)v[4] * 256 + (long long)(v[5] + ((v[6] + 128) >> 8));
            const double a = __hiloint2double((int)hi[y], (int)lo[y]) +
                             fixed_rn(V, er + (int)(sh.colexp[c & 15][yb + y] >> 20));
            lo[y] = (unsigned)__double2loint(a);
            hi[y] = (unsigned)__double2hiint(a);
          }
          if (!last) {
            kt_st8(tlo + yb, lo);
            kt_st8(thi + yb, hi);
          } else if (!bad && s < kp.S) {
#pragma unroll
            for (int y = 0; y < 8; y++)
              if (yb + y < ny) ka.C[s + ka.ldc * (y0 + yb + y)] = __hiloint2double((int)hi[y], (int)lo[y]);
          }
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(&sh.acc_empty[c & 1]);
      }
      ok = kt_sync<2, 128>(ok);
      if (!ok) break;
      if (row == 0) {
        ka.flag[tile] = bad;
        if (bad) sh.bad[it & 7] = 0;
      }
    }
  } else if (warp == MMA_WARP) {
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
            if (!mbar_wait(&sh.st_full[n & 1], (n >> 1) & 1, lim) || !mbar_wait(&sh.w_full[n & 1], (n >> 1) & 1, lim)) {
              ok = false;
              break;
            }
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
      // no matrix instruction is in flight when the accumulators are given back, also where
      // a wait ran out
      kt_commit(&sh.drain);
      ok = mbar_wait(&sh.drain, 0, kDrainLimit) && ok;
    }
    __syncwarp();
  } else if (warp == MMA_WARP + 1) {
    // ---- the chunks' tuples and W's scales, ahead of the producers ----
    int c = 0;
    for (int64_t tile = blockIdx.x; ok && tile < ka.tiles; tile += gridDim.x)
      for (int ch = 0; ok && ch < ka.nchunk; ch++, c++) {
        if (!mbar_wait(&sh.tab_empty[c % 3], ((c / 3) & 1) ^ 1, lim)) { ok = false; break; }
        const int64_t s0 = tile / ka.ytiles * KT_ROWS;
        const unsigned bytes = (unsigned)(min((int64_t)KT_ROWS, kp.S - s0) * 8) & ~15u;
        for (int e = lane; e < KT_CHUNK; e += 32) {
          const int t = ka.tix[ch * KT_CHUNK + e];
          sh.tix[c % 3][e] = t;
          // the tuple's rows of A on their way to L2
          const double* a = static_cast<const double*>(kp.A) + (int64_t)t * kp.S + s0;
          if (((uintptr_t)a & 15) == 0 && bytes > 0)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(bytes) : "memory");
        }
        if (lane < KT_UPC) sh.pat[c % 3][lane] = ka.pat[ch * KT_UPC + lane];
        if (lane == 0) sh.room[c % 3] = ka.room[tile % ka.ytiles * ka.nchunk + ch];
        sh.colexp[c & 15][lane] = ka.wexp[(tile % ka.ytiles * ka.nchunk + ch) * KT_COLS + lane];
        mbar_arrive(&sh.tab_full[c % 3]);
      }
  }
  if (!ok) report_timeout(kp);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // KC, which waits for this grid
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == MMA_WARP) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// what the pool below keeps
constexpr int64_t KT_POOL = 128 << 20;

// The library's memory pool for KT's workspaces on a device: freed blocks up to 128 MB
// stay with it between calls (the default pool would return them to the system at every
// synchronisation and map them again, milliseconds). Null if the device has no pools.
inline cudaMemPool_t kt_pool(int dev) {
  static DeviceCache cache;
  long long v = 0;
  const int rc = cache.get(dev, &v, [&](long long* val) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    // (another thread may be capturing: creating a pool touches no stream)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    cudaError_t err = cudaMemPoolCreate(&p, &props);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (err != cudaSuccess) return (int)err;
    unsigned long long keep = KT_POOL;
    err = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    *val = (long long)(uintptr_t)p;
    return (int)err;
  });
  if (rc != 0) {
    cudaGetLastError();
    return nullptr;
  }
  return (cudaMemPool_t)(uintptr_t)v;
}

// Workspaces of captured calls. Allocation nodes would keep a graph from being
// instantiated twice or put into another, and KC, which needs none, takes up to twelve
// times as long; so the graph holds a workspace from the pool as a user object, and a later
// call gives it back (no CUDA call may be made where the graph's end is reported).
struct KtHeld {
  void* ws;
  int dev;
  KtHeld* next;
};
inline std::atomic<KtHeld*>& kt_dead() {
  static std::atomic<KtHeld*> head{nullptr};
  return head;
}
inline void CUDART_CB kt_retire(void* held) {
  KtHeld* h = static_cast<KtHeld*>(held);
  h->next = kt_dead().load(std::memory_order_relaxed);
  while (!kt_dead().compare_exchange_weak(h->next, h, std::memory_order_release, std::memory_order_relaxed)) {
  }
}
// the workspaces of device dev whose graphs are gone, back to the pool in st's order
inline void kt_reap(int dev, cudaStream_t st) {
  if (kt_dead().load(std::memory_order_relaxed) == nullptr) return;
  for (KtHeld* h = kt_dead().exchange(nullptr, std::memory_order_acquire); h != nullptr;) {
    KtHeld* const next = h->next;
    if (h->dev != dev) {
      kt_retire(h);
    } else {
      if (cudaFreeAsync(h->ws, st) != cudaSuccess) cudaGetLastError();
      delete h;
    }
    h = next;
  }
}
inline bool kt_graph_workspace(cudaMemPool_t pool, int dev, cudaGraph_t graph, size_t bytes, unsigned char** ws) {
  // the allocation goes to a stream of its own, outside the capture
  static DeviceCache cache;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return false;
  long long v = 0;
  const int rc = cache.get(dev, &v, [](long long* val) {
    cudaStream_t s = nullptr;
    const cudaError_t err = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    *val = (long long)(uintptr_t)s;
    return (int)err;
  });
  const cudaStream_t own = (cudaStream_t)(uintptr_t)v;
  KtHeld* const held = new (std::nothrow) KtHeld{nullptr, dev, nullptr};
  bool ok = rc == 0 && held != nullptr && cudaMallocFromPoolAsync((void**)ws, bytes, pool, own) == cudaSuccess;
  if (ok) {
    held->ws = *ws;
    cudaUserObject_t obj = nullptr;
    ok = cudaStreamSynchronize(own) == cudaSuccess &&
         cudaUserObjectCreate(&obj, held, kt_retire, 1, cudaUserObjectNoDestructorSync) == cudaSuccess;
    if (!ok) {
      cudaFreeAsync(*ws, own);
      delete held;
    } else if (cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove) != cudaSuccess) {
      cudaUserObjectRelease(obj, 1);  // kt_retire: given back by a later call
      ok = false;
    }
  } else {
    delete held;
  }
  cudaThreadExchangeStreamCaptureMode(&mode);
  return ok;
}

// Whether KT takes the contraction: exact arithmetic with integer coefficients
// (the operator's 1-norm is then at most 127, so the limb sums stay below 2^31),
// more than two row tiles (smaller calls stay with KC, whose FP64 sums equal those of
// the summation followed by the contraction alone bit for bit), and where it is the
// faster one. Per spectator position KT costs 4.9 ps per tuple of its whole chunks and 32
// columns, KC 1.8 ps per tuple and column of its column tiles (A[48^3,16^3]: KT 2.23 ms up to
// 32 columns, KC 3.4 ms up to 4; A[100,90,80,6^3], 216 tuples in two chunks: KT 1.34 ms, KC
// 1.08 ms up to 4 columns and 2.09 up to 8); and below a million tuple-columns both are shorter
// than the call, KC with one launch and no workspace.
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
  if (T < 1 || T > 0x7FFFFFFF || kp.S <= 2 * KT_ROWS || (kp.flags & KF_ALPHA_MUL) || L > 127) return false;
  int lg = 0;
  while ((double)(1 << lg) < L) lg++;
  KtArgs ka{};
  ka.ldw = ldw;
  ka.ldc = ldc;
  ka.ytiles = (int)((Y + KT_COLS - 1) / KT_COLS);
  ka.tiles = (kp.S + KT_ROWS - 1) / KT_ROWS * ka.ytiles;
  ka.bits = lg > 2 ? 54 - lg : 52;  // (a mantissa has 53 bits, one of them for rounding)
  // kp.cexp = (53 - 2 W + kdrop + aexp) << 20 + 0x80000, aexp = the coefficients' scale;
  // a joined sum counts 2^56 of the products' units 2^(E_A + 1 - bits + aexp) 2^(E_W - 53)
  const int aexp = ((kp.cexp - 0x80000) >> 20) - 53 + 2 * kp.W - kp.kdrop;
  ka.kappa = 16 * (ka.bits - 43);
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
  const int64_t ct = Y <= 4 ? 4 : (Y <= 8 ? 8 : (Y <= 16 || D == 4 ? 16 : 32)), kc_cols = (Y + ct - 1) / ct * ct;
  if (2.7 * KT_CHUNK * ka.nchunk * ka.ytiles > (double)T * kc_cols || (double)kp.S * T * kc_cols < 1e6) return false;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaGraph_t graph = nullptr;  // that the call is captured into
  if (cudaStreamGetCaptureInfo(st, &cap, nullptr, &graph) != cudaSuccess || cap == cudaStreamCaptureStatusInvalidated) {
    cudaGetLastError();
    return false;
  }
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
  // workspace: the digits, scales and tuples; stream-ordered, so that calls on different
  // streams and threads have their own and nothing outlives the call. A workspace above what
  // the pool keeps is unmapped at the next synchronisation and mapped again by the next call
  // (63 MB, A[300,30^3] with 133 columns, each call synchronised: 2436 us against 2199), so
  // columns that need more are taken in slabs, as long as a slab gives every SM two tiles (in
  // slabs of six tiles that call takes 6529 us).
  const int64_t rows = ka.tiles / ka.ytiles, ytiles = ka.ytiles;
  const int64_t bt = (int64_t)ka.nchunk * KT_CHUNK * 4, bp = (int64_t)ka.nchunk * KT_UPC * 4;
  const int64_t per = (int64_t)ka.nchunk * (4 * KT_WST + KT_COLS * 4 + 8) + rows;  // of a column tile
  const int64_t fit = std::min<int64_t>(32768, std::max<int64_t>((KT_POOL - bt - bp) / per, (2 * sms + rows - 1) / rows));
  const int64_t nslab = (ka.ytiles + fit - 1) / fit, slab = (ka.ytiles + nslab - 1) / nslab;  // column tiles
  const int64_t nd = slab * ka.nchunk, bw = nd * 4 * KT_WST, be = nd * KT_COLS * 4, br = nd * 8;
  unsigned char* ws = nullptr;
  cudaMemPool_t pool = kt_pool(dev);
  const size_t bytes = (size_t)(bw + be + br + bt + bp + slab * rows);
  if (!pool || bw > (2LL << 30) ||
      (graph ? !kt_graph_workspace(pool, dev, graph, bytes, &ws)
             : cudaMallocFromPoolAsync((void**)&ws, bytes, pool, st) != cudaSuccess)) {
    cudaGetLastError();
    return false;  // KC needs no workspace
  }
  if (!graph) kt_reap(dev, st);
  ka.wdig = ws;
  ka.wexp = reinterpret_cast<unsigned*>(ws + bw);
  ka.room = reinterpret_cast<int*>(ws + bw + be);
  ka.vote = reinterpret_cast<unsigned*>(ka.room + nd);
  ka.tix = reinterpret_cast<int*>(ws + bw + be + br);
  ka.pat = reinterpret_cast<int*>(ws + bw + be + br + bt);
  ka.flag = ws + bw + be + br + bt + bp;
  for (int64_t t0 = 0; t0 < ytiles && *e == cudaSuccess; t0 += slab) {
    const int64_t y0 = t0 * KT_COLS;
    ka.W = W + y0;
    ka.C = C + ldc * y0;
    ka.Y = std::min(Y - y0, slab * KT_COLS);
    ka.ytiles = (int)((ka.Y + KT_COLS - 1) / KT_COLS);
    ka.tiles = rows * ka.ytiles;
    const int64_t grid = ka.tiles < sms ? ka.tiles : sms;
    kt_prep_kernel<D><<<dim3((unsigned)ka.nchunk, (unsigned)ka.ytiles), 256, 0, st>>>(kp, ka);
    *e = cudaGetLastError();
    if (*e == cudaSuccess) {
      launch_under(kt_kernel<D>, dim3((unsigned)grid), KT_THREADS, 2 * KT_STAGE, st, kp, ka);
      *e = cudaGetLastError();
    }
    if (*e == cudaSuccess) *e = launch_kc_impl<D, AR_EXACT, true>(kp, ka.W, ka.Y, ldw, ka.C, ldc, st, ka.flag);
  }
  count_launches((int)(3 * nslab - 1));
  if (!graph) {
    const cudaError_t f = cudaFreeAsync(ws, st);
    if (*e == cudaSuccess) *e = f;
  }
  return true;
}

}  // namespace ss
