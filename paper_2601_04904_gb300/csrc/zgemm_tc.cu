// Complex GEMM with FP64-level accuracy on the tcgen05 tensor cores.
//
// GB300's FP64 pipe delivers about 1 TFLOP/s, while its BF16 tensor cores
// deliver ~2 PFLOP/s.  The block products of the sweeps are therefore
// emulated with a modular-integer scheme (the "Ozaki scheme II" of Ozaki,
// Uchino and Imamura, 2025, restated here for complex operands):
//
//   1. scale: for a problem D = beta*C + sum_t alpha_t op(A_t) op(B_t) every
//      row m of the op(A_t) and every column n of the op(B_t) gets one common
//      power-of-two scale 2^e_m, 2^f_n (max over the terms), and the operands
//      are rounded to integers a = round(x 2^(t - e_m)), |a| < 2^t (t <= 62
//      bits, the largest for which the exact integer product fits the CRT
//      range: 58-60 bits for the products here, so that entries well below
//      their row maximum still keep FP64-level precision);
//   2. reduce: each integer is replaced by its residues modulo NMOD = 17
//      pairwise coprime moduli 191 <= p_i <= 256 (M ~ 2^132.95), kept in
//      [-128, 128]; integers of that size are exact in BF16;
//   3. multiply: per modulus, Cr = Ar Br - Ai Bi and Ci = Ar Bi + Ai Br are
//      tensor-core GEMMs with FP32 accumulation in TMEM; every partial sum is an
//      integer of magnitude at most 2^24, so the accumulation is exact (at most
//      1024 products of magnitude <= 2^14 per accumulator; longer K is split
//      into chunks whose residues are added);
//   4. reconstruct: the residues of the exact integer product give it back by
//      the Chinese remainder theorem, C/M = frac(sum_i s_i / p_i) with
//      s_i = r_i y_i mod p_i, y_i = (M/p_i)^{-1} mod p_i, evaluated in 96-bit
//      fixed point (error below 2^-83 of the CRT range); the result is
//      scaled by 2^(e_m + f_n - 2t) and added to beta*C in FP64.
// The only FP64 arithmetic is the final scaling and the beta*C update.
//
// The number of moduli is a parameter of each call: all 17 give FP64-level
// products (QSI_FP64_EMU); a prefix of the list (9..16 moduli, 13 by default
// for QSI_MIXED) shrinks the CRT range, hence t (about 43 bits with 13 moduli
// for the products of the sweeps), and with it the conversion, MMA and
// reconstruction work in proportion.  The error of one product is then about
// 2^-t relative to max|row of A| * max|column of B|.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <mutex>

#include "qsi_internal.h"
#include "tc_common.cuh"

namespace {

constexpr int NMOD = 17;           // moduli of the FP64-accurate scheme (the full list)
constexpr int NMOD_MIN = 9;        // smallest prefix of the list offered
constexpr int NSET = NMOD - NMOD_MIN + 1;
constexpr int NPLANE = 2 * NMOD;  // re/im residue planes per operand (at most)
constexpr int MODS[NMOD] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193, 191};
constexpr int RES_MAX = 128;   // residues are kept in [-128, 128] (operands) / [-128, 127] (int8 results)
constexpr int TBITS_MAX = 62;  // scaled integers are int64
constexpr int NPIECE = 5;      // 13-bit pieces of a scaled integer (65 bits >= TBITS_MAX)
constexpr int PIECE_BITS = 13;

// per-modulus constants (the same for every prefix of the list)
struct CrtConst {
  float p[NMOD];
  float inv_p[NMOD];
  float w[NMOD][NPIECE];         // 2^(13 j) mod p_i, in (-p_i / 2, p_i / 2]
  float2 w2[NMOD][NPIECE];       // (w, w): operands of the packed conversion arithmetic
  float2 inv_p2[NMOD], negp2[NMOD];  // (1/p_i, 1/p_i), (-p_i, -p_i)
};
__constant__ CrtConst c_crt;
// reconstruction constants of the first nm moduli, M = p_0 ... p_{nm-1}
struct CrtSet {
  unsigned H[NMOD][3];           // round(2^96 frac(y_i / p_i)), y_i = (M / p_i)^{-1} mod p_i; 32-bit limbs
  unsigned Hoff[3];              // 2^96 - (128 sum_i H_i mod 2^96): undoes the +128 offset of the residues
  int m_shift;                   // M = m_top * 2^m_shift + (remainder < 2^m_shift)
  unsigned long long m_top;      // the 64 leading bits of M (leading one at bit 63)
  double m_over_2_64;            // M / 2^64
  double log2_m;
};
__constant__ CrtSet c_set[NSET];  // c_set[nm - NMOD_MIN]

constexpr int BM = 128, BN = 128, BK = 64;  // complex output tile, K step (bf16 elements)
constexpr int STAGES = 3;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;  // re and im planes of A and B
constexpr int KPAD = 64;   // row stride of a residue plane: whole 128-byte lines (a box row is one line)
constexpr int CHUNK_KT = 16;  // k-tiles per exact accumulation: 16 * 64 products of magnitude <= 2^14 stay <= 2^24
constexpr int NUM_SMS = 152;
constexpr long long CRT_V4_OUTPUTS = 4ll * 256 * 8 * NUM_SMS;  // reconstruction: four outputs per thread from here on
// Mixed mode (3-term split): each FP64 operand is cut into three BF16 terms
// (the top 24 bits of its mantissa); the six products with i + j <= 2 are
// accumulated in FP32.  Pair groups per CTA:
constexpr int SPLIT_PLANES = 6;  // 3 terms x (re, im)
constexpr int SPLIT_GROUPS = 2;
constexpr int SPLIT_PAIRS = 3;   // pairs per group
__constant__ int c_split_pairs[SPLIT_GROUPS][SPLIT_PAIRS][2] = {{{0, 0}, {0, 1}, {1, 0}}, {{0, 2}, {1, 1}, {2, 0}}};
enum Scheme { SCHEME_CRT = 0, SCHEME_SPLIT3 = 1 };
constexpr int EPI_WARPS = 8;  // two per TMEM lane quarter, each converting one half of the columns
constexpr int THREADS = 64 + 32 * EPI_WARPS;  // producer warp, MMA warp, epilogue warps
constexpr int STAGING_BYTES = 2 * BM * BN;    // int8 residues, re and im
constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + STAGING_BYTES + 1024 + 256;
constexpr int EXP_SENTINEL = (int)0x80808080;  // exponent of a row/column that is all zero

struct TcTerm {
  CUtensorMap ma, mb;  // residue planes [NPLANE][rows][K] (row stride Kp), bf16
  int K, pad[15];
};

struct TcProb {
  TcTerm t[QSI_MAX_TERMS];
  int M, N, nterms, tiles_n, ngroups, cta0;
  int nmod;           // CRT: moduli of this problem (residue planes 2 * nmod per operand)
  int mpc;            // CRT: moduli per CTA (ngroups = ceil(nmod / mpc))
  int ctas_per_b;     // CTAs of one batch entry (tiles x ngroups)
  int stage_bytes;    // bytes of the four boxes of a pipeline stage
  int ldr;            // CRT: row length of res (N rounded up to 16)
  long long out_bs;   // batch stride of res / part (elements)
  int8_t *res;        // CRT: residues [batch][nmod][2][M][ldr]
  float *part;        // SPLIT3: FP32 partial products [batch][SPLIT_GROUPS][2][M][N]
};

struct TcGroup {
  TcProb p[QSI_MAX_PROB];
  int nprob, total_ctas;
};

// --------------------------------------------------------------------------
// conversion helpers (integer arithmetic on the FP64 bit pattern)
// --------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// |round(x * 2^(t - e))| for |x| < 2^e (below 2^t), and its sign (the sign
// bit of x) in neg: the magnitude and sign of the scaled integer.
__device__ __forceinline__ unsigned long long scaled_mag(double x, int e, int t, bool &neg) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  neg = (b >> 63) != 0;
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) return 0;
  const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = E - 1075 + t - e;
  if (sh >= 0) return mant << min(sh, 10);
  if (sh <= -64) return 0;
  return (mant + (1ull << (-sh - 1))) >> (-sh);
}

// d = a * b + c and d = a + b on two FP32 lanes at once (packed f32x2
// arithmetic of sm_100+; each lane rounds exactly like fmaf / __fadd_rn)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*(const unsigned long long *)&a), "l"(*(const unsigned long long *)&b),
        "l"(*(const unsigned long long *)&c));
  return *(const float2 *)&d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(*(const unsigned long long *)&a), "l"(*(const unsigned long long *)&b));
  return *(const float2 *)&d;
}

// One launch converts every operand of a grouped product: a job per side of a
// problem, all of its terms together (they share the rows' exponents).
struct ConvTerm {
  const zc *X;
  long long ld, sX;         // leading dimension, batch stride (elements)
  __nv_bfloat16 *planes;
  long long pl_bs;          // batch stride of the planes (bf16 elements)
  int K, Kp;                // depth, row stride of the planes (K rounded up to 64)
  int tile0;                // the term's first 64-k tile among the job's
  int row_contig, conj, negate;
};
struct ConvJob {
  ConvTerm t[QSI_MAX_TERMS];
  int *eexp;                // CRT: exponent bound per row of the op(X), one array per batch entry (R ints)
  int R, nterms, ntiles;
  int blk0, nblk;           // first cluster of this job in the launch, clusters per batch entry
  int tbits, nmod;          // CRT: bits of the scaled integers, moduli (residue planes 2 * nmod)
};
constexpr int MAX_JOBS = 2 * QSI_MAX_PROB;
struct ConvJobs {
  ConvJob j[MAX_JOBS];
  int njobs;
  int cs, keep;             // CTAs per cluster, tiles a CTA keeps in shared memory
};

// ---------------------------------------------------------------------------
// 1. and 2. exponents and residue planes, one pass over the operands.
//    e_r = the FP64 exponent bound (|x| < 2^e_r) of row r of the op(X) over all
//    terms; planes[2i + c][r][k] (bf16) = residue mod p_i of the scaled integer
//    of Re (c = 0) / Im (c = 1) of s * op(X)[r][k], r < R, k < K (row stride Kp,
//    K rounded up to 64, so that every row of a box is one 128-byte line: with
//    rows of 1040 bytes the products at K = 520 took 33.3 instead of 31.3 us).
//    The padding is never written: the maps end at R rows and K columns, and TMA
//    fills the rest of a box with zeros.  At b = 46 that leaves out 4 of 5 bytes
//    of the planes padded to whole boxes.  s = -1 when negate, op(X) conjugated
//    when conj; row_contig: op(X)[r][k] = X[r ld + k], else X[k ld + r].
//
//    A cluster takes 16 rows: its CTAs load the rows' 16 x 64 tiles in turn into
//    shared memory (coalesced either way), take the rows' maxima as they pass,
//    exchange them through distributed shared memory, and convert the tiles they
//    hold (those beyond J.keep are read again).  A separate scan, with the memset
//    its atomics needed, was two more launches per group, 8 to 9 us of every
//    group's chain, and a second read of every operand.
// ---------------------------------------------------------------------------
constexpr int CV_R = 16, CV_K = 64;  // tile: rows x k, four consecutive k of one row per thread
constexpr int CV_G = 18;             // tile column of k: (k & 3) * CV_G + (k >> 2), free of bank conflicts both ways
constexpr int CV_TILE = CV_R * 4 * CV_G;  // elements of a tile
constexpr int CV_MAXCS = 8, CV_MAXKEEP = 4;

// order-preserving 32-bit key of |x|: its exponent in bits 20.., nonzero unless x = 0
__device__ __forceinline__ unsigned mag_key(double x) {
  const unsigned long long b = abs_bits(x);
  return (unsigned)(b >> 32) | ((unsigned)b != 0u ? 1u : 0u);
}

constexpr int CV_PER = CV_R * CV_K / 256;  // elements of a tile per thread

// row and k within the tile of a thread's element it
__device__ __forceinline__ void tile_pos(const ConvTerm &T, int it, int &r, int &k) {
  const int idx = threadIdx.x + 256 * it;
  r = T.row_contig ? idx / CV_K : idx % CV_R;
  k = T.row_contig ? idx % CV_K : idx / CV_R;
}

// this thread's elements of the op(X) tile at (r0, k0), zero outside R x K
__device__ __forceinline__ void load_tile(zc (&v)[CV_PER], const ConvTerm &T, const zc *X, int R, int r0, int k0) {
#pragma unroll
  for (int it = 0; it < CV_PER; ++it) {
    int r, k;
    tile_pos(T, it, r, k);
    v[it] = make_double2(0.0, 0.0);
    if (r0 + r < R && k0 + k < T.K)
      v[it] = T.row_contig ? X[(long long)(r0 + r) * T.ld + k0 + k] : X[(long long)(k0 + k) * T.ld + r0 + r];
  }
}
__device__ __forceinline__ void keep_tile(zc *dst, const zc (&v)[CV_PER], const ConvTerm &T) {
#pragma unroll
  for (int it = 0; it < CV_PER; ++it) {
    int r, k;
    tile_pos(T, it, r, k);
    dst[r * 4 * CV_G + (k & 3) * CV_G + (k >> 2)] = v[it];
  }
}
// maxima of the rows' keys -> s_key
__device__ __forceinline__ void tile_keys(unsigned *s_key, const zc (&v)[CV_PER], const ConvTerm &T) {
  unsigned cm = 0;
#pragma unroll
  for (int it = 0; it < CV_PER; ++it) {
    const unsigned key = max(mag_key(v[it].x), mag_key(v[it].y));
    if (T.row_contig) {  // a warp's 32 elements share the row
      const unsigned m = __reduce_max_sync(0xffffffffu, key);
      if ((threadIdx.x & 31) == 0 && m != 0u) atomicMax(&s_key[(threadIdx.x + 256 * it) / CV_K], m);
    } else {
      cm = max(cm, key);  // a thread's elements share the row
    }
  }
  if (!T.row_contig) {
    cm = max(cm, __shfl_xor_sync(0xffffffffu, cm, 16));
    if ((threadIdx.x & 31) < 16 && cm != 0u) atomicMax(&s_key[threadIdx.x & 15], cm);
  }
}

__device__ __forceinline__ float pow2f(int k) {
  if (k < -126) return 0.f;
  if (k > 127) return INFINITY;
  return __int_as_float((k + 127) << 23);
}

__device__ __forceinline__ void split3(double x, float (&t)[3]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) {
    t[0] = t[1] = t[2] = 0.f;
    return;
  }
  const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int ex = E - 1023;  // x = mant * 2^(ex - 52)
  const float sgn = (b >> 63) ? -1.f : 1.f;
  t[0] = sgn * (float)(unsigned)(mant >> 45) * pow2f(ex - 7);
  t[1] = sgn * (float)(unsigned)((mant >> 37) & 0xFF) * pow2f(ex - 15);
  t[2] = sgn * (float)(unsigned)((mant >> 29) & 0xFF) * pow2f(ex - 23);
}

// 2b. mixed mode (3-term split): three BF16 terms per real number,
//     planes[2s + c][r][k]; four consecutive k of one row
__device__ __forceinline__ void split_four(const zc (&x)[4], const ConvTerm &T, uint2 *out, long long qplane) {
  float t[2][4][3];  // [re, im][k][term]
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    double re = x[h].x, im = T.conj ? -x[h].y : x[h].y;
    if (T.negate) {
      re = -re;
      im = -im;
    }
    split3(re, t[0][h]);
    split3(im, t[1][h]);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(t[c][0][q], t[c][1][q]),
                           hi = __floats2bfloat162_rn(t[c][2][q], t[c][3][q]);
      out[(2 * q + c) * qplane] = make_uint2(*(const unsigned *)&lo, *(const unsigned *)&hi);
    }
}

// residues of four consecutive k of one row, as two pairs that share every
// instruction of the residue arithmetic (packed lanes .x, .y); each modulus's
// constants are loaded once for the four pair streams (2 pairs x re, im).
// NM: moduli (0: nmod at run time), NP: 13-bit pieces that cover tbits + 1
template <int NM, int NP>
__device__ __forceinline__ void convert_four(const zc (&x)[4], int e, int tbits, const ConvTerm &T, int nmod,
                                             uint2 *out, long long qplane) {
  float2 pc[2][2][NP];  // [pair][re, im][piece]
  const int nm = NM > 0 ? NM : nmod;
#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {
    // magnitudes and signs of the scaled integers; conj and negate flip the
    // signs (integer ops, not FP64 negations); zero beyond K (loaded as zero)
    unsigned long long mg[2][2];  // [element][re, im]
    bool ng[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const zc v = x[2 * pr + h];
      mg[h][0] = scaled_mag(v.x, e, tbits, ng[h][0]);
      mg[h][1] = scaled_mag(v.y, e, tbits, ng[h][1]);
      ng[h][0] = ng[h][0] != (T.negate != 0);
      ng[h][1] = ng[h][1] != ((T.conj != 0) != (T.negate != 0));
    }
    // signed 13-bit pieces: a = sum_j piece_j 2^(13 j), the sign of a folded
    // into every piece (converted through 32-bit integers: a conversion from
    // a 64-bit integer would run on the FP64 unit)
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float sg = ng[h][c] ? -1.0f : 1.0f;
        const unsigned long long u = mg[h][c];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          const float pj = sg * (float)(unsigned)((u >> (PIECE_BITS * j)) & ((1ull << PIECE_BITS) - 1ull));
          if (h == 0)
            pc[pr][c][j].x = pj;
          else
            pc[pr][c][j].y = pj;
        }
      }
  }
#pragma unroll
  for (int i = 0; i < (NM > 0 ? NM : NMOD); ++i) {
    if (NM == 0 && i >= nm) break;
    // s = sum_j piece_j w_ij with |w_ij| <= 128: |s| <= 8191 (1 + 4 * 128)
    // < 2^23, every partial sum exact in FP32.  One FMA against 1.5 * 2^23
    // rounds s * fl(1/p_i) to the nearest integer q; as |s / p_i| < 2^15,
    // fl(1/p_i) moves it by less than 0.0013, so r = s - q p_i (exact) has
    // |r| <= 0.5013 p_i, i.e. |r| <= 128 for every modulus here (exact in
    // BF16, and the bound the MMA chunks assume).
    float2 w[NP];
#pragma unroll
    for (int j = 1; j < NP; ++j) w[j] = c_crt.w2[i][j];
    const float2 ip = c_crt.inv_p2[i], np = c_crt.negp2[i];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      unsigned o[2];
#pragma unroll
      for (int pr = 0; pr < 2; ++pr) {
        float2 sv = pc[pr][c][0];
#pragma unroll
        for (int j = 1; j < NP; ++j) sv = ffma2(pc[pr][c][j], w[j], sv);
        const float2 q = fadd2(ffma2(sv, ip, make_float2(12582912.0f, 12582912.0f)),
                               make_float2(-12582912.0f, -12582912.0f));
        const float2 res = ffma2(q, np, sv);
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(res.x, res.y);
        o[pr] = *(const unsigned *)&b2;
      }
      out[(2 * i + c) * qplane] = make_uint2(o[0], o[1]);
    }
  }
}

// NM > 0: that many moduli, 0: the job's count, -1: the 3-term split (no exponents)
template <int NM, int NP>
__global__ void __launch_bounds__(256) tc_convert_kernel(const __grid_constant__ ConvJobs J) {
  extern __shared__ zc tiles[];  // J.keep tiles
  __shared__ unsigned s_key[CV_R], s_all[CV_R];  // this CTA's rows' maxima, the cluster's
  const int cs = J.cs, rank = blockIdx.x % cs, cl = blockIdx.x / cs, tid = threadIdx.x;
  tc::pdl_wait();
  int ji = 0;
  while (ji + 1 < J.njobs && cl >= J.j[ji + 1].blk0) ++ji;
  const ConvJob &job = J.j[ji];
  const int bi = (cl - job.blk0) / job.nblk, r0 = ((cl - job.blk0) % job.nblk) * CV_R;
  const int R = job.R, r = tid >> 4, kq = tid & 15, gr = r0 + r;
  // term of tile tl
  auto term_of = [&](int tl) -> const ConvTerm & {
    int t = 0;
    while (t + 1 < job.nterms && tl >= job.t[t + 1].tile0) ++t;
    return job.t[t];
  };
  int e = 0;
  if (NM >= 0) {
    if (tid < CV_R) s_key[tid] = s_all[tid] = 0u;
    __syncthreads();
    zc v[CV_PER];
    if (rank < job.ntiles) {
      const ConvTerm &T = term_of(rank);
      load_tile(v, T, T.X + bi * T.sX, R, r0, (rank - T.tile0) * CV_K);
    }
#pragma unroll 1
    for (int tl = rank, slot = 0; tl < job.ntiles; tl += cs, ++slot) {
      zc nv[CV_PER];  // the next tile's loads are in flight meanwhile
      if (tl + cs < job.ntiles) {
        const ConvTerm &N = term_of(tl + cs);
        load_tile(nv, N, N.X + bi * N.sX, R, r0, (tl + cs - N.tile0) * CV_K);
      }
      const ConvTerm &T = term_of(tl);
      if (slot < J.keep) keep_tile(tiles + slot * CV_TILE, v, T);
      tile_keys(s_key, v, T);
#pragma unroll
      for (int it = 0; it < CV_PER; ++it) v[it] = nv[it];
    }
    __syncthreads();
    unsigned key = 0;
    if (cs > 1) {
      tc::cluster_sync();
      if (tid < CV_R * cs) {
        unsigned a, v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(a)
                     : "r"(tc::su32(&s_key[tid % CV_R])), "r"(tid / CV_R));
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
        if (v != 0u) atomicMax(&s_all[tid % CV_R], v);
      }
      // no CTA leaves (or reuses s_key) while another may still read it: waited for at the end
      tc::cluster_arrive();
      __syncthreads();
      key = s_all[r];
    } else {
      key = s_key[r];
    }
    e = key != 0u ? (int)(key >> 20) - 1022 : EXP_SENTINEL;
    if (rank == 0 && kq == 0 && gr < R) job.eexp[(long long)bi * R + gr] = e;
  }
#pragma unroll 1
  for (int tl = rank, slot = 0; tl < job.ntiles; tl += cs, ++slot) {
    const ConvTerm &T = term_of(tl);
    const int k0 = (tl - T.tile0) * CV_K, gk = k0 + 4 * kq;
    zc *tile = tiles + min(slot, J.keep - 1) * CV_TILE;
    if (NM < 0 || slot >= J.keep) {
      __syncthreads();
      zc v[CV_PER];
      load_tile(v, T, T.X + bi * T.sX, R, r0, k0);
      keep_tile(tile, v, T);
      __syncthreads();
    }
    if (gr >= R || gk >= T.K) continue;  // Kp is a multiple of 64: four values stay inside the row
    const long long qplane = (long long)R * T.Kp / 4;  // one plane in groups of four
    uint2 *out = (uint2 *)(T.planes + bi * T.pl_bs + (long long)gr * T.Kp + gk);
    zc x[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) x[h] = tile[r * 4 * CV_G + h * CV_G + kq];
    if (NM < 0)
      split_four(x, T, out, qplane);
    else
      convert_four<NM < 0 ? 0 : NM, NP>(x, e, job.tbits, T, job.nmod, out, qplane);
  }
  if (NM >= 0 && cs > 1) tc::cluster_wait();
}

// ---------------------------------------------------------------------------
// 3. tensor-core products per modulus -> int8 residues of the exact integer
//    product.  One CTA: one 128 x 128 complex output tile, mpc moduli (chosen
//    per launch so that the CTAs fill the SMs in as few waves as possible).
//    Warp 0: TMA producer; warp 1: TMEM owner + MMA issuer; warps 2..9:
//    epilogue (TMEM -> residues -> shared staging -> coalesced global stores).
//    TMEM: two buffers x (Cr | Ci), 4 x 128 columns.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int reduce_res(float v, int i) {
  // representative of v mod p_i in [-128, 127] (fits int8): the rounded
  // quotient leaves |r| <= p_i/2 + 1, one correction step folds it in
  int r = (int)(v - rintf(v * c_crt.inv_p[i]) * c_crt.p[i]);
  const int p = (int)c_crt.p[i];
  if (r > RES_MAX - 1) r -= p;
  if (r < -RES_MAX) r += p;
  return r;
}

// (term, k-tile) of linear k-tile index j over the terms of a problem
__device__ __forceinline__ void locate_kt(const TcProb &P, int j, int &t, int &kt) {
  t = 0;
  while (t + 1 < P.nterms) {
    const int nkt = (P.t[t].K + BK - 1) / BK;
    if (j < nkt) break;
    j -= nkt;
    ++t;
  }
  kt = j;
}

template <int SCHEME>
__global__ void __launch_bounds__(THREADS, 1) tc_mma_kernel(const __grid_constant__ TcGroup g, int *err) {
  using namespace tc;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *staging = smem + STAGES * STAGE_BYTES;
  uint64_t *full = (uint64_t *)(staging + STAGING_BYTES);
  uint64_t *empty = full + STAGES;
  uint64_t *accf = empty + STAGES;     // [2] MMA -> epilogue
  uint64_t *accfree = accf + 2;        // [2] epilogue -> MMA
  uint32_t *tslot = (uint32_t *)(accfree + 2);
  volatile int *abort_flag = (volatile int *)(tslot + 1);
  volatile int *epi_ok = (volatile int *)(tslot + 2);  // [EPI_WARPS]

  // locate problem / tile / modulus group
  int pi = 0;
  while (pi + 1 < g.nprob && (int)blockIdx.x >= g.p[pi + 1].cta0) ++pi;
  const TcProb &P = g.p[pi];
  const int lcta = blockIdx.x - P.cta0;
  const int bi = lcta / P.ctas_per_b;  // batch entry: residue planes bi * nplanes.., outputs bi * out_bs..
  const int local = lcta - bi * P.ctas_per_b;
  const int grp = local % P.ngroups, tile = local / P.ngroups;
  const int zoff = bi * (SCHEME == SCHEME_CRT ? 2 * P.nmod : SPLIT_PLANES);
  const int m0 = (tile / P.tiles_n) * BM, n0 = (tile % P.tiles_n) * BN;
  const int mod_lo = grp * P.mpc, mod_hi = min(P.nmod, mod_lo + P.mpc);
  // columns of this tile that exist, rounded up to the MMA's step of 16: the
  // products and the epilogue leave out the rest (and the k beyond a term's K,
  // in steps of 16)
  const int ncol = min(BN, (P.N - n0 + 15) & ~15);

  // accumulation units.  CRT: (modulus, chunk), chunks of at most CHUNK_KT
  // k-tiles over all terms.  SPLIT3: one unit, SPLIT_PAIRS x all k-tiles.
  int kt_total = 0;
  for (int t = 0; t < P.nterms; ++t) kt_total += (P.t[t].K + BK - 1) / BK;
  const int chunks = (kt_total + CHUNK_KT - 1) / CHUNK_KT;
  const int units = SCHEME == SCHEME_CRT ? (mod_hi - mod_lo) * chunks : (kt_total > 0 ? 1 : 0);
  auto unit_stages = [&](int u) {
    if (SCHEME == SCHEME_CRT) {
      const int ch = u % chunks;
      return min(kt_total, (ch + 1) * CHUNK_KT) - ch * CHUNK_KT;
    }
    return SPLIT_PAIRS * kt_total;
  };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ew = warp - 2;  // epilogue warp index 0..EPI_WARPS-1
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&accfree[b], EPI_WARPS);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tslot, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = *tslot;
  pdl_wait();  // the operands' planes are complete

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    int it = 0, issued = 0;
    for (int u = 0; u < units && !*abort_flag; ++u) {
      const int nst = unit_stages(u);
      for (int k = 0; k < nst; ++k) {
        int t, kt, za, zb;
        if (SCHEME == SCHEME_CRT) {
          const int mod = mod_lo + u / chunks, ch = u % chunks;
          locate_kt(P, ch * CHUNK_KT + k, t, kt);
          za = zb = mod;
        } else {
          const int pr = k / kt_total;
          locate_kt(P, k % kt_total, t, kt);
          za = c_split_pairs[grp][pr][0];
          zb = c_split_pairs[grp][pr][1];
        }
        const int s = it % STAGES;
        if (it >= STAGES && !mbar_wait(&empty[s], ((it / STAGES) - 1) & 1)) {
          *abort_flag = 1;
          atomicExch(err, 1);
          break;
        }
        uint8_t *st = smem + s * STAGE_BYTES;
        mbar_expect_tx(&full[s], P.stage_bytes);
        tma_load_3d(st, &P.t[t].ma, &full[s], kt * BK, m0, zoff + 2 * za);
        tma_load_3d(st + A_BYTES, &P.t[t].ma, &full[s], kt * BK, m0, zoff + 2 * za + 1);
        tma_load_3d(st + 2 * A_BYTES, &P.t[t].mb, &full[s], kt * BK, n0, zoff + 2 * zb);
        tma_load_3d(st + 2 * A_BYTES + B_BYTES, &P.t[t].mb, &full[s], kt * BK, n0, zoff + 2 * zb + 1);
        ++it;
        ++issued;
      }
    }
    // wait for every copy issued (they complete without the consumer)
    for (int k = (issued > STAGES ? issued - STAGES : 0); k < issued; ++k)
      if (!mbar_wait(&full[k % STAGES], (k / STAGES) & 1)) atomicExch(err, 2);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    const uint32_t ID_POS = idesc_bf16_f32(BM, ncol, false), ID_NEG = idesc_bf16_f32(BM, ncol, true);
    int it = 0;
    for (int u = 0; u < units; ++u) {
      const int buf = u & 1;
      if (u >= 2 && !mbar_wait(&accfree[buf], ((u >> 1) - 1) & 1)) {
        *abort_flag = 1;
        atomicExch(err, 3);
        break;
      }
      fence_after();
      const uint32_t d_re = tbase + buf * 2 * BN, d_im = d_re + BN;
      const int nst = unit_stages(u);
      bool ok = true;
      int t, kt;  // term and k-tile of this stage
      locate_kt(P, SCHEME == SCHEME_CRT ? (u % chunks) * CHUNK_KT : 0, t, kt);
      int krem = P.t[t].K - kt * BK;  // k left in the term
      for (int k = 0; k < nst; ++k, ++it) {
        const int s = it % STAGES;
        if (!mbar_wait(&full[s], (it / STAGES) & 1)) {
          ok = false;
          break;
        }
        fence_after();
        const uint32_t sa_re = su32(smem + s * STAGE_BYTES);
        // descriptors of the four operand tiles; a step of 16 k is 32 bytes (2 units) on
        const uint64_t ar = sdesc_sw128(sa_re), ai = sdesc_sw128(sa_re + A_BYTES),
                       br = sdesc_sw128(sa_re + 2 * A_BYTES), bi_ = sdesc_sw128(sa_re + 2 * A_BYTES + B_BYTES);
        auto step = [&](int kk) {
          const uint32_t acc = (k | kk) != 0;
          umma_bf16(d_re, ar + 2 * kk, br + 2 * kk, ID_POS, acc);
          umma_bf16(d_re, ai + 2 * kk, bi_ + 2 * kk, ID_NEG, 1);
          umma_bf16(d_im, ar + 2 * kk, bi_ + 2 * kk, ID_POS, acc);
          umma_bf16(d_im, ai + 2 * kk, br + 2 * kk, ID_POS, 1);
        };
        if (krem >= BK) {  // a whole k-tile: no branches between the products
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) step(kk);
        } else {
#pragma unroll 1
          for (int kk = 0; kk * 16 < krem; ++kk) step(kk);
        }
        krem -= BK;
        if (krem <= 0 && k + 1 < nst) {  // next term (SPLIT3: or the next pair's first)
          t = t + 1 < P.nterms ? t + 1 : 0;
          krem = P.t[t].K;
        }
        umma_commit(&empty[s]);
      }
      umma_commit(&accf[buf]);
      if (!ok) {
        *abort_flag = 1;
        atomicExch(err, 4);
        break;
      }
    }
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int q = warp & 3;  // TMEM lane quarter (a warp reads the lanes of warp index mod 4)
    const int row = q * 32 + lane;
    const int col0 = (ew >> 2) * (BN / 2);  // this warp's half of the accumulator columns
    const long long MN = (long long)P.M * P.N;
    for (int u = 0; u < units; ++u) {
      const int buf = u & 1;
      bool ok = mbar_wait(&accf[buf], (u >> 1) & 1);
      fence_after();
      ok = __all_sync(0xffffffffu, ok && !*abort_flag);
      // all epilogue warps take the same decision before any further barrier
      if (lane == 0) epi_ok[ew] = ok ? 1 : 0;
      named_sync(1, 32 * EPI_WARPS);
      bool all_ok = true;
#pragma unroll
      for (int w = 0; w < EPI_WARPS; ++w) all_ok = all_ok && epi_ok[w];
      if (!all_ok) {
        if (lane == 0) atomicExch(err, 5);
        break;
      }
      if (SCHEME == SCHEME_SPLIT3) {
        // FP32 partial products: 32 columns at a time through the staging
        // buffer (a warp's 32 rows x 32 floats, rows XOR-swizzled by 16-byte
        // chunk), then stored row by row, 128 contiguous bytes per warp store
        float *stg = (float *)staging + ew * 32 * 32;  // this warp's 4 KB
        for (int c = 0; c < 2; ++c) {
          float *gpl = P.part + bi * P.out_bs + ((long long)grp * 2 + c) * MN;
#pragma unroll 1
          for (int col = col0; col < min(ncol, col0 + BN / 2); col += 32) {
            uint32_t r[32];
            tmem_ld32(tbase + ((uint32_t)(q * 32) << 16) + buf * 2 * BN + c * BN + col, r);
            tmem_wait_ld();
#pragma unroll
            for (int ck = 0; ck < 8; ++ck)
              *(uint4 *)(stg + lane * 32 + 4 * (ck ^ (lane & 7))) =
                  make_uint4(r[4 * ck], r[4 * ck + 1], r[4 * ck + 2], r[4 * ck + 3]);
            __syncwarp();
            // row rr of this warp's quarter; lane = column
            const int n = n0 + col + lane;
#pragma unroll 4
            for (int rr = 0; rr < 32; ++rr) {
              const int m = m0 + q * 32 + rr;
              const float v = stg[rr * 32 + 4 * ((lane >> 2) ^ (rr & 7)) + (lane & 3)];
              if (m < P.M && n < P.N) gpl[(long long)m * P.N + n] = v;
            }
            __syncwarp();
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&accfree[buf]);
        continue;
      }
      const int mod = mod_lo + u / chunks, ch = u % chunks;
      // TMEM -> residues -> staging[c][row][col] (rows and columns that exist)
      const int cend = m0 + q * 32 < P.M ? min(ncol, col0 + BN / 2) : 0;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
#pragma unroll 1
        for (int col = col0; col < cend; col += 32) {
          uint32_t r[32];
          tmem_ld32(tbase + ((uint32_t)(q * 32) << 16) + buf * 2 * BN + c * BN + col, r);
          tmem_wait_ld();
          // residues of the exact integer sums (|v| <= 2^24), two per packed
          // instruction: q = v * fl(1/p) rounded to an integer by one FMA
          // against 1.5 * 2^23, x = v - q p (exact), |x| <= 0.5052 p, so x is
          // in [-128, 127] except x = 128 for p = 256 (whose byte -128 is the
          // same residue) and p = 255 (folded to -127); the byte of x is the
          // low byte of x + 1.5 * 2^23
          const float2 ip = c_crt.inv_p2[mod], np = c_crt.negp2[mod];
          const bool p255 = c_crt.p[mod] == 255.0f;
          uint32_t packed[8];
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            uint32_t bits[4];
#pragma unroll
            for (int h = 0; h < 4; h += 2) {
              const float2 v2 = make_float2(__uint_as_float(r[4 * w + h]), __uint_as_float(r[4 * w + h + 1]));
              const float2 q2 = fadd2(ffma2(v2, ip, make_float2(12582912.0f, 12582912.0f)),
                                      make_float2(-12582912.0f, -12582912.0f));
              float2 x2 = ffma2(q2, np, v2);
              if (p255) {
                x2.x = x2.x > 127.5f ? x2.x - 255.0f : x2.x;
                x2.y = x2.y > 127.5f ? x2.y - 255.0f : x2.y;
              }
              const float2 m2 = fadd2(x2, make_float2(12582912.0f, 12582912.0f));
              bits[h] = __float_as_uint(m2.x);
              bits[h + 1] = __float_as_uint(m2.y);
            }
            packed[w] = __byte_perm(__byte_perm(bits[0], bits[1], 0x0040), __byte_perm(bits[2], bits[3], 0x0040),
                                    0x5410);
          }
          // 16-byte chunks of a staging row are XOR-swizzled by (row & 7), so
          // that the 32 rows of a warp do not all hit the same banks
          uint8_t *srow_ = staging + c * BM * BN + row * BN;
          *(uint4 *)(srow_ + 16 * ((col / 16) ^ (row & 7))) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
          *(uint4 *)(srow_ + 16 * ((col / 16 + 1) ^ (row & 7))) =
              make_uint4(packed[4], packed[5], packed[6], packed[7]);
        }
      }
      // the accumulator buffer may be reused once every epilogue warp has read it
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accfree[buf]);
      named_sync(1, 32 * EPI_WARPS);  // staging complete (epilogue warps only)
      {
        // 16 bytes per lane, four rows per warp instruction (whole 32-byte
        // sectors): rows of res are a multiple of 16 long, so the last 16
        // columns of a ragged tile are stored whole
        const int sub = lane >> 3, kq = lane & 7;
        const int rows = min(BM, P.M - m0);
        if (16 * kq < ncol)
          for (int c = 0; c < 2; ++c) {
            int8_t *gres = P.res + bi * P.out_bs + ((long long)mod * 2 + c) * P.M * P.ldr;
            for (int rr = 4 * ew + sub; rr < rows; rr += 4 * EPI_WARPS) {
              uint4 v = *(const uint4 *)(staging + c * BM * BN + rr * BN + 16 * (kq ^ (rr & 7)));
              uint4 *pdst = (uint4 *)(gres + (long long)(m0 + rr) * P.ldr + n0 + 16 * kq);
              if (ch > 0) {  // add the earlier chunk's residues, modulo p
                const uint4 o = *pdst;
                const uint32_t nv[4] = {v.x, v.y, v.z, v.w}, ov[4] = {o.x, o.y, o.z, o.w};
                uint32_t outw[4];
#pragma unroll
                for (int wq = 0; wq < 4; ++wq) {
                  uint32_t pk = 0;
#pragma unroll
                  for (int bb = 0; bb < 4; ++bb) {
                    const int a = (int)(int8_t)(nv[wq] >> (8 * bb)), b2 = (int)(int8_t)(ov[wq] >> (8 * bb));
                    pk |= ((uint32_t)(uint8_t)(int8_t)reduce_res((float)(a + b2), mod)) << (8 * bb);
                  }
                  outw[wq] = pk;
                }
                v = make_uint4(outw[0], outw[1], outw[2], outw[3]);
              }
              *pdst = v;
            }
          }
      }
      named_sync(1, 32 * EPI_WARPS);  // staging may be overwritten
    }
  }
  __syncwarp();  // the producer's and the issuer's lane rejoin their warps
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tbase, 512);
  }
}

// ---------------------------------------------------------------------------
// 4. CRT reconstruction + scaling + beta*C, one thread per complex element.
// ---------------------------------------------------------------------------
struct CrtJob {
  const int8_t *res;
  const int *ea, *eb;
  const zc *C;
  zc *D;
  long long ldc, ldd;
  long long res_bs, sC, sD;  // batch strides (res: elements; C, D: complex elements)
  zc beta;
  int M, N, tbits, elem0;    // elem0: first unit of this job (batch x M rows of ceil(N / V) units)
  int nmod, ldr;             // ldr: row length of res
  int add;                   // beta C: 0 none, 1 C (beta = 1), 2 any beta
};
struct CrtJobs {
  CrtJob j[QSI_MAX_PROB];
  int njobs, total;
};

__device__ __forceinline__ double pow2(int k) {
  if (k < -1022) return 0.0;
  if (k > 1023) return INFINITY;
  return __longlong_as_double((long long)(k + 1023) << 52);
}

// top * M * 2^(s - 64) as a double, rounded to nearest-even from the 128-bit
// product of top (leading one at bit 63) and the 64 leading bits of M
// (relative truncation error of M below 2^-63).  Falls back to FP64
// arithmetic outside the normal exponent range.
__device__ __forceinline__ double crt_to_double(const CrtSet &cs, unsigned long long top, int s, bool neg) {
  const unsigned long long lo = top * cs.m_top, hi = __umul64hi(top, cs.m_top);
  const int hb = 126 + (int)(hi >> 63);  // the product is in [2^126, 2^128)
  const int sh = hb - 116;               // m53 = P >> (hb - 52) = hi >> sh (sh = 10 or 11)
  unsigned long long m53 = hi >> sh;
  const bool rnd = (hi >> (sh - 1)) & 1ull;
  const bool sticky = ((hi & ((1ull << (sh - 1)) - 1ull)) | lo) != 0ull;
  int E = hb + cs.m_shift - 64 + s;  // value = 1.f * 2^E
  if (rnd && (sticky || (m53 & 1ull))) {
    ++m53;
    if (m53 == (1ull << 53)) {
      m53 >>= 1;
      ++E;
    }
  }
  if (E < -1022 || E > 1023) {
    const double d = (double)top * cs.m_over_2_64 * pow2(s);
    return neg ? -d : d;
  }
  const unsigned long long bits =
      ((unsigned long long)neg << 63) | ((unsigned long long)(E + 1023) << 52) | (m53 & ((1ull << 52) - 1ull));
  return __longlong_as_double((long long)bits);
}

// V consecutive elements of one row per thread (the residues of a plane load as
// one word: rows of res are padded to 16; elements beyond N are not stored).
// frac(sum_i s_i / p_i) with s_i = r_i y_i mod p_i equals frac(sum_i r_i y_i / p_i):
// every residue byte, offset by 128 to [0, 255], multiplies the 96-bit
// frac(y_i / p_i) directly, and one constant removes the offset.
// NM: moduli (0: job.nmod at run time; a launch's jobs share one count).
template <int V, int NM>
__global__ void __launch_bounds__(256) tc_crt_kernel(const __grid_constant__ CrtJobs J) {
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;  // unit of V elements
  tc::pdl_wait();
  if (gid >= J.total) return;
  int ji = 0;
  while (ji + 1 < J.njobs && gid >= J.j[ji + 1].elem0) ++ji;
  const CrtJob &job = J.j[ji];
  const int nm = NM > 0 ? NM : job.nmod;
  const CrtSet &cs = c_set[nm - NMOD_MIN];
  const int rowu = (job.N + V - 1) / V, local = gid - job.elem0;
  const int row = local / rowu, n = (local - row * rowu) * V;
  const int bi = row / job.M, m = row - bi * job.M;
  const long long MN = (long long)job.M * job.ldr;  // one residue plane
  const int ea = job.ea ? job.ea[bi * job.M + m] : EXP_SENTINEL;
  const int8_t *res = job.res + bi * job.res_bs + (long long)m * job.ldr + n;
  int eb[V];
  bool zero[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    eb[v] = job.eb && n + v < job.N ? job.eb[bi * job.N + n + v] : EXP_SENTINEL;
    zero[v] = ea == EXP_SENTINEL || eb[v] == EXP_SENTINEL;  // (ea, eb NULL: no product term)
  }
  zc out[V];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    // frac(sum_i (r_i + 128) y_i / p_i) in 96-bit fixed point: one 32 x 32
    // -> 64-bit multiply-add per limb and modulus (each limb sum < 2^45),
    // carries propagated once, then the offset removed modulo 2^96.  The
    // rounding of the nm <= 17 constants moves the fraction by less than
    // 2^-84, i.e. below 2^-(84 - log2 M + 2t) of the product's scale 2^(2t):
    // 2^-70 for 17 moduli (t >= 58), 2^-67 for 13 (t <= 43).
    unsigned long long a0[V], a1[V], a2[V];
#pragma unroll
    for (int v = 0; v < V; ++v) a0[v] = a1[v] = a2[v] = 0;
#pragma unroll
    for (int i = 0; i < (NM > 0 ? NM : NMOD); ++i) {
      if (NM == 0 && i >= nm) break;
      const int8_t *pl = res + ((long long)i * 2 + c) * MN;
      unsigned word;
      if (V == 4)
        word = *(const unsigned *)pl;
      else if (V == 2)
        word = (unsigned)*(const unsigned short *)pl;
      else
        word = (unsigned)(unsigned char)pl[0];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const unsigned ru = ((word >> (8 * v)) & 255u) ^ 128u;  // int8 residue + 128
        a0[v] += (unsigned long long)ru * cs.H[i][0];
        a1[v] += (unsigned long long)ru * cs.H[i][1];
        a2[v] += (unsigned long long)ru * cs.H[i][2];
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      a0[v] += cs.Hoff[0];
      a1[v] += cs.Hoff[1];
      a2[v] += cs.Hoff[2];
      a1[v] += a0[v] >> 32;
      a2[v] += a1[v] >> 32;
      // 96-bit two's-complement fraction x = hi:lo (64 + 32 bits), centred:
      // [-1/2, 1/2); its magnitude, then the leading 64 bits of x << lz
      unsigned long long hi = ((unsigned long long)(unsigned)a2[v] << 32) | (unsigned)a1[v];
      unsigned lo = (unsigned)a0[v];
      const bool neg = (hi >> 63) != 0;
      if (neg) {  // x <- 2^96 - x
        hi = ~hi + (lo == 0u ? 1ull : 0ull);
        lo = 0u - lo;
      }
      double d = 0.0;
      if (!zero[v] && (hi | lo) != 0) {
        int lz;
        unsigned long long top;  // leading one at bit 63
        if (hi) {
          lz = __clzll((long long)hi);
          top = lz ? (hi << lz) | (((unsigned long long)lo << 32) >> (64 - lz)) : hi;
        } else {
          lz = 64 + __clz((int)lo);
          top = (unsigned long long)lo << (lz - 32);
        }
        // value = frac * M * 2^(ea+eb-2t), frac = top * 2^(-64-lz): the double is
        // assembled with integer arithmetic (the FP64 pipe runs at 1/64 rate)
        d = crt_to_double(cs, top, ea + eb[v] - 2 * job.tbits - lz, neg);
      }
      if (c == 0)
        out[v].x = d;
      else
        out[v].y = d;
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (n + v >= job.N) break;
    zc o = out[v];
    if (job.add != 0) {  // (an integer: comparing beta here took five FP64 instructions per element)
      const zc cc = job.C[bi * job.sC + (long long)m * job.ldc + n + v];
      if (job.add == 1) {
        o.x += cc.x;
        o.y += cc.y;
      } else {
        o.x += job.beta.x * cc.x - job.beta.y * cc.y;
        o.y += job.beta.x * cc.y + job.beta.y * cc.x;
      }
    }
    job.D[bi * job.sD + (long long)m * job.ldd + n + v] = o;
  }
}

// 4b. mixed mode: D = beta*C + sum over pair groups of the FP32 partials (FP64 sum).
struct SplitJob {
  const float *part;  // nullptr when the problem has no product term (D = beta*C)
  const zc *C;
  zc *D;
  long long ldc, ldd;
  long long part_bs, sC, sD;  // batch strides
  zc beta;
  int M, N, elem0;
};
struct SplitJobs {
  SplitJob j[QSI_MAX_PROB];
  int njobs, total;
};

__global__ void tc_split_final_kernel(const __grid_constant__ SplitJobs J) {
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  tc::pdl_wait();
  if (gid >= J.total) return;
  int ji = 0;
  while (ji + 1 < J.njobs && gid >= J.j[ji + 1].elem0) ++ji;
  const SplitJob &job = J.j[ji];
  const long long MN = (long long)job.M * job.N;
  const int eg = gid - job.elem0;
  const int bi = (int)(eg / MN), e = (int)(eg - bi * MN);
  const int m = e / job.N, n = e % job.N;
  zc out = make_double2(0.0, 0.0);
  if (job.part) {
    const float *part = job.part + bi * job.part_bs;
#pragma unroll
    for (int gq = 0; gq < SPLIT_GROUPS; ++gq) {
      out.x += (double)part[(gq * 2 + 0) * MN + e];
      out.y += (double)part[(gq * 2 + 1) * MN + e];
    }
  }
  if (job.C && (job.beta.x != 0.0 || job.beta.y != 0.0)) {
    const zc cc = job.C[bi * job.sC + (long long)m * job.ldc + n];
    out.x += job.beta.x * cc.x - job.beta.y * cc.y;
    out.y += job.beta.x * cc.y + job.beta.y * cc.x;
  }
  job.D[bi * job.sD + (long long)m * job.ldd + n] = out;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
size_t rup(size_t x, size_t a) { return (x + a - 1) / a * a; }

long long inv_mod(long long a, long long p) {
  long long t = 0, nt = 1, r = p, nr = ((a % p) + p) % p;
  while (nr) {
    const long long q = r / nr;
    long long tmp = t - q * nt;
    t = nt;
    nt = tmp;
    tmp = r - q * nr;
    r = nr;
    nr = tmp;
  }
  return (t % p + p) % p;
}

CrtConst make_consts() {
  CrtConst c;
  for (int i = 0; i < NMOD; ++i) {
    const long long p = MODS[i];
    c.p[i] = (float)p;
    c.inv_p[i] = 1.0f / (float)p;
    c.inv_p2[i] = make_float2(c.inv_p[i], c.inv_p[i]);
    c.negp2[i] = make_float2(-(float)p, -(float)p);
    for (int j = 0; j < NPIECE; ++j) {
      long long w = 1;
      for (int s = 0; s < PIECE_BITS * j; ++s) w = (w * 2) % p;
      if (2 * w > p) w -= p;  // symmetric: |w| <= p / 2 <= 128
      c.w[i][j] = (float)w;
      c.w2[i][j] = make_float2((float)w, (float)w);
    }
  }
  return c;
}

// reconstruction constants of the first nm moduli
CrtSet make_set(int nm) {
  CrtSet c;
  memset(&c, 0, sizeof c);
  // M = prod p_i (up to ~2^132.95, beyond 128-bit integers): accumulate
  // M / 2^64 in long double (at least a 64-bit mantissa: relative error
  // < 17 * 2^-64), then round once to double
  long double m64 = 1.0L;
  for (int i = 0; i < nm; ++i) m64 *= (long double)MODS[i];
  m64 = std::ldexp(m64, -64);
  c.m_over_2_64 = (double)m64;
  c.log2_m = 64.0 + std::log2(c.m_over_2_64);
  {
    // exact M as 32-bit limbs, then its 64 leading bits
    unsigned limb[8] = {1u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    for (int i = 0; i < nm; ++i) {
      unsigned long long carry = 0;
      for (int l = 0; l < 8; ++l) {
        const unsigned long long t = (unsigned long long)limb[l] * (unsigned)MODS[i] + carry;
        limb[l] = (unsigned)t;
        carry = t >> 32;
      }
    }
    int top = 7;
    while (top > 0 && limb[top] == 0) --top;
    int bits = 32 * top + 32 - __builtin_clz(limb[top]);  // bit length of M (> 64 for nm >= 9)
    c.m_shift = bits - 64;
    unsigned long long mt = 0;
    for (int k = 0; k < 64; ++k) {
      const int bit = bits - 1 - k;
      mt = (mt << 1) | ((limb[bit / 32] >> (bit % 32)) & 1u);
    }
    c.m_top = mt;
  }
  for (int i = 0; i < nm; ++i) {
    const long long p = MODS[i];
    long long mi = 1;  // (M / p_i) mod p_i
    for (int j = 0; j < nm; ++j)
      if (j != i) mi = (mi * (MODS[j] % p)) % p;
    // round(2^96 y_i / p_i), y_i = (M / p_i)^{-1} mod p_i < p_i (below 2^96)
    const unsigned __int128 yi = (unsigned __int128)(unsigned long long)inv_mod(mi, p);
    const unsigned __int128 h = ((yi << 96) + (unsigned __int128)(p / 2)) / (unsigned __int128)p;
    for (int l = 0; l < 3; ++l) c.H[i][l] = (unsigned)(h >> (32 * l));
  }
  {
    // the residue bytes are offset by 128: remove 128 * sum_i H_i modulo 2^96
    const unsigned __int128 mask96 = ((unsigned __int128)1 << 96) - 1;
    unsigned __int128 sum = 0;
    for (int i = 0; i < nm; ++i)
      sum += ((unsigned __int128)c.H[i][2] << 64) | ((unsigned __int128)c.H[i][1] << 32) | c.H[i][0];
    const unsigned __int128 off = (((unsigned __int128)1 << 96) - ((sum * 128) & mask96)) & mask96;
    for (int l = 0; l < 3; ++l) c.Hoff[l] = (unsigned)(off >> (32 * l));
  }
  return c;
}

double log2_modulus(int nm) {
  static double tab[NSET];
  static std::once_flag once;
  std::call_once(once, [] {
    for (int k = 0; k < NSET; ++k) tab[k] = make_set(NMOD_MIN + k).log2_m;
  });
  return tab[nm - NMOD_MIN];
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    cudaDriverEntryPointQueryResult q;
    void *p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  });
  return fn;
}

// planes [nplanes][rows][K] bf16, row stride Kp (a multiple of 64), box {64, box_rows, 1},
// 128-byte swizzle; what a box holds beyond rows and K is filled with zeros
bool make_map(CUtensorMap *m, void *base, int K, int Kp, int rows, int nplanes, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)nplanes};
  cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)Kp * 2 * rows};
  cuuint32_t box[3] = {BK, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// rows of a box: a tile's 128, or all rows of a smaller operand in steps of 16
// (the product reads 128 rows of A whatever the box holds: a row of the output
// depends on its own row of A alone, and rows beyond M are never stored)
int box_rows(int rows) { return rows < BM ? (rows + 15) & ~15 : BM; }

cudaError_t ensure_setup() {
  static unsigned long long done = 0;
  static std::mutex mu;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  const unsigned long long bit = 1ull << (dev & 63);
  if (done & bit) return cudaSuccess;
  const CrtConst c = make_consts();
  CrtSet sets[NSET];
  for (int k = 0; k < NSET; ++k) sets[k] = make_set(NMOD_MIN + k);
  e = cudaMemcpyToSymbol(c_crt, &c, sizeof c);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_set, sets, sizeof sets);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tc_mma_kernel<SCHEME_CRT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tc_mma_kernel<SCHEME_SPLIT3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)SMEM_BYTES);
  const auto smem = [&](auto kernel) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(CV_MAXKEEP * CV_TILE * sizeof(zc)));
  };
  smem(tc_convert_kernel<NMOD, 5>);
  smem(tc_convert_kernel<QSI_TC_MODULI_MIXED, 4>);
  smem(tc_convert_kernel<0, 5>);
  smem(tc_convert_kernel<-1, 1>);
  if (e == cudaSuccess) done |= bit;
  return e;
}

}  // namespace

double qsi_tc_log2_modulus(int nmod) { return log2_modulus(nmod); }

namespace {
// One bounded wait exactly as the tensor-core kernels wait (mbar_wait with a
// wall-clock limit), on an mbarrier that nothing arrives at: it runs out after
// limit_ns and records stage QSI_TC_STAGE_PROBE in *err, then the kernel
// returns (no trap, no endless loop).
__global__ void wait_probe_kernel(int *err, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !tc::mbar_wait(&bar, 0, limit_ns)) atomicExch(err, QSI_TC_STAGE_PROBE);
}
}  // namespace

cudaError_t qsi_tc_wait_probe(int *d_err, unsigned long long limit_ns, cudaStream_t s) {
  wait_probe_kernel<<<1, 32, 0, s>>>(d_err, limit_ns);
  return cudaGetLastError();
}

cudaError_t qsi_tc_setup() { return ensure_setup(); }

size_t qsi_tc_scratch_bytes(int M, int N, int K, int batch, int scheme) {
  // the layout qsi_zgemm_tc builds for one single-term problem
  const bool crt = scheme != QSI_TC_SPLIT3;
  const int nplanes = crt ? 2 * scheme : SPLIT_PLANES;
  size_t bytes = rup(sizeof(int) * (size_t)M * batch, 256) + rup(sizeof(int) * (size_t)N * batch, 256);
  bytes = rup(bytes, 1024);
  const size_t out_bs =
      crt ? rup((size_t)scheme * 2 * M * rup(N, 16), 1024) : rup((size_t)SPLIT_GROUPS * 2 * M * N, 256);
  bytes += crt ? out_bs * batch : out_bs * 4 * batch;
  const size_t Kp = rup(K, KPAD);
  bytes += rup((size_t)nplanes * M * Kp * 2 * batch, 1024) + rup((size_t)nplanes * N * Kp * 2 * batch, 1024);
  return bytes;
}

size_t qsi_tc_scratch_per_point(int b, int a) {
  // at most 8 problems of at most two terms, each operand (rows and depth at
  // most w = max(b, a)) as NPLANE bf16 planes, plus the int8 residues
  // and the exponents of every problem
  const size_t w = (size_t)std::max(b, a);
  const size_t planes = (size_t)NPLANE * w * rup(w, KPAD) * 2 + 1024;
  return QSI_MAX_PROB *
             (2 * 2 * planes + rup((size_t)NMOD * 2 * w * rup(w, 16), 1024) + 2 * rup(sizeof(int) * w, 256)) +
         (1 << 16);
}

cudaError_t qsi_zgemm_tc(ZGroup &g, int batch, cudaStream_t s, QsiProf *prof, cudaMemPool_t pool, int *d_err,
                         int scheme, TcArena *arena, const TcKnobs *knobs) {
  const bool crt = scheme != QSI_TC_SPLIT3;
  const int nm = crt ? scheme : 0;  // moduli of the CRT scheme
  if (crt && (nm < NMOD_MIN || nm > NMOD)) return cudaErrorInvalidValue;
  const int nplanes = crt ? 2 * nm : SPLIT_PLANES;
  if (batch < 1) return cudaErrorInvalidValue;
  cudaError_t e = ensure_setup();
  if (e != cudaSuccess) return e;
  if (!encode_fn()) return cudaErrorNotSupported;
  const double log2m = crt ? log2_modulus(nm) : 0.0;

  // keep non-empty problems; terms with K > 0; alpha must be +-1
  struct PInfo {
    ZProb p;
    int tbits;
    size_t off_ea, off_eb, off_res, off_a[QSI_MAX_TERMS], off_b[QSI_MAX_TERMS];
    int Kp[QSI_MAX_TERMS];
    int ldr;                         // row length of the residues
    long long out_bs;                // batch stride of the residues / partials (elements)
    int share_a = -1, share_b = -1;  // problem whose converted A / B operands this one reuses
    int map_a[QSI_MAX_TERMS], map_b[QSI_MAX_TERMS];  // and that problem's term for each of this one's
  } info[QSI_MAX_PROB];
  int np = 0;
  for (int i = 0; i < g.nprob; ++i) {
    ZProb p = g.p[i];
    if (p.M <= 0 || p.N <= 0) continue;
    int nt = 0;
    long long ksum = 0;
    for (int t = 0; t < p.nterms; ++t) {
      if (p.t[t].K <= 0) continue;
      const zc al = p.t[t].alpha;
      if (al.y != 0.0 || std::fabs(al.x) != 1.0) return cudaErrorNotSupported;
      ksum += p.t[t].K;
      p.t[nt++] = p.t[t];
    }
    p.nterms = nt;
    PInfo &I = info[np++];
    I.p = p;
    I.tbits = crt ? std::min(TBITS_MAX, (int)std::floor((log2m - 2.0 - std::log2(2.0 * std::max(1LL, ksum))) / 2.0))
                  : 0;
    // the mixed-mode conversion cuts the scaled integers (below 2^(tbits + 1))
    // into four 13-bit pieces: tbits <= 51 (13 moduli, log2 M = 102.4, give at most 49)
    if (crt && nm == QSI_TC_MODULI_MIXED && I.tbits > 4 * PIECE_BITS - 1) return cudaErrorInvalidValue;
  }
  // Problems that multiply the same operands on the same side (pointer, leading
  // dimension, op, sign, shape and bits; the terms in any order) get identical
  // exponents, which are common to all terms, and identical residue planes:
  // they are converted once.  The sweeps form whole block rows and columns of
  // compound products, e.g. Q A^H - L1 B_i,t - B L^H beside Q A^H - ... for the
  // next diagonal block, so this removes 21 % of the converted elements of a
  // step at a = b / 2.
  if (crt)
    for (int i = 0; i < np; ++i) {
      const ZProb &p = info[i].p;
      if (p.nterms == 0) continue;
      for (int j = 0; j < i; ++j) {
        const ZProb &o = info[j].p;
        if (o.nterms != p.nterms || info[j].tbits != info[i].tbits) continue;
        const bool try_a = info[i].share_a < 0 && info[j].share_a < 0 && o.M == p.M,
                   try_b = info[i].share_b < 0 && info[j].share_b < 0 && o.N == p.N;
        for (int side = 0; side < 2; ++side) {
          if (!(side == 0 ? try_a : try_b)) continue;
          int map[QSI_MAX_TERMS];
          unsigned taken = 0;
          bool all = true;
          for (int t = 0; t < p.nterms && all; ++t) {
            const ZTerm &T = p.t[t];
            map[t] = -1;
            for (int u = 0; u < o.nterms && map[t] < 0; ++u) {
              const ZTerm &O = o.t[u];
              if (((taken >> u) & 1u) || O.K != T.K) continue;
              const bool same = side == 0 ? O.A == T.A && O.lda == T.lda && O.sA == T.sA && O.opA == T.opA &&
                                                (O.alpha.x < 0.0) == (T.alpha.x < 0.0)
                                          : O.B == T.B && O.ldb == T.ldb && O.sB == T.sB && O.opB == T.opB;
              if (same) {
                map[t] = u;
                taken |= 1u << u;
              }
            }
            all = map[t] >= 0;
          }
          if (!all) continue;
          (side == 0 ? info[i].share_a : info[i].share_b) = j;
          for (int t = 0; t < p.nterms; ++t) (side == 0 ? info[i].map_a : info[i].map_b)[t] = map[t];
        }
      }
    }
  // scratch layout: every exponent array, then residues / partials and planes
  size_t bytes = 0;
  for (int i = 0; i < np; ++i) {
    if (info[i].share_a < 0) {
      info[i].off_ea = bytes;
      bytes += rup(sizeof(int) * info[i].p.M * batch, 256);
    }
    if (info[i].share_b < 0) {
      info[i].off_eb = bytes;
      bytes += rup(sizeof(int) * info[i].p.N * batch, 256);
    }
  }
  for (int i = 0; i < np; ++i) {
    if (info[i].share_a >= 0) info[i].off_ea = info[info[i].share_a].off_ea;
    if (info[i].share_b >= 0) info[i].off_eb = info[info[i].share_b].off_eb;
  }
  bytes = rup(bytes, 1024);
  for (int i = 0; i < np; ++i) {
    PInfo &I = info[i];
    const ZProb &p = I.p;
    I.off_res = bytes;
    I.ldr = (int)rup(p.N, 16);
    I.out_bs = crt ? (long long)rup((size_t)nm * 2 * p.M * I.ldr, 1024)
                   : (long long)rup((size_t)SPLIT_GROUPS * 2 * p.M * p.N, 256);  // int8 / float elements
    bytes += crt ? (size_t)I.out_bs * batch : (size_t)I.out_bs * 4 * batch;
    for (int t = 0; t < p.nterms; ++t) {
      I.Kp[t] = (int)rup(p.t[t].K, KPAD);
      if (I.share_a >= 0) {
        I.off_a[t] = info[I.share_a].off_a[I.map_a[t]];
      } else {
        I.off_a[t] = bytes;
        bytes += rup((size_t)nplanes * p.M * I.Kp[t] * 2 * batch, 1024);
      }
      if (I.share_b >= 0) {
        I.off_b[t] = info[I.share_b].off_b[I.map_b[t]];
      } else {
        I.off_b[t] = bytes;
        bytes += rup((size_t)nplanes * p.N * I.Kp[t] * 2 * batch, 1024);
      }
    }
  }
  if (np == 0) return cudaSuccess;
  uint8_t *scratch = nullptr;
  if (arena) arena->max_need = std::max(arena->max_need, bytes);
  const bool own = !(arena && arena->base);
  if (own) {
    e = cudaMallocFromPoolAsync((void **)&scratch, bytes, pool, s);
    if (e != cudaSuccess) return e;
  } else {
    if (bytes > arena->bytes) return cudaErrorMemoryAllocation;
    scratch = arena->base;
  }

  // operand-conversion / reconstruction launches: counted and (timing on) timed
  auto aux_begin = [&](int kind = QsiProf::TC_AUX) -> cudaError_t {
    if (!prof) return cudaSuccess;
    prof->launches++;
    prof->tc_aux_launches++;
    return prof->begin(kind, s);
  };
  auto aux_end = [&](cudaError_t e) -> cudaError_t {
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess && prof) e = prof->end(s);
    return e;
  };
  // operand jobs: A and B of every problem, all terms
  ConvJobs J;
  memset(&J, 0, sizeof J);
  for (int i = 0; i < np; ++i) {
    PInfo &I = info[i];
    if (I.p.nterms == 0) continue;
    for (int side = 0; side < 2; ++side) {
      if ((side == 0 ? I.share_a : I.share_b) >= 0) continue;  // converted with an earlier problem
      ConvJob &j = J.j[J.njobs++];
      j.R = side == 0 ? I.p.M : I.p.N;
      j.nterms = I.p.nterms;
      j.tbits = I.tbits;
      j.nmod = nm;
      j.eexp = (int *)(scratch + (side == 0 ? I.off_ea : I.off_eb));
      for (int t = 0; t < I.p.nterms; ++t) {
        const ZTerm &T = I.p.t[t];
        ConvTerm &c = j.t[t];
        if (side == 0) {  // rows of op(A): op N -> rows of A; op H -> conjugated columns of A
          c.X = T.A;
          c.sX = T.sA;
          c.ld = T.lda;
          c.row_contig = T.opA == ZOP_N;
          c.conj = T.opA == ZOP_H;
          c.negate = T.alpha.x < 0.0;
          c.planes = (__nv_bfloat16 *)(scratch + I.off_a[t]);
        } else {  // columns of op(B): op N -> columns of B; op H -> conjugated rows of B
          c.X = T.B;
          c.sX = T.sB;
          c.ld = T.ldb;
          c.row_contig = T.opB == ZOP_H;
          c.conj = T.opB == ZOP_H;
          c.negate = 0;
          c.planes = (__nv_bfloat16 *)(scratch + I.off_b[t]);
        }
        c.K = T.K;
        c.Kp = I.Kp[t];
        c.pl_bs = (long long)nplanes * j.R * c.Kp;
        c.tile0 = j.ntiles;
        j.ntiles += (T.K + CV_K - 1) / CV_K;
      }
    }
  }
  if (J.njobs > 0) {
    // clusters of as many CTAs as the longest row has tiles, or that many in two,
    // three, ... rounds of at most 8 CTAs (the split exchanges nothing: its CTAs
    // are launched without clusters)
    int tiles = 1, clusters = 0;
    for (int k = 0; k < J.njobs; ++k) {
      tiles = std::max(tiles, J.j[k].ntiles);
      J.j[k].blk0 = clusters;
      J.j[k].nblk = (J.j[k].R + CV_R - 1) / CV_R;
      clusters += J.j[k].nblk * batch;
    }
    const int rounds = crt ? (tiles + CV_MAXCS - 1) / CV_MAXCS : 1;
    J.cs = (tiles + rounds - 1) / rounds;
    J.keep = std::min(rounds, CV_MAXKEEP);
    e = aux_begin();
    if (e == cudaSuccess) {
      cudaLaunchConfig_t lc = {};
      cudaLaunchAttribute at[2];
      int na = 0;
      if (!own && arena->direct) at[na++] = tc::pdl_attr();
      if (crt) {
        at[na].id = cudaLaunchAttributeClusterDimension;
        at[na].val.clusterDim.x = J.cs;
        at[na].val.clusterDim.y = 1;
        at[na++].val.clusterDim.z = 1;
      }
      lc.gridDim = dim3(clusters * J.cs);
      lc.blockDim = dim3(256);
      lc.dynamicSmemBytes = J.keep * CV_TILE * sizeof(zc);
      lc.stream = s;
      lc.attrs = at;
      lc.numAttrs = na;
      e = cudaLaunchKernelEx(&lc,
                             !crt                        ? tc_convert_kernel<-1, 1>
                             : nm == NMOD                ? tc_convert_kernel<NMOD, 5>
                             : nm == QSI_TC_MODULI_MIXED ? tc_convert_kernel<QSI_TC_MODULI_MIXED, 4>
                                                         : tc_convert_kernel<0, 5>,
                             J);
    }
    e = aux_end(e);
  }
  // tensor-core products
  if (e == cudaSuccess) {
    TcGroup G;
    memset(&G, 0, sizeof G);
    G.nprob = np;
    // moduli per CTA: fewest estimated CTA waves x the longest CTA (one CTA
    // per SM; a CTA costs mpc x its k-tiles plus a fixed overhead of pipeline
    // fill and final epilogue, counted as 6 k-tiles: on the n=64, b=512,
    // a=256 step 1 / 3 / 6 / 12 gave 147.2 / 144.0 / 143.5 / 143.6 ms)
    int mpc = 1;
    if (crt) {
      long long tiles = 0;
      int kt_max = 1;
      for (int i = 0; i < np; ++i) {
        tiles += (long long)((info[i].p.M + BM - 1) / BM) * ((info[i].p.N + BN - 1) / BN) * batch;
        int kt = 0;
        for (int t = 0; t < info[i].p.nterms; ++t) kt += (info[i].p.t[t].K + BK - 1) / BK;
        kt_max = std::max(kt_max, kt);
      }
      double best = 0.0, fill = 6.0;  // knobs, then QSI_TC_CTA_FILL, set the per-CTA overhead (k-tiles)
      if (knobs && knobs->cta_fill >= 0.0) fill = knobs->cta_fill;
      if (const char *ef = getenv("QSI_TC_CTA_FILL")) fill = std::max(0.0, atof(ef));
      for (int m = 1; m <= nm; ++m) {
        const long long c = tiles * ((nm + m - 1) / m);
        const double est = (double)((c + NUM_SMS - 1) / NUM_SMS) * (m * (double)kt_max + fill);
        if (m == 1 || est < best) {
          best = est;
          mpc = m;
        }
      }
    }
    int ctas = 0;
    for (int i = 0; i < np && e == cudaSuccess; ++i) {
      PInfo &I = info[i];
      TcProb &P = G.p[i];
      P.M = I.p.M;
      P.N = I.p.N;
      P.nterms = I.p.nterms;
      P.tiles_n = (P.N + BN - 1) / BN;
      P.mpc = mpc;
      P.nmod = nm;
      P.ngroups = crt ? (nm + mpc - 1) / mpc : SPLIT_GROUPS;
      P.cta0 = ctas;
      P.res = crt ? (int8_t *)(scratch + I.off_res) : nullptr;
      P.part = crt ? nullptr : (float *)(scratch + I.off_res);
      P.out_bs = I.out_bs;
      P.ldr = I.ldr;
      P.stage_bytes = 2 * (box_rows(P.M) + box_rows(P.N)) * BK * 2;
      P.ctas_per_b = ((P.M + BM - 1) / BM) * P.tiles_n * P.ngroups;
      ctas += P.ctas_per_b * batch;
      for (int t = 0; t < P.nterms; ++t) {
        P.t[t].K = I.p.t[t].K;
        const int K = P.t[t].K;
        if (!make_map(&P.t[t].ma, scratch + I.off_a[t], K, I.Kp[t], P.M, nplanes * batch, box_rows(P.M)) ||
            !make_map(&P.t[t].mb, scratch + I.off_b[t], K, I.Kp[t], P.N, nplanes * batch, box_rows(P.N)))
          e = cudaErrorInvalidValue;
      }
    }
    G.total_ctas = ctas;
    if (e == cudaSuccess) {
      if (prof) {
        prof->launches++;
        prof->tc_launches++;
        for (int i = 0; i < np; ++i)
          for (int t = 0; t < info[i].p.nterms; ++t)
            prof->tc_flops += 8.0 * info[i].p.M * info[i].p.N * info[i].p.t[t].K * batch;
        e = prof->begin(QsiProf::TC, s);
      }
      if (e == cudaSuccess) {
        e = tc::launch_after(crt ? tc_mma_kernel<SCHEME_CRT> : tc_mma_kernel<SCHEME_SPLIT3>, ctas, THREADS, SMEM_BYTES, s,
                         J.njobs > 0, G, d_err);
      }
      if (e == cudaSuccess && prof) e = prof->end(s);
    }
  }
  // mixed mode: sum of the partial products
  if (e == cudaSuccess && !crt) {
    SplitJobs J;
    memset(&J, 0, sizeof J);
    J.njobs = np;
    int total = 0;
    for (int i = 0; i < np; ++i) {
      PInfo &I = info[i];
      SplitJob &j = J.j[i];
      j.part = I.p.nterms > 0 ? (const float *)(scratch + I.off_res) : nullptr;
      j.part_bs = I.out_bs;
      j.C = I.p.C;
      j.D = I.p.D;
      j.ldc = I.p.ldc;
      j.ldd = I.p.ldd;
      j.sC = I.p.sC;
      j.sD = I.p.sD;
      j.beta = I.p.beta;
      j.M = I.p.M;
      j.N = I.p.N;
      j.elem0 = total;
      total += I.p.M * I.p.N * batch;
    }
    J.total = total;
    e = aux_begin(QsiProf::TC_CRT);
    if (e == cudaSuccess) e = tc::launch_after(tc_split_final_kernel, (total + 255) / 256, 256, 0, s, true, J);
    e = aux_end(e);
  }
  // reconstruction
  if (e == cudaSuccess && crt) {
    CrtJobs J;
    memset(&J, 0, sizeof J);
    J.njobs = np;
    int total = 0;
    for (int i = 0; i < np; ++i) {
      PInfo &I = info[i];
      CrtJob &j = J.j[i];
      j.res = (const int8_t *)(scratch + I.off_res);
      j.res_bs = I.out_bs;
      j.ea = I.p.nterms > 0 ? (const int *)(scratch + I.off_ea) : nullptr;
      j.eb = I.p.nterms > 0 ? (const int *)(scratch + I.off_eb) : nullptr;
      j.C = I.p.C;
      j.D = I.p.D;
      j.ldc = I.p.ldc;
      j.ldd = I.p.ldd;
      j.sC = I.p.sC;
      j.sD = I.p.sD;
      j.beta = I.p.beta;
      j.add = !I.p.C || (j.beta.x == 0.0 && j.beta.y == 0.0) ? 0 : j.beta.x == 1.0 && j.beta.y == 0.0 ? 1 : 2;
      j.M = I.p.M;
      j.N = I.p.N;
      j.tbits = I.tbits;
      j.nmod = nm;
      j.ldr = I.ldr;
    }
    // V consecutive elements per thread: 2, or 4 where that still leaves eight
    // blocks per SM and more (32 points of (32, 256, 128): 239.0 ms with 4 against
    // 241.4 with 2; (64, 512, 256) solve: 88.6 against 88.5, 91.7 with 1); QSI_CRT_V
    // overrides
    long long outputs = 0;
    for (int i = 0; i < np; ++i) outputs += (long long)info[i].p.M * info[i].p.N * batch;
    int V = outputs >= CRT_V4_OUTPUTS ? 4 : 2;
    if (knobs && (knobs->crt_v == 1 || knobs->crt_v == 2 || knobs->crt_v == 4)) V = knobs->crt_v;
    if (const char *ev = getenv("QSI_CRT_V")) {
      const int want = atoi(ev);
      if (want == 1 || want == 2 || want == 4) V = want;
    }
    if (nm != NMOD && nm != QSI_TC_MODULI_MIXED) V = 1;  // the run-time moduli count has V = 1 only
    for (int i = 0; i < np; ++i) {
      J.j[i].elem0 = total;
      total += info[i].p.M * ((info[i].p.N + V - 1) / V) * batch;
    }
    J.total = total;
    e = aux_begin(QsiProf::TC_CRT);
    if (e == cudaSuccess) {
      const int nb = (total + 255) / 256;
      const bool full = nm == NMOD, mixed = nm == QSI_TC_MODULI_MIXED;
      e = tc::launch_after(full    ? V == 4 ? tc_crt_kernel<4, NMOD> : V == 2 ? tc_crt_kernel<2, NMOD> : tc_crt_kernel<1, NMOD>
                       : mixed ? V == 4   ? tc_crt_kernel<4, QSI_TC_MODULI_MIXED>
                                 : V == 2 ? tc_crt_kernel<2, QSI_TC_MODULI_MIXED>
                                          : tc_crt_kernel<1, QSI_TC_MODULI_MIXED>
                               : tc_crt_kernel<1, 0>,
                       nb, 256, 0, s, true, J);
    }
    e = aux_end(e);
  }
  if (arena) arena->direct = !own && e == cudaSuccess;  // the stream's last operation is a kernel of ours
  cudaError_t e2 = own ? cudaFreeAsync(scratch, s) : cudaSuccess;
  return e != cudaSuccess ? e : e2;
}
