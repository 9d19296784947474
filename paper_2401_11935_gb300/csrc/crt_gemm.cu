// FP64 contractions on the tensor cores by modular arithmetic.
//
// The FP64 pipe of this GPU retires 2 FMA per clock and SM (1.25 TFLOP/s);
// its tensor cores do 4096 BF16 FMA.  A product of integers modulo a small
// p needs only BF16: residues of magnitude <= 128 are exact in BF16, their
// products are at most 2^14, and sums of up to 1024 of them are exact in the
// FP32 accumulator.  So (Ozaki, Uchino and Imamura, "Ozaki Scheme II",
// arXiv 2504.08009):
//   1. every row of A and B (over k) is scaled by a power of two to integers
//      with 2-norm below 2^62 and 2^61 (elements rounded to the nearest
//      integer, the only approximation);
//   2. the integer rows are reduced modulo 16 pairwise coprime p_i <= 256;
//   3. one tcgen05 GEMM per modulus gives C mod p_i exactly;
//   4. C is put together by the Chinese remainder theorem: |C| <= |a| |b| <
//      2^123 < P / 4 with P = prod p_i = 2^125.4, in integer arithmetic, then
//      rounded once to FP64.
// The rounding of step 1 leaves an error relative to |a| |b|: in the units
// where the norms' bounds are 1, at most 0.75 sqrt(K) 2^-61, 0.3 2^-61 in the
// root mean square.  A chain of FMAs errs relative to S = sum_k |a_k b_k|,
// which is far below |a| |b| where large elements of a meet small ones of b.
// So one more GEMM, over the magnitudes rounded down to BF16, gives S; where it
// is below 2^-7 in the same units (and not zero), the element is computed as a
// chain of FMAs instead (k_crt_patch).  The others err by at most
// 0.375 sqrt(K) 2^-53 S, 2e-17 S in the root mean square, as much as a chain
// does for products of random sign.  Rows and columns with Inf or NaN go to
// the chain, too.
//
// Measured (GB300), CUDA cores -> this path: (M, N, K) = (432, 2196, 14884)
// 23.6 -> 0.91 ms, of which GEMM 0.33 (1.46 PFLOP/s of BF16), residues 0.38,
// norms 0.18; (2196, 14884, 360) 19.2 -> 0.98 ms, of which GEMM 0.43 (short
// k) and output 0.41; (1464, 1464, 1464) 5.18 -> 0.20 ms.  The whole FP64
// residual at (10, 120, 360): 445 -> 23.0 ms, of which the patch takes 1.7
// (0.28 ms of a contraction whose i = j columns are zero in one operand where
// the other is largest); before the sums of magnitudes and the patch, with 15
// moduli, 21.1 ms.  Operands that fall by 12 decades along k, against each
// other, take the CUDA cores' time and 7 to 20 % (50 to 90 us where it is short).
#include "common.h"
#include "tc_ptx.h"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>

namespace dcsd {

namespace {

// ---------------------------------------------------------------------------
// moduli and derived constants
// ---------------------------------------------------------------------------
constexpr int kMods = 16;
constexpr int kModulus[kMods] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};
constexpr int kPlanes = kMods + 1;             // residues, and the magnitudes
constexpr int kLimbs = 6;                      // 20-bit limbs of P and P / p_i
constexpr int kBetaA = 62, kBetaB = 61;        // log2 bounds of the integer rows' 2-norms
constexpr int kSegBlocks = 16;                 // 64-deep k-blocks per exact FP32 sum (16 * 64 = 1024)

// Sums of magnitudes as a byte per split of K: 0 for a zero sum, else S 2^13 +
// 0.75 to the nearest integer, 1 to 255.  A result is kept where the splits'
// sum is 0 (all products are zero) or at least 74: S >= (74 - 8 x 1.25) 2^-13 = 2^-7.
constexpr float kSumScale = 8192.0f;
constexpr int kSumKept = 74, kMaxSplit = 8;
__device__ __forceinline__ bool sum_kept(int code) { return code == 0 || code >= kSumKept; }

constexpr long sym_mod(long x, long p) {       // residue in [-(p - 1) / 2, p / 2]
    long r = x % p;
    if (r < 0) r += p;
    return r > p / 2 ? r - p : r;
}

constexpr long sym_byte(long x, long p) {      // the same in [-128, 127]
    const long r = sym_mod(x, p);
    return r == 128 ? -128 : r;                // p = 256
}

struct Tables {
    float p[kPlanes], inv_p[kPlanes];          // (magnitudes: 0, which reduce_mod leaves as they are)
    // byte weights of a 64-bit integer, 2^(8 j) mod p (side B: times
    // (P / p_i)^-1), signed bytes; the start value -2^63 of a biased integer,
    // already offset by the FP32 pattern of kRint
    unsigned w_lo[2][kMods], w_hi[2][kMods];
    int w_start[2][kMods];
    int limb[kMods][kLimbs];                   // P / p_i
    int plimb[kLimbs];                         // P
};

constexpr Tables make_tables() {
    Tables t{};
    unsigned __int128 P = 1;
    for (int i = 0; i < kMods; ++i) P *= (unsigned)kModulus[i];
    for (int i = 0; i < kMods; ++i) {
        const long p = kModulus[i];
        const unsigned __int128 Mi = P / (unsigned)p;
        const long mi = (long)(Mi % (unsigned)p);
        long inv = 1;
        while ((mi * inv) % p != 1) ++inv;
        t.p[i] = (float)p;
        t.inv_p[i] = 1.0f / (float)p;
        for (int side = 0; side < 2; ++side) {
            long w = side == 0 ? 1 : inv;
            for (int j = 0; j < 8; ++j) {
                const unsigned b = (unsigned)(sym_byte(w, p) & 0xFF);
                if (j < 4) t.w_lo[side][i] |= b << (8 * j);
                else t.w_hi[side][i] |= b << (8 * (j - 4));
                if (j == 7) t.w_start[side][i] = 0x4B400000 - (int)sym_mod(128 * w, p);
                w = (w << 8) % p;
            }
        }
        for (int l = 0; l < kLimbs; ++l) t.limb[i][l] = (int)((Mi >> (20 * l)) & 0xFFFFF);
    }
    for (int l = 0; l < kLimbs; ++l) t.plimb[l] = (int)((P >> (20 * l)) & (l + 1 < kLimbs ? 0xFFFFF : 0x7FFFFFFF));
    return t;
}

__constant__ Tables d_tab = make_tables();

constexpr float kRint = 12582912.0f;           // 1.5 * 2^23: x + kRint - kRint rounds |x| < 2^22 to an integer

// x mod p (|x| <= 2^24 an integer), within p / 2 + 3; exact in FP32
__device__ __forceinline__ float reduce_mod(float x, float p, float inv_p) {
    const float q = __fadd_rn(__fmaf_rn(x, inv_p, kRint), -kRint);
    return __fmaf_rn(-p, q, x);
}

// ---------------------------------------------------------------------------
// operands: a strided FP64 matrix [rows][K] (modes as in GemmPlan)
// ---------------------------------------------------------------------------
struct Operand {
    const double* p;
    int nr, nk;
    long rsz[kMaxMode], rs[kMaxMode], rc[kMaxMode];  // row modes: size, stride in the operand, stride in C
    long ksz[kMaxMode], ks[kMaxMode];
    long rows, K;       // of this pass
    long r0, k0;        // first row and k of this pass
    int kfast;          // the k index is the contiguous one
    int beta;           // log2 bound of the integer rows' 2-norm
    int side;           // digit table
    // outputs
    double* part_ss;            // [nchunk][rows] sums of squares
    unsigned long long* part_mx;  // [nchunk][rows] magnitudes' bit patterns
    int* shift;                 // [rows] power-of-two scale, kNonFinite where a row holds Inf or NaN
    long* coff;                 // [rows] offset in C
    uint16_t* dst;              // [plane][K / 64][rows][64] residues and magnitudes (BF16)
    int nchunk, nkb;
    int kchunk;                 // k per partial norm
    int kbper;                  // k-blocks per block of the pack launch
    long blocks;                // thread blocks of this operand in the norm / pack launch
};

constexpr int kNonFinite = INT_MIN;
constexpr int kNormK = 512;     // k offsets staged at a time by the norm kernel

__device__ __forceinline__ long mode_offset(unsigned idx, int n, const long* size, const long* s) {
    long o = 0;
#pragma unroll
    for (int j = kMaxMode - 1; j >= 0; --j)
        if (j < n) {
            const unsigned sz = (unsigned)size[j], q = idx / sz;
            o += (long)(idx - q * sz) * s[j];
            idx = q;
        }
    return o;
}

__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

// Row norms over pieces of kchunk k: the sum of squares (FP64) and the
// largest magnitude (bit pattern).  One warp per row when k is contiguous (8
// rows per block), else 64 rows per block with four groups of k.  Bound by
// reading the operand once; kchunk keeps at most 32 pieces, and enough blocks.
__global__ void __launch_bounds__(256) k_crt_norm(const Operand oa, const Operand ob) {
    __shared__ long koff[kNormK];
    __shared__ double sh_s[4][64];
    __shared__ unsigned long long sh_m[4][64];
    const bool first = (long)blockIdx.x < oa.blocks;
    const Operand& o = first ? oa : ob;
    const long b = first ? blockIdx.x : blockIdx.x - oa.blocks;
    const long rb = b / o.nchunk;
    const int ch = (int)(b - rb * o.nchunk);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, rl = threadIdx.x & 63, g = threadIdx.x >> 6;
    const long r = o.kfast ? rb * 8 + w : rb * 64 + rl;
    const int k_first = o.kfast ? lane : g, k_step = o.kfast ? 32 : 4;
    const unsigned long long mask = 0x7FFFFFFFFFFFFFFFull;
    const double* src = o.p + (r < o.rows ? mode_offset((unsigned)(o.r0 + r), o.nr, o.rsz, o.rs) : 0);
    double s0 = 0.0, s1 = 0.0;
    unsigned long long m = 0;
    const long kb = (long)ch * o.kchunk, ke = min(o.K, kb + o.kchunk);
    for (long k0 = kb; k0 < ke; k0 += kNormK) {
        const int kn = (int)min((long)kNormK, ke - k0);
        __syncthreads();
        for (int k = threadIdx.x; k < kn; k += 256) koff[k] = mode_offset((unsigned)(o.k0 + k0 + k), o.nk, o.ksz, o.ks);
        __syncthreads();
        if (r >= o.rows) continue;
        int k = k_first;
        for (; k + 3 * k_step < kn; k += 4 * k_step) {
            const double x0 = src[koff[k]], x1 = src[koff[k + k_step]], x2 = src[koff[k + 2 * k_step]],
                         x3 = src[koff[k + 3 * k_step]];
            s0 = fma(x0, x0, s0);
            s1 = fma(x1, x1, s1);
            s0 = fma(x2, x2, s0);
            s1 = fma(x3, x3, s1);
            m = umax64(umax64(m, __double_as_longlong(x0) & mask), umax64(__double_as_longlong(x1) & mask,
                       umax64(__double_as_longlong(x2) & mask, __double_as_longlong(x3) & mask)));
        }
        for (; k < kn; k += k_step) {
            const double x = src[koff[k]];
            s0 = fma(x, x, s0);
            m = umax64(m, __double_as_longlong(x) & mask);
        }
    }
    s0 += s1;
    if (o.kfast) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, d);
            m = umax64(m, __shfl_xor_sync(0xffffffffu, m, d));
        }
        if (lane == 0 && r < o.rows) {
            o.part_ss[(long)ch * o.rows + r] = s0;
            o.part_mx[(long)ch * o.rows + r] = m;
        }
    } else {
        sh_s[g][rl] = s0;
        sh_m[g][rl] = m;
        __syncthreads();
        if (g == 0 && r < o.rows) {
            o.part_ss[(long)ch * o.rows + r] = (sh_s[0][rl] + sh_s[1][rl]) + (sh_s[2][rl] + sh_s[3][rl]);
            o.part_mx[(long)ch * o.rows + r] = umax64(umax64(sh_m[0][rl], sh_m[1][rl]), umax64(sh_m[2][rl], sh_m[3][rl]));
        }
    }
}

// scale exponent of a row: the largest s with 2-norm * 2^s <= 2^beta (up to
// one bit).  Outside the range where squares are exact enough, the norm is
// bounded by the largest magnitude times sqrt(K).
__device__ __forceinline__ int row_shift(double ss, unsigned long long mx, long K, int beta) {
    if (mx == 0) return 0;
    const int e = (int)(mx >> 52);  // biased exponent of the largest magnitude
    if (e == 0x7FF) return kNonFinite;
    int L;  // norm < 2^L
    if (e > 1023 - 400 && e < 1023 + 400) {
        const int e2 = (int)((__double_as_longlong(ss * (1.0 + 1e-9)) >> 52) & 0x7FF) - 1023;
        L = (e2 + 2) >> 1;
    } else {
        L = max(e, 1) - 1022 + (65 - __clzll((unsigned long long)K)) / 2;
    }
    return beta - L;
}

// x * 2^s rounded to the nearest integer (|result| <= 2^62 by the row's scale)
__device__ __forceinline__ long long scaled_int(double x, int s) {
    const long long b = __double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7FF);
    unsigned long long m = (unsigned long long)b & 0xFFFFFFFFFFFFFull;
    if (ef) m |= 1ull << 52;
    const int sh = (ef ? ef : 1) - 1075 + s;
    unsigned long long v;
    if (sh >= 0) v = m << min(sh, 63);
    else if (sh > -55) v = (m + (1ull << (-sh - 1))) >> (-sh);
    else v = 0;
    return b < 0 ? -(long long)v : (long long)v;
}

// kRint + (v mod p up to a few hundred p): the eight bytes of v + 2^63 times
// their weights, two four-way byte products; |sum| <= 8 * 255 * 128 < 2^19
__device__ __forceinline__ int byte_dot(unsigned bytes, unsigned weights, int acc) {
    int r;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(bytes), "r"(weights), "r"(acc));
    return r;
}

// |v| 2^-beta rounded down to BF16, in the upper half of a word; at least
// 2^(2 - beta) where the element is not zero, so that only sums whose products
// are all zero vanish (the products stay normal in FP32: >= 2^-119)
__device__ __forceinline__ unsigned magnitude(long long v, double x, int beta) {
    if (x == 0.0) return 0u;
    const float f = fmaxf(__ull2float_rz((unsigned long long)(v < 0 ? -v : v)), 4.0f);
    return __float_as_uint(f) - ((unsigned)beta << 23);
}

// Residues of one operand: per 64 rows x 64 k, scale to integers, reduce
// modulo every p_i, store BF16 K-blocked [plane][k block][row][64], the
// magnitudes after the residues.  Writes 34 bytes per element read; two byte
// products and five FP32 operations per element and modulus.  Clears the
// nclear words of the patch's flags as well.
__global__ void __launch_bounds__(256) k_crt_pack(const Operand oa, const Operand ob, unsigned* clear, long nclear) {
    for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < nclear; i += (long)gridDim.x * 256) clear[i] = 0u;
    __shared__ double tile[64][65];
    __shared__ long roff[64], koff[64];
    __shared__ int sh[64];
    const bool first = (long)blockIdx.x < oa.blocks;
    const Operand& o = first ? oa : ob;
    const long b = first ? blockIdx.x : blockIdx.x - oa.blocks;
    const int nkg = (o.nkb + o.kbper - 1) / o.kbper;
    const long rb = b / nkg;
    const int kt0 = (int)(b - rb * nkg) * o.kbper, kt1 = min(o.nkb, kt0 + o.kbper);
    const long row0 = rb * 64;
    const int tid = threadIdx.x;
    if (tid < 64) {
        const long r = row0 + tid;
        roff[tid] = -1;
        sh[tid] = 0;
        if (r < o.rows) {
            roff[tid] = mode_offset((unsigned)(o.r0 + r), o.nr, o.rsz, o.rs);
            double ss = 0.0;
            unsigned long long mx = 0;
            for (int c = 0; c < o.nchunk; ++c) {
                ss += o.part_ss[(long)c * o.rows + r];
                mx = umax64(mx, o.part_mx[(long)c * o.rows + r]);
            }
            const int s = row_shift(ss, mx, o.K, o.beta);
            sh[tid] = s;
            if (kt0 == 0) {
                o.shift[r] = s;
                o.coff[r] = mode_offset((unsigned)(o.r0 + r), o.nr, o.rsz, o.rc);
            }
        }
    }
    const int lane = tid & 31, w = tid >> 5;
    const long plane = (long)o.nkb * o.rows * 64;
    const bool side = o.side != 0;
    for (int kt = kt0; kt < kt1; ++kt) {
        __syncthreads();  // the tile and the offsets are free (and roff, sh written)
        if (tid < 64) {
            const long k = (long)kt * 64 + tid;
            koff[tid] = k < o.K ? mode_offset((unsigned)(o.k0 + k), o.nk, o.ksz, o.ks) : -1;
        }
        __syncthreads();
#pragma unroll 8
        for (int e = tid; e < 64 * 64; e += 256) {
            const int f = e & 63, g = e >> 6;
            const int rr = o.kfast ? g : f, kk = o.kfast ? f : g;
            const long ro = roff[rr], ko = koff[kk];
            tile[rr][kk] = (ro >= 0 && ko >= 0) ? o.p[ro + ko] : 0.0;
        }
        __syncthreads();
#pragma unroll 1
        for (int rr = 0; rr < 8; ++rr) {
            const int rl = w * 8 + rr;
            const long r = row0 + rl;
            if (r >= o.rows) break;
            const int s = sh[rl];
            const double e0 = s == kNonFinite ? 0.0 : tile[rl][2 * lane], e1 = s == kNonFinite ? 0.0 : tile[rl][2 * lane + 1];
            const long long i0 = scaled_int(e0, s), i1 = scaled_int(e1, s);
            const unsigned long long v0 = (unsigned long long)i0 ^ 0x8000000000000000ull;
            const unsigned long long v1 = (unsigned long long)i1 ^ 0x8000000000000000ull;
            uint32_t* dst = (uint32_t*)(o.dst + ((long)kt * o.rows + r) * 64) + lane;
#pragma unroll
            for (int i = 0; i < kMods; ++i) {
                const unsigned wl = side ? d_tab.w_lo[1][i] : d_tab.w_lo[0][i], wh = side ? d_tab.w_hi[1][i] : d_tab.w_hi[0][i];
                const int ws = side ? d_tab.w_start[1][i] : d_tab.w_start[0][i];
                const float x0 = __int_as_float(byte_dot((unsigned)v0, wl, byte_dot((unsigned)(v0 >> 32), wh, ws))) - kRint;
                const float x1 = __int_as_float(byte_dot((unsigned)v1, wl, byte_dot((unsigned)(v1 >> 32), wh, ws))) - kRint;
                const float y0 = reduce_mod(x0, d_tab.p[i], d_tab.inv_p[i]);
                const float y1 = reduce_mod(x1, d_tab.p[i], d_tab.inv_p[i]);
                // integers of magnitude <= 128: the upper half of the FP32 word is the BF16 value
                dst[(long)i * (plane / 2)] = __byte_perm(__float_as_uint(y0), __float_as_uint(y1), 0x7632);
            }
            dst[(long)kMods * (plane / 2)] = __byte_perm(magnitude(i0, e0, o.beta), magnitude(i1, e1, o.beta), 0x7632);
        }
    }
}

// ---------------------------------------------------------------------------
// the modular GEMM
// ---------------------------------------------------------------------------
constexpr int CG_BM = 128, CG_BK = 64;
constexpr uint32_t CG_A = CG_BM * CG_BK * 2;
// stages of 16 KB of A and up to 32 KB of B; in a pair half of B
__host__ __device__ constexpr int cg_stages(bool pair) { return pair ? 6 : 4; }
__host__ __device__ constexpr uint32_t cg_stage(bool pair) { return CG_A + (pair ? 128 : 256) * CG_BK * 2; }
constexpr int kEpiWarps = 8, kThreads = 32 * (2 + kEpiWarps);
constexpr size_t kCrtSmem = 6 * cg_stage(true) + 2048;  // (= 4 * cg_stage(false) + 2048)

struct GemmShape {
    long M, N;              // rows and columns
    int nkb, kper;          // 64-deep k-blocks, k-blocks per split
    int nsplit;
    int tilesM, tilesN, BN; // n-tiles of BN columns (a multiple of 16, in a pair of 32; at most 256)
    int group;
    uint32_t* planes;       // [split][plane][ceil(N / 4)][M] four residues or sums (bytes) of consecutive n
};

// Persistent tcgen05 GEMM over (split, plane, m-tile, n-tile).  The pipeline
// is that of k_tc_gemm: warp 0 loads K-blocked tiles by TMA, warp 1 issues
// the MMAs into one of two TMEM accumulators, eight warps drain the other.
// The accumulator is drained every 1024 k, where its integer sum is still
// exact, and kept modulo p in FP32 registers (four FP32 operations per
// element, hidden behind the 16 k-blocks of MMAs), so a long k costs no
// memory traffic; the residues leave as bytes.
// PAIR: two CTAs on neighbouring m-tiles of one n-tile as a cta_group::2 pair,
// as in k_tc_gemm: each loads its rows of A and half of B, and a k-block takes
// 600 clocks instead of 784 with 256 columns.  (10, 120, 360): the ladder's
// M = 2196, K = 14884 contraction of a chunk 373 -> 268 us, its integrals,
// M = 14884, K = 360, 455 -> 405 us, with what electing the issuing lane gave
// (both over 15 planes; 328 and 429 us over 17).
template <bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
    k_crt_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmShape g,
               int* err) {
    constexpr int CG_STAGES = cg_stages(PAIR);
    constexpr uint32_t CG_STAGE = cg_stage(PAIR);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + CG_STAGES * CG_STAGE);
    uint64_t* empty = full + CG_STAGES;
    uint64_t* accf = empty + CG_STAGES;  // [2] MMA -> epilogue
    uint64_t* acce = accf + 2;           // [2] epilogue -> MMA
    uint32_t* tslot = (uint32_t*)(acce + 2);
    volatile int* issued = (volatile int*)(tslot + 1);
    volatile int* consumed = issued + 1;

    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int crank = PAIR ? (int)cluster_rank() : 0;
    const int tile0 = PAIR ? (int)blockIdx.x / 2 : (int)blockIdx.x;
    const int tstep = PAIR ? (int)gridDim.x / 2 : (int)gridDim.x;
    const int tilesMs = PAIR ? (g.tilesM + 1) / 2 : g.tilesM;
    const int nmn = tilesMs * g.tilesN;
    const int ntiles = nmn * kPlanes * g.nsplit;
    const int BN = g.BN;
    if (threadIdx.x == 0) {
        for (int s = 0; s < CG_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf[b], 1);
            mbar_init(&acce[b], PAIR ? 2 * kEpiWarps : kEpiWarps);
        }
        *issued = 0;
        *consumed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        if (PAIR) tmem_alloc_pair(tslot, 512);
        else tmem_alloc(tslot, 512);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (PAIR) cluster_sync();
    const uint32_t tmem = *tslot;

    // tile -> (m-tile, n-tile, plane, split)
    auto locate = [&](int tile, int& tm, int& tn, int& mod, int& ks) {
        const int z = tile / nmn, mn = tile - z * nmn;
        ks = z / kPlanes;
        mod = z - ks * kPlanes;
        const int gr = max(1, min(g.group, tilesMs));
        const int band = mn / (gr * g.tilesN), r = mn - band * gr * g.tilesN;
        const int rows = min(gr, tilesMs - band * gr);
        tm = band * gr + r % rows;
        tn = r / rows;
        if (PAIR) tm = 2 * tm + crank;
    };

    if (warp == 0) {
        if (elect_one()) {
            int it = 0;
            bool ok = true;
            for (int tile = tile0; tile < ntiles && ok; tile += tstep) {
                int tm, tn, mod, ks;
                locate(tile, tm, tn, mod, ks);
                const int kb = ks * g.kper, ke = min(g.nkb, kb + g.kper);
                for (int kt = kb; kt < ke; ++kt, ++it) {
                    const int s = it % CG_STAGES, round = it / CG_STAGES;
                    if (round > 0 && !mbar_wait(&empty[s], (round - 1) & 1)) {
                        atomicExch(err, 1);
                        ok = false;
                        break;
                    }
                    const int z = mod * g.nkb + kt;
                    uint8_t* st = smem + s * CG_STAGE;
                    if (PAIR) {
                        // both CTAs' bytes complete on the leader's barrier
                        if (crank == 0) mbar_expect_tx(&full[s], 2 * CG_A + (uint32_t)BN * CG_BK * 2);
                        const uint32_t bar = leader_addr(&full[s]);
                        tma_load_3d_pair(st, &tmA, bar, 0, tm * CG_BM, z);
                        tma_load_3d_pair(st + CG_A, &tmB, bar, 0, tn * BN + crank * (BN / 2), z);
                    } else {
                        mbar_expect_tx(&full[s], CG_A + (uint32_t)BN * CG_BK * 2);
                        tma_load_3d(st, &tmA, &full[s], 0, tm * CG_BM, z);
                        tma_load_3d(st + CG_A, &tmB, &full[s], 0, tn * BN, z);
                    }
                    *issued = it + 1;
                }
            }
            if (PAIR) {
                // every slot free in both CTAs before the cluster may end
                for (int i = max(0, it - CG_STAGES); i < it; ++i)
                    if (!mbar_wait(&empty[i % CG_STAGES], (i / CG_STAGES) & 1)) atomicExch(err, 5);
            }
        }
    } else if (warp == 1) {
        if (crank == 0 && elect_one()) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                   ((uint32_t)((PAIR ? 2 * CG_BM : CG_BM) >> 4) << 24);
            int it = 0, j = 0;
            bool ok = true;
            for (int tile = tile0; tile < ntiles && ok; tile += tstep) {
                int tm, tn, mod, ks;
                locate(tile, tm, tn, mod, ks);
                const int kb = ks * g.kper, ke = min(g.nkb, kb + g.kper);
                for (int k0 = kb; k0 < ke && ok; k0 += kSegBlocks, ++j) {
                    const int buf = j & 1, u = j >> 1;
                    if (u > 0 && !mbar_wait(&acce[buf], (u - 1) & 1)) {
                        atomicExch(err, 4);
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(buf * 256);
                    const int k1 = min(ke, k0 + kSegBlocks);
                    for (int kt = k0; kt < k1; ++kt, ++it) {
                        const int s = it % CG_STAGES, round = it / CG_STAGES;
                        if (!mbar_wait(&full[s], round & 1)) {
                            atomicExch(err, 2);
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a0 = smem_u32(smem + s * CG_STAGE), b0 = a0 + CG_A;
#pragma unroll
                        for (int kk = 0; kk < CG_BK / 16; ++kk) {
                            const uint32_t acc = (kt > k0 || kk > 0) ? 1u : 0u;
                            if (PAIR) mma_bf16_pair(d, smem_desc(a0 + kk * 32), smem_desc(b0 + kk * 32), idesc, acc);
                            else mma_bf16(d, smem_desc(a0 + kk * 32), smem_desc(b0 + kk * 32), idesc, acc);
                        }
                        if (PAIR) mma_commit_pair(&empty[s]);
                        else mma_commit(&empty[s]);
                        *consumed = it + 1;
                    }
                    if (ok) {
                        if (PAIR) mma_commit_pair(&accf[buf]);
                        else mma_commit(&accf[buf]);
                    }
                }
            }
            if (!ok) {
                // let issued MMAs finish and drain copies that were not consumed
                if (PAIR) mma_commit_pair(&accf[j & 1]);
                else mma_commit(&accf[j & 1]);
                for (int i = *consumed; i < *issued; ++i) mbar_wait(&full[i % CG_STAGES], (i / CG_STAGES) & 1);
            }
        }
    } else {
        // warps 2..9: TMEM lane quarter warp % 4; warps 2..5 take the first
        // half of the tile's columns, warps 6..9 the second
        const int q = warp & 3, half = BN >> 1, c0 = ((warp - 2) >> 2) * half;
        const int nch = (half + 31) >> 5;
        const long N4 = (g.N + 3) >> 2;
        int j = 0;
        bool ok = true;
        for (int tile = tile0; tile < ntiles && ok; tile += tstep) {
            int tm, tn, mod, ks;
            locate(tile, tm, tn, mod, ks);
            const float p = d_tab.p[mod], ip = d_tab.inv_p[mod];
            const int kb = ks * g.kper, ke = min(g.nkb, kb + g.kper);
            float acc[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int x = 0; x < 32; ++x) acc[c][x] = 0.0f;
            for (int k0 = kb; k0 < ke; k0 += kSegBlocks, ++j) {
                const int buf = j & 1, u = j >> 1;
                ok = mbar_wait(&accf[buf], u & 1);
                tc_fence_after();
                if (!ok) {
                    atomicExch(err, 3);
                    break;
                }
                const uint32_t tb = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * 256 + c0);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (c < nch) {
                        uint32_t r[32];
                        tmem_ld32(tb + (uint32_t)(c * 32), r);
#pragma unroll
                        for (int x = 0; x < 32; ++x) acc[c][x] += reduce_mod(__uint_as_float(r[x]), p, ip);
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (PAIR) mbar_arrive_cluster(leader_addr(&acce[buf]));
                    else mbar_arrive(&acce[buf]);
                }
            }
            if (!ok) break;
            const long m = (long)tm * CG_BM + 32 * q + lane;
            if (m >= g.M) continue;
            uint32_t* out = g.planes + (long)(ks * kPlanes + mod) * N4 * g.M + m;
            const long n4 = ((long)tn * BN + c0) >> 2;
            // low byte of an FP32 word + kRint: the residue, or the sum's byte
            // (two loops: one with the choice inside issued both and took 1.8
            // times as long over a short k)
            auto store = [&](auto byte) {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (c < nch) {
#pragma unroll
                        for (int x = 0; x < 32; x += 4) {
                            if (c * 32 + x >= half || n4 + c * 8 + x / 4 >= N4) continue;
                            uint32_t w[4];
#pragma unroll
                            for (int y = 0; y < 4; ++y) w[y] = byte(acc[c][x + y]);
                            const uint32_t lo = __byte_perm(w[0], w[1], 0x0040), hi = __byte_perm(w[2], w[3], 0x0040);
                            out[(n4 + c * 8 + x / 4) * g.M] = __byte_perm(lo, hi, 0x5410);
                        }
                    }
            };
            if (mod == kMods)
                store([](float s) {
                    return s == 0.0f ? 0u : __float_as_uint(fminf(255.0f, fmaf(s, kSumScale, 0.75f)) + kRint);
                });
            else
                store([&](float r) { return __float_as_uint(reduce_mod(r, p, ip) + kRint); });
        }
    }
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    if (PAIR) cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem, 512);
        else tmem_dealloc(tmem, 512);
    }
}

// ---------------------------------------------------------------------------
// Chinese remainder and output
// ---------------------------------------------------------------------------
struct OutArgs {
    const uint32_t* planes;
    long M, N;
    int nsplit;
    const int *shift_m, *shift_n;
    const long *off_m, *off_n;
    double* C;
    double alpha, beta;
    unsigned* flags;        // [n / 16][m / 16] tiles with elements left to k_crt_patch
    long tilesM;
};

// sum_i q_i (P / p_i) mod P in 20-bit limbs, as a double times 2^-e
__device__ __forceinline__ double crt_value(const int* S, int e) {
    int c[kLimbs];
    int t = 0;
#pragma unroll
    for (int l = 0; l < kLimbs; ++l) {
        t += S[l];
        c[l] = t & 0xFFFFF;
        if (l + 1 < kLimbs) t >>= 20;
    }
    long long hi = ((long long)t << 40) | ((long long)c[4] << 20) | c[3];
    unsigned long long lo = ((unsigned long long)c[2] << 40) | ((unsigned long long)c[1] << 20) | (unsigned)c[0];
    const unsigned long long neg = hi < 0 ? 0x8000000000000000ull : 0ull;
    if (neg) {
        hi = ~hi + (lo == 0);
        lo = ((1ull << 60) - lo) & ((1ull << 60) - 1);
    }
    unsigned long long w1 = (unsigned long long)hi >> 4, w0 = ((unsigned long long)hi << 60) | lo;
    int ex;
    if (w1) {
        const int z = __clzll((long long)w1);
        if (z) {
            w1 = (w1 << z) | (w0 >> (64 - z));
            w0 <<= z;
        }
        ex = 127 - z;
    } else if (w0) {
        const int z = __clzll((long long)w0);
        w1 = w0 << z;
        w0 = 0;
        ex = 63 - z;
    } else {
        return 0.0;
    }
    unsigned long long m = w1 >> 11;
    const unsigned rem = (unsigned)w1 & 0x7FFu;
    if (rem > 0x400u || (rem == 0x400u && (w0 || (m & 1)))) ++m;  // to nearest, ties to even
    ex -= e;
    if (ex >= -1022 && ex <= 1022)
        return __longlong_as_double((long long)(neg | (((unsigned long long)(ex + 1023) << 52) + (m - (1ull << 52)))));
    const double v = scalbn((double)m, max(-4000, min(4000, ex - 52)));
    return neg ? -v : v;
}

// One thread per m and four n: 15 words of residues in, four elements out.
// About 40 integer operations per modulus and word, bound by the integer
// pipe; the words and C are read and written along m.  SPLIT: the residues
// of the k splits are added first (biased bytes in 16-bit lanes).
template <bool SPLIT>
__global__ void __launch_bounds__(128, 8) k_crt_out(const OutArgs a) {
    const long m = (long)blockIdx.x * 128 + threadIdx.x;
    if (m >= a.M) return;
    const long N4 = (a.N + 3) >> 2;
    const int sm = a.shift_m[m];
    const long om = a.off_m[m];
    for (long n4 = blockIdx.y; n4 < N4; n4 += gridDim.y) {
        int S[4][kLimbs];
        float kf[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int l = 0; l < kLimbs; ++l) S[y][l] = 0;
        const uint32_t* src = a.planes + n4 * a.M + m;
        const long plane = N4 * a.M;
        uint32_t w[kMods], even[SPLIT ? kMods : 1], odd[SPLIT ? kMods : 1];
        uint32_t sum = src[kMods * plane], sume = 0, sumo = 0;
#pragma unroll
        for (int i = 0; i < kMods; ++i) w[i] = src[i * plane];
        if (SPLIT) {
#pragma unroll
            for (int i = 0; i < kMods; ++i) {
                even[i] = (w[i] ^ 0x80808080u) & 0x00FF00FFu;
                odd[i] = ((w[i] ^ 0x80808080u) >> 8) & 0x00FF00FFu;
            }
            sume = sum & 0x00FF00FFu;
            sumo = (sum >> 8) & 0x00FF00FFu;
            for (int s = 1; s < a.nsplit; ++s) {
#pragma unroll
                for (int i = 0; i < kMods; ++i) w[i] = src[((long)s * kPlanes + i) * plane];
                sum = src[((long)s * kPlanes + kMods) * plane];
                sume += sum & 0x00FF00FFu;
                sumo += (sum >> 8) & 0x00FF00FFu;
#pragma unroll
                for (int i = 0; i < kMods; ++i) {
                    even[i] += (w[i] ^ 0x80808080u) & 0x00FF00FFu;
                    odd[i] += ((w[i] ^ 0x80808080u) >> 8) & 0x00FF00FFu;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kMods; ++i) {
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                int qi = (int)(int8_t)(w[i] >> (8 * y));
                if (SPLIT) {
                    qi = (int)(((y & 1 ? odd[i] : even[i]) >> (8 * (y & 2))) & 0xFFFFu) - 128 * a.nsplit;
                    const float f = __int_as_float(0x4B400000 + qi) - kRint;
                    qi = __float_as_int(reduce_mod(f, d_tab.p[i], d_tab.inv_p[i]) + kRint) - 0x4B400000;
                }
                kf[y] = fmaf(__int_as_float(0x4B400000 + qi) - kRint, d_tab.inv_p[i], kf[y]);
#pragma unroll
                for (int l = 0; l < kLimbs; ++l) S[y][l] += qi * d_tab.limb[i][l];
            }
        }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const long n = 4 * n4 + y;
            if (n >= a.N) break;
            const int k = __float_as_int(kf[y] + kRint) - 0x4B400000;
#pragma unroll
            for (int l = 0; l < kLimbs; ++l) S[y][l] -= k * d_tab.plimb[l];
            const int sn = a.shift_n[n];
            const int code = (int)(SPLIT ? ((y & 1 ? sumo : sume) >> (8 * (y & 2))) & 0xFFFFu : (sum >> (8 * y)) & 0xFFu);
            if (sm == kNonFinite || sn == kNonFinite || !sum_kept(code)) {
                a.flags[(n4 >> 2) * a.tilesM + (m >> 4)] = 1u;
                continue;
            }
            double v = crt_value(S[y], sm + sn);
            double* cp = a.C + om + a.off_n[n];
            v *= a.alpha;
            if (a.beta != 0.0) v = fma(a.beta, *cp, v);
            *cp = v;
        }
    }
}

// The elements that k_crt_out left, by 16 x 16 tiles.  A tile with up to 64 of
// them (a row or a column, a diagonal: exchange-antisymmetric amplitudes vanish
// where a diagonal of the other operand is large): a warp per element, its lanes over k.  Else the
// whole tile as FMAs of a chain per element.  K in pieces where few tiles are
// to share the chip (kchunk; the last block of a tile adds the pieces in
// order).  A block looks through the flags of its tiles 256 at a time.
struct PatchArgs {
    unsigned *flags, *count;  // [tile], count: arrivals of a tile's pieces
    long ntiles;
    int nsplit;
    long kchunk;
    double* ws;               // [tile][piece][256]
};

__global__ void __launch_bounds__(256) k_crt_patch(const Operand oa, const Operand ob, const OutArgs a,
                                                   const PatchArgs g) {
    constexpr int T = 16, KC = 32;
    __shared__ double As[KC][T + 1], Bs[KC][T + 1];
    __shared__ long ra[T], rb[T];
    __shared__ int list[256], nlist, elem[256], nelem;
    __shared__ double sums[256];
    __shared__ bool last;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const long N4 = (a.N + 3) >> 2, plane = N4 * a.M;
    const long kb = blockIdx.y * g.kchunk, ke = min(oa.K, kb + g.kchunk);
    for (long r = 0; r * gridDim.x + blockIdx.x < g.ntiles; r += 256) {
        const long mine = (r + tid) * gridDim.x + blockIdx.x;
        if (tid == 0) nlist = 0;
        __syncthreads();
        if (mine < g.ntiles && g.flags[mine]) list[atomicAdd(&nlist, 1)] = (int)mine;
        __syncthreads();
        for (int i = 0; i < nlist; ++i) {
            const long t = list[i], m0 = t % a.tilesM * T, n0 = t / a.tilesM * T, m = m0 + tx, n = n0 + ty;
            if (tid < T) ra[tid] = m0 + tid < a.M ? mode_offset((unsigned)(oa.r0 + m0 + tid), oa.nr, oa.rsz, oa.rs) : -1;
            else if (tid < 2 * T)
                rb[tid - T] = n0 + tid - T < a.N ? mode_offset((unsigned)(ob.r0 + n0 + tid - T), ob.nr, ob.rsz, ob.rs) : -1;
            else if (tid == 2 * T) nelem = 0;
            bool wanted = false;
            if (m < a.M && n < a.N) {
                int code = 0;
                for (int s = 0; s < a.nsplit; ++s)
                    code += (a.planes[((long)s * kPlanes + kMods) * plane + (n >> 2) * a.M + m] >> (8 * (n & 3))) & 0xFFu;
                wanted = a.shift_m[m] == kNonFinite || a.shift_n[n] == kNonFinite || !sum_kept(code);
            }
            __syncthreads();
            if (wanted) elem[atomicAdd(&nelem, 1)] = tid;
            __syncthreads();
            double acc = 0.0;
            if (nelem <= 64) {
                for (int e = tid >> 5; e < nelem; e += 8) {
                    const double *pa = oa.p + ra[elem[e] & 15], *pb = ob.p + rb[elem[e] >> 4];
                    double s = 0.0;
                    for (long k = kb + (tid & 31); k < ke; k += 32)
                        s = fma(pa[mode_offset((unsigned)(oa.k0 + k), oa.nk, oa.ksz, oa.ks)],
                                pb[mode_offset((unsigned)(ob.k0 + k), ob.nk, ob.ksz, ob.ks)], s);
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
                    if ((tid & 31) == 0) sums[elem[e]] = s;
                }
                __syncthreads();
                if (wanted) acc = sums[tid];
            } else {
                double x[2], y[2];
                auto fetch = [&](long k0) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int e = tid + 256 * h;
                        const int ka = oa.kfast ? e & 31 : e >> 4, ma = oa.kfast ? e >> 5 : e & 15;
                        const int kn = ob.kfast ? e & 31 : e >> 4, mn = ob.kfast ? e >> 5 : e & 15;
                        x[h] = k0 + ka < ke && ra[ma] >= 0
                                   ? oa.p[ra[ma] + mode_offset((unsigned)(oa.k0 + k0 + ka), oa.nk, oa.ksz, oa.ks)] : 0.0;
                        y[h] = k0 + kn < ke && rb[mn] >= 0
                                   ? ob.p[rb[mn] + mode_offset((unsigned)(ob.k0 + k0 + kn), ob.nk, ob.ksz, ob.ks)] : 0.0;
                    }
                };
                fetch(kb);
                for (long k0 = kb; k0 < ke; k0 += KC) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int e = tid + 256 * h;
                        if (oa.kfast) As[e & 31][e >> 5] = x[h];
                        else As[e >> 4][e & 15] = x[h];
                        if (ob.kfast) Bs[e & 31][e >> 5] = y[h];
                        else Bs[e >> 4][e & 15] = y[h];
                    }
                    __syncthreads();
                    if (k0 + KC < ke) fetch(k0 + KC);
                    const int kn = (int)min((long)KC, ke - k0);
                    for (int k = 0; k < kn; ++k) acc = fma(As[k][tx], Bs[k][ty], acc);
                    __syncthreads();
                }
            }
            bool write = wanted;
            if (g.nsplit > 1) {
                double* w = g.ws + t * g.nsplit * 256;
                w[blockIdx.y * 256 + tid] = acc;
                __threadfence();
                __syncthreads();
                if (tid == 0) last = atomicAdd(g.count + t, 1u) == (unsigned)g.nsplit - 1;
                __syncthreads();
                write = wanted && last;
                if (write) {
                    __threadfence();
                    acc = 0.0;
                    for (int s = 0; s < g.nsplit; ++s) acc += __ldcg(w + s * 256 + tid);
                }
            }
            if (write) {
                double* cp = a.C + a.off_m[m] + a.off_n[n];
                double v = acc * a.alpha;
                if (a.beta != 0.0) v = fma(a.beta, *cp, v);
                *cp = v;
            }
            __syncthreads();  // the tile's tables are free
        }
        __syncthreads();
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct CrtEngine {
    PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    uint8_t* ws = nullptr;  // workspace, allocated by the first contraction that pays
    size_t bytes = 0, want = 0;
    bool refused = false;   // it could not be allocated, or was given back
    int clusters = 0;       // resident two-CTA clusters (-1: none)
};

static long up(long x, long m) { return (x + m - 1) / m * m; }

// Workspace: every contraction's operands, residues and outputs whole up to
// 2 GB (larger ones run in pieces), at least 32 MB.  It is optional: a context
// whose calls stay in BF16 never has it, and without it every contraction
// stays on the CUDA cores.
dcsd_status crt_init(Ctx* c) {
    CrtEngine* e = new CrtEngine();
    c->crt = e;
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        c->err = "cuTensorMapEncodeTiled unavailable";
        return DCSD_ERR_CUDA;
    }
    e->encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    const double V = c->V, OV = (double)c->O * c->V, rows = 4.0 * c->O * c->O;
    const double want = 2.0 * kPlanes * 2.0 * ((V * V + rows) * (V * V + 64) + 2 * OV * (OV + 64)) + kPlanes * OV * OV;
    e->want = (size_t)std::min(2147483648.0, std::max(33554432.0, want)) / 1024 * 1024;
    DCSD_CUDA(c, cudaFuncSetAttribute(k_crt_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCrtSmem));
    DCSD_CUDA(c, cudaFuncSetAttribute(k_crt_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCrtSmem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(c->num_sms / 2 * 2));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kCrtSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&e->clusters, k_crt_gemm<true>, &cfg) != cudaSuccess || e->clusters < 1) {
        cudaGetLastError();
        e->clusters = -1;
    }
    return DCSD_OK;
}

void crt_free(Ctx* c) {
    if (!c->crt) return;
    if (c->crt->ws) cudaFree(c->crt->ws);
    delete c->crt;
    c->crt = nullptr;
}

static dcsd_status make_map(Ctx* c, CUtensorMap* map, const uint16_t* p, long rows, long nz, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)CG_BK, (cuuint64_t)rows, (cuuint64_t)nz};
    cuuint64_t strides[2] = {(cuuint64_t)(CG_BK * 2), (cuuint64_t)(rows * CG_BK * 2)};
    cuuint32_t box[3] = {CG_BK, (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    const CUresult r = c->crt->encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)p, dims, strides, box, es,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        c->err = "cuTensorMapEncodeTiled (residues) failed (" + std::to_string((int)r) + ")";
        return DCSD_ERR_CUDA;
    }
    return DCSD_OK;
}

bool crt_ready(Ctx* c) {
    CrtEngine* e = c->crt;
    if (!e) return false;
    if (!e->ws && !e->refused) {
        // (nothing can be allocated while the caller or graph_record captures the stream)
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(c->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
            cudaGetLastError();
            return false;
        }
        if (cudaMalloc((void**)&e->ws, e->want) == cudaSuccess) {
            e->bytes = e->want;
        } else {
            cudaGetLastError();
            e->ws = nullptr;
            e->refused = true;
        }
    }
    return e->ws != nullptr;
}

const void* crt_workspace(const Ctx* c) { return c->crt ? c->crt->ws : nullptr; }

cudaError_t dev_malloc(Ctx* c, void** p, size_t bytes) {
    cudaError_t st = cudaMalloc(p, bytes);
    CrtEngine* e = c->crt;
    if (st != cudaErrorMemoryAllocation || !e || !e->ws) return st;
    cudaGetLastError();
    cudaFree(e->ws);  // (waits for the launches that use it)
    e->ws = nullptr;
    e->bytes = 0;
    e->refused = true;
    return cudaMalloc(p, bytes);
}

// k per partial norm: a multiple of 128, at most 32 pieces
static int norm_chunk(long K) { return (int)std::max<long>(128, up((K + 31) / 32, 128)); }

static long patch_tiles(long M, long N) { return ((M + 15) / 16) * ((N + 15) / 16); }

// bytes of a pass: residues of both operands, row tables, residues of the output, flags
static size_t pass_bytes(long M, long N, long K, long nsplit) {
    const size_t nkb = (size_t)(K + 63) / 64, nch = (size_t)(K + norm_chunk(K) - 1) / norm_chunk(K);
    return (size_t)(M + N) * (nkb * 64 * 2 * kPlanes + nch * 16 + 16) + (size_t)nsplit * kPlanes * 4 * ((N + 3) / 4) * M +
           8 * (size_t)patch_tiles(M, N) + 16 * 256;
}

// one pass: rows [m0, m0 + M), columns [n0, n0 + N), k [k0, k0 + K)
static dcsd_status crt_pass(Ctx* c, const char* spec, const GemmPlan& p, const double* Ap, const double* Bp,
                            double* Cp, double alpha, double beta, long m0, long M, long n0, long N, long k0, long K) {
    CrtEngine* e = c->crt;
    GemmShape g;
    g.M = M;
    g.N = N;
    g.nkb = (int)((K + 63) / 64);
    g.tilesM = (int)((M + CG_BM - 1) / CG_BM);
    g.tilesN = (int)((N + 255) / 256);
    const bool pair = c->tc_pairs && e->clusters > 0 && g.tilesM > 1;
    g.BN = (int)up((N + g.tilesN - 1) / g.tilesN, pair ? 32 : 16);
    const long tilesMs = pair ? (g.tilesM + 1) / 2 : g.tilesM;
    const long slots = pair ? e->clusters : c->num_sms;
    const long t1 = tilesMs * g.tilesN * kPlanes;
    // few output tiles: k split over the idle SMs (a pass reduces the splits' residues)
    long ns = std::max<long>(1, std::min<long>({slots / t1, (long)g.nkb / 8, (long)kMaxSplit}));
    while (ns > 1 && pass_bytes(M, N, K, ns) > e->bytes) --ns;
    g.kper = (int)((g.nkb + ns - 1) / ns);
    g.nsplit = (g.nkb + g.kper - 1) / g.kper;
    g.group = (int)std::max<long>(1, std::min<long>(tilesMs, std::lround(std::sqrt((double)slots * g.BN / CG_BM / (pair ? 2 : 1)))));
    // (recorded: a piece of the workspace of its own when it is large enough)
    const size_t need = pass_bytes(M, N, K, g.nsplit);
    const size_t at = need <= e->bytes / 2 ? dag_slice(c, 3, (need + 255) / 256 * 256, e->bytes) : 0;
    uint8_t* w = e->ws + at;
    auto take = [&](size_t bytes) {
        uint8_t* r = w;
        w += (bytes + 255) / 256 * 256;
        return r;
    };
    Operand o[2];
    std::memset(o, 0, sizeof(o));
    for (int s = 0; s < 2; ++s) {
        Operand& x = o[s];
        x.p = s == 0 ? Ap : Bp;
        x.nr = s == 0 ? p.nm : p.nn;
        x.nk = p.nk;
        for (int i = 0; i < kMaxMode; ++i) {
            x.rsz[i] = s == 0 ? p.m_size[i] : p.n_size[i];
            x.rs[i] = s == 0 ? p.m_sa[i] : p.n_sb[i];
            x.rc[i] = s == 0 ? p.m_sc[i] : p.n_sc[i];
            x.ksz[i] = p.k_size[i];
            x.ks[i] = s == 0 ? p.k_sa[i] : p.k_sb[i];
        }
        x.rows = s == 0 ? M : N;
        x.r0 = s == 0 ? m0 : n0;
        x.K = K;
        x.k0 = k0;
        const long rf = x.nr > 0 ? std::labs(x.rs[x.nr - 1]) : LONG_MAX;
        const long kf = x.nk > 0 ? std::labs(x.ks[x.nk - 1]) : LONG_MAX;
        x.kfast = kf <= rf ? 1 : 0;
        x.beta = s == 0 ? kBetaA : kBetaB;
        x.side = s;
        x.nkb = g.nkb;
        x.kchunk = norm_chunk(K);
        x.nchunk = (int)((K + x.kchunk - 1) / x.kchunk);
        x.dst = (uint16_t*)take((size_t)kPlanes * g.nkb * 64 * x.rows * 2);
        x.part_ss = (double*)take((size_t)x.nchunk * x.rows * 8);
        x.part_mx = (unsigned long long*)take((size_t)x.nchunk * x.rows * 8);
        x.shift = (int*)take((size_t)x.rows * 4);
        x.coff = (long*)take((size_t)x.rows * 8);
    }
    const long N4 = (N + 3) / 4;
    g.planes = (uint32_t*)take((size_t)g.nsplit * kPlanes * 4 * N4 * M);
    const long ptiles = patch_tiles(M, N);
    unsigned* flags = (unsigned*)take((size_t)ptiles * 8);
    if ((size_t)(w - e->ws) > e->bytes || (size_t)(w - e->ws) > at + need) {
        c->err = std::string(spec) + ": modular GEMM workspace";
        return DCSD_ERR_INVALID_ARG;
    }
    auto view_of = [](const double* p0, int na, const long* sa, const long* ta, int nb, const long* sb, const long* tb,
                      bool write) {
        long n = 1;
        for (int i = 0; i < na; ++i) n += (sa[i] - 1) * ta[i];
        for (int i = 0; i < nb; ++i) n += (sb[i] - 1) * tb[i];
        return Span{p0, p0 + n, write};
    };
    const DagOp op(c, {view_of(Ap, p.nm, p.m_size, p.m_sa, p.nk, p.k_size, p.k_sa, false),
                       view_of(Bp, p.nn, p.n_size, p.n_sb, p.nk, p.k_size, p.k_sb, false),
                       view_of(Cp, p.nm, p.m_size, p.m_sc, p.nn, p.n_size, p.n_sc, true),
                       wr(e->ws + at, (size_t)(w - e->ws) - at)});
    prof_begin(c, DCSD_PROF_FP64);
    auto label = [&](const char* what) {
        return std::string(what) + spec + " M=" + std::to_string(M) + " N=" + std::to_string(N) + " K=" +
               std::to_string(K) + (g.nsplit > 1 ? " split=" + std::to_string(g.nsplit) : "");
    };
    for (int s = 0; s < 2; ++s) o[s].blocks = (o[s].rows + (o[s].kfast ? 7 : 63)) / (o[s].kfast ? 8 : 64) * o[s].nchunk;
    if (c->trace) trace_begin(c, label("crt-norm "));
    k_crt_norm<<<(unsigned)(o[0].blocks + o[1].blocks), 256, 0, c->stream>>>(o[0], o[1]);
    trace_end(c);
    DCSD_TRY(launch_check(c, "crt_norm"));
    for (int s = 0; s < 2; ++s) {
        // several k-blocks per block while at least eight blocks per SM remain
        const long rb = (o[s].rows + 63) / 64;
        o[s].kbper = (int)std::max<long>(1, std::min<long>(8, rb * o[s].nkb / (8l * c->num_sms)));
        o[s].blocks = rb * ((o[s].nkb + o[s].kbper - 1) / o[s].kbper);
    }
    if (c->trace) trace_begin(c, label("crt-pack "));
    k_crt_pack<<<(unsigned)(o[0].blocks + o[1].blocks), 256, 0, c->stream>>>(o[0], o[1], flags, 2 * ptiles);
    trace_end(c);
    DCSD_TRY(launch_check(c, "crt_pack"));
    CUtensorMap ma, mb;
    DCSD_TRY(make_map(c, &ma, o[0].dst, M, (long)kPlanes * g.nkb, CG_BM));
    DCSD_TRY(make_map(c, &mb, o[1].dst, N, (long)kPlanes * g.nkb, pair ? g.BN / 2 : g.BN));
    if (c->trace) trace_begin(c, label(pair ? "crt-gemm-pairs " : "crt-gemm "));
    const long nt = tilesMs * g.tilesN * kPlanes * g.nsplit;
    if (pair) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(2 * std::min<long>(nt, slots)));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kCrtSmem;
        cfg.stream = c->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        DCSD_CUDA(c, cudaLaunchKernelEx(&cfg, k_crt_gemm<true>, ma, mb, g, c->tc_err));
    } else {
        k_crt_gemm<false><<<(unsigned)std::min<long>(nt, slots), kThreads, kCrtSmem, c->stream>>>(ma, mb, g, c->tc_err);
    }
    trace_end(c);
    DCSD_TRY(launch_check(c, "crt_gemm"));
    OutArgs a;
    a.planes = g.planes;
    a.M = M;
    a.N = N;
    a.nsplit = g.nsplit;
    a.shift_m = o[0].shift;
    a.shift_n = o[1].shift;
    a.off_m = o[0].coff;
    a.off_n = o[1].coff;
    a.C = Cp;
    a.alpha = alpha;
    a.beta = beta;
    a.flags = flags;
    a.tilesM = (M + 15) / 16;
    if (c->trace) trace_begin(c, label("crt-out "));
    dim3 grid((unsigned)((M + 127) / 128), (unsigned)std::min<long>(N4, 65535));
    if (g.nsplit > 1) k_crt_out<true><<<grid, 128, 0, c->stream>>>(a);
    else k_crt_out<false><<<grid, 128, 0, c->stream>>>(a);
    trace_end(c);
    DCSD_TRY(launch_check(c, "crt_out"));
    // the residues of A are not needed any more: pieces of the patch's sums
    PatchArgs q;
    q.flags = flags;
    q.count = flags + ptiles;
    q.ntiles = ptiles;
    q.nsplit = 1;
    q.ws = (double*)o[0].dst;
    if (ptiles < 2l * c->num_sms) {
        const long room = (long)((size_t)kPlanes * g.nkb * 64 * M * 2 / (2048ul * ptiles));
        q.nsplit = (int)std::max<long>(1, std::min<long>({(2l * c->num_sms + ptiles - 1) / ptiles, K / 256, room}));
    }
    q.kchunk = up((K + q.nsplit - 1) / q.nsplit, 32);
    q.nsplit = (int)((K + q.kchunk - 1) / q.kchunk);
    if (c->trace) trace_begin(c, label("crt-patch "));
    k_crt_patch<<<dim3((unsigned)std::min<long>(ptiles, 6l * c->num_sms), (unsigned)q.nsplit), 256, 0, c->stream>>>(
        o[0], o[1], a, q);
    trace_end(c);
    prof_end(c, DCSD_PROF_FP64);
    return launch_check(c, "crt_patch");
}

// C = alpha A B + beta C on the modular GEMM (NB = 1, crt_ready)
dcsd_status einsum_crt(Ctx* c, const char* spec, const GemmPlan& plan, const double* Ap, const double* Bp, double* Cp,
                       double alpha, double beta) {
    GemmPlan p = plan;
    // row orders within M and N are free: by decreasing stride in C
    auto order = [](int n, long* size, long* so, long* sc) {
        for (int a = 1; a < n; ++a)
            for (int b = a; b > 0 && std::labs(sc[b - 1]) < std::labs(sc[b]); --b) {
                std::swap(size[b - 1], size[b]);
                std::swap(so[b - 1], so[b]);
                std::swap(sc[b - 1], sc[b]);
            }
    };
    order(p.nm, p.m_size, p.m_sa, p.m_sc);
    order(p.nn, p.n_size, p.n_sb, p.n_sc);
    // the m side (lanes) takes C's contiguous axis, unless the tiles of the
    // other assignment hold a fifth less padding over a long k
    const long mf = p.nm > 0 ? std::labs(p.m_sc[p.nm - 1]) : LONG_MAX, nf = p.nn > 0 ? std::labs(p.n_sc[p.nn - 1]) : LONG_MAX;
    auto padded = [](long m, long n) {
        const long t = (n + 255) / 256;
        return (double)up(m, CG_BM) * (double)(t * up((n + t - 1) / t, 16));
    };
    bool swap = nf < mf;
    const double now = swap ? padded(p.N, p.M) : padded(p.M, p.N), alt = swap ? padded(p.M, p.N) : padded(p.N, p.M);
    if (p.K >= 512 && alt < 0.8 * now) swap = !swap;
    if (swap) {
        const GemmPlan q = p;
        p.nm = q.nn; p.nn = q.nm; p.M = q.N; p.N = q.M;
        for (int i = 0; i < kMaxMode; ++i) {
            p.m_size[i] = q.n_size[i]; p.m_sa[i] = q.n_sb[i]; p.m_sc[i] = q.n_sc[i];
            p.n_size[i] = q.m_size[i]; p.n_sb[i] = q.m_sa[i]; p.n_sc[i] = q.m_sc[i];
            p.k_sa[i] = q.k_sb[i]; p.k_sb[i] = q.k_sa[i];
        }
        std::swap(Ap, Bp);
    }
    // pieces that fit the workspace: k first (a piece's sum is exact, the
    // pieces add in FP64), then n, then m
    const size_t cap = c->crt->bytes;
    long Kc = p.K, Nc = p.N, Mc = p.M;
    while (pass_bytes(Mc, Nc, Kc, 1) > cap) {
        if (Kc > 16384) Kc = up((Kc + 1) / 2, 1024);
        else if (Mc > 4096 || (Mc >= Nc && Mc > 128)) Mc = up((Mc + 1) / 2, 128);
        else if (Nc > 256) Nc = up((Nc + 1) / 2, 256);
        else if (Kc > 1024) Kc = up((Kc + 1) / 2, 1024);
        else {
            c->err = std::string(spec) + ": modular GEMM workspace";
            return DCSD_ERR_INVALID_ARG;
        }
    }
    for (long k0 = 0; k0 < p.K; k0 += Kc)
        for (long n0 = 0; n0 < p.N; n0 += Nc)
            for (long m0 = 0; m0 < p.M; m0 += Mc)
                DCSD_TRY(crt_pass(c, spec, p, Ap, Bp, Cp, alpha, k0 == 0 ? beta : 1.0, m0, std::min(Mc, p.M - m0), n0,
                                  std::min(Nc, p.N - n0), k0, std::min(Kc, p.K - k0)));
    return DCSD_OK;
}

}  // namespace dcsd
