// gemm_crt.cu -- exact ring GEMM mod 2^64 and mod 2^128 from residue products
// (Chinese remainder theorem) on the fp16 tensor cores, for layers large in
// both output dimensions.
//
// Computes Z = C + L . R mod 2^(64 W) with L = [E | X + cE] (M x 2K) and
// R = [B ; F] (2K x N), the same product as gemm_tc.cu.  There every element is
// split into 8 W byte digits, which takes 36 (W = 1) or 136 (W = 2) digit
// products.  Here the integer product V = L . R of the signed representatives
// is computed modulo NP = 16 or 31 pairwise coprime moduli p_i <= 512 whose
// product exceeds 2 |V|, one fp16 product each, and rebuilt (the integer
// modular scheme of Ozaki, Uchino and Imamura, "Ozaki Scheme II", 2025):
//     c_i = V (P/p_i)^-1 mod p_i,   V = sum_i c_i (P/p_i) - q P,
//     q = round(sum_i c_i / p_i),   P = prod p_i.
// Only V mod 2^(64 W) is needed, so P/p_i and P enter mod 2^(64 W).  The factor
// (P/p_i)^-1 mod p_i is folded into the residues of R.
//
// Exactness.  Representatives lie within 2^63 (1 + 2^-4 + 2^-13) (W = 1) or
// 2^127 (1 + 2^-7) (W = 2) in magnitude, so |V| <= 1.13 2K 2^126 (1.02 2K 2^254);
// P = 2^142.96 (2^273.59) leaves |V| / P < 0.30 up to 2K = 2^15, so rounding
// sum c_i / p_i, computed with an error below 0.02, to the nearest integer gives
// q exactly.  Residues are integers of magnitude <= 256, exact in fp16; 256
// products of 2^16 sum to at most 2^24, so the fp32 accumulation over 256 K
// values is exact, and the accumulators are reduced mod p_i every 256 K values.
//
// Three launches on the caller's stream, each a programmatic dependent of the
// one before:
//   1. residue_kernel  L and R as NP fp16 residue planes in the workspace, in
//      the shared-memory image of the MMA (K-major, no swizzle, 8 x 16-byte core
//      matrices).  Elements are split into 10-bit pieces; small warp-level MMAs
//      multiply the pieces by 2^(10 j) mod p_i, and the sums are reduced in
//      packed fp32.  Bound: memory (8 W bytes read, 2 NP written per element);
//      measured 7.2 ps per element in Z_2^64 (floor 5.9), 13.6 in Z_2^128 (15.6
//      where cE is added; 11.5).
//      With fp32 multiply-adds in place of the small MMAs Z_2^128 took 31 ps.
//   2. residue_gemm_kernel  plain fp16 GEMMs, one per (modulus, output tile):
//      CTA pairs (cta_group::2) on 256 x 256 tiles, because one CTA per tile
//      would read and fill its shared memory faster than its 128 bytes a clock;
//      two 256-column accumulator sets alternate, drained every 256 K values
//      by eight warps per CTA that reduce mod p_i in packed fp32.  Bound: the
//      tensor cores; measured 0.85-0.95 of the fp16 rate on 4096 x 4096 x 4096
//      in Z_2^64.  (Layers whose planes exceed L2 but that have few outputs are
//      bound by reading the planes, as in Z_2^128 at 2048 x 2304 x 256.)
//   3. combine_kernel  Z = C + V mod 2^(64 W) from the NP residues of each
//      output, by small MMAs again.  Bound: memory (2 NP + 16 W bytes per output).
//
// Share calls, digit tiles (gemm_tc.cu) -> this path, measured on GB300:
// Z_2^64 2048 x 1024 x 4096 841 -> 507 us, 2048 x 1024 x 1024 233 -> 158 us,
// 4096 x 4096 x 4096 6.6 -> 3.3 ms, 1000 x 999 x 1001 (odd N, integer pipes)
// 928 -> 115 us; Z_2^128 2048 x 2304 x 256 606 -> 331 us, 512 x 4608 x 512
// 503 -> 274 us, 512 x 512 x 512 80 -> 46 us.  Splitting the operands costs
// (M + N) 2K elements against 2 M N K multiply-adds, so layers with one small
// side (128 x 4096 x 4096, convolutions with 64 outputs) stay with the digits.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "kernels.h"
#include "sm100_ptx.cuh"

namespace mpcl {

namespace {

__device__ unsigned int g_crt_timeout = 0;

// ---------------------------------------------------------------------------
// moduli and derived tables

constexpr int MAXNP = 31;
constexpr int kModuli[MAXNP] = {512, 511, 509, 505, 503, 501, 499, 493, 491, 487, 481, 479, 473, 467, 463, 461,
                                457, 449, 443, 439, 437, 433, 431, 421, 419, 409, 401, 397, 389, 383, 379};

template <int W> struct Crt {
    static constexpr int NP = W == 1 ? 16 : 31;       // moduli
    static constexpr int NPT = W == 1 ? 2 : 4;        // groups of 8 moduli (MMA columns), the last padded
    static constexpr int PIECES = W == 1 ? 7 : 13;    // 10-bit pieces of an element
    static constexpr int OUT = W == 1 ? 6 : 12;       // 11-bit pieces of P / p_i mod 2^(64 W)
};

constexpr int gcd_(int a, int b) { return b == 0 ? a : gcd_(b, a % b); }
constexpr bool coprime_all() {
    for (int i = 0; i < MAXNP; ++i)
        for (int j = 0; j < i; ++j)
            if (gcd_(kModuli[i], kModuli[j]) != 1) return false;
    return true;
}
static_assert(coprime_all(), "the moduli are pairwise coprime");
constexpr double product(int n) {
    double p = 1;
    for (int i = 0; i < n; ++i) p *= kModuli[i];
    return p;
}
constexpr double pow2(int n) { return n == 0 ? 1.0 : 2.0 * pow2(n - 1); }
constexpr int64_t CRT_MAX_K2 = int64_t(1) << 15;   // padded inner dimension 2K
static_assert(0.30 * product(16) > 1.13 * pow2(15) * pow2(126) && 0.30 * product(31) > 1.02 * pow2(15) * pow2(254),
              "|V| / P stays below 0.30");

// symmetric residue of a (a >= 0)
constexpr int sym(int64_t a, int p) {
    int r = (int)(a % p);
    return 2 * r > p ? r - p : r;
}

// fp16 bits of an integer |v| <= 1024 (exact)
constexpr uint16_t half_bits(int v) {
    if (v == 0) return 0;
    const int a = v < 0 ? -v : v;
    int e = 0;
    while ((2 << e) <= a) ++e;                        // 2^e <= a < 2^(e + 1)
    return (uint16_t)((v < 0 ? 0x8000 : 0) | ((e + 15) << 10) | ((a << (10 - e)) & 0x3FF));
}

// Right operands of the small MMAs that split elements into residues and put
// residues together, as fp16 pairs of consecutive K in the fragment order
// (value [k / 2][n] holds rows k, k + 1 of column n), and the moduli.
template <int W> struct Tables {
    uint32_t w[2][8][8 * Crt<W>::NPT];    // k: piece j, n: modulus i: 2^(10 j) mod p_i; side 1 times (P/p_i)^-1
    uint32_t out[4 * Crt<W>::NPT][8 * W]; // k: modulus i, n: piece j of P/p_i; column OUT: 1 / p_i
    float ip[8 * Crt<W>::NPT], np[8 * Crt<W>::NPT];   // 1 / p_i, -p_i
    float P[8 * W];                       // pieces of P
    uint32_t ip2[8 * Crt<W>::NPT], np2[8 * Crt<W>::NPT];   // fp16 pairs (1 / p_i twice, -p_i twice)
};

// fp16 bits of 1 / p rounded down to 11 bits (relative error below 2^-10)
constexpr uint16_t inv_bits(int p) {
    int e = 0;
    while ((1 << e) < p) ++e;                         // 2^(e - 1) < p <= 2^e: 1 / p in [2^-e, 2^(1 - e))
    const int m = (int)((int64_t(1) << (e + 10)) / p);   // 1024 <= m <= 2047: 1 / p ~ m 2^(-e - 10)
    return (uint16_t)(((15 - e) << 10) | (m & 0x3FF));
}

template <int W> constexpr Tables<W> make_tables() {
    constexpr int NP = Crt<W>::NP;
    Tables<W> t{};
    for (int i = 0; i <= NP; ++i) {
        // P / p_i (row NP: P) mod 2^128 and mod p_i
        unsigned __int128 c = 1;
        int64_t m = 1;
        for (int j = 0; j < NP; ++j)
            if (j != i) {
                c *= (unsigned)kModuli[j];
                if (i < NP) m = m * kModuli[j] % kModuli[i];
            }
        // signed 11-bit pieces, the carry out of the top one dropped mod 2^(64 W)
        for (int j = 0; j < Crt<W>::OUT; ++j) {
            int d = (int)(c & 2047);
            c >>= 11;
            if (d >= 1024) {
                d -= 2048;
                c += 1;
            }
            if (i == NP) t.P[j] = (float)d;
            else t.out[i / 2][j] |= (uint32_t)half_bits(d) << (16 * (i & 1));
        }
        if (i == NP) break;
        const int p = kModuli[i];
        t.out[i / 2][Crt<W>::OUT] |= (uint32_t)inv_bits(p) << (16 * (i & 1));
        int64_t inv = 1;
        while (inv * m % p != 1) ++inv;
        int64_t w = 1;
        for (int j = 0; j < Crt<W>::PIECES; ++j) {
            t.w[0][j / 2][i] |= (uint32_t)half_bits(sym(w, p)) << (16 * (j & 1));
            t.w[1][j / 2][i] |= (uint32_t)half_bits(sym(w * inv % p, p)) << (16 * (j & 1));
            w = w * 1024 % p;
        }
        t.ip[i] = (float)(1.0 / p);
        t.np[i] = (float)-p;
        t.ip2[i] = inv_bits(p) * 0x10001u;
        t.np2[i] = half_bits(-p) * 0x10001u;
    }
    return t;
}

// read per lane, so in global and not in constant memory
__device__ const Tables<1> d_tab1 = make_tables<1>();
__device__ const Tables<2> d_tab2 = make_tables<2>();
template <int W> __device__ __forceinline__ const Tables<W>& tab() {
    if constexpr (W == 1) return d_tab1;
    else return d_tab2;
}

// D += A . B for one 16 x 8 tile: fp16 operands, fp32 sums, exact for the
// integers used here
__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// packed fp32 arithmetic on two values (half the issue slots)
__device__ __forceinline__ u64 pack2(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ u64 add_f32x2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fma_f32x2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// two integers |v| <= 2^24 mod p, within (p + 1) / 2 of zero: adding 1.5 2^23
// rounds v / p to an integer
__device__ __forceinline__ u64 reduce_mod2(u64 v, u64 ip, u64 np) {
    constexpr u64 R = 0x4B4000004B400000ull, NR = 0xCB400000CB400000ull;   // +-1.5 2^23 twice
    return fma_f32x2(add_f32x2(fma_f32x2(v, ip, R), NR), np, v);
}

// ---------------------------------------------------------------------------
// 1. residue planes

constexpr int KS = 16;      // K of one MMA step
constexpr int KB = 64;      // K of one operand stage (4 steps)
constexpr int KD = 256;     // K between reductions of the accumulators

struct ResidueSide {
    uint8_t* planes;
    int64_t mod_stride;     // bytes between the planes of consecutive moduli
    int64_t rows;           // M (left) or N (right)
    int rt;                 // rows per tile image (128 or 64)
    int tiles;              // tiles converted: ceil(rows / rt)
    int side;               // 0: the left operand, 1: the right one
    int blocks;
};

struct ResidueParams {
    const u64 *E, *X, *B, *F, *alpha;
    int coef, one_half;
    int64_t M, K, N, Kp;
    int kb;                 // 64-deep stages per tile
    ResidueSide s[2];       // s[0]: A tiles of the MMA, s[1]: B tiles
};

// Pieces of an element x for this lane's A fragment.  Adding `bias` makes the
// signed 10-bit pieces non-negative: x + bias = sum_j u_j 2^(10 j), and the
// representative sum_j (u_j - o_j) 2^(10 j) = x mod 2^(64 W) lies in
// [-bias, 2^(64 W) - bias), o_j = 512 (the top piece: 8 or 128, so that bias is
// close to half of the ring).  A pair of pieces becomes fp16 by placing each
// under 0x64 (1024 + u) and subtracting 1024 + o.  Lane t = lane % 4 holds
// pieces 2t, 2t + 1 and (W = 2) 8 + 2t, 9 + 2t; pieces past the last have zero
// weights.
constexpr u64 BIAS_LO = (1ull << 9) | (1ull << 19) | (1ull << 29) | (1ull << 39) | (1ull << 49) | (1ull << 59);
template <int W> struct Splitter {
    uint32_t sh, sub, sh2, sub2;
    int t;
    __device__ __forceinline__ explicit Splitter(int t_) : t(t_) {
        if constexpr (W == 1) {
            sh = (20 * t) & 31;                                       // bits 20 t: words (0, 1) or (1, -)
            sub = t == 3 ? 0x64006408u : 0x66006600u;                 // piece 6: 1024 + 8
            sh2 = sub2 = 0;
        } else {
            sh = t < 2 ? 20 * t : 20 * t - 32;                        // bits 20 t: words (0, 1) or (1, 2)
            sub = 0x66006600u;
            sh2 = t == 0 ? 16 : t == 1 ? 4 : 24;                      // bits 80 + 20 t: words (2, 3) or (3, -)
            sub2 = t == 2 ? 0x64006480u : 0x66006600u;                // piece 12: 1024 + 128
        }
    }
    static __device__ __forceinline__ uint32_t pair(uint32_t f, uint32_t sub) {
        const uint32_t r = (f & 0x3FFu) | 0x64006400u | ((f << 6) & 0x03FF0000u);
        uint32_t h;
        asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(r), "r"(sub));
        return h;
    }
    __device__ __forceinline__ void split(typename Elem<W>::T x, uint32_t& a, uint32_t& a2) const {
        if constexpr (W == 1) {
            const u64 y = x + (BIAS_LO | (1ull << 63));
            const uint32_t w0 = (uint32_t)y, w1 = (uint32_t)(y >> 32);
            a = pair(__funnelshift_r(t < 2 ? w0 : w1, t < 2 ? w1 : 0u, sh), sub);
            a2 = 0;
        } else {
            constexpr u64 HI = (1ull << 5) | (1ull << 15) | (1ull << 25) | (1ull << 35) | (1ull << 45) | (1ull << 55) |
                               (1ull << 63);                          // 2^(9 + 10 j), j = 6 .. 11, and 2^127
            const u128 y = x + ((u128)BIAS_LO | ((u128)HI << 64));
            const uint32_t w0 = (uint32_t)y, w1 = (uint32_t)(y >> 32), w2 = (uint32_t)(y >> 64), w3 = (uint32_t)(y >> 96);
            a = pair(__funnelshift_r(t < 2 ? w0 : w1, t < 2 ? w1 : w2, sh), sub);
            a2 = pair(__funnelshift_r(t == 0 ? w2 : w3, t == 0 ? w3 : 0u, sh2), sub2);
        }
    }
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// A chunk of a warp: 16 rows of L (columns of R) x CK values of K, staged in
// shared memory as 16 lines of 128 bytes (padded by 16, so that the fragment
// reads hit distinct banks): line = row of L, or K value of R (W = 2: K value
// and half of the 16 columns).  The X half of L also stages E when cE is added.
template <int W> struct Chunk {
    static constexpr int CK = W == 1 ? 16 : 8;
    static constexpr int LINE = 144, BYTES = 16 * LINE;
    static constexpr int DEPTH = 3;                       // chunks in flight
    static constexpr int WARPS = 8;
    static constexpr int SMEM = WARPS * DEPTH * 2 * BYTES;
};

struct ChunkAt {
    uint32_t tile, ks, rg;     // tile image, CK-deep step, group of 16 rows
};

// A warp takes chunks in turn.  For each K value one small MMA per 8 moduli
// multiplies the rows' pieces by the pieces' weights, so lane (g, t) ends with
// rows g and g + 8 of moduli 2t, 2t + 1 and packs 8 K values of each into one
// 16-byte row of a core matrix.
template <int W>
__global__ void __launch_bounds__(256, 2) residue_kernel(const __grid_constant__ ResidueParams p) {
    using T = typename Elem<W>::T;
    using Ch = Chunk<W>;
    constexpr int NPT = Crt<W>::NPT, CK = Ch::CK, DEPTH = Ch::DEPTH;
    extern __shared__ __align__(1024) uint8_t smem[];
    ptx::grid_dep_launch();
    const bool second = (int)blockIdx.x >= p.s[0].blocks;
    const ResidueSide& sd = p.s[second ? 1 : 0];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const Splitter<W> sp(t);
    uint32_t b[NPT][W];
    u64 ip[NPT], np[NPT];
#pragma unroll
    for (int n = 0; n < NPT; ++n) {
        b[n][0] = tab<W>().w[sd.side][t][8 * n + g];
        if constexpr (W == 2) b[n][1] = tab<W>().w[sd.side][t + 4][8 * n + g];
        ip[n] = pack2(tab<W>().ip[8 * n + 2 * t], tab<W>().ip[8 * n + 2 * t + 1]);
        np[n] = pack2(tab<W>().np[8 * n + 2 * t], tab<W>().np[8 * n + 2 * t + 1]);
    }
    const uint32_t per = (uint32_t)sd.rt / 16u, steps = (uint32_t)p.kb * (KB / CK);
    const uint32_t total = (uint32_t)sd.tiles * steps * per, nw = (uint32_t)sd.blocks * Ch::WARPS;
    const uint32_t w0 = ((uint32_t)blockIdx.x - (second ? p.s[0].blocks : 0)) * Ch::WARPS + warp;
    const bool left = sd.side == 0, pairs = W == 2 || ((left ? p.K : p.N) & 1) == 0;
    const uint32_t sbase = ptx::smem_u32(smem) + warp * (DEPTH * 2 * Ch::BYTES);
    auto at = [&](uint32_t id) {
        const uint32_t ts = id / per;
        const uint32_t tile = ts / steps;
        return ChunkAt{tile, ts - tile * steps, id - ts * per};
    };
    ptx::grid_dep_wait();
    const T c = p.coef == COEF_ALPHA ? ld_elem<W>(p.alpha, 0) : (T)1;

    // copies of chunk id into stage s (zeros outside the matrix)
    auto fetch = [&](uint32_t id, uint32_t s) {
        if (id < total) {
            const ChunkAt x = at(id);
            const int64_t kp0 = (int64_t)x.ks * CK, row0 = (int64_t)x.tile * sd.rt + x.rg * 16;
            const bool first = !p.one_half && kp0 < p.Kp;
            const int64_t kk = (first || p.one_half) ? kp0 : kp0 - p.Kp;
            const bool add = left && !first && p.coef != COEF_ZERO;
            const u64* src = left ? (first ? p.E : p.X) : (first ? p.B : p.F);
            const uint32_t dst = sbase + s * (2 * Ch::BYTES) + (lane & 7) * 16;
            constexpr int EPV = 2 / W;                  // elements per 16 bytes
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int line = i * 4 + (lane >> 3);
                int64_t e, n;                           // first element, elements inside the matrix
                if (left) {
                    const int64_t k = kk + (lane & 7) * EPV;
                    e = (row0 + line) * p.K + k;
                    n = row0 + line < sd.rows ? p.K - k : 0;
                } else {
                    const int64_t k = kk + (W == 1 ? line : line >> 1);
                    const int64_t col = row0 + (lane & 7) * EPV + (W == 1 ? 0 : (line & 1) * 8);
                    e = k * p.N + col;
                    n = k < p.K ? p.N - col : 0;
                }
                const int cnt = n <= 0 ? 0 : n >= EPV ? EPV : 1;
                const uint32_t d = dst + line * Ch::LINE;
                const int64_t o = cnt > 0 ? e * W : 0;
                if (pairs) {
                    cp_async16(d, src + o, cnt * 8 * W);
                    if (add) cp_async16(d + Ch::BYTES, p.E + o, cnt * 8 * W);
                } else {
                    const int64_t o1 = cnt > 1 ? o + 1 : 0;
                    cp_async8(d, src + o, cnt > 0 ? 8 : 0);
                    cp_async8(d + 8, src + o1, cnt > 1 ? 8 : 0);
                    if (add) {
                        cp_async8(d + Ch::BYTES, p.E + o, cnt > 0 ? 8 : 0);
                        cp_async8(d + Ch::BYTES + 8, p.E + o1, cnt > 1 ? 8 : 0);
                    }
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    for (uint32_t s = 0; s < DEPTH - 1; ++s) fetch(w0 + s * nw, s);
    uint32_t s = 0;
#pragma unroll 1
    for (uint32_t id = w0; id < total; id += nw, s = s + 1 == DEPTH ? 0 : s + 1) {
        fetch(id + (DEPTH - 1) * nw, s == 0 ? DEPTH - 1 : s - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH - 1) : "memory");
        __syncwarp();
        const ChunkAt x = at(id);
        const int64_t kp0 = (int64_t)x.ks * CK;
        const bool add = left && (p.one_half || kp0 >= p.Kp) && p.coef != COEF_ZERO;
        const uint8_t* raw = smem + warp * (DEPTH * 2 * Ch::BYTES) + s * (2 * Ch::BYTES);
        uint8_t* dst = sd.planes + ((int64_t)x.tile * p.kb * (KB / KS) + kp0 / KS) * (sd.rt * 32) + x.rg * 512 + g * 16 +
                       (W == 2 ? (x.ks & 1) * 128 : 0) + 2 * t * sd.mod_stride;
#pragma unroll 1
        for (int kh = 0; kh < CK / 8; ++kh) {
            T x0[8], x1[8];
            auto gather = [&](const uint8_t* q, T (&y0)[8], T (&y1)[8]) {
                if constexpr (W == 1) {
                    if (left) {
#pragma unroll
                        for (int j = 0; j < 8; j += 2) {
                            const uint8_t* a = q + g * Ch::LINE + kh * 64 + j * 8;
                            const ulonglong2 v0 = *reinterpret_cast<const ulonglong2*>(a);
                            const ulonglong2 v1 = *reinterpret_cast<const ulonglong2*>(a + 8 * Ch::LINE);
                            y0[j] = v0.x, y0[j + 1] = v0.y, y1[j] = v1.x, y1[j + 1] = v1.y;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const uint8_t* a = q + (kh * 8 + j) * Ch::LINE + g * 8;
                            y0[j] = *reinterpret_cast<const u64*>(a);
                            y1[j] = *reinterpret_cast<const u64*>(a + 64);
                        }
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint8_t* a = left ? q + g * Ch::LINE + j * 16 : q + 2 * j * Ch::LINE + g * 16;
                        y0[j] = ld_elem<2>(reinterpret_cast<const u64*>(a), 0);
                        y1[j] = ld_elem<2>(reinterpret_cast<const u64*>(a + (left ? 8 : 1) * Ch::LINE), 0);
                    }
                }
            };
            gather(raw, x0, x1);
            if (add) {
                T e0[8], e1[8];
                gather(raw + Ch::BYTES, e0, e1);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    x0[j] += c * e0[j];
                    x1[j] += c * e1[j];
                }
            }
            uint32_t a[8][4];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                sp.split(x0[j], a[j][0], a[j][2]);
                sp.split(x1[j], a[j][1], a[j][3]);
            }
#pragma unroll
            for (int n = 0; n < NPT; ++n) {
                uint32_t h[4][4];                   // [fragment value][K pair]
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    float d[2][4], r[2][4];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) d[e][q] = 0.0f;
                        if constexpr (W == 1) mma_k8(d[e], a[j + e][0], a[j + e][1], b[n][0]);
                        else mma_k16(d[e], a[j + e], b[n][0], b[n][W - 1]);
#pragma unroll
                        for (int q = 0; q < 4; q += 2)
                            unpack2(reduce_mod2(pack2(d[e][q], d[e][q + 1]), ip[n], np[n]), r[e][q], r[e][q + 1]);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h[q][j / 2]) : "f"(r[1][q]), "f"(r[0][q]));
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (8 * n + 2 * t + (q & 1) < Crt<W>::NP)
                        *reinterpret_cast<uint4*>(dst + (8 * n + (q & 1)) * sd.mod_stride + (q >> 1) * 256 + kh * 128) =
                            make_uint4(h[q][0], h[q][1], h[q][2], h[q][3]);
            }
        }
        __syncwarp();      // the stage is read before the next fetch into it
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------------------
// 2. the residue GEMMs

constexpr int STAGES = 6;
constexpr uint32_t A_STAGE = 128 * KB * 2;       // 16 KB: 128 rows of the A tile per CTA
constexpr int NWARPS = 12;                       // 0: producer, 1: MMA (rank 0), 4-11: drain
constexpr int NT = NWARPS * 32;
constexpr uint32_t TMEM_COLS = 512;
constexpr long long WAIT_LIMIT = 4000000000LL;   // clock cycles (about 2 s)
constexpr int TM = 256;                          // rows of the pair's tile

template <int BN> struct GemmLayout {
    static constexpr uint32_t B_STAGE = BN / 2 * KB * 2;      // BN / 2 rows of the B tile per CTA
    static constexpr uint32_t STAGE = A_STAGE + B_STAGE;
    static constexpr uint32_t OFF_BAR = STAGES * STAGE;
    static constexpr int NBARS = 2 * STAGES + 2 + 2 + 1;
    static constexpr uint32_t SMEM = OFF_BAR + NBARS * 8 + 16;
};
static_assert(GemmLayout<256>::SMEM <= 227 * 1024, "shared memory");

// The planes are read through 2-D tensor maps with 128-byte rows (a tile image
// is a run of consecutive rows), because only tensor copies may complete on the
// barrier of the pair's other CTA.
constexpr int MAP_ROW = 128;

struct GemmParams {
    CUtensorMap tmA, tmB;
    int a_mod, b_mod;         // map rows between the planes of consecutive moduli
    uint8_t* res;
    int a_tiles, b_tiles;     // tile images present (128 rows; BN / 2 rows)
    int mt, nt;               // tiles of TM x BN
    int kb;                   // 64-deep stages of the inner dimension
    int splits, kps;          // K splits and stages per split (a multiple of 4)
    int units;                // NP splits mt nt
};

struct UnitAt {
    int mod, split, m, n, kb0, nkb;
};
__device__ __forceinline__ UnitAt unit_at(const GemmParams& p, int u) {
    UnitAt x;
    const int T = p.mt * p.nt, ms = u / T, t = u - ms * T;
    x.mod = ms / p.splits;
    x.split = ms - x.mod * p.splits;
    x.n = t / p.mt;
    x.m = t - x.n * p.mt;
    x.kb0 = x.split * p.kps;
    x.nkb = min(p.kb - x.kb0, p.kps);
    return x;
}

__device__ __forceinline__ void gave_up(volatile int* abort_flag) {
    *abort_flag = 1;
    atomicExch(&g_crt_timeout, 1u);
}

template <int W, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NT, 1)
residue_gemm_kernel(const __grid_constant__ GemmParams p) {
    using Lay = GemmLayout<BN>;
    constexpr uint32_t STAGE = Lay::STAGE;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + Lay::OFF_BAR);   // rank 0: both CTAs' copies have landed
    uint64_t* empty = full + STAGES;      // the MMAs that read the stage are done
    uint64_t* accFull = empty + STAGES;
    uint64_t* accEmpty = accFull + 2;     // rank 0: both CTAs' drains have read the set
    uint64_t* done = accEmpty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_rank();
    const int pair = blockIdx.x >> 1, npair = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&accFull[b], 1);
            ptx::mbar_init(&accEmpty[b], 16);   // eight drain warps in each CTA
        }
        ptx::mbar_init(done, 1);
        *abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0) {
        ptx::tmem_alloc_pair(tmem_slot, TMEM_COLS);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync();   // both CTAs' barriers are initialised
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    ptx::grid_dep_wait();  // the residue planes

    if (warp == 0) {
        int it = 0;
        bool ok = true;
        if (lane == 0) {
            ptx::prefetch_tmap(&p.tmA);
            ptx::prefetch_tmap(&p.tmB);
        }
        const uint32_t full0 = ptx::mapa(full, 0);
        for (int u = pair; u < p.units && ok; u += npair) {
            const UnitAt x = unit_at(p, u);
            const int ta = min(2 * x.m + (int)rank, p.a_tiles - 1), tb = min(2 * x.n + (int)rank, p.b_tiles - 1);
            constexpr int AR = A_STAGE / MAP_ROW, BR = Lay::B_STAGE / MAP_ROW;   // map rows per stage
            const int a = x.mod * p.a_mod + (ta * p.kb + x.kb0) * AR, b = x.mod * p.b_mod + (tb * p.kb + x.kb0) * BR;
            for (int j = 0; j < x.nkb; ++j, ++it) {
                const int s = it % STAGES;
                if (!__all_sync(0xffffffffu,
                                ptx::mbar_wait(&empty[s], ((it / STAGES) & 1) ^ 1, abort_flag, WAIT_LIMIT))) {
                    if (lane == 0) gave_up(abort_flag);
                    ok = false;
                    break;
                }
                // both CTAs' copies complete on rank 0's barrier, which expects
                // their bytes together
                const uint32_t leader = ptx::elect_one();
                ptx::mbar_arrive_expect_tx_if(leader && rank == 0, &full[s], 2 * STAGE);
                ptx::tma_load_2d_pair_if(leader, smem + s * STAGE, &p.tmA, 0, a + j * AR, full0 + s * 8);
                ptx::tma_load_2d_pair_if(leader, smem + s * STAGE + A_STAGE, &p.tmB, 0, b + j * BR, full0 + s * 8);
            }
        }
        // copies still in flight land before either CTA exits
        if (rank == 0)
            for (int j = max(0, it - STAGES); j < it; ++j)
                ptx::mbar_wait_cluster(&full[j % STAGES], (j / STAGES) & 1, abort_flag, WAIT_LIMIT);
    } else if (warp == 1 && rank == 1) {
        ptx::mbar_wait(done, 0, abort_flag, WAIT_LIMIT);   // the last arrival from rank 0 has landed
    } else if (warp == 1) {
        const uint32_t base = ptx::smem_u32(smem);
        constexpr uint32_t idesc = ptx::idesc_f16_f32(TM, BN);
        int it = 0, v = 0;
        bool ok = true;
        for (int u = pair; u < p.units && ok; u += npair) {
            const UnitAt x = unit_at(p, u);
            for (int j = 0; j < x.nkb; ++j, ++it) {
                const int set = v & 1;
                if (j % (KD / KB) == 0) {
                    if (!__all_sync(0xffffffffu, ptx::mbar_wait_cluster(&accEmpty[set], ((v >> 1) & 1) ^ 1, abort_flag,
                                                                        WAIT_LIMIT))) {
                        if (lane == 0) gave_up(abort_flag);
                        ok = false;
                        break;
                    }
                }
                const int s = it % STAGES;
                if (!__all_sync(0xffffffffu,
                                ptx::mbar_wait_cluster(&full[s], (it / STAGES) & 1, abort_flag, WAIT_LIMIT))) {
                    if (lane == 0) gave_up(abort_flag);
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const uint32_t leader = ptx::elect_one();
#pragma unroll
                for (int k = 0; k < KB / KS; ++k) {
                    const uint64_t ad = ptx::smem_desc_kmajor(base + s * STAGE + k * 4096, 128, 256);
                    const uint64_t bd = ptx::smem_desc_kmajor(base + s * STAGE + A_STAGE + k * (BN / 2 * 32), 128, 256);
                    ptx::mma_f16_pair_if(leader, tmem + set * 256, ad, bd, idesc,
                                         (j % (KD / KB) == 0 && k == 0) ? 0u : 1u);
                }
                ptx::mma_commit_pair_if(leader, &empty[s]);
                if (j % (KD / KB) == KD / KB - 1 || j == x.nkb - 1) {
                    ptx::mma_commit_pair_if(leader, &accFull[set]);
                    ++v;
                }
            }
        }
        // every MMA of the pair completes before either CTA's memory is released
        ptx::mma_commit_pair_if(ptx::elect_one(), done);
        ptx::mbar_wait(done, 0, abort_flag, WAIT_LIMIT);
    } else if (warp >= 4) {
        // lane l of quadrant q: row 32 q + l of this CTA's half, BN / 2 of the tile's columns
        const int quad = warp & 3, half = (warp - 4) >> 2;
        constexpr int NC = BN / 2;
        const uint32_t empty0[2] = {ptx::mapa(&accEmpty[0], 0), ptx::mapa(&accEmpty[1], 0)};
        u64 acc[NC / 2];       // sums of residues, two fp32 columns each
        int v = 0;
        bool ok = true;
        for (int u = pair; u < p.units && ok; u += npair) {
            const UnitAt x = unit_at(p, u);
            const float ip1 = tab<W>().ip[x.mod], np1 = tab<W>().np[x.mod];
            const u64 ip = pack2(ip1, ip1), np = pack2(np1, np1);
#pragma unroll
            for (int c = 0; c < NC / 2; ++c) acc[c] = 0;
            for (int j = 0; j < x.nkb; j += KD / KB, ++v) {
                const int set = v & 1;
                if (!__all_sync(0xffffffffu, ptx::mbar_wait(&accFull[set], (v >> 1) & 1, abort_flag, WAIT_LIMIT))) {
                    if (lane == 0) gave_up(abort_flag);
                    ok = false;
                    break;
                }
                ptx::tc_fence_after();
                const uint32_t t0 = tmem + ((uint32_t)(quad * 32) << 16) + set * 256 + half * NC;
#pragma unroll
                for (int c0 = 0; c0 < NC; c0 += 32) {
                    uint32_t f[32];
                    ptx::tmem_ld32(t0 + c0, f);
                    ptx::tmem_wait_ld();
                    if (c0 + 32 == NC) {
                        ptx::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive_cluster(empty0[set]);
                    }
#pragma unroll
                    for (int c = 0; c < 32; c += 2)
                        acc[(c0 + c) / 2] = add_f32x2(
                            acc[(c0 + c) / 2],
                            reduce_mod2(pack2(__uint_as_float(f[c]), __uint_as_float(f[c + 1])), ip, np));
                }
            }
            if (!ok) break;
            // residues of 8 columns per 16-byte vector, rows contiguous
            const int64_t tile = ((int64_t)(x.mod * p.splits + x.split) * p.mt + x.m) * p.nt + x.n;
            uint8_t* dst = p.res + ((tile * (BN / 8) + half * (NC / 8)) * TM + rank * 128 + quad * 32 + lane) * 16;
#pragma unroll
            for (int c = 0; c < NC; c += 8) {
                uint32_t h[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float a0, a1;
                    unpack2(reduce_mod2(acc[c / 2 + q], ip, np), a0, a1);
                    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h[q]) : "f"(a1), "f"(a0));
                }
                *reinterpret_cast<uint4*>(dst + (int64_t)(c / 8) * TM * 16) = make_uint4(h[0], h[1], h[2], h[3]);
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync();   // neither CTA leaves while the other may still use its memory
    ptx::tc_fence_after();
    if (warp == 0) ptx::tmem_dealloc_pair(tmem, TMEM_COLS);
}

// ---------------------------------------------------------------------------
// 3. Z = C + V mod 2^(64 W)

struct CombineParams {
    const uint8_t* res;
    const u64* C;       // NULL: no addend
    u64* Z;
    int64_t M, N;
    int swap;           // the A tiles hold columns of R: tile rows are output columns
    int mt, nt, bn, splits;
};

// A warp rebuilds the outputs of 16 tile rows x 8 tile columns.  Its residues (a
// 16-byte vector of 8 columns per row and modulus) are staged in shared memory
// and read back transposed as A fragments of small MMAs (rows = 16 outputs, K =
// moduli) whose columns are the pieces S_j = sum_i c_i (P/p_i)_j and sum_i c_i /
// p_i (fp16 inverses, 2^-10 relative: error below 31 / 2 2^-10 in the sum).  Every S_j is an integer below 2^23.
// The four lanes of a quad then hold the pieces of the same outputs; they
// exchange partial sums so that each ends with one row's output.
template <int W> struct Combine {
    static constexpr int WARPS = 8, ROWS = 16;
    static constexpr int MODS = 8 * Crt<W>::NPT;
    static constexpr int STRIDE = ROWS * 16 + 16;     // bytes per modulus (padded: conflict-free transposed reads)
    static constexpr int SMEM = WARPS * MODS * STRIDE;
};

__device__ __forceinline__ uint32_t add2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// two fp16 integers (|v| < 2048) mod p, within p / 2 + 1 of zero: rounding to
// an integer by adding 1536
__device__ __forceinline__ uint32_t reduce2(uint32_t v, uint32_t ip, uint32_t np) {
    uint32_t q;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(q) : "r"(v), "r"(ip), "r"(0x66006600u));
    q = add2(q, 0xE600E600u);
    asm("fma.rn.f16x2 %0, %0, %1, %2;" : "+r"(q) : "r"(np), "r"(v));
    return q;
}

// 16-byte load at this point of the program (plain ones are moved about by the
// compiler: the split sums below then spilled 100 bytes)
__device__ __forceinline__ uint4 ld_vec(const uint8_t* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

template <typename T>
__device__ __forceinline__ T shfl_xor_elem(T v, int o) {
    if constexpr (sizeof(T) == 8) {
        return __shfl_xor_sync(0xffffffffu, v, o);
    } else {
        const u64 lo = __shfl_xor_sync(0xffffffffu, (u64)v, o), hi = __shfl_xor_sync(0xffffffffu, (u64)(v >> 64), o);
        return (u128)lo | ((u128)hi << 64);
    }
}

template <int W>
__global__ void __launch_bounds__(256, W == 1 ? 4 : 3) combine_kernel(const __grid_constant__ CombineParams p) {
    constexpr int NP = Crt<W>::NP, NPT = Crt<W>::NPT, OUT = Crt<W>::OUT, STRIDE = Combine<W>::STRIDE;
    constexpr int KT = NPT / 2;          // 16-deep MMA steps over the moduli
    constexpr int TC = OUT % 8;          // column of sum c_i / p_i in the last 8-column tile
    using T = typename Elem<W>::T;
    extern __shared__ __align__(1024) uint8_t smem[];
    ptx::grid_dep_launch();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    uint32_t b[W][KT][2];
#pragma unroll
    for (int n = 0; n < W; ++n)
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            b[n][k][0] = tab<W>().out[8 * k + t][8 * n + g];
            b[n][k][1] = tab<W>().out[8 * k + t + 4][8 * n + g];
        }
    float P[W][2];
#pragma unroll
    for (int n = 0; n < W; ++n)
#pragma unroll
        for (int q = 0; q < 2; ++q) P[n][q] = tab<W>().P[8 * n + 2 * t + q];
    ptx::grid_dep_wait();   // the residues
    // warp task: (8-column group of a tile, 16 tile rows)
    constexpr int ROWS = Combine<W>::ROWS;
    const int task = blockIdx.x * Combine<W>::WARPS + warp;
    const int gi = task / (TM / ROWS), r0 = (task % (TM / ROWS)) * ROWS;
    const int gpt = p.bn / 8, tile = gi / gpt, gc = gi - tile * gpt;
    if (tile >= p.mt * p.nt) return;
    const int tm = tile / p.nt, tn = tile - tm * p.nt;
    const int64_t a0 = (int64_t)tm * TM + r0, b0 = (int64_t)tn * p.bn + gc * 8;
    const int64_t na = p.swap ? p.N : p.M, nb = p.swap ? p.M : p.N;
    if (a0 >= na || b0 >= nb) return;
    uint8_t* st = smem + warp * (Combine<W>::MODS * STRIDE);
    const int64_t stride = (int64_t)p.mt * p.nt * gpt * TM * 16;      // bytes per (modulus, split)
    // half-warps take alternate moduli, lanes consecutive rows
    const int lr = lane & 15, lm = lane >> 4;
    const uint8_t* src = p.res + ((int64_t)gi * TM + r0 + lr) * 16;
    if (p.splits == 1) {
#pragma unroll
        for (int i = 0; i < 8 * NPT; i += 2) {
            const int m = i + lm;
            cp_async16(ptx::smem_u32(st) + m * STRIDE + lr * 16, src + (int64_t)(m < NP ? m : 0) * stride,
                       m < NP ? 16 : 0);
        }
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    } else {
        // add the splits' residues (at most MAX_SPLITS 257 < 2048: exact in
        // fp16) and reduce them again, so that the sums below stay exact
#pragma unroll 4
        for (int i = 0; i < 8 * NPT; i += 2) {
            const int m = i + lm;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (m < NP) {
                const uint8_t* a = src + (int64_t)m * p.splits * stride;
                v = ld_vec(a);
                for (int s = 1; s < p.splits; ++s) {
                    const uint4 y = ld_vec(a + s * stride);
                    v = make_uint4(add2(v.x, y.x), add2(v.y, y.y), add2(v.z, y.z), add2(v.w, y.w));
                }
                const uint32_t ip = tab<W>().ip2[m], np = tab<W>().np2[m];
                v = make_uint4(reduce2(v.x, ip, np), reduce2(v.y, ip, np), reduce2(v.z, ip, np), reduce2(v.w, ip, np));
            }
            *reinterpret_cast<uint4*>(st + m * STRIDE + lr * 16) = v;
        }
    }
    __syncwarp();
    // four rows at a time: two MMA tiles of two rows (16 outputs) each
    const uint32_t fbase = ptx::smem_u32(st) + (uint32_t)((lane & 7) + ((lane >> 4) & 1) * 8) * STRIDE +
                           (uint32_t)((lane >> 3) & 1) * 16;
#pragma unroll 2
    for (int r = 0; r < ROWS; r += 4) {
        T part[4];      // this lane's part of output column g of rows r .. r + 3
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float d[W][4];
#pragma unroll
            for (int n = 0; n < W; ++n)
#pragma unroll
                for (int q = 0; q < 4; ++q) d[n][q] = 0.0f;
#pragma unroll
            for (int k = 0; k < KT; ++k) {
                uint32_t a[4];   // matrices: (row, moduli 0-7), (row + 1, 0-7), (row, 8-15), (row + 1, 8-15)
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                             : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                             : "r"(fbase + (uint32_t)(k * 16) * STRIDE + (uint32_t)(r + 2 * h) * 16)
                             : "memory");
#pragma unroll
                for (int n = 0; n < W; ++n) mma_k16(d[n], a, b[n][k][0], b[n][k][1]);
            }
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                // q = round(sum c_i / p_i) from the lane that holds that column
                const float qf = -rintf(__shfl_sync(0xffffffffu, d[W - 1][2 * v + (TC & 1)], (lane & 28) | (TC / 2)));
                T s = 0;
#pragma unroll
                for (int n = 0; n < W; ++n) {
                    const int d0 = __float2int_rn(__fmaf_rn(qf, P[n][0], d[n][2 * v]));
                    const int d1 = __float2int_rn(__fmaf_rn(qf, P[n][1], d[n][2 * v + 1]));
                    const long long w = (long long)d0 + (long long)d1 * 2048;
                    if (8 * n + 2 * t < OUT) s += (T)w << (88 * n + 22 * t);
                }
                part[2 * h + v] = s;
            }
        }
        // this lane's output; its addend arrives during the exchange below
        const int64_t ar = a0 + r + t, bc = b0 + g, e = p.swap ? bc * p.N + ar : ar * p.N + bc;
        const T c = p.C && ar < na && bc < nb ? ld_elem<W>(p.C, e) : (T)0;
        // lane t keeps row r + t: pairs exchange halves, then the pairs' halves
        const bool t0 = t & 1, t1 = t & 2;
        const T k0 = (t0 ? part[1] : part[0]) + shfl_xor_elem<T>(t0 ? part[0] : part[1], 1);
        const T k1 = (t0 ? part[3] : part[2]) + shfl_xor_elem<T>(t0 ? part[2] : part[3], 1);
        const T z = (t1 ? k1 : k0) + shfl_xor_elem<T>(t1 ? k0 : k1, 2);
        if (ar < na && bc < nb) st_elem<W>(p.Z, e, z + c);
    }
}

// ---------------------------------------------------------------------------
// host side

int sm_pairs() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 74;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 2) return 74;
    return n / 2;
}

constexpr int MAX_SPLITS = 6;

struct CrtPlan {
    int swap, bn, np;
    int64_t ra, rb;                // rows of the A side and of the B side
    int a_tiles, b_tiles, mt, nt;
    int64_t Kp;
    int kb, splits, kps;
    int64_t a_mod, b_mod;
    size_t off_b, off_res, total;
    double us;                     // estimated time of the call
};

// Measured on GB300: one 64-deep stage of 256 columns on a CTA pair (0.93 of
// the measured fp16 rate under its power limit), and storing and reading one
// residue of one output.
constexpr double STAGE_US = 0.35, RESIDUE_US = 6.0e-7;

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

CrtPlan crt_plan(int64_t M, int64_t K, int64_t N, int words, int one_half) {
    CrtPlan q{};
    q.np = words == 1 ? Crt<1>::NP : Crt<2>::NP;
    // A side: 256-row tiles; the operand that fills them better, L unless R^T does
    const int64_t padL = cdiv(M, TM) * TM, padR = cdiv(N, TM) * TM;
    q.swap = M < 256 && (double)padL / M > (double)padR / N;
    q.ra = q.swap ? N : M;
    q.rb = q.swap ? M : N;
    // B side: 256 columns unless 128 leave much less padding (a 128-column tile
    // reads the A operand twice as often)
    q.bn = cdiv(q.rb, 128) * 128 * 5 < cdiv(q.rb, 256) * 256 * 4 ? 128 : 256;
    q.a_tiles = (int)cdiv(q.ra, 128);
    q.b_tiles = (int)cdiv(q.rb, q.bn / 2);
    q.mt = (int)cdiv(q.ra, TM);
    q.nt = (int)cdiv(q.rb, q.bn);
    q.Kp = cdiv(K, KS) * KS;
    q.kb = (int)cdiv((one_half ? 1 : 2) * q.Kp, KB);
    q.a_mod = (int64_t)q.a_tiles * q.kb * A_STAGE;
    q.b_mod = (int64_t)q.b_tiles * q.kb * (q.bn / 2 * KB * 2);
    // K splits: the number with the least time of the GEMM's waves of units over
    // 76 pairs plus that of storing and reading its residues
    const int64_t T = (int64_t)q.mt * q.nt * q.np;
    q.us = -1.0;
    for (int s = 1; s <= MAX_SPLITS; ++s) {
        const int kps = (int)cdiv(cdiv(q.kb, s), KD / KB) * (KD / KB);
        if ((int)cdiv(q.kb, kps) != s) continue;
        const double us = (double)cdiv(T * s, 76) * kps * STAGE_US * q.bn / 256 +
                          (double)s * q.mt * q.nt * TM * q.bn * q.np * RESIDUE_US;
        if (q.us < 0 || us < q.us) {
            q.us = us;
            q.splits = s;
            q.kps = kps;
        }
    }
    // estimate of the whole call, fitted to 45 share calls per ring (mean error 6-7 %)
    const double el = (double)(q.a_tiles * 128 + q.b_tiles * (q.bn / 2)) * q.kb * KB;
    const double stages = (double)cdiv(T * q.splits, 76) * q.kps * q.bn / 256;
    const double res = (double)q.splits * q.mt * q.nt * TM * q.bn * q.np;
    q.us = words == 1 ? 14.4 + 1.01e-5 * el + 0.293 * stages + 1.15e-6 * res
                      : 12.9 + 2.25e-5 * el + 0.209 * stages + 0.80e-6 * res;
    auto up = [](int64_t b) { return (size_t)((b + 255) / 256 * 256); };
    q.off_b = up(q.a_mod * q.np);
    q.off_res = q.off_b + up(q.b_mod * q.np);
    q.total = q.off_res + up((int64_t)q.np * q.splits * q.mt * q.nt * TM * q.bn * 2);
    return q;
}

// map over a side's planes: 128-byte rows, one box per stage image
bool make_plane_map(CUtensorMap* map, const uint8_t* base, int64_t bytes, int64_t stage) {
    auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tensor_map_encoder());
    if (!fn) return false;
    cuuint64_t dims[2] = {MAP_ROW / 2, (cuuint64_t)(bytes / MAP_ROW)};
    cuuint64_t strides[1] = {MAP_ROW};
    cuuint32_t box[2] = {MAP_ROW / 2, (cuuint32_t)(stage / MAP_ROW)};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint8_t*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// the dynamic shared-memory opt-in of a kernel, once per device
template <auto Kernel> cudaError_t allow_smem(int bytes) {
    static std::atomic<bool> set[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    if (dev >= 0 && dev < 64 && set[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && dev >= 0 && dev < 64) set[dev].store(true, std::memory_order_relaxed);
    return e;
}

template <int W, int BN>
cudaError_t launch_residue_gemm(const GemmParams& gp, cudaStream_t st) {
    const cudaError_t e = allow_smem<residue_gemm_kernel<W, BN>>(GemmLayout<BN>::SMEM);
    if (e != cudaSuccess) return e;
    const int pairs = std::min(sm_pairs(), gp.units);
    return launch_dependent(residue_gemm_kernel<W, BN>, dim3(2 * pairs), dim3(NT), GemmLayout<BN>::SMEM, st, gp);
}

template <int W>
cudaError_t run(const GemmArgs& a, const CrtPlan& q, uint8_t* ws, cudaStream_t st) {
    ResidueParams rp{a.E, a.X, a.B, a.F, a.alpha, a.coef, a.one_half, a.M, a.K, a.N, q.Kp, q.kb, {}};
    // two blocks per SM, shared out between the sides by their sizes
    const int64_t ca = (int64_t)q.a_tiles * 128, cb = (int64_t)q.b_tiles * (q.bn / 2);    // rows converted
    const int64_t warps = (ca + cb) / 16 * q.kb * (KB / Chunk<W>::CK);
    const int nblk = (int)std::min<int64_t>(4 * sm_pairs(), std::max<int64_t>(2, cdiv(warps, Chunk<W>::WARPS)));
    const int nb0 = std::min(nblk - 1, std::max(1, (int)((double)nblk * ca / (ca + cb) + 0.5)));
    rp.s[0] = ResidueSide{ws, q.a_mod, q.ra, 128, q.a_tiles, q.swap ? 1 : 0, nb0};
    rp.s[1] = ResidueSide{ws + q.off_b, q.b_mod, q.rb, q.bn / 2, q.b_tiles, q.swap ? 0 : 1, nblk - nb0};
    cudaError_t e = allow_smem<residue_kernel<W>>(Chunk<W>::SMEM);
    if (e != cudaSuccess) return e;
    e = launch_dependent(residue_kernel<W>, dim3((unsigned)nblk), dim3(256), Chunk<W>::SMEM, st, rp);
    if (e != cudaSuccess) return e;
    GemmParams gp{};
    if (!make_plane_map(&gp.tmA, ws, q.a_mod * q.np, A_STAGE) ||
        !make_plane_map(&gp.tmB, ws + q.off_b, q.b_mod * q.np, q.bn / 2 * KB * 2))
        return cudaErrorInvalidValue;
    gp = GemmParams{gp.tmA, gp.tmB, (int)(q.a_mod / MAP_ROW), (int)(q.b_mod / MAP_ROW), ws + q.off_res, q.a_tiles, q.b_tiles, q.mt, q.nt, q.kb,
                  q.splits, q.kps, q.np * q.splits * q.mt * q.nt};
    e = q.bn == 256 ? launch_residue_gemm<W, 256>(gp, st) : launch_residue_gemm<W, 128>(gp, st);
    if (e != cudaSuccess) return e;
    CombineParams cp{ws + q.off_res, a.C, a.Z, a.M, a.N, q.swap, q.mt, q.nt, q.bn, q.splits};
    using Cm = Combine<W>;
    e = allow_smem<combine_kernel<W>>(Cm::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t tasks = (int64_t)q.mt * q.nt * (q.bn / 8) * (TM / Cm::ROWS);
    e = launch_dependent(combine_kernel<W>, dim3((unsigned)cdiv(tasks, Cm::WARPS)), dim3(256), Cm::SMEM, st,
                         cp);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

namespace {
// the plan of a shape that the kernels can run
bool feasible_plan(int64_t M, int64_t K, int64_t N, int words, int one_half, CrtPlan& q) {
    if ((words != 1 && words != 2) || M < 1 || N < 1 || K < 1) return false;
    if (2 * cdiv(K, KS) * KS > CRT_MAX_K2) return false;
    q = crt_plan(M, K, N, words, one_half);
    // 32-bit block, unit and thread counts
    const double threads = (double)(q.a_tiles * 128.0 + q.b_tiles * (q.bn / 2.0)) * q.kb * 8;
    if (q.total / MAP_ROW >= (size_t(1) << 31)) return false;   // map coordinates
    return threads < 4.0e9 && (double)q.np * q.splits * q.mt * q.nt < 1e9 &&
           (double)q.mt * q.nt * (q.bn / 8) * 2 < 2e9;
}

// Estimated time of the other paths, fitted to the same calls: the digit tiles
// (a constant, the left operand's digit planes, and the waves of Kd-deep units
// over 152 SMs), or the integer pipes for the Z_2^64 layers with odd N that the
// digit tiles do not take.
double digit_us(int64_t M, int64_t K, int64_t N, int words) {
    if (!gemm_tc_feasible(M, K, N, words)) return 15.0 + 2.0 * M * K * N / (words == 1 ? 2.15e6 : 0.5e6);
    const int64_t nd = words == 1 ? 32 : 16, kd = words == 1 ? 128 : 64;
    const int64_t U = cdiv(M, 128) * cdiv(N, nd) * cdiv(2 * cdiv(K, KS) * KS, kd);
    const double mb = 2.0 * M * K * 16e-6 * words;
    return words == 1 ? 14.9 + 0.127 * mb + 0.43 * cdiv(U, 152) + 3.51 * U / 152
                      : 21.5 + 0.216 * mb + 1.91 * cdiv(U, 152) + 1.86 * U / 152;
}
constexpr size_t MAX_WORKSPACE = size_t(12) << 30;
// The residue path's time over the other paths'.  In a group the digit tiles'
// launch, set-up and last wave are shared with the other layers.
// 1e9: not run there; `total`: its workspace.
double crt_ratio(int64_t M, int64_t K, int64_t N, int words, bool grouped = false, size_t* total = nullptr) {
    CrtPlan q;
    if (M <= 8 || N <= 8 || !feasible_plan(M, K, N, words, 0, q) || q.total > MAX_WORKSPACE) return 1e9;
    if (total) *total = q.total;
    // up to 64 rows the wide and 64-row digit tiles waste less than 256-row tiles
    if (M <= 64 && gemm_tc_feasible(M, K, N, words)) return 1e8;
    const double shared = grouped ? (words == 1 ? 12.0 : 18.0) : 0.0;
    return q.us / (digit_us(M, K, N, words) - shared);
}
}  // namespace

bool gemm_crt_near(int64_t M, int64_t K, int64_t N, int words) { return crt_ratio(M, K, N, words) < 1.1; }
bool gemm_crt_candidate(int64_t M, int64_t K, int64_t N, int words) {
    size_t total = 0;
    const double r = crt_ratio(M, K, N, words, false, &total);
    return r < 1.1 || (r < 1e9 && total <= (size_t(32) << 20));
}
bool gemm_crt_preferred(int64_t M, int64_t K, int64_t N, int words, bool grouped) {
    return M > 32 && N > 64 && crt_ratio(M, K, N, words, grouped) < 0.93;   // within the measured sizes
}

size_t gemm_crt_workspace(int64_t M, int64_t K, int64_t N, int words, int one_half) {
    return crt_plan(M, K, N, words, one_half).total;
}

cudaError_t launch_gemm_crt(const GemmArgs& a, void* ws, size_t ws_bytes, cudaStream_t st) {
    CrtPlan q;
    if (!feasible_plan(a.M, a.K, a.N, a.words, a.one_half, q)) return cudaErrorNotSupported;
    if (!ws || ws_bytes < q.total) return cudaErrorInvalidValue;
    return a.words == 1 ? run<1>(a, q, (uint8_t*)ws, st) : run<2>(a, q, (uint8_t*)ws, st);
}

namespace {
__device__ unsigned int g_crt_taken = 0;
__global__ void take_crt_timeout_kernel() { g_crt_taken = atomicExch(&g_crt_timeout, 0u); }
}  // namespace

// as tc_timeout_flag, for this file's kernels, on stream `s`
int crt_timeout_flag(bool* set, cudaStream_t s) {
    take_crt_timeout_kernel<<<1, 1, 0, s>>>();
    if (cudaGetLastError() != cudaSuccess) return -1;
    unsigned int v = 0;
    if (cudaMemcpyFromSymbolAsync(&v, g_crt_taken, sizeof(v), 0, cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
    if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
    *set = v != 0;
    return 0;
}

namespace {
__device__ int g_crt_selftest_gave_up = 0;

// the wait of the pair's kernel on a barrier that nothing arrives at
__global__ void crt_wait_selftest_kernel(long long limit) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bar, 1);
        abort_flag = 0;
        ptx::fence_barrier_init();
        g_crt_selftest_gave_up = 0;
        if (!ptx::mbar_wait_cluster(&bar, 0, &abort_flag, limit)) {
            gave_up(&abort_flag);
            g_crt_selftest_gave_up = 1;
        }
    }
}
}  // namespace

int crt_wait_selftest(long long limit, cudaStream_t st) {
    int v = 0;
    crt_wait_selftest_kernel<<<1, 32, 0, st>>>(limit);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyFromSymbolAsync(&v, g_crt_selftest_gave_up, sizeof(v), 0, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return -1;
    return v;
}

}  // namespace mpcl
