// gemm_simt.cu -- exact ring GEMM on the integer pipes (CUDA cores).
//
// Computes Z = C + [E | X + c E] . [B ; F] mod 2^(64 W) (the 2K form of
// Eq. (compute-z) and Eq. (compute-ztag), §2.5) for layers the tensor-core
// kernel (gemm_tc.cu) does not take: Z_2^64 layers with odd N, layers too small
// to amortise a 128-row MMA tile, and skinny layers (M <= 8, e.g. dense layers
// at batch 1) whose cost is streaming [B ; F] from memory.
//
// Three kernels, all optionally split along K over grid.z:
//   * ring_gemm_simt_kernel<W, TM, CLUSTER, J>: TM x 64 outputs per 256-thread
//     block (TM = 64, or 16 for layers whose 64-row tiles would leave most SMs
//     idle), 16-deep K slices staged in shared memory, each thread owns a
//     (TM / 16) x J strided sub-tile (conflict-free shared reads); J = 1 for
//     layers of at most 16 columns.
//   * ring_gemv_kernel (M <= 8): a block's eight warps take interleaved rows of
//     its K range for 32 or 64 output columns and add their sums up in shared
//     memory, so that a block contributes one partial per output.
//   * ring_gemv_wide_kernel (M <= 8, wide layers with a long K): one thread per
//     output column or pair keeps M sums; the right operand is read once,
//     coalesced along N.
// The K splits of an output that fit one thread-block cluster (of up to 16) are
// added up through distributed shared memory: one launch, nothing set up before
// it.  With more of them, Z is first set to C (a device-to-device copy) and
// every block adds its partial sums with exact wrapping atomics.  Without a
// split the block writes C + sum.  Out-of-range rows/columns/K are zero-filled.
//
// A block's time goes with its K slices (a 16-deep one takes about 1 us in
// Z_2^64, 3-4 us in Z_2^128: the low 64 or 128 bits of a product need 1 or 6
// wide multiply-adds, which issue at 15 per clock cycle and SM), so small layers
// spread K over as many blocks as fit the chip once.  Shares, us, with a copy of C
// and atomics and now: 64 x 128 x 64 11.1, 4.4 (Z_2^128: 17.9, 8.2); 33 x 70 x 40 9.3,
// 4.3; 16 x 512 x 10 11.2, 6.6; 8 x 299 x 368 12.4, 6.4 (18.5, 10.0); 16 x 50000 x 10
// 57.9, 27.3.
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "kernels.h"
#include "sm100_ptx.cuh"

namespace mpcl {

namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;
constexpr int BM_SMALL = 16;     // tile rows of the small-grid variant
constexpr int GV_M = 8;         // rows handled by the skinny kernel
constexpr int GV_KC = 128;      // K chunk staged in shared memory
constexpr int PORTABLE_CLUSTER = 8, MAX_CLUSTER = 16;
constexpr int GV_NARROW = 256;  // N up to here: ring_gemv_kernel for any K
constexpr int GV_GRID = 200;    // blocks up to which wider layers take it too, when their K splits fit one
                                // cluster (measured: 4 x 512 x 1000, 128 blocks, 11.5 -> 8.9 us; 1 x 512 x 4096,
                                // 512 blocks, would go from 6.7 to 9.4)


// element kv of row m of the left operand [E | X + cE] (one_half: X + cE)
template <int W>
__device__ __forceinline__ typename Elem<W>::T left(const GemmArgs& a, typename Elem<W>::T c,
                                                   int64_t m, int64_t kv) {
    using T = typename Elem<W>::T;
    if (a.one_half) kv += a.K;
    if (kv < a.K) return ld_elem<W>(a.E, m * a.K + kv);
    const int64_t kx = kv - a.K;
    T v = ld_elem<W>(a.X, m * a.K + kx);
    if (a.coef != COEF_ZERO) v += c * ld_elem<W>(a.E, m * a.K + kx);
    return v;
}

template <int W>
__device__ __forceinline__ typename Elem<W>::T coef_value(const GemmArgs& a) {
    if (a.coef == COEF_ONE) return 1;
    if (a.coef == COEF_ALPHA) return ld_elem<W>(a.alpha, 0);
    return 0;
}

// The blocks of a cluster (all of grid.z of one output tile) have written their
// sums of the same `count` outputs to `part` in their own shared memory: block r
// adds up one contiguous share of the outputs over the cluster and stores it in Z
// with the addend.  at(index): the output's place, or -1.
template <int W, typename At>
__device__ __forceinline__ void cluster_sums(const GemmArgs& a, const typename Elem<W>::T* part, int count, At at) {
    using T = typename Elem<W>::T;
    const int cs = (int)ptx::cluster_size(), rank = (int)ptx::cluster_rank();
    const int per = (count + cs - 1) / cs;
    const int end = min(count, (rank + 1) * per);
    __syncwarp();
    ptx::cluster_sync();        // every block's sums are written
    for (int i = rank * per + (int)threadIdx.x; i < end; i += NT) {
        const int64_t e = at(i);
        const T c = e >= 0 && a.C ? ld_elem<W>(a.C, e) : (T)0;
        T s = 0;
#pragma unroll 4
        for (int r = 0; r < cs; ++r) {
            const uint32_t p = ptx::cluster_addr(part + i, (uint32_t)r);
            if constexpr (W == 1) {
                s += ptx::ld_cluster_u64(p);
            } else {
                s += (T)ptx::ld_cluster_u64(p) | ((T)ptx::ld_cluster_u64(p + 8) << 64);
            }
        }
        if (e >= 0) st_elem<W>(a.Z, e, s + c);
    }
    __syncwarp();
    ptx::cluster_sync();        // and read, before a block leaves
}

// element e of the addend; 0 where Z += sum (Z was set to C) or there is none.
// A thread reads the addend of all of its outputs before it stores the first, so
// that the loads are in flight together.
template <int W>
__device__ __forceinline__ typename Elem<W>::T addend(const GemmArgs& a, int64_t e, int atomic) {
    using T = typename Elem<W>::T;
    return a.C && !atomic ? ld_elem<W>(a.C, e) : (T)0;
}

// Z = sum (the addend included), or Z += sum where several blocks share the output
template <int W>
__device__ __forceinline__ void put(const GemmArgs& a, int64_t e, typename Elem<W>::T v, int atomic) {
    if (atomic) atomic_add_elem<W>(a.Z, e, v);
    else st_elem<W>(a.Z, e, v);
}

// The operands of the next K slice are loaded while the present one is
// multiplied; not in 16-row Z_2^128 tiles of more than 16 columns, which are
// bound by their wide multiply-adds (300 x 300 x 300: 84.6 us with it, 82.5
// without).  CLUSTER: the K splits of a tile are the blocks of a cluster.
template <int W, int TM, bool CLUSTER, int J>
__global__ void __launch_bounds__(NT) ring_gemm_simt_kernel(GemmArgs a, int64_t kchunk, int atomic) {
    using T = typename Elem<W>::T;
    constexpr int RI = TM / 16;        // rows of a thread's sub-tile
    constexpr int LV = TM * BK / NT, RV = BK * BN / NT;     // values a thread stages
    __shared__ T Ls[BK][TM + 1];
    __shared__ T Rs[BK][BN];           // at the end, the sums of a 16-row tile
    static_assert(!CLUSTER || TM <= BK, "the sums fit the staged right operand");

    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t m0 = (int64_t)blockIdx.y * TM, n0 = (int64_t)blockIdx.x * BN;
    const int64_t M = a.M, K = a.K, N = a.N, K2 = a.one_half ? a.K : 2 * a.K;
    const int64_t kbeg = (int64_t)blockIdx.z * kchunk;
    const int64_t kend = kbeg + kchunk < K2 ? kbeg + kchunk : K2;
    const T c = coef_value<W>(a);
    const int64_t kr = a.one_half ? K : 0;   // row offset into [B ; F]

    T acc[RI][4];
#pragma unroll
    for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;

    auto left_at = [&](int idx, int64_t k0) {
        const int64_t m = m0 + idx / BK, kv = k0 + idx % BK;
        return (m < M && kv < kend) ? left<W>(a, c, m, kv) : (T)0;
    };
    auto right_at = [&](int idx, int64_t k0) {
        const int64_t n = n0 + idx % BN, kv = k0 + idx / BN;
        if (n >= N || kv >= kend) return (T)0;
        const int64_t kq = kv + kr;
        return kq < K ? ld_elem<W>(a.B, kq * N + n) : ld_elem<W>(a.F, (kq - K) * N + n);
    };
    auto multiply = [&] {
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            T av[RI], bv[J];
#pragma unroll
            for (int i = 0; i < RI; ++i) av[i] = Ls[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < J; ++j) bv[j] = Rs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < RI; ++i)
#pragma unroll
                for (int j = 0; j < J; ++j) acc[i][j] += av[i] * bv[j];
        }
    };
    if constexpr (W == 1 || TM == BM || J == 1 || CLUSTER) {
        T lv[LV], rv[RV];
        auto fetch = [&](int64_t k0) {
#pragma unroll
            for (int r = 0; r < LV; ++r) lv[r] = left_at(tid + r * NT, k0);
#pragma unroll
            for (int r = 0; r < RV; ++r) rv[r] = right_at(tid + r * NT, k0);
        };
        if (kbeg < kend) fetch(kbeg);
        for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
            for (int r = 0; r < LV; ++r) Ls[(tid + r * NT) % BK][(tid + r * NT) / BK] = lv[r];
#pragma unroll
            for (int r = 0; r < RV; ++r) Rs[(tid + r * NT) / BN][(tid + r * NT) % BN] = rv[r];
            __syncthreads();
            if (k0 + BK < kend) fetch(k0 + BK);
            multiply();
            __syncthreads();
        }
    } else {
        for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
            for (int r = 0; r < LV; ++r)
                Ls[(tid + r * NT) % BK][(tid + r * NT) / BK] = left_at(tid + r * NT, k0);
#pragma unroll
            for (int r = 0; r < RV; ++r)
                Rs[(tid + r * NT) / BN][(tid + r * NT) % BN] = right_at(tid + r * NT, k0);
            __syncthreads();
            multiply();
            __syncthreads();
        }
    }
    if constexpr (CLUSTER) {
#pragma unroll
        for (int j = 0; j < 4; ++j) Rs[ty][tx + 16 * j] = acc[0][j];
        cluster_sums<W>(a, &Rs[0][0], BM_SMALL * BN, [&](int i) {
            const int64_t m = m0 + i / BN, n = n0 + i % BN;
            return m < M && n < N ? m * N + n : (int64_t)-1;
        });
    } else {
        auto each = [&](auto f) {
#pragma unroll
            for (int i = 0; i < RI; ++i) {
                const int64_t m = m0 + ty + 16 * i;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int64_t n = n0 + tx + 16 * j;
                    if (m < M && n < N) f(acc[i][j], m * N + n);
                }
            }
        };
        each([&](T& v, int64_t e) { v += addend<W>(a, e, atomic); });
        each([&](T& v, int64_t e) { put<W>(a, e, v, atomic); });
    }
}

// acc += the left operand's staged rows times rows `first`, first + STEP, ... below
// kc of a K chunk of [B ; F] that starts at row k0, at columns n .. n + VEC - 1.
// The loads of U rows are in flight together; in Z_2^128 with more than two rows of
// the left operand, which is bound by its multiply-adds, the compiler's own order
// is as good (shares, us, with one and the other: 8 x 4608 x 512 53.1, 52.0;
// 2 x 4096 x 4096 112, 162; Z_2^64: 3 x 1832 x 632 17.6, 22.3).  PRED: the last
// batch of a chunk too, with zeros past its end (Ls is zero there).
template <int W, int VEC, int MM, int STEP, bool PRED>
__device__ __forceinline__ void gemv_rows(const GemmArgs& a, const typename Elem<W>::T* Ls, int64_t k0, int first,
                                          int kc, int64_t n, typename Elem<W>::T (&acc)[MM][VEC]) {
    using T = typename Elem<W>::T;
    constexpr int U = W == 2 && MM > 2 ? 1 : 8 / W;
    static_assert(!PRED || GV_KC % (U * STEP) == 0, "whole batches");
    int k1 = first;
    auto rows = [&](auto count) {
        constexpr int B = decltype(count)::value;
        T r[B][VEC];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const int64_t kv = k0 + k1 + u * STEP;
            const u64* row = kv < a.K ? a.B + kv * a.N * W : a.F + (kv - a.K) * a.N * W;
            if constexpr (VEC == 2) {
                ulonglong2 v = make_ulonglong2(0, 0);
                if (!PRED || k1 + u * STEP < kc) v = *reinterpret_cast<const ulonglong2*>(row + n);
                r[u][0] = v.x;
                r[u][1] = v.y;
            } else {
                r[u][0] = ld_elem<W>(row, n);
            }
        }
#pragma unroll
        for (int u = 0; u < B; ++u)
#pragma unroll
            for (int i = 0; i < MM; ++i)
#pragma unroll
                for (int v = 0; v < VEC; ++v) acc[i][v] += Ls[i * GV_KC + k1 + u * STEP] * r[u][v];
    };
    if constexpr (U > 1) {
#pragma unroll 1
        for (; k1 + (PRED ? 0 : (U - 1) * STEP) < kc; k1 += U * STEP) rows(std::integral_constant<int, U>());
#pragma unroll 1
        for (; k1 < kc; k1 += STEP) rows(std::integral_constant<int, 1>());
    } else {
#pragma unroll 8
        for (; k1 < kc; k1 += STEP) rows(std::integral_constant<int, 1>());
    }
}

// GEMV for wide layers: one thread per VEC output columns keeps M sums over
// every row of the block's K range (deep independent loads along K).  VEC = 2:
// two adjacent Z_2^64 columns per thread, read as one 16-byte vector (needs
// even N); VEC = 1 otherwise.  MM >= M rows are accumulated (1, 2, 4 or 8).  PRED
// (one row, Z_2^64): 30 registers in place of 48 and eight blocks per SM, faster by
// itself (1 x 4096 x 4096 42.6, 43.8 us; 1 x 512 x 2048 5.9, 6.7) but not beside
// the tensor-core kernels of a group, whose SMs it fills (VGG-16 at batch 1 329,
// 311 us).
template <int W, int VEC, int MM, bool PRED>
__global__ void __launch_bounds__(NT) ring_gemv_wide_kernel(GemmArgs a, int64_t kchunk, int atomic) {
    using T = typename Elem<W>::T;
    __shared__ T Ls[MM][GV_KC];
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int64_t n = ((int64_t)blockIdx.x * NT + threadIdx.x) * VEC;
    const int64_t K = a.K, N = a.N, K2 = a.one_half ? a.K : 2 * a.K;
    const int64_t kr = a.one_half ? K : 0;   // row offset into [B ; F]
    const int M = (int)a.M;
    const int64_t kbeg = (int64_t)blockIdx.z * kchunk;
    const int64_t kend = kbeg + kchunk < K2 ? kbeg + kchunk : K2;
    const T c = coef_value<W>(a);
    T acc[MM][VEC];
#pragma unroll
    for (int i = 0; i < MM; ++i)
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[i][v] = 0;
    for (int64_t k0 = kbeg; k0 < kend; k0 += GV_KC) {
        const int kc = (int)(kend - k0 < GV_KC ? kend - k0 : GV_KC);
        for (int idx = threadIdx.x; idx < MM * GV_KC; idx += NT) {
            const int mm = idx / GV_KC, kk = idx % GV_KC;
            Ls[mm][kk] = (mm < M && kk < kc) ? left<W>(a, c, mm, k0 + kk) : (T)0;
        }
        __syncthreads();
        if (n < N) gemv_rows<W, VEC, MM, 1, PRED>(a, &Ls[0][0], k0 + kr, 0, kc, n, acc);
        __syncthreads();
    }
    auto each = [&](auto f) {
#pragma unroll
        for (int v = 0; v < VEC; ++v)
#pragma unroll
            for (int i = 0; i < MM; ++i)
                if (i < M && n + v < N) f(acc[i][v], (int64_t)i * N + n + v);
    };
    each([&](T& v, int64_t e) { v += addend<W>(a, e, atomic); });
    each([&](T& v, int64_t e) { put<W>(a, e, v, atomic); });
}

// GEMV (M <= GV_M): a block covers 32 lanes x VEC output columns (VEC = 2: two
// adjacent Z_2^64 columns as one 16-byte vector, which needs even N) and its
// eight warps take rows w, w + 8, ... of each staged K chunk; MM >= M rows are
// accumulated (1, 2, 4 or 8).  The warps' sums are added in shared memory and
// the cluster's blocks, which split K, add theirs through distributed shared
// memory.
template <int W, int VEC, int MM>
__global__ void __launch_bounds__(NT) ring_gemv_kernel(GemmArgs a, int64_t kchunk, int atomic) {
    using T = typename Elem<W>::T;
    constexpr int NW = NT / 32;                 // warps per block
    constexpr int NCOL = 32 * VEC;              // columns per block
    __shared__ T Ls[MM][GV_KC];
    __shared__ T red[NW - 1][MM][NCOL];         // sums of warps 1 .. NW - 1
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = (int64_t)blockIdx.x * NCOL + lane * VEC;
    const int64_t K = a.K, N = a.N, K2 = a.one_half ? a.K : 2 * a.K;
    const int64_t kr = a.one_half ? K : 0;   // row offset into [B ; F]
    const int M = (int)a.M;
    const int64_t kbeg = (int64_t)blockIdx.z * kchunk;
    const int64_t kend = kbeg + kchunk < K2 ? kbeg + kchunk : K2;
    const T c = coef_value<W>(a);
    T acc[MM][VEC];
#pragma unroll
    for (int i = 0; i < MM; ++i)
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[i][v] = 0;
    for (int64_t k0 = kbeg; k0 < kend; k0 += GV_KC) {
        const int kc = (int)(kend - k0 < GV_KC ? kend - k0 : GV_KC);
        for (int idx = threadIdx.x; idx < MM * GV_KC; idx += NT) {
            const int mm = idx / GV_KC, kk = idx % GV_KC;
            Ls[mm][kk] = (mm < M && kk < kc) ? left<W>(a, c, mm, k0 + kk) : (T)0;
        }
        __syncthreads();
        if (n < N) gemv_rows<W, VEC, MM, NW, false>(a, &Ls[0][0], k0 + kr, warp, kc, n, acc);
        __syncthreads();
    }
    if (warp > 0) {
#pragma unroll
        for (int i = 0; i < MM; ++i)
#pragma unroll
            for (int v = 0; v < VEC; ++v) red[warp - 1][i][lane * VEC + v] = acc[i][v];
    }
    __syncthreads();
    T* part = &Ls[0][0];                        // every warp is done with the staged rows
    if (warp == 0) {
#pragma unroll
        for (int w = 0; w < NW - 1; ++w)
#pragma unroll
            for (int i = 0; i < MM; ++i)
#pragma unroll
                for (int v = 0; v < VEC; ++v) acc[i][v] += red[w][i][lane * VEC + v];
        if (ptx::cluster_size() == 1) {
            auto each = [&](auto f) {
#pragma unroll
                for (int i = 0; i < MM; ++i)
#pragma unroll
                    for (int v = 0; v < VEC; ++v)
                        if (i < M && n + v < N) f(acc[i][v], (int64_t)i * N + n + v);
            };
            each([&](T& v, int64_t e) { v += addend<W>(a, e, atomic); });
            each([&](T& v, int64_t e) { put<W>(a, e, v, atomic); });
        } else {
#pragma unroll
            for (int i = 0; i < MM; ++i)
#pragma unroll
                for (int v = 0; v < VEC; ++v) part[i * NCOL + lane * VEC + v] = acc[i][v];
        }
    }
    if (ptx::cluster_size() == 1) return;
    cluster_sums<W>(a, part, MM * NCOL, [&](int i) {
        const int row = i / NCOL;
        const int64_t col = (int64_t)blockIdx.x * NCOL + i % NCOL;
        return row < M && col < N ? row * N + col : (int64_t)-1;
    });
}

// K chunks (multiples of `step`, at least `min_chunk`) so that the grid covers
// about `waves` x 152 blocks
int64_t choose_kchunk(int64_t blocks_2d, int64_t K2, int64_t step, int64_t min_chunk, int64_t waves) {
    int64_t splits = waves * 152 / (blocks_2d > 0 ? blocks_2d : 1);
    const int64_t max_splits = (K2 + min_chunk - 1) / min_chunk;
    if (splits > max_splits) splits = max_splits;
    if (splits < 1) splits = 1;
    int64_t chunk = (K2 + splits - 1) / splits;
    chunk = ((chunk + step - 1) / step) * step;
    return chunk > 0 ? chunk : step;
}

}  // namespace

// Tile rows of the integer-pipe GEMM: the launch table's choice (64 or 16),
// else 16 when 64-row tiles would give fewer blocks than SMs.
int simt_tile_rows(int64_t M, int64_t N, int rows) {
    if (rows == 64 || rows == BM_SMALL) return rows;
    return ((M + BM - 1) / BM) * ((N + BN - 1) / BN) < 152 ? BM_SMALL : BM;
}

namespace {

using Kernel = void (*)(GemmArgs, int64_t, int);

template <int W, int J> Kernel tile_kernel(int tm, bool cluster) {
    if (tm == BM) return ring_gemm_simt_kernel<W, BM, false, J>;
    return cluster ? ring_gemm_simt_kernel<W, BM_SMALL, true, J> : ring_gemm_simt_kernel<W, BM_SMALL, false, J>;
}

template <int W, int VEC> Kernel gemv_kernel(int64_t M, bool wide, bool alone) {
    if (wide)
        return M <= 1   ? (alone ? ring_gemv_wide_kernel<W, VEC, 1, VEC == 2> : ring_gemv_wide_kernel<W, VEC, 1, false>)
               : M <= 2 ? ring_gemv_wide_kernel<W, VEC, 2, false>
               : M <= 4 ? ring_gemv_wide_kernel<W, VEC, 4, false>
                        : ring_gemv_wide_kernel<W, VEC, 8, false>;
    return M <= 1   ? ring_gemv_kernel<W, VEC, 1>
           : M <= 2 ? ring_gemv_kernel<W, VEC, 2>
           : M <= 4 ? ring_gemv_kernel<W, VEC, 4>
                    : ring_gemv_kernel<W, VEC, 8>;
}

// Whether the device places clusters of MAX_CLUSTER blocks of `kernel`, a size that
// is not portable (a partition of the SMs may hold none): asked once per device and
// kernel, together with the kernel's leave to have them.
bool places_max_cluster(Kernel kernel) {
    static std::mutex mu;
    static std::map<std::pair<Kernel, int>, bool> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lk(mu);
    const auto it = known.find({kernel, dev});
    if (it != known.end()) return it->second;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, 1, MAX_CLUSTER);
    cfg.blockDim = dim3(NT);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = MAX_CLUSTER;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, (const void*)kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();          // the portable size serves
        return false;
    }
    return known[{kernel, dev}] = n > 0;
}

// dependent: a call by itself, launched as a dependent of the kernel before it (in
// a group on a side stream it is not); most: the largest cluster
template <int W>
cudaError_t run(const GemmArgs& a, cudaStream_t st, bool dependent, int most = MAX_CLUSTER) {
    const int64_t K2 = a.one_half ? a.K : 2 * a.K;
    const bool skinny = a.M <= GV_M;
    const int vec = (skinny && W == 1 && a.N % 2 == 0) ? 2 : 1;
    const int tm = simt_tile_rows(a.M, a.N, a.rows);
    const int64_t by = skinny ? 1 : (a.M + tm - 1) / tm;
    if (by > 65535) return cudaErrorInvalidConfiguration;
    const int64_t waves = a.simt_waves > 0 ? a.simt_waves : (skinny ? 4 : 2);
    int64_t bx = skinny ? (a.N + 32 * vec - 1) / (32 * vec) : (a.N + BN - 1) / BN;
    // one cluster per output tile with all of its K splits, where that gives
    // blocks little work: no atomics, and no pass to set Z to C before them
    const int64_t least = skinny ? 128 : BK;         // K of a block, at least
    int64_t splits = (K2 + least - 1) / least;
    if (skinny && a.N <= GV_NARROW) splits = std::min(splits, std::max<int64_t>(1, waves * 152 / bx));
    int cs = 1;
    while (cs < splits && cs < most) cs *= 2;
    if (!skinny)
        while (cs > 1 && bx * by * cs > 152) cs /= 2;
    // a table entry with a K-split target gets that many splits, added up by atomics
    const bool cluster = a.simt_waves == 0 &&
                         (skinny ? cs >= splits && (a.N <= GV_NARROW || bx * cs <= GV_GRID)
                                 // 48 (16): beyond three (one) slices per block more splits with
                                 // atomics are faster: 16 x 400 x 160 in Z_2^64 9.9 us as clusters, 8.5 so
                                 : tm == BM_SMALL && cs > 1 && K2 <= cs * (W == 1 ? 48 : 16));
    const bool wide = skinny && a.N > GV_NARROW && !cluster;
    int64_t kchunk, bz;
    if (cluster) {
        bz = cs;
        kchunk = ((K2 + bz - 1) / bz + 15) / 16 * 16;
    } else {
        // the grid covers about `waves` x 152 blocks (launch table, else 4 / 2); GEMV chunks
        // give each of a block's eight warps at least 16 rows
        cs = 1;
        if (wide) bx = (a.N + NT * vec - 1) / (NT * vec);
        kchunk = choose_kchunk(bx * by, K2, 16, wide ? 32 : skinny ? 128 : 4 * BK, waves);
        bz = K2 > 0 ? (K2 + kchunk - 1) / kchunk : 1;
    }
    if (bz > 65535) return cudaErrorInvalidConfiguration;
    const Kernel kernel = !skinny     ? (a.N <= 16 ? tile_kernel<W, 1>(tm, cluster) : tile_kernel<W, 4>(tm, cluster))
                          : vec == 2 ? gemv_kernel<W, 3 - W>(a.M, wide, dependent)
                                     : gemv_kernel<W, 1>(a.M, wide, dependent);
    if (cs > PORTABLE_CLUSTER && !places_max_cluster(kernel)) return run<W>(a, st, dependent, PORTABLE_CLUSTER);
    const int atomic = bz > cs ? 1 : 0;
    if (atomic) {
        const size_t bytes = (size_t)a.M * a.N * 8 * W;
        cudaError_t e = a.C ? cudaMemcpyAsync(a.Z, a.C, bytes, cudaMemcpyDeviceToDevice, st)
                            : cudaMemsetAsync(a.Z, 0, bytes, st);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)bx, (unsigned)by, (unsigned)bz);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(NT);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (dependent) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cs > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = 1;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs++].val.clusterDim.z = (unsigned)cs;
    }
    return cudaLaunchKernelEx(&cfg, kernel, a, kchunk, atomic);
}

}  // namespace

cudaError_t launch_gemm_simt(const GemmArgs& a, cudaStream_t st, bool dependent) {
    if (a.M == 0 || a.N == 0) return cudaSuccess;
    return a.words == 1 ? run<1>(a, st, dependent) : run<2>(a, st, dependent);
}

}  // namespace mpcl
