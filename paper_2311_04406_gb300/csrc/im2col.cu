// im2col.cu -- the im2col view of a convolution (§2.6): a convolution of an
// f x f filter over a batch of C x H x W ring-element images (NCHW) becomes
// the ring GEMM  out (B H' W' x C f f) . W (C f f x O).  Row (b, oy, ox),
// column (c, ky, kx) of `out` is in[b][c][oy s + ky - p][ox s + kx - p], or 0
// where that falls in the zero padding.  Zero is a sharing of 0 and its tag
// (§2.4), so each party applies this to its own shares and tags locally.
#include "common.cuh"
#include "kernels.h"
#include "sm100_ptx.cuh"

namespace mpcl {

namespace {

constexpr int NT = 256;
constexpr int64_t BLOCKS = 152 * 64;     // upper target of the grid

struct Im2colArgs {
    // dimensions, rows and columns are at most 2^31: a coordinate in the padding
    // before the image wraps above any H or W
    uint32_t C, H, W, f, pad, stride, Ho, Wo;
    uint32_t sb, sy, sx;        // NT / tx rows as images, rows and columns of the output
    const u64* in;
    u64* out;
};

// A block covers `tx` columns (a power of two, at most NT) of a run of rows: a
// thread keeps one column, whose (c, ky, kx) it works out once, and steps
// through rows ty, ty + NT / tx, ... by carrying (ox, oy, b) along, so that an
// element costs a few comparisons and no division.  FAR: the step is wider than a
// row of the output, and is added as images, rows and columns (200,000 images of
// one value: 2.2 us; with a loop over the carries 36, with divisions 3.8).
// Consecutive threads take consecutive columns, so the writes are coalesced, and
// the reads of neighbouring rows share lines.  One thread per element with six 64-bit
// divisions each was bound by their instructions: 1 x 64 x 32 x 32 with f = 3
// took 7.5 us and takes 3.8, 128 such images 532 and 127 (Z_2^128: 538 and 208,
// 5.8 TB/s written).
constexpr int UNROLL = 4;       // loads in flight per thread

template <int WW, bool FAR>
__global__ void __launch_bounds__(NT) im2col_kernel(const Im2colArgs a, uint32_t rows, uint32_t Kc, uint32_t tx,
                                                    uint32_t col_blocks, uint32_t run) {
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();   // launched as a dependent of the kernel before it
    using T = typename Elem<WW>::T;
    const uint32_t rb = blockIdx.x / col_blocks;
    const uint32_t col = (blockIdx.x - rb * col_blocks) * tx + (threadIdx.x & (tx - 1));
    const uint32_t ty = threadIdx.x / tx, step = NT / tx;
    const uint32_t first = rb * run, end = rows - first < run ? rows : first + run;
    uint32_t row = first + ty;
    if (col >= Kc || row >= end) return;
    const uint32_t ff = a.f * a.f, hw = a.Ho * a.Wo;
    const uint32_t c = col / ff, kk = col - c * ff;
    const uint32_t ky = kk / a.f, kx = kk - ky * a.f;
    uint32_t b = row / hw, oy = (row - b * hw) / a.Wo, ox = row - b * hw - oy * a.Wo;
    u64* out = a.out + ((int64_t)row * Kc + col) * WW;
    const int64_t jump = (int64_t)step * Kc * WW;
    while (row < end) {
        T v[UNROLL];
#pragma unroll
        for (int j = 0; j < UNROLL; ++j) {
            const uint32_t y = oy * a.stride + ky - a.pad, x = ox * a.stride + kx - a.pad;
            v[j] = 0;
            if (j * step < end - row && y < a.H && x < a.W)
                v[j] = ld_elem<WW>(a.in, (((int64_t)b * a.C + c) * a.H + y) * a.W + x);
            if constexpr (FAR) {
                ox += a.sx;
                oy += a.sy;
                b += a.sb;
                if (ox >= a.Wo) {
                    ox -= a.Wo;
                    ++oy;
                }
                if (oy >= a.Ho) {       // below 2 Ho
                    oy -= a.Ho;
                    ++b;
                }
            } else {
                for (ox += step; ox >= a.Wo; ox -= a.Wo)    // once at most
                    if (++oy == a.Ho) {
                        oy = 0;
                        ++b;
                    }
            }
        }
#pragma unroll
        for (int j = 0; j < UNROLL; ++j) {
            if (j * step < end - row) st_elem<WW>(out, 0, v[j]);
            out += jump;
        }
        if (end - row <= UNROLL * step) break;
        row += UNROLL * step;
    }
}

}  // namespace

cudaError_t launch_im2col(int64_t B, int64_t C, int64_t H, int64_t W, int f, int pad, int stride, int words,
                          const u64* in, u64* out, cudaStream_t st) {
    const int64_t Ho = (H - f + 2 * pad) / stride + 1, Wo = (W - f + 2 * pad) / stride + 1;
    const int64_t total = B * Ho * Wo * C * f * f;
    if (total <= 0) return cudaSuccess;
    const int64_t rows = B * Ho * Wo, Kc = C * f * f;
    int64_t tx = 1;
    while (tx < Kc && tx < NT) tx *= 2;
    const int64_t col_blocks = (Kc + tx - 1) / tx, step = NT / tx;
    const int64_t hw = Ho * Wo;
    const Im2colArgs a{(uint32_t)C,      (uint32_t)H,  (uint32_t)W,  (uint32_t)f,           (uint32_t)pad,
                       (uint32_t)stride, (uint32_t)Ho, (uint32_t)Wo, (uint32_t)(step / hw), (uint32_t)(step % hw / Wo),
                       (uint32_t)(step % Wo), in,      out};
    // rows of a block: UNROLL per thread, and more where that alone would give
    // more than BLOCKS blocks (a thread's divisions then serve more rows)
    const int64_t passes = (rows + step * UNROLL - 1) / (step * UNROLL);
    const int64_t per = (passes * col_blocks + BLOCKS - 1) / BLOCKS;
    const int64_t run = per * step * UNROLL, blocks = (rows + run - 1) / run * col_blocks;
    auto* kernel = step > Wo ? (words == 1 ? im2col_kernel<1, true> : im2col_kernel<2, true>)
                             : (words == 1 ? im2col_kernel<1, false> : im2col_kernel<2, false>);
    return launch_dependent(kernel, dim3((unsigned)blocks), dim3(NT), 0, st, a,
                            (uint32_t)rows, (uint32_t)Kc, (uint32_t)tx, (uint32_t)col_blocks, (uint32_t)run);
}

}  // namespace mpcl
