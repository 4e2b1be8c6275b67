// Draft-token draw (Algorithm 3, the step that samples the K draft blocks): one token per logit row from
// softmax(z/T) by inverse CDF, softmax and draw fused in one pass over the row (per-tile maxima and sums, the
// tile located through them, one tile recomputed).
//
// A cluster of C CTAs per row.  What bounds the kernel is the latency of one pass over a row by the CTAs it is shared out
// to, so few rows are spread over as many CTAs as fill the device (two of 512 threads per SM) and still give every warp
// pair a tile.  With one CTA of 1024 threads per row and three block-wide searches before, and now, per call of a replayed
// graph: 3 rows of 32256 float32 8.4 -> 6.1 us, 4 of 128256 bfloat16 15.9 -> 6.5, 128 of them 16.6 -> 14.8 (2.2 TB/s; the
// special-function pipe alone takes 4.2 of it, the launch and the three searches 6), 2048 of 32000 bfloat16 109 -> 55.
#include "sgbv_sample.cuh"

namespace sgbv {

namespace {

constexpr int kThreads = 512;
constexpr int kSlots = 2 * 148;        // CTAs the device holds (64 registers per thread)
constexpr int kTilesInSmem = 1024;     // tiles per CTA whose statistics stay in shared memory, else in global scratch

template <typename T>
__global__ void __launch_bounds__(kThreads, 2)
draw_rows_kernel(const T *__restrict__ z_all, const float *__restrict__ u, Shape s, int C, float *__restrict__ tile_scratch,
                 int32_t *__restrict__ out_token, double *__restrict__ out_logp, int32_t *__restrict__ out_status) {
    __shared__ DrawScratch sc;
    __shared__ float sh_tiles[2][kTilesInSmem];
    const int r = blockIdx.x / C, rank = C > 1 ? (int)cluster_ctarank() : 0;
    if (C > 1) cluster_arrive();
    const int per = (s.ntiles + C - 1) / C;
    float *tile_s = sh_tiles[0], *tile_m = sh_tiles[1];
    if (per > kTilesInSmem) {
        tile_s = tile_scratch + (size_t)r * 2 * s.ntiles + min(s.ntiles, rank * per);
        tile_m = tile_s + s.ntiles;
    }
    const T *z = z_all + (size_t)r * s.V;
    const double us = (double)u[r];
    if (C > 1) cluster_wait();  // (the peers are running)
    const Drawn d = draw_row<T>(z, s, us, rank, C, tile_s, tile_m, &sc);
    if (threadIdx.x == 0 && (d.bad ? rank == 0 : d.y >= 0)) {
        out_token[r] = d.y;
        if (out_status) out_status[r] = d.bad ? SGBV_STATUS_NONFINITE_LOGIT : 0;
        // log softmax of the drawn token
        if (out_logp) out_logp[r] = d.bad ? NAN : ((double)ld_logit(z, d.y) - (double)d.m) * s.inv_T - log(d.total);
    }
}

}  // namespace

int launch_draw_rows(const void *z, int dtype, const float *u, const Shape &s, float *tile_scratch, int32_t *out_token,
                     double *out_logp, int32_t *out_status, cudaStream_t stream) {
    int C = 1;
    while (2 * C <= kMaxRowCtas && (long)s.B * 2 * C <= kSlots && s.ntiles >= 2 * C * kThreads / 64) C *= 2;
    const unsigned grid = (unsigned)s.B * (unsigned)C;
    const cudaError_t e =
        dtype == SGBV_DTYPE_BF16
            ? launch_clusters(draw_rows_kernel<uint16_t>, grid, kThreads, 0, C, stream, (const uint16_t *)z, u, s, C,
                              tile_scratch, out_token, out_logp, out_status)
            : launch_clusters(draw_rows_kernel<float>, grid, kThreads, 0, C, stream, (const float *)z, u, s, C, tile_scratch,
                              out_token, out_logp, out_status);
    if (e == cudaSuccess) return 1;
    cudaGetLastError();
    return SGBV_ERR_CUDA;
}

}  // namespace sgbv
