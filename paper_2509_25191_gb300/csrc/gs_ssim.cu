// Photometric loss with D-SSIM (Section 3.1): L = (1 - lambda) mean|x - y|
// + lambda (1 - mean SSIM(x, y)), SSIM from local statistics under an 11x11
// Gaussian window (sigma 1.5) with zero padding, per channel of every view,
// and its gradient with respect to the rendered image x.
//
// One kernel does the forward and the backward for a 32x32 output tile and
// all three channels: it stages x and y with a 10-pixel halo in shared
// memory, blurs x, y, (x - y)^2, xy (separable: a horizontal then a vertical
// 11-tap pass) over the tile plus a 5-pixel halo, forms SSIM and the three
// per-pixel derivative fields a = dS/dmu_x, b = dS/dE[x^2], c = dS/dE[xy]
// there, blurs those over the tile, and writes
//   dL/dx = (1 - lambda) sign(x - y) / n - lambda / n (G a + 2 x G b + y G c).
// SSIM and its derivatives need the two variances only as their sum, which is
// var(x - y) + 2 cov(x, y): the second half is the covariance of the numerator, so
// that its rounding (a difference of numbers a thousand times larger where the image
// is flat) leaves their ratio nearly alone, and an image against itself has SSIM 1.
// Every pass keeps a run of outputs per thread in registers so that each
// staged value is read from shared memory once per run, not once per tap.
// Bound by instruction issue, with a barrier after each of the five passes: it
// needs several blocks per SM to cover them, so a, b, c take the staged inputs'
// place (the centre pixels are read again from the caches) and registers are
// capped for four blocks. Two 1237x822 images, back to back: 133 us (137 with a blur of
// x^2 + y^2 for (x - y)^2, and then 141 with three blocks, 157 with two); 173 us with
// five blurs, its own room for a, b, c and two blocks per SM. Error of the gradient
// against 64 bits, five blurs -> (x - y)^2: 2.4e-6 -> 1.9e-6 for images 0.1 apart,
// 1.2e-5 -> 6.0e-6 for 0.01, 2.5e-4 -> 8.1e-5 for a bright flat image 1e-3 apart.
#include "gs_common.cuh"

namespace gsk {

constexpr int SS_T = 32;                 // output tile (square)
constexpr int SS_R = 5;                  // window radius
constexpr int SS_S1 = SS_T + 2 * SS_R;   // 42: tile + halo where SSIM is formed
constexpr int SS_IN = SS_T + 4 * SS_R;   // 52: staged input
constexpr int SS_THREADS = 256;
constexpr int SS_CH = 3;                 // channels
constexpr float SS_C1 = 0.0001f, SS_C2 = 0.0009f;

struct SsimLaunch {
    int n_views;
    int tiles_x[GS_MAX_VIEWS], tiles_y[GS_MAX_VIEWS];
    int W[GS_MAX_VIEWS], H[GS_MAX_VIEWS];
    long long tile_base[GS_MAX_VIEWS + 1];
    long long pix_base[GS_MAX_VIEWS];
    float g[2 * SS_R + 1];
    float lambda, inv_n;
};

struct SsimSmem {
    union {
        float xy[2][SS_IN][SS_IN];    // x, y
        float abc[3][SS_S1][SS_S1];
    } in;
    union {
        float h1[4][SS_IN][SS_S1];    // horizontal blurs of x, y, (x - y)^2, xy
        float h2[3][SS_S1][SS_T];     // horizontal blurs of a, b, c
    } u;
    float red[2][SS_THREADS / 32];
    float part[2][SS_CH];             // (split tiles, the first channel's block) each channel's sums
};

// Barrier over the channels of a tile (a cluster of blocks).
__device__ __forceinline__ void tile_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void tile_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// BLOCKS: the blocks per SM that the registers leave room for. SPLIT: a cluster of
// three blocks per tile, one per channel; else a block per tile.
template <int BLOCKS, bool SPLIT>
__global__ void __launch_bounds__(SS_THREADS, BLOCKS)
    k_l1_dssim(const SsimLaunch L, const float *__restrict__ image, const float *__restrict__ target,
               float *__restrict__ grad, float *loss) {
    extern __shared__ __align__(16) unsigned char ss_raw[];
    SsimSmem &sm = *reinterpret_cast<SsimSmem *>(ss_raw);
    const long long tile = SPLIT ? blockIdx.x / SS_CH : blockIdx.x;
    const int rank = SPLIT ? blockIdx.x % SS_CH : 0;   // in the cluster
    if (SPLIT) tile_arrive();
    int v = 0;
    while (v + 1 < L.n_views && L.tile_base[v + 1] <= tile) ++v;
    const int lt = (int)(tile - L.tile_base[v]);
    const int W = L.W[v], H = L.H[v];
    const int ox = (lt % L.tiles_x[v]) * SS_T, oy = (lt / L.tiles_x[v]) * SS_T;
    const int tid = threadIdx.x;
    float g[2 * SS_R + 1];
#pragma unroll
    for (int k = 0; k <= 2 * SS_R; ++k) g[k] = L.g[k];
    float acc_s = 0.f, acc_l1 = 0.f;

    for (int ch = rank; ch < (SPLIT ? rank + 1 : SS_CH); ++ch) {
        const float *X = image + L.pix_base[v] + (long long)ch * W * H;
        const float *Y = target + L.pix_base[v] + (long long)ch * W * H;
        float *G = grad + L.pix_base[v] + (long long)ch * W * H;
        // stage x, y with a 10-pixel halo (0 outside the image)
        for (int i = tid; i < SS_IN * SS_IN; i += SS_THREADS) {
            const int r = i / SS_IN, c = i % SS_IN;
            const int gy = oy - 2 * SS_R + r, gx = ox - 2 * SS_R + c;
            const bool in = gy >= 0 && gy < H && gx >= 0 && gx < W;
            sm.in.xy[0][r][c] = in ? X[(long long)gy * W + gx] : 0.f;
            sm.in.xy[1][r][c] = in ? Y[(long long)gy * W + gx] : 0.f;
        }
        __syncthreads();
        // horizontal pass: 52 rows x 42 columns, runs of 7 columns per thread
        constexpr int RUN1 = 7;
        for (int i = tid; i < SS_IN * (SS_S1 / RUN1); i += SS_THREADS) {
            const int r = i / (SS_S1 / RUN1), c0 = (i % (SS_S1 / RUN1)) * RUN1;
            float a[4][RUN1];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < RUN1; ++j) a[q][j] = 0.f;
#pragma unroll
            for (int k = 0; k < RUN1 + 2 * SS_R; ++k) {
                const float xv = sm.in.xy[0][r][c0 + k], yv = sm.in.xy[1][r][c0 + k];
                const float df = xv - yv, sq = df * df, xy = xv * yv;
#pragma unroll
                for (int j = 0; j < RUN1; ++j) {
                    const int t = k - j;
                    if (t >= 0 && t <= 2 * SS_R) {
                        a[0][j] = fmaf(g[t], xv, a[0][j]);
                        a[1][j] = fmaf(g[t], yv, a[1][j]);
                        a[2][j] = fmaf(g[t], sq, a[2][j]);
                        a[3][j] = fmaf(g[t], xy, a[3][j]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < RUN1; ++j) sm.u.h1[q][r][c0 + j] = a[q][j];
        }
        __syncthreads();
        // vertical pass over the 42x42 region, runs of 7 rows: SSIM and a, b, c
        for (int i = tid; i < SS_S1 * (SS_S1 / RUN1); i += SS_THREADS) {
            const int c = i % SS_S1, r0 = (i / SS_S1) * RUN1;
            float a[4][RUN1];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < RUN1; ++j) a[q][j] = 0.f;
#pragma unroll
            for (int k = 0; k < RUN1 + 2 * SS_R; ++k) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float hv = sm.u.h1[q][r0 + k][c];
#pragma unroll
                    for (int j = 0; j < RUN1; ++j) {
                        const int t = k - j;
                        if (t >= 0 && t <= 2 * SS_R) a[q][j] = fmaf(g[t], hv, a[q][j]);
                    }
                }
            }
            const int gx = ox - SS_R + c;
#pragma unroll
            for (int j = 0; j < RUN1; ++j) {
                const int r = r0 + j;
                const int gy = oy - SS_R + r;
                float da = 0.f, db = 0.f, dc = 0.f;
                if (gy >= 0 && gy < H && gx >= 0 && gx < W) {
                    const float mx = a[0][j], my = a[1][j];
                    const float dm = mx - my, sxy = a[3][j] - mx * my;
                    const float l1 = 2.f * mx * my + SS_C1, l2 = 2.f * sxy + SS_C2;
                    const float d1 = dm * dm + l1, d2 = (a[2][j] - dm * dm) + l2;
                    const float rd1 = 1.f / d1, rd2 = 1.f / d2, rq = rd1 * rd2;
                    const float S = l1 * l2 * rq;
                    // dS/dmu_x with E[x^2] and E[xy] held fixed, written without
                    // dividing by l1 or l2 (l2 = 2 s_xy + C2 can be ~0):
                    // S (2 my / l1 - 2 my / l2) = 2 my (l2 - l1) / (d1 d2)
                    da = 2.f * my * (l2 - l1) * rq + 2.f * mx * S * (rd2 - rd1);
                    db = -S * rd2;
                    dc = 2.f * l1 * rq;
                    if (r >= SS_R && r < SS_R + SS_T && c >= SS_R && c < SS_R + SS_T) acc_s += S;
                }
                sm.in.abc[0][r][c] = da;
                sm.in.abc[1][r][c] = db;
                sm.in.abc[2][r][c] = dc;
            }
        }
        __syncthreads();
        // horizontal pass of a, b, c: 42 rows x 32 columns, runs of 4
        constexpr int RUN2 = 4;
        for (int i = tid; i < SS_S1 * (SS_T / RUN2); i += SS_THREADS) {
            const int r = i / (SS_T / RUN2), c0 = (i % (SS_T / RUN2)) * RUN2;
            float a[3][RUN2];
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int j = 0; j < RUN2; ++j) a[q][j] = 0.f;
#pragma unroll
            for (int k = 0; k < RUN2 + 2 * SS_R; ++k) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const float hv = sm.in.abc[q][r][c0 + k];
#pragma unroll
                    for (int j = 0; j < RUN2; ++j) {
                        const int t = k - j;
                        if (t >= 0 && t <= 2 * SS_R) a[q][j] = fmaf(g[t], hv, a[q][j]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int j = 0; j < RUN2; ++j) sm.u.h2[q][r][c0 + j] = a[q][j];
        }
        __syncthreads();
        // vertical pass to the 32x32 tile, runs of 4 rows; write the gradient
        for (int i = tid; i < SS_T * (SS_T / RUN2); i += SS_THREADS) {
            const int c = i % SS_T, r0 = (i / SS_T) * RUN2;
            float a[3][RUN2];
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int j = 0; j < RUN2; ++j) a[q][j] = 0.f;
#pragma unroll
            for (int k = 0; k < RUN2 + 2 * SS_R; ++k) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const float hv = sm.u.h2[q][r0 + k][c];
#pragma unroll
                    for (int j = 0; j < RUN2; ++j) {
                        const int t = k - j;
                        if (t >= 0 && t <= 2 * SS_R) a[q][j] = fmaf(g[t], hv, a[q][j]);
                    }
                }
            }
            const int gx = ox + c;
#pragma unroll
            for (int j = 0; j < RUN2; ++j) {
                const int gy = oy + r0 + j;
                if (gy < H && gx < W) {
                    const float xv = X[(long long)gy * W + gx], yv = Y[(long long)gy * W + gx];
                    const float d = xv - yv;
                    acc_l1 += fabsf(d);
                    const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
                    const float gs = a[0][j] + 2.f * xv * a[1][j] + yv * a[2][j];
                    G[(long long)gy * W + gx] = L.inv_n * ((1.f - L.lambda) * sg - L.lambda * gs);
                }
            }
        }
        __syncthreads();
    }
    // sums of SSIM and |x - y| over the tile (fixed order), one atomic each
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc_s += __shfl_xor_sync(0xffffffffu, acc_s, o);
        acc_l1 += __shfl_xor_sync(0xffffffffu, acc_l1, o);
    }
    if ((tid & 31) == 0) {
        sm.red[0][tid >> 5] = acc_s;
        sm.red[1][tid >> 5] = acc_l1;
    }
    __syncthreads();
    if (SPLIT) {
        // the channels' sums meet in the first channel's block
        tile_wait();   // (every block of the cluster has started: its shared memory may be written)
        if (tid < 2) {
            float sum = 0.f;
            for (int w = 0; w < SS_THREADS / 32; ++w) sum += sm.red[tid][w];
            uint32_t at;
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(&sm.part[tid][rank])), "r"(0));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(at), "f"(sum) : "memory");
        }
        __syncwarp();
        tile_arrive();
        tile_wait();
    }
    if (rank == 0 && tid == 0) {
        float s = 0.f, l = 0.f;
        for (int w = 0; w < (SPLIT ? SS_CH : SS_THREADS / 32); ++w) {
            s += SPLIT ? sm.part[0][w] : sm.red[0][w];
            l += SPLIT ? sm.part[1][w] : sm.red[1][w];
        }
        // The additions to the loss round to the whole, and there are thousands of
        // them: a full tile with SSIM above 1/2 adds its distance from 1 and is
        // counted (an image against itself adds nothing but rounding; two 1237x822
        // images 0.1 apart: error 3e-7 either way, 8e-7 with every distance from 1).
        constexpr float FULL = SS_CH * SS_T * SS_T;
        const unsigned int tiles = (unsigned int)L.tile_base[L.n_views];
        const bool count_ones = tiles < 0x10000u;   // (two 16-bit counts in loss[0], zero before)
        const bool one = count_ones && W - ox >= SS_T && H - oy >= SS_T && s > 0.5f * FULL;
        atomicAdd(&loss[1], l * L.inv_n);
        atomicAdd(&loss[2], (one ? s - FULL : s) * L.inv_n);
        // the last tile forms the loss
        __threadfence();
        const unsigned int n = atomicAdd(reinterpret_cast<unsigned int *>(loss), one ? 0x10001u : 1u);
        if ((count_ones ? n & 0xffffu : n) == tiles - 1) {
            __threadfence();
            const float ones = count_ones ? (float)((n >> 16) + (one ? 1u : 0u)) : 0.f;
            const float l1 = __ldcg(loss + 1), dssim = (1.f - ones * FULL * L.inv_n) - __ldcg(loss + 2);
            loss[2] = dssim;
            loss[0] = (1.f - L.lambda) * l1 + L.lambda * dssim;
        }
    }
}

int launch_l1_dssim(const int *W, const int *H, int n_views, const float *image, const float *target, float lambda,
                    float *loss, float *grad, cudaStream_t st) {
    SsimLaunch L{};
    L.n_views = n_views;
    long long tiles = 0, pix = 0;
    for (int v = 0; v < n_views; ++v) {
        L.W[v] = W[v];
        L.H[v] = H[v];
        L.tiles_x[v] = (W[v] + SS_T - 1) / SS_T;
        L.tiles_y[v] = (H[v] + SS_T - 1) / SS_T;
        L.tile_base[v] = tiles;
        L.pix_base[v] = pix;
        tiles += (long long)L.tiles_x[v] * L.tiles_y[v];
        pix += 3LL * W[v] * H[v];
    }
    L.tile_base[n_views] = tiles;
    double gs[2 * SS_R + 1], tot = 0.0;
    for (int k = 0; k <= 2 * SS_R; ++k) {
        const double d = k - SS_R;
        gs[k] = exp(-d * d / (2.0 * 1.5 * 1.5));
        tot += gs[k];
    }
    for (int k = 0; k <= 2 * SS_R; ++k) L.g[k] = (float)(gs[k] / tot);
    L.lambda = lambda;
    L.inv_n = pix > 0 ? (float)(1.0 / (double)pix) : 0.f;
    if (cudaMemsetAsync(loss, 0, 3 * sizeof(float), st) != cudaSuccess) return GS_ERR_CUDA;
    const size_t smem = sizeof(SsimSmem);
    // Few tiles do not fill the chip: up to 1.5 per SM a block per channel (176 tiles
    // 21 us against 27 with a block per tile, 256 tiles 29 against 27), up to 2 per SM
    // two blocks per SM with twice the registers (304 tiles 27 us against 31, 400 tiles
    // 41 against 37).
    const bool split = 2 * tiles <= 3LL * num_sms(), few = tiles <= 2LL * num_sms();
    const auto kernel = split ? k_l1_dssim<4, true> : few ? k_l1_dssim<2, false> : k_l1_dssim<4, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return GS_ERR_CUDA;
    // (views are at least 1x1: there is a tile)
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = SS_CH;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    lc.gridDim = dim3((unsigned)(split ? SS_CH * tiles : tiles));
    lc.blockDim = dim3(SS_THREADS);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    lc.attrs = at;
    lc.numAttrs = split ? 1 : 0;
    if (cudaLaunchKernelEx(&lc, kernel, L, image, target, grad, loss) != cudaSuccess) return GS_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // namespace gsk
