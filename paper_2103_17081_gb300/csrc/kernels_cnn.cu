// kernels_cnn.cu — the learned warm start: a 4-layer 3x3 convolutional network (32 channels,
// BF16 weights, FP32 accumulation) mapping a restricted subdomain right-hand side to an initial
// guess for its deflated GMRES, with its training kernels (backward passes and Adam).
//
// Images are the solver's tasks: task t is an nx x ny image stored channels-last at pixel
// offsets Task::foff (activation index (foff + y·nx + x)·C + c).  Zero padding at the box edge
// matches the zero Dirichlet values around a subdomain.
#include "hdd_common.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace hdd {

constexpr int CT = 256;                    // threads per conv CTA

__device__ __forceinline__ float bf2f(__nv_bfloat16 v) { return __bfloat162float(v); }

// Per-task scale σ_t = sqrt(mean |f̃|²) (one CTA per task) and the input image
// (Re f̃/σ, Im f̃/σ, k·h, 0).
template <typename R>
__global__ void __launch_bounds__(CT)
k_cnn_input(const Task *__restrict__ tasks, const c2<R> *__restrict__ f, float kh,
            float *__restrict__ sigma, float *__restrict__ X0, float2 *__restrict__ Fh) {
    __shared__ float red[CT / 32];
    __shared__ float sig_s;
    const Task T = tasks[blockIdx.x];
    const int n = T.nx * T.ny;
    float s = 0.f;
    for (int i = threadIdx.x; i < n; i += CT) {
        const c2<R> v = f[T.foff + i];
        s = fmaf((float)v.x, (float)v.x, fmaf((float)v.y, (float)v.y, s));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int q = 0; q < CT / 32; q++) t += red[q];
        float sg = sqrtf(t / (float)n);
        sig_s = sg > 0.f ? sg : 1.f;
        sigma[blockIdx.x] = sig_s;
    }
    __syncthreads();
    const float inv = 1.f / sig_s;
    for (int i = threadIdx.x; i < n; i += CT) {
        const c2<R> v = f[T.foff + i];
        float4 o = make_float4((float)v.x * inv, (float)v.y * inv, kh, 0.f);
        reinterpret_cast<float4 *>(X0)[T.foff + i] = o;
        if (Fh) Fh[T.foff + i] = make_float2(o.x, o.y);
    }
}

// Y = conv3x3(X) + b, optionally ReLU; one fine tile per CTA, one output pixel per thread step,
// all COUT channels accumulated in registers; weights (BF16 → FP32) staged in shared memory.
template <int CIN, int COUT, bool RELU>
__global__ void __launch_bounds__(CT)
k_conv_fwd(const Task *__restrict__ tasks, const Tile *__restrict__ tiles,
           const __nv_bfloat16 *__restrict__ Wb, const float *__restrict__ bias,
           const float *__restrict__ X, float *__restrict__ Y) {
    __shared__ float Ws[COUT * 9 * CIN];
    __shared__ float Bs[COUT];
    for (int i = threadIdx.x; i < COUT * 9 * CIN; i += CT) Ws[i] = bf2f(Wb[i]);
    for (int i = threadIdx.x; i < COUT; i += CT) Bs[i] = bias[i];
    __syncthreads();
    const Tile tl = tiles[blockIdx.x];
    const Task T = tasks[tl.task];
    const int nx = T.nx, ny = T.ny;
    for (int e = threadIdx.x; e < tl.nr * nx; e += CT) {
        const int y = tl.r0 + e / nx, x = e % nx;
        float acc[COUT];
#pragma unroll
        for (int c = 0; c < COUT; c++) acc[c] = Bs[c];
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const int yy = y + k / 3 - 1, xx = x + k % 3 - 1;
            if (yy < 0 || yy >= ny || xx < 0 || xx >= nx) continue;
            const float4 *xp = reinterpret_cast<const float4 *>(X + (T.foff + (long long)yy * nx + xx) * CIN);
#pragma unroll
            for (int c4 = 0; c4 < CIN / 4; c4++) {
                const float4 v = __ldg(xp + c4);
#pragma unroll
                for (int co = 0; co < COUT; co++) {
                    const float *w = Ws + (co * 9 + k) * CIN + 4 * c4;
                    acc[co] = fmaf(w[0], v.x, fmaf(w[1], v.y, fmaf(w[2], v.z, fmaf(w[3], v.w, acc[co]))));
                }
            }
        }
        float *yp = Y + (T.foff + (long long)y * nx + x) * COUT;
#pragma unroll
        for (int co = 0; co < COUT; co++) yp[co] = RELU ? fmaxf(acc[co], 0.f) : acc[co];
    }
}

// dX[p][ci] = Σ_k Σ_co W[co][k][ci] dY'[p - d_k][co], dY' = dY masked by the ReLU of the
// layer's output (act_out > 0) when act_out is given.
template <int CIN, int COUT>
__global__ void __launch_bounds__(CT)
k_conv_bwd_data(const Task *__restrict__ tasks, const Tile *__restrict__ tiles,
                const __nv_bfloat16 *__restrict__ Wb, const float *__restrict__ dY,
                const float *__restrict__ act_out, float *__restrict__ dX) {
    __shared__ float Ws[COUT * 9 * CIN];
    for (int i = threadIdx.x; i < COUT * 9 * CIN; i += CT) Ws[i] = bf2f(Wb[i]);
    __syncthreads();
    const Tile tl = tiles[blockIdx.x];
    const Task T = tasks[tl.task];
    const int nx = T.nx, ny = T.ny;
    for (int e = threadIdx.x; e < tl.nr * nx; e += CT) {
        const int y = tl.r0 + e / nx, x = e % nx;
        float acc[CIN];
#pragma unroll
        for (int c = 0; c < CIN; c++) acc[c] = 0.f;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            // output pixel q with q + d_k = p
            const int yy = y - (k / 3 - 1), xx = x - (k % 3 - 1);
            if (yy < 0 || yy >= ny || xx < 0 || xx >= nx) continue;
            const long long q = T.foff + (long long)yy * nx + xx;
#pragma unroll
            for (int co = 0; co < COUT; co++) {
                float g = dY[q * COUT + co];
                if (act_out && !(act_out[q * COUT + co] > 0.f)) g = 0.f;
                const float *w = Ws + (co * 9 + k) * CIN;
#pragma unroll
                for (int ci = 0; ci < CIN; ci++) acc[ci] = fmaf(w[ci], g, acc[ci]);
            }
        }
        float *xp = dX + (T.foff + (long long)y * nx + x) * CIN;
#pragma unroll
        for (int ci = 0; ci < CIN; ci++) xp[ci] = acc[ci];
    }
}

// The 32 → 32 channel convolutions of training: Y = conv3x3(X) + b with ReLU (BWD false), or the
// gradient with respect to the input, dX[p][ci] = Σ_k Σ_co W[co][k][ci] dY'[p - d_k][co], dY' = dY
// masked by the ReLU of the layer's output (BWD true: the convolution of dY' with the taps turned
// round and the weights transposed).  CTA: one fine tile in strips of at most `srows` rows, whose
// input rows with their halo (zeros outside the box) lie in shared memory as 32 channel planes
// beside the FP32 weights; a warp takes 128 pixels x 8 output channels, a thread 4 pixels x 8
// channels in registers, so that 32 FMAs share 4 + 2 shared-memory loads (one pixel x 32 channels
// per thread, reading pixels from L2 and a weight per FMA, ran at a fifth of the FP32 rate).  The
// forward sums run in the order tap, then channels 3 2 1 0, 7 6 5 4, ..., that of k_conv_fwd: the
// loss amplifies the rounding of the network's output.  Measured on 64 boxes of 83 x 83 (k=200):
// 303 us forward (505 before), 330 us backward (1320 before); 4.1 G FMAs, 106 us at the FP32 peak.
constexpr int CONV_CH = 8;                 // output channels per thread
constexpr int CONV_PX = 4;                 // pixels per thread, 32 apart
// floats of one channel plane of r rows of a box nx wide: ≡ 1 (mod 32), so that the 8 channels x 4
// pixels a warp writes at a time when it turns the rows into planes fall in distinct banks
__host__ __device__ __forceinline__ int conv_plane(int r, int nx) {
    const int n = (r + 2) * (nx + 2);
    return n + ((33 - n % 32) & 31);
}
constexpr int CONV_T = 384;                // 24 warp tasks of a tile of 8 rows x 83: two rounds of 12 warps
template <bool BWD>
__global__ void __launch_bounds__(CONV_T, 1)
k_conv32(const Task *__restrict__ tasks, const Tile *__restrict__ tiles, int ntiles, const __nv_bfloat16 *__restrict__ Wb,
         const float *__restrict__ bias, const float *__restrict__ X, const float *__restrict__ mask,
         float *__restrict__ Y, int srows) {
    extern __shared__ __align__(16) float csm[];
    float *Ws = csm;                                       // [tap][in][out]
    float *Xs = csm + 9 * 32 * 32;
    for (int i = threadIdx.x; i < 9 * 32 * 32; i += CONV_T) {
        const int ci = i % 32, k = (i / 32) % 9, co = i / 288;
        Ws[BWD ? ((8 - k) * 32 + co) * 32 + ci : (k * 32 + ci) * 32 + co] = bf2f(Wb[i]);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int b = blockIdx.x; b < ntiles; b += gridDim.x) {
    const Tile tl = tiles[b];
    const Task T = tasks[tl.task];
    const int nx = T.nx, ny = T.ny, px = nx + 2;
    for (int s0 = tl.r0; s0 < tl.r0 + tl.nr; s0 += srows) {
        const int sr = min(srows, tl.r0 + tl.nr - s0), plane = conv_plane(sr, nx);
        __syncthreads();                                   // the previous strip is done with (or the weights are there)
        for (int i = threadIdx.x; i < (sr + 2) * px * 8; i += CONV_T) {
            const int q = i >> 3, c = i & 7, yy = s0 - 1 + q / px, xx = q % px - 1;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (yy >= 0 && yy < ny && xx >= 0 && xx < nx) {
                const long long p = (T.foff + (long long)yy * nx + xx) * 8 + c;
                v = __ldg(reinterpret_cast<const float4 *>(X) + p);
                if (BWD) {
                    const float4 m = __ldg(reinterpret_cast<const float4 *>(mask) + p);
                    if (!(m.x > 0.f)) v.x = 0.f;
                    if (!(m.y > 0.f)) v.y = 0.f;
                    if (!(m.z > 0.f)) v.z = 0.f;
                    if (!(m.w > 0.f)) v.w = 0.f;
                }
            }
            float *d = Xs + (size_t)(4 * c) * plane + q;
            d[0] = v.x; d[plane] = v.y; d[2 * plane] = v.z; d[3 * plane] = v.w;
        }
        __syncthreads();
        const int npix = sr * nx, nchunk = (npix + 32 * CONV_PX - 1) / (32 * CONV_PX);
        for (int w = warp; w < nchunk * (32 / CONV_CH); w += CONV_T / 32) {
            const int cog = (w & 3) * CONV_CH, e0 = (w >> 2) * 32 * CONV_PX + lane;
            int off[CONV_PX];
#pragma unroll
            for (int j = 0; j < CONV_PX; j++) {
                const int e = min(e0 + 32 * j, npix - 1), yy = e / nx;
                off[j] = yy * px + (e - yy * nx);          // of tap (-1, -1)
            }
            float acc[CONV_PX][CONV_CH];
#pragma unroll
            for (int j = 0; j < CONV_PX; j++)
#pragma unroll
                for (int c = 0; c < CONV_CH; c++) acc[j][c] = BWD ? 0.f : __ldg(bias + cog + c);
            for (int k = 0; k < 9; k++) {
                const float *xk = Xs + (k / 3) * px + k % 3;
                const float *wk = Ws + k * 1024 + cog;
                for (int c4 = 0; c4 < 8; c4++) {
#pragma unroll
                    for (int r = 3; r >= 0; r--) {
                        const int ci = 4 * c4 + r;
                        const float4 w0 = *reinterpret_cast<const float4 *>(wk + ci * 32);
                        const float4 w1 = *reinterpret_cast<const float4 *>(wk + ci * 32 + 4);
                        const float *xp = xk + (size_t)ci * plane;
#pragma unroll
                        for (int j = 0; j < CONV_PX; j++) {
                            const float v = xp[off[j]];
                            acc[j][0] = fmaf(w0.x, v, acc[j][0]); acc[j][1] = fmaf(w0.y, v, acc[j][1]);
                            acc[j][2] = fmaf(w0.z, v, acc[j][2]); acc[j][3] = fmaf(w0.w, v, acc[j][3]);
                            acc[j][4] = fmaf(w1.x, v, acc[j][4]); acc[j][5] = fmaf(w1.y, v, acc[j][5]);
                            acc[j][6] = fmaf(w1.z, v, acc[j][6]); acc[j][7] = fmaf(w1.w, v, acc[j][7]);
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < CONV_PX; j++) {
                const int e = e0 + 32 * j;
                if (e >= npix) continue;
                float4 *yp = reinterpret_cast<float4 *>(Y + (T.foff + (long long)s0 * nx + e) * 32 + cog);
                float o[CONV_CH];
#pragma unroll
                for (int c = 0; c < CONV_CH; c++) o[c] = BWD ? acc[j][c] : fmaxf(acc[j][c], 0.f);
                yp[0] = make_float4(o[0], o[1], o[2], o[3]);
                yp[1] = make_float4(o[4], o[5], o[6], o[7]);
            }
        }
    }
    }
}

// Weight gradients, partial sums of one CTA's fine tiles b, b + gridDim.x, ...:
//   part[b][(co·9 + k)·CIN + ci] = Σ_q dY'[q][co] X[q + d_k][ci],  part[b][W + co] = Σ_q dY'[q][co].
// A thread owns one input channel, CPT output channels and all nine taps (36 sums for 32 x 32) of
// one of NSEG stretches of every row, and walks along the row with the 3 x 3 window of its channel
// in registers: per pixel three values of X and its dY' from shared memory for 9·CPT FMAs.  The
// rows are staged a row ahead: X by cp.async in a ring of four rows (with a zero column at both ends
// and zero rows outside the box), dY' in two.  Sums are added up per tile first, then over the
// CTA's tiles, the stretches and the CTAs, in a fixed order.  One weight per thread over all pixels
// of a tile, reading dY and X from L2 for every FMA, took 17 ms for a 32 x 32 layer of 64 boxes of
// 83 x 83 (k=200), this 239 us; 4.1 G FMAs, 106 us at the FP32 peak.
template <int CIN, int COUT, int CPT, int NSEG>
__global__ void __launch_bounds__(CT)
k_conv_bwd_w(const Task *__restrict__ tasks, const Tile *__restrict__ tiles, int ntiles, const float *__restrict__ dY,
             const float *__restrict__ act_out, const float *__restrict__ X, float *__restrict__ part, int max_nx) {
    static_assert(CIN * (COUT / CPT) * NSEG == CT, "every thread has its sums");
    constexpr int NW = COUT * 9 * CIN;
    extern __shared__ __align__(16) float csm[];
    const int xrow = (max_nx + 2) * CIN, grow = max_nx * COUT;
    float *Xr = csm, *Gr = csm + 4 * xrow;         // X ring, masked dY rows
    const int tid = threadIdx.x, ci = tid % CIN, cob = (tid / CIN) % (COUT / CPT) * CPT, seg = tid / (CIN * (COUT / CPT));
    float tot[CPT][9], btot[CPT];
#pragma unroll
    for (int c = 0; c < CPT; c++) {
        btot[c] = 0.f;
#pragma unroll
        for (int k = 0; k < 9; k++) tot[c][k] = 0.f;
    }
    auto cp = [](float *d, const float *src, bool in) {       // 16 bytes, zeros where not in
        const unsigned a = (unsigned)__cvta_generic_to_shared(d);
        const int n = in ? 16 : 0;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(a), "l"(src), "r"(n) : "memory");
    };
    for (int b = blockIdx.x; b < ntiles; b += gridDim.x) {
        const Tile tl = tiles[b];
        const Task T = tasks[tl.task];
        const int nx = T.nx, ny = T.ny;
        const int x0 = seg * nx / NSEG, x1 = (seg + 1) * nx / NSEG;
        auto load_x = [&](int y) {                             // row y into ring slot (y + 4) % 4
            float *d = Xr + ((y + 4) & 3) * xrow;
            const bool in = y >= 0 && y < ny;
            const float *src = X + (T.foff + (long long)(in ? y : 0) * nx) * CIN;
            for (int i = tid; i < nx * CIN / 4; i += CT) cp(d + CIN + 4 * i, src + 4 * i, in);
            for (int i = tid; i < CIN; i += CT) { d[i] = 0.f; d[(nx + 1) * CIN + i] = 0.f; }
        };
        auto load_g = [&](int y) {
            const long long o = (T.foff + (long long)y * nx) * COUT;
            float *d = Gr + (y & 1) * grow;
            if (COUT % 4 == 0) {                               // (a row of 2 channels starts on 8 bytes only)
                for (int i = tid; i < nx * COUT / 4; i += CT) {
                    float4 v = __ldg(reinterpret_cast<const float4 *>(dY + o) + i);
                    if (act_out) {
                        const float4 m = __ldg(reinterpret_cast<const float4 *>(act_out + o) + i);
                        if (!(m.x > 0.f)) v.x = 0.f;
                        if (!(m.y > 0.f)) v.y = 0.f;
                        if (!(m.z > 0.f)) v.z = 0.f;
                        if (!(m.w > 0.f)) v.w = 0.f;
                    }
                    reinterpret_cast<float4 *>(d)[i] = v;
                }
            } else {
                for (int i = tid; i < nx * COUT; i += CT) d[i] = act_out && !(act_out[o + i] > 0.f) ? 0.f : dY[o + i];
            }
        };
        __syncthreads();                                       // the previous tile's rows are done with
        load_x(tl.r0 - 1); load_x(tl.r0); load_x(tl.r0 + 1); load_g(tl.r0);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        float acc[CPT][9], bacc[CPT];
#pragma unroll
        for (int c = 0; c < CPT; c++) {
            bacc[c] = 0.f;
#pragma unroll
            for (int k = 0; k < 9; k++) acc[c][k] = 0.f;
        }
        for (int y = tl.r0; y < tl.r0 + tl.nr; y++) {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            __syncthreads();
            if (y + 1 < tl.r0 + tl.nr) { load_x(y + 2); load_g(y + 1); }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            const float *r[3];
#pragma unroll
            for (int d = 0; d < 3; d++) r[d] = Xr + ((y + 3 + d) & 3) * xrow + ci;
            const float *g = Gr + (y & 1) * grow + cob;
            float win[3][3];                                   // [row][column], column (x + j) % 3 holds x + j - 1
#pragma unroll
            for (int d = 0; d < 3; d++) {
                win[d][0] = r[d][x0 * CIN];
                win[d][1] = r[d][(x0 + 1) * CIN];
            }
            auto pixel = [&](int x, int p) {                   // p: (x - x0) % 3
                float gv[CPT];
#pragma unroll
                for (int c = 0; c < CPT; c++) gv[c] = g[x * COUT + c];
#pragma unroll
                for (int d = 0; d < 3; d++) win[d][(p + 2) % 3] = r[d][(x + 2) * CIN];
#pragma unroll
                for (int c = 0; c < CPT; c++) {
                    bacc[c] += gv[c];
#pragma unroll
                    for (int k = 0; k < 9; k++) acc[c][k] = fmaf(gv[c], win[k / 3][(p + k % 3) % 3], acc[c][k]);
                }
            };
            int x = x0;
            for (; x + 2 < x1; x += 3) { pixel(x, 0); pixel(x + 1, 1); pixel(x + 2, 2); }
            if (x < x1) pixel(x, 0);
            if (x + 1 < x1) pixel(x + 1, 1);
        }
#pragma unroll
        for (int c = 0; c < CPT; c++) {
            btot[c] += bacc[c];
#pragma unroll
            for (int k = 0; k < 9; k++) tot[c][k] += acc[c][k];
        }
    }
    float *mine = part + (long long)blockIdx.x * (NW + COUT);
    if (NSEG == 1) {
#pragma unroll
        for (int c = 0; c < CPT; c++) {
            for (int k = 0; k < 9; k++) mine[((cob + c) * 9 + k) * CIN + ci] = tot[c][k];
            if (ci == 0) mine[NW + cob + c] = btot[c];
        }
        return;
    }
    __syncthreads();                                           // rows done with: their space takes the stretches' sums
    float *sums = csm + (size_t)seg * (NW + COUT);
#pragma unroll
    for (int c = 0; c < CPT; c++) {
        for (int k = 0; k < 9; k++) sums[((cob + c) * 9 + k) * CIN + ci] = tot[c][k];
        if (ci == 0) sums[NW + cob + c] = btot[c];
    }
    __syncthreads();
    for (int w = tid; w < NW + COUT; w += CT) {
        float s = 0.f;
        for (int q = 0; q < NSEG; q++) s += csm[(size_t)q * (NW + COUT) + w];
        mine[w] = s;
    }
}

// grad[w] = scale · Σ_p part[p][w]: 32 weights x 8 shares of the partial sums per CTA, shares and
// their sums in a fixed order.
__global__ void __launch_bounds__(256)
k_sum_partials(const float *__restrict__ part, int npart, int nw, float scale, float *__restrict__ grad) {
    __shared__ float red[8][32];
    const int lane = threadIdx.x & 31, sh = threadIdx.x >> 5, w = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (w < nw)
        for (int t = sh; t < npart; t += 8) s += part[(long long)t * nw + w];
    red[sh][lane] = s;
    __syncthreads();
    if (sh == 0 && w < nw) {
        for (int q = 1; q < 8; q++) s += red[q][lane];
        grad[w] = s * scale;
    }
}

// Residual of the guess in normalised units, r = f̃/σ - A (a + i b) (A real, zero outside the
// box), from the input image X0 (channels 0, 1) and the network output Y4 (2 channels); per-tile
// partial Σ|r|²/n_t.
__global__ void __launch_bounds__(CT)
k_cnn_resid(const Task *__restrict__ tasks, const Tile *__restrict__ tiles, Stencil st,
            const float *__restrict__ X0, const float *__restrict__ Y4, float *__restrict__ Rr,
            float *__restrict__ lpart) {
    __shared__ float red[CT / 32];
    const Tile tl = tiles[blockIdx.x];
    const Task T = tasks[tl.task];
    const int nx = T.nx, ny = T.ny;
    const float c0 = (float)st.c0, c1 = (float)st.c1, c2v = (float)st.c2;
    float s = 0.f;
    for (int e = threadIdx.x; e < tl.nr * nx; e += CT) {
        const int y = tl.r0 + e / nx, x = e % nx;
        auto U = [&](int xx, int yy) -> float2 {
            if (xx < 0 || xx >= nx || yy < 0 || yy >= ny) return make_float2(0.f, 0.f);
            return reinterpret_cast<const float2 *>(Y4)[T.foff + (long long)yy * nx + xx];
        };
        const float2 cc = U(x, y), ee = U(x + 1, y), ww = U(x - 1, y), nn = U(x, y + 1), ss = U(x, y - 1);
        float2 d1, d2;
        if (st.diag == 0) { d1 = U(x + 1, y + 1); d2 = U(x - 1, y - 1); }
        else { d1 = U(x + 1, y - 1); d2 = U(x - 1, y + 1); }
        const long long p = T.foff + (long long)y * nx + x;
        const float4 in = reinterpret_cast<const float4 *>(X0)[p];
        float2 r;
        r.x = in.x - (c0 * cc.x + c1 * (((ee.x + ww.x) + nn.x) + ss.x) + c2v * (d1.x + d2.x));
        r.y = in.y - (c0 * cc.y + c1 * (((ee.y + ww.y) + nn.y) + ss.y) + c2v * (d1.y + d2.y));
        reinterpret_cast<float2 *>(Rr)[p] = r;
        s = fmaf(r.x, r.x, fmaf(r.y, r.y, s));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int q = 0; q < CT / 32; q++) t += red[q];
        lpart[blockIdx.x] = t / (float)(nx * ny);
    }
}

// dL/d(a, b) = scale_t · A v (A real symmetric, so Aᵀ = A) for the vector v of the loss.
__global__ void __launch_bounds__(CT)
k_cnn_out_grad(const Task *__restrict__ tasks, const Tile *__restrict__ tiles, Stencil st,
               const float *__restrict__ Rr, const float *__restrict__ scale, float *__restrict__ dY4) {
    const Tile tl = tiles[blockIdx.x];
    const Task T = tasks[tl.task];
    const int nx = T.nx, ny = T.ny;
    const float c0 = (float)st.c0, c1 = (float)st.c1, c2v = (float)st.c2;
    const float sc = scale[tl.task];
    for (int e = threadIdx.x; e < tl.nr * nx; e += CT) {
        const int y = tl.r0 + e / nx, x = e % nx;
        auto U = [&](int xx, int yy) -> float2 {
            if (xx < 0 || xx >= nx || yy < 0 || yy >= ny) return make_float2(0.f, 0.f);
            return reinterpret_cast<const float2 *>(Rr)[T.foff + (long long)yy * nx + xx];
        };
        const float2 cc = U(x, y), ee = U(x + 1, y), ww = U(x - 1, y), nn = U(x, y + 1), ss = U(x, y - 1);
        float2 d1, d2;
        if (st.diag == 0) { d1 = U(x + 1, y + 1); d2 = U(x - 1, y - 1); }
        else { d1 = U(x + 1, y - 1); d2 = U(x - 1, y + 1); }
        float2 g;
        g.x = sc * (c0 * cc.x + c1 * (((ee.x + ww.x) + nn.x) + ss.x) + c2v * (d1.x + d2.x));
        g.y = sc * (c0 * cc.y + c1 * (((ee.y + ww.y) + nn.y) + ss.y) + c2v * (d1.y + d2.y));
        reinterpret_cast<float2 *>(dY4)[T.foff + (long long)y * nx + x] = g;
    }
}

// Loss of the batch: L = mean_t ||P r_t||² / ||P f̂_t||², f̂ = f̃/σ, r = f̂ - A(a + i b) (the
// relative deflated residual the local GMRES starts from).  scale_t = -2 / (ntask ||P f̂_t||²)
// from the per-tile partial norms of P f̂ (slot LDP-1 of each tile's partial-sum block).
__global__ void k_cnn_task_scale(const Task *__restrict__ tasks, int ntask, const float2 *__restrict__ p3f,
                                 float *__restrict__ scale) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntask) return;
    const Task T = tasks[t];
    float s = 0.f;
    for (int q = 0; q < T.ntiles; q++) s += p3f[(long long)(T.tile0 + q) * LOCAL_LDP + LOCAL_LDP - 1].x;
    scale[t] = s > 0.f ? -2.f / ((float)ntask * s) : 0.f;
}
__global__ void k_cnn_task_loss(const Task *__restrict__ tasks, int ntask, const float2 *__restrict__ p3r,
                                const float2 *__restrict__ p3f, float *__restrict__ loss) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntask) return;
    const Task T = tasks[t];
    float a = 0.f, b = 0.f;
    for (int q = 0; q < T.ntiles; q++) {
        a += p3r[(long long)(T.tile0 + q) * LOCAL_LDP + LOCAL_LDP - 1].x;
        b += p3f[(long long)(T.tile0 + q) * LOCAL_LDP + LOCAL_LDP - 1].x;
    }
    loss[t] = b > 0.f ? a / b : 0.f;
}

// x0 = σ_t (a + i b) into the packed local iterate (precision R)
template <typename R>
__global__ void k_cnn_output(const Task *__restrict__ tasks, const Tile *__restrict__ tiles,
                             const float *__restrict__ sigma, const float *__restrict__ Y4,
                             c2<R> *__restrict__ x0, const int *__restrict__ flag) {
    const Tile tl = tiles[blockIdx.x];
    if (flag && !flag[tl.task]) return;
    const Task T = tasks[tl.task];
    const float sg = sigma[tl.task];
    for (int e = threadIdx.x; e < tl.nr * T.nx; e += blockDim.x) {
        const long long p = T.foff + (long long)tl.r0 * T.nx + e;
        const float2 v = reinterpret_cast<const float2 *>(Y4)[p];
        x0[p] = mk<R>((R)(sg * v.x), (R)(sg * v.y));
    }
}

// Adam on the FP32 master weights (Kingma & Ba 2015), then the BF16 copy used by the kernels.
__global__ void k_adam(int n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, __nv_bfloat16 *__restrict__ pb, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi; v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    pb[i] = __float2bfloat16(pi);
}

__global__ void k_to_bf16(int n, const float *__restrict__ p, __nv_bfloat16 *__restrict__ pb) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) pb[i] = __float2bfloat16(p[i]);
}

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------
template <typename R>
void launch_cnn_input(const Task *tasks, int ntasks, const c2<R> *f, float kh, float *sigma, float *X0,
                      float2 *Fh, cudaStream_t s) {
    k_cnn_input<R><<<ntasks, CT, 0, s>>>(tasks, f, kh, sigma, X0, Fh);
}
void launch_cnn_task_scale(const Task *tasks, int ntasks, const float2 *p3f, float *scale, cudaStream_t s) {
    k_cnn_task_scale<<<(ntasks + 127) / 128, 128, 0, s>>>(tasks, ntasks, p3f, scale);
}
void launch_cnn_task_loss(const Task *tasks, int ntasks, const float2 *p3r, const float2 *p3f, float *loss,
                          cudaStream_t s) {
    k_cnn_task_loss<<<(ntasks + 127) / 128, 128, 0, s>>>(tasks, ntasks, p3r, p3f, loss);
}
template <typename R>
void launch_cnn_output(const Task *tasks, const Tile *tiles, int ntiles, const float *sigma,
                       const float *Y4, c2<R> *x0, const int *flag, cudaStream_t s) {
    k_cnn_output<R><<<ntiles, 256, 0, s>>>(tasks, tiles, sigma, Y4, x0, flag);
}
static int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
        n = 152;
    return n;
}
template <bool BWD>
static void conv32(const Task *tasks, const Tile *tiles, int ntiles, int max_nx, int frows, const __nv_bfloat16 *W,
                   const float *b, const float *X, const float *mask, float *Y, cudaStream_t s) {
    // the most rows per strip that fit 220 KB beside the weights
    int sr = frows;
    auto smem = [&](int r) { return (size_t)(9 * 32 * 32 + 32 * conv_plane(r, max_nx)) * sizeof(float); };
    while (sr > 1 && smem(sr) > 220 * 1024) sr--;
    // (narrower boxes, or fewer rows, may have a larger stride than their size by the padding)
    const size_t sm = smem(sr) + 32 * 32 * sizeof(float);
    if (allow_smem(k_conv32<BWD>) != cudaSuccess) return;          // (the error stays for the caller to find)
    k_conv32<BWD><<<std::min(ntiles, sm_count()), CONV_T, sm, s>>>(tasks, tiles, ntiles, W, b, X, mask, Y, sr);
}
void launch_conv_fwd(int layer, const Task *tasks, const Tile *tiles, int ntiles, int max_nx, int frows,
                     const __nv_bfloat16 *W, const float *b, const float *X, float *Y, cudaStream_t s) {
    switch (layer) {
        case 0: k_conv_fwd<4, 32, true><<<ntiles, CT, 0, s>>>(tasks, tiles, W, b, X, Y); break;
        case 1:
        case 2: conv32<false>(tasks, tiles, ntiles, max_nx, frows, W, b, X, nullptr, Y, s); break;
        default: k_conv_fwd<32, 2, false><<<ntiles, CT, 0, s>>>(tasks, tiles, W, b, X, Y); break;
    }
}
void launch_conv_bwd_data(int layer, const Task *tasks, const Tile *tiles, int ntiles, int max_nx, int frows,
                          const __nv_bfloat16 *W, const float *dY, const float *act_out, float *dX,
                          cudaStream_t s) {
    switch (layer) {
        case 1:
        case 2: conv32<true>(tasks, tiles, ntiles, max_nx, frows, W, nullptr, dY, act_out, dX, s); break;
        case 3: k_conv_bwd_data<32, 2><<<ntiles, CT, 0, s>>>(tasks, tiles, W, dY, act_out, dX); break;
        default: break;                       // the input image needs no gradient
    }
}
// CTAs (and partial sums) of the weight gradients: two per SM
int conv_bwd_w_parts(int ntiles) { return std::min(ntiles, 2 * sm_count()); }
template <int CIN, int COUT, int CPT, int NSEG>
static void bwd_w(const Task *tasks, const Tile *tiles, int ntiles, int max_nx, const float *dY, const float *act_out,
                  const float *X, float *part, cudaStream_t s) {
    const size_t rows = (size_t)4 * (max_nx + 2) * CIN + (size_t)2 * max_nx * COUT;
    const size_t sums = NSEG > 1 ? (size_t)NSEG * (COUT * 9 * CIN + COUT) : 0;
    const size_t sm = std::max(rows, sums) * sizeof(float);
    if (allow_smem(k_conv_bwd_w<CIN, COUT, CPT, NSEG>) != cudaSuccess) return;
    k_conv_bwd_w<CIN, COUT, CPT, NSEG><<<conv_bwd_w_parts(ntiles), CT, sm, s>>>(tasks, tiles, ntiles, dY, act_out, X,
                                                                               part, max_nx);
}
void launch_conv_bwd_w(int layer, const Task *tasks, const Tile *tiles, int ntiles, int max_nx, const float *dY,
                       const float *act_out, const float *X, float *part, cudaStream_t s) {
    switch (layer) {
        case 0: bwd_w<4, 32, 4, 8>(tasks, tiles, ntiles, max_nx, dY, act_out, X, part, s); break;
        case 1:
        case 2: bwd_w<32, 32, 4, 1>(tasks, tiles, ntiles, max_nx, dY, act_out, X, part, s); break;
        default: bwd_w<32, 2, 2, 8>(tasks, tiles, ntiles, max_nx, dY, act_out, X, part, s); break;
    }
}
void launch_sum_partials(const float *part, int npart, int nw, float scale, float *grad, cudaStream_t s) {
    k_sum_partials<<<(nw + 31) / 32, 256, 0, s>>>(part, npart, nw, scale, grad);
}
void launch_cnn_resid(const Task *tasks, const Tile *tiles, int ntiles, const Stencil &st, const float *X0,
                      const float *Y4, float *Rr, float *lpart, cudaStream_t s) {
    k_cnn_resid<<<ntiles, CT, 0, s>>>(tasks, tiles, st, X0, Y4, Rr, lpart);
}
void launch_cnn_out_grad(const Task *tasks, const Tile *tiles, int ntiles, const Stencil &st, const float *Rr,
                         const float *scale, float *dY4, cudaStream_t s) {
    k_cnn_out_grad<<<ntiles, CT, 0, s>>>(tasks, tiles, st, Rr, scale, dY4);
}
void launch_adam(int n, float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, float lr, float b1,
                 float b2, float eps, int step, cudaStream_t s) {
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_adam<<<(n + 255) / 256, 256, 0, s>>>(n, p, g, m, v, pb, lr, b1, b2, eps, c1, c2);
}
void launch_to_bf16(int n, const float *p, __nv_bfloat16 *pb, cudaStream_t s) {
    k_to_bf16<<<(n + 255) / 256, 256, 0, s>>>(n, p, pb);
}

template void launch_cnn_input<float>(const Task *, int, const float2 *, float, float *, float *, float2 *, cudaStream_t);
template void launch_cnn_input<double>(const Task *, int, const double2 *, float, float *, float *, float2 *, cudaStream_t);
template void launch_cnn_output<float>(const Task *, const Tile *, int, const float *, const float *, float2 *, const int *, cudaStream_t);
template void launch_cnn_output<double>(const Task *, const Tile *, int, const float *, const float *, double2 *, const int *, cudaStream_t);

}  // namespace hdd
