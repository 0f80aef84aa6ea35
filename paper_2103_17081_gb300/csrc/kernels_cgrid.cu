// kernels_cgrid.cu — the grid coarse space of the two-level RAS variant (the conclusions, §4,
// name a coarse space as the next step): restriction Pᵀ and interpolation P between the fine
// interior nodes and the P1 nodes of the mesh of spacing H = c·h (same diagonal direction), and
// A_H⁻¹ for the lumped coarse operator A_H = K_H - k²H² I through the 2D sine transform.
//
// Layouts: fine vectors complex128, (N-1)² interior nodes, x fastest, nrhs consecutive vectors
// (stride ldv); coarse vectors m² entries (m = N/c - 1), x fastest, stride ldh.
#include <algorithm>

#include "hdd_common.cuh"

namespace hdd {

// Numerator of the coarse hat function at a fine offset (dx, dy) in fine cells from its node:
// φ = num / c with num = max(0, c - max(|dx|, |dy|, |dx ∓ dy|)) (diag 0: dx - dy, the mesh's
// diagonals run along (1, 1); diag 1: dx + dy, along (1, -1)).
__device__ __forceinline__ int hat_num(int dx, int dy, int c, int diag) {
    const int ad = diag ? abs(dx + dy) : abs(dx - dy);
    const int mx = max(max(abs(dx), abs(dy)), ad);
    return mx < c ? c - mx : 0;
}

// The weights num / c as a table in shared memory (c below CG_TAB; a division costs some 15 FP64
// instructions at 64 clocks a warp, the rest of a node's work 8 to 14)
constexpr int CG_T = 128, CG_TAB = 256;
__device__ __forceinline__ void hat_table(double *tab, int c) {
    if (c < CG_TAB)
        for (int q = threadIdx.x; q <= c; q += CG_T) tab[q] = (double)q / c;
    __syncthreads();
}
__device__ __forceinline__ double hat_weight(const double *tab, int num, int c) {
    return c < CG_TAB ? tab[num] : (double)num / c;
}

// vH = Pᵀ v: a coarse node gathers its (2c-1)² fine neighbours weighted by its hat function
// (all interior nodes for 1 <= I, J <= m), rows of the stencil in increasing fine index.  A CTA takes
// rpb rows of CG_T nodes.  Bound by the FP64 pipe (14 instructions a node at c = 2); N = 640, c = 2:
// 19 us with a division per weight and 64-bit index divisions, 10 now.
template <typename T>
__global__ void __launch_bounds__(CG_T)
k_cg_restrict(CGrid g, const double2 *__restrict__ v, c2<T> *__restrict__ vH, long long ldv, long long ldh,
              const int *__restrict__ active, int rpb) {
    __shared__ double tab[CG_TAB];
    const int m = g.m, c = g.c, w = g.N - 1;
    hat_table(tab, c);
    CHAIN_ENTER();
    LAUNDER(v); LAUNDER(active);
    if (active && !active[blockIdx.z]) return;
    v += blockIdx.z * ldv;
    vH += blockIdx.z * ldh;
    const int I = blockIdx.x * CG_T + threadIdx.x + 1;
    if (I > m) return;
    for (long long j0 = (long long)blockIdx.y * rpb; j0 < m; j0 += (long long)gridDim.y * rpb)
        for (int J = (int)j0 + 1; J <= min(m, (int)j0 + rpb); J++) {
            double sx = 0.0, sy = 0.0;
            for (int dy = 1 - c; dy < c; dy++) {
                const double2 *row = v + (long long)(c * J + dy - 1) * w + (c * I - 1);
#pragma unroll 4
                for (int dx = 1 - c; dx < c; dx++) {
                    const int num = hat_num(dx, dy, c, g.diag);
                    if (num == 0) continue;
                    const double wt = hat_weight(tab, num, c);
                    const double2 a = row[dx];
                    sx = fma(wt, a.x, sx);
                    sy = fma(wt, a.y, sy);
                }
            }
            vH[(I - 1) + (long long)(J - 1) * m] = narrow_c<T>(make_double2(sx, sy));
        }
}

// z = P xH (accumulate = 0) or z += P xH (1): a fine node interpolates the corners of the coarse
// cell that contains it (the corner off its triangle has weight 0; boundary corners hold 0).  CTAs
// as above; N = 640, c = 2: 32 us before, 13 now.
template <typename T>
__global__ void __launch_bounds__(CG_T)
k_cg_prolong(CGrid g, const c2<T> *__restrict__ xH, double2 *__restrict__ z, int accumulate, long long ldv, long long ldh,
             const int *__restrict__ active, int rpb) {
    __shared__ double tab[CG_TAB];
    const int m = g.m, c = g.c, w = g.N - 1;
    hat_table(tab, c);
    const int i = blockIdx.x * CG_T + threadIdx.x + 1, cx0 = i / c;
    CHAIN_ENTER();
    LAUNDER(xH); LAUNDER(active);
    if (active && !active[blockIdx.z]) return;
    z += blockIdx.z * ldv;
    xH += blockIdx.z * ldh;
    if (i > w) return;
    for (long long j0 = (long long)blockIdx.y * rpb; j0 < w; j0 += (long long)gridDim.y * rpb)
        for (int j = (int)j0 + 1; j <= min(w, (int)j0 + rpb); j++) {
            const int cy0 = j / c;
            const long long e = (i - 1) + (long long)(j - 1) * w;
            double2 o = make_double2(0.0, 0.0);
            if (accumulate) o = z[e];
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int b = 0; b < 2; b++) {
                const int J = cy0 + b;
                if (J < 1 || J > m) continue;
#pragma unroll
                for (int a = 0; a < 2; a++) {
                    const int I = cx0 + a;
                    if (I < 1 || I > m) continue;
                    const int num = hat_num(i - c * I, j - c * J, c, g.diag);
                    if (num == 0) continue;
                    const double wt = hat_weight(tab, num, c);
                    const double2 u = widen_c(xH[(I - 1) + (long long)(J - 1) * m]);
                    sx = fma(wt, u.x, sx);
                    sy = fma(wt, u.y, sy);
                }
            }
            z[e] = accumulate ? make_double2(o.x + sx, o.y + sy) : make_double2(sx, sy);
        }
}

// One pass of the separable sine transform: out = (S · in)ᵀ, optionally scaled entrywise by
// Dinv, for an m x m complex matrix `in` (row j, column x) and the real symmetric S:
// out[x][i] = Dinv[x][i] · Σ_j S[i][j] in[j][x].  Two passes give S X S; the solve is
// A_H⁻¹ Y = S (D⁻¹ ∘ (S Y S)) S (S orthonormal and symmetric, D symmetric), four passes.
// The sines of row i are even (i odd, counted from 1) or odd (i even) about the middle of the range,
// S[i][Nc-j] = ±S[i][j], so with e± = in[j] ± in[Nc-j] (the middle entry of an even Nc alone)
// the sum runs over j <= Nc/2 only: half the products.  CTA: a DT x DT output tile (rows i sorted
// by parity in shared memory), four groups of 64 threads that each take a quarter of the j range,
// 4 rows of one parity x 4 columns per thread (16 complex sums for three 16-byte loads); the
// groups' sums are added up through shared memory in a fixed order.  Bound by latency: at m = 319
// there are 100 CTAs, one per SM, so a CTA brings its whole operands (DKC pairs of rows at a time)
// in one go and its eight warps share one tile: 13 us per pass (29 with chunks of 32 rows, four
// warps and all 319 products per output; 0.8 us at the FP32 peak).
constexpr int DT = 32, DTHREADS = 256, DGROUPS = 4;
template <typename T> constexpr int DKC = sizeof(T) == 4 ? 160 : 80;     // pairs of rows staged at a time
template <typename T> constexpr size_t dst_smem() { return (size_t)DKC<T> * DT * (2 * sizeof(c2<T>) + sizeof(T)); }
template <typename T>
__global__ void __launch_bounds__(DTHREADS)
k_dst_pass(int m, long long ldh, const T *__restrict__ S, const T *__restrict__ Dinv,
           const c2<T> *__restrict__ in, c2<T> *__restrict__ out, const int *__restrict__ active) {
    CHAIN_ENTER();
    LAUNDER(in); LAUNDER(active);
    if (active && !active[blockIdx.z]) return;
    in += blockIdx.z * ldh;
    out += blockIdx.z * ldh;
    extern __shared__ __align__(16) unsigned char dsm[];
    c2<T> *E = reinterpret_cast<c2<T> *>(dsm);                           // [parity][pair][column]
    T *Ss = reinterpret_cast<T *>(E + (size_t)2 * DKC<T> * DT);          // [pair][parity · 16 + row / 2]
    const int tid = threadIdx.x, grp = tid >> 6, ti = tid & 7, tx = (tid >> 3) & 7, par = ti >> 2;
    const int i0 = blockIdx.x * DT, x0 = blockIdx.y * DT;
    const int Nc = m + 1, K = Nc / 2;                                    // pairs 1..K (the last without partner if Nc is even)
    c2<T> acc[4][4];                                                     // [column][row]
#pragma unroll
    for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[p][q] = mk<T>((T)0, (T)0);
    for (int k0 = 0; k0 < K; k0 += DKC<T>) {
        const int nk = min(DKC<T>, K - k0);
        if (k0) __syncthreads();
#pragma unroll 4
        for (int e = tid; e < nk * DT; e += DTHREADS) {
            const int kk = e / DT, cc = e % DT, j = k0 + kk + 1, x = x0 + cc, i = i0 + cc;
            c2<T> u = mk<T>((T)0, (T)0), v = u;
            if (x < m) {
                u = in[(long long)(j - 1) * m + x];
                if (2 * j != Nc) v = in[(long long)(Nc - j - 1) * m + x];
            }
            // row index i counts from 0: sine number i + 1, even about the middle for even i
            E[(size_t)kk * DT + cc] = cadd<T>(u, v);
            E[(size_t)(DKC<T> + kk) * DT + cc] = 2 * j != Nc ? csub<T>(u, v) : mk<T>((T)0, (T)0);
            Ss[kk * DT + (cc & 1) * 16 + (cc >> 1)] = i < m ? S[(long long)(j - 1) * m + i] : (T)0;
        }
        __syncthreads();
        // (i0 is a multiple of DT, so a row's parity is that of its place in the tile)
        const c2<T> *Ep = E + (size_t)par * DKC<T> * DT + 4 * tx;
        const T *Sp = Ss + par * 16 + 4 * (ti & 3);
        const int ka = grp * nk / DGROUPS, kb = (grp + 1) * nk / DGROUPS;
#pragma unroll 4
        for (int kk = ka; kk < kb; kk++) {
            T sv[4];
            c2<T> xv[4];
#pragma unroll
            for (int q = 0; q < 4; q++) { sv[q] = Sp[kk * DT + q]; xv[q] = Ep[(size_t)kk * DT + q]; }
#pragma unroll
            for (int p = 0; p < 4; p++)
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    acc[p][q].x = fma(sv[q], xv[p].x, acc[p][q].x);
                    acc[p][q].y = fma(sv[q], xv[p].y, acc[p][q].y);
                }
        }
    }
    __syncthreads();                                                     // the operands' space takes the groups' sums
    c2<T> *R = E;                                                        // [group][column][row], rows padded to 33
    constexpr int RP = DT + 1;
#pragma unroll
    for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) R[((size_t)grp * DT + 4 * tx + p) * RP + 2 * (4 * (ti & 3) + q) + par] = acc[p][q];
    __syncthreads();
    for (int e = tid; e < DT * DT; e += DTHREADS) {
        const int cx = e / DT, ci = e % DT, x = x0 + cx, i = i0 + ci;
        if (x >= m || i >= m) continue;
        c2<T> r = R[(size_t)cx * RP + ci];
#pragma unroll
        for (int g = 1; g < DGROUPS; g++) r = cadd<T>(r, R[((size_t)g * DT + cx) * RP + ci]);
        if (Dinv) {
            const T d = Dinv[(long long)x * m + i];
            r.x *= d;
            r.y *= d;
        }
        out[(long long)x * m + i] = r;
    }
}

template <typename TI, typename TO>
__global__ void k_cg_convert(long long n, const TI *__restrict__ in, TO *__restrict__ out) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const TI a = in[e];
        TO b;
        b.x = a.x;
        b.y = a.y;
        out[e] = b;
    }
}

static int cg_grid(long long n) {
    long long g = (n + 255) / 256;
    if (g > 8 * 152) g = 8 * 152;
    return g < 1 ? 1 : (int)g;
}

template <typename T>
void launch_cg_restrict(const CGrid &g, const double2 *v, c2<T> *vH, int nrhs, long long ldv, long long ldh,
                        const int *active, cudaStream_t s) {
    const int rpb = 2;
    launch_chained(k_cg_restrict<T>, dim3((g.m + CG_T - 1) / CG_T, std::min((g.m + rpb - 1) / rpb, 65535), nrhs), CG_T, 0, s, g,
                   v, vH, ldv, ldh, active, rpb);
}
template <typename T>
void launch_cg_prolong(const CGrid &g, const c2<T> *xH, double2 *z, int accumulate, int nrhs, long long ldv,
                       long long ldh, const int *active, cudaStream_t s) {
    const int w = g.N - 1, rpb = 4;
    launch_chained(k_cg_prolong<T>, dim3((w + CG_T - 1) / CG_T, std::min((w + rpb - 1) / rpb, 65535), nrhs), CG_T, 0, s, g, xH,
                   z, accumulate, ldv, ldh, active, rpb);
}
template <typename T>
void launch_dst_pass(int m, const T *S, const T *Dinv, const c2<T> *in, c2<T> *out, int nrhs, long long ldh,
                     const int *active, cudaStream_t s) {
    const int t = (m + DT - 1) / DT;
    static_assert((size_t)DGROUPS * DT * (DT + 1) * sizeof(c2<T>) <= dst_smem<T>(), "the groups' sums fit");
    allow_smem(k_dst_pass<T>);
    launch_chained(k_dst_pass<T>, dim3(t, t, nrhs), DTHREADS, dst_smem<T>(), s, m, ldh, S, Dinv, in, out, active);
}
void launch_cg_widen(long long n, const float2 *in, double2 *out, cudaStream_t s) {
    k_cg_convert<float2, double2><<<cg_grid(n), 256, 0, s>>>(n, in, out);
}
void launch_cg_narrow(long long n, const double2 *in, float2 *out, cudaStream_t s) {
    k_cg_convert<double2, float2><<<cg_grid(n), 256, 0, s>>>(n, in, out);
}

template void launch_cg_restrict<float>(const CGrid &, const double2 *, float2 *, int, long long, long long,
                                        const int *, cudaStream_t);
template void launch_cg_restrict<double>(const CGrid &, const double2 *, double2 *, int, long long, long long,
                                         const int *, cudaStream_t);
template void launch_cg_prolong<float>(const CGrid &, const float2 *, double2 *, int, int, long long, long long,
                                       const int *, cudaStream_t);
template void launch_cg_prolong<double>(const CGrid &, const double2 *, double2 *, int, int, long long, long long,
                                        const int *, cudaStream_t);
template void launch_dst_pass<float>(int, const float *, const float *, const float2 *, float2 *, int, long long,
                                     const int *, cudaStream_t);
template void launch_dst_pass<double>(int, const double *, const double *, const double2 *, double2 *, int,
                                      long long, const int *, cudaStream_t);

}  // namespace hdd
