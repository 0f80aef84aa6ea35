// kernels_local.cu — batched kernels of the inner deflated GMRES (§2 Eq. 4–5, §3), one CTA per
// tile of one task, every task of every subdomain (and right-hand side) in one launch.
//
// Fine tiles cover up to LocalArgs::frows box rows of one task (frows·nx <= LOCAL_THREADS·EPT);
// coarse tiles cover up to LocalArgs::crows coarse rows.  Kernels read each tile's height from the
// tile table; the host sizes shared memory for the largest heights.
// Reductions are two-stage and deterministic: each tile writes its partial sums to a slot of
// its own, and every consumer adds the partials of a task in tile order.
#include <type_traits>

#include "hdd_common.cuh"

namespace hdd {

constexpr int LDP = MAX_RESTART + 2;     // partial-sum slots per tile
constexpr int EPT = FINE_EPT;            // fine elements per thread (frows*max_nx <= 2048)
constexpr int NWARP = LOCAL_THREADS / 32;

// 1D Bézier deflation weight (Eq. 5 factor): fine node f, coarse node c (0-based); column c is
// centred on fine node 2c+1 with weights (1,4,6,4,1)/8 on f = 2c-1 .. 2c+3.
__device__ __forceinline__ float zw_f(int t) {
    return t == 0 || t == 4 ? 0.125f : (t == 2 ? 0.75f : 0.5f);
}
template <typename R> __device__ __forceinline__ R zw(int t) { return (R)zw_f(t); }

template <typename R> __device__ __forceinline__ c2<R> load_c(const c2<R> *p) { return *p; }

// Row of a boundary node (impedance condition): Σ_q cf[q] v_q over the 7 stencil slots.
template <typename R>
__device__ __forceinline__ c2<R> boundary_row(const double2 *__restrict__ cf, c2<R> v0, c2<R> v1, c2<R> v2,
                                           c2<R> v3, c2<R> v4, c2<R> v5, c2<R> v6) {
    const c2<R> v[7] = {v0, v1, v2, v3, v4, v5, v6};
    c2<R> r = mk<R>(0, 0);
#pragma unroll
    for (int q = 0; q < 7; q++) {
        const double2 a = cf[q];
        r = cadd<R>(r, cmul<R>(mk<R>((R)a.x, (R)a.y), v[q]));
    }
    return r;
}

// w = A u at local (x, y) from a shared-memory row buffer u[rows][nx] whose row 0 is box row
// `ybase`; rows outside [0, ny) and columns outside [0, nx) are zero (Dirichlet around the box).
// (gx0, gy0): mesh node of the box's local (0, 0); under the impedance condition the rows of
// nodes on the boundary of the square take their class's complex coefficients.
// IMP: compiled for the impedance condition (the Dirichlet instantiation carries no boundary code).
template <typename R, bool IMP>
__device__ __forceinline__ c2<R> stencil_smem(const Stencil &st, const c2<R> *u, int ybase,
                                              int nrows, int nx, int ny, int x, int y, int gx0, int gy0) {
    const R c0 = (R)st.c0, c1 = (R)st.c1, c2v = (R)st.c2;
    auto U = [&](int xx, int yy) -> c2<R> {
        if (xx < 0 || xx >= nx || yy < 0 || yy >= ny) return mk<R>(0, 0);
        int r = yy - ybase;
        if (r < 0 || r >= nrows) return mk<R>(0, 0);
        return u[r * nx + xx];
    };
    c2<R> cc = U(x, y);
    c2<R> e = U(x + 1, y), wv = U(x - 1, y), n = U(x, y + 1), s = U(x, y - 1);
    c2<R> d1, d2;
    if (st.diag == 0) { d1 = U(x + 1, y + 1); d2 = U(x - 1, y - 1); }
    else { d1 = U(x + 1, y - 1); d2 = U(x - 1, y + 1); }
    c2<R> r;
    if (IMP) {
        const int cls = node_class(st.N, gx0 + x, gy0 + y);
        if (cls != 4) return boundary_row<R>(st.bcoef + cls * 7, cc, e, wv, n, s, d1, d2);
    }
    r.x = c0 * cc.x + c1 * (((e.x + wv.x) + n.x) + s.x) + c2v * (d1.x + d2.x);
    r.y = c0 * cc.y + c1 * (((e.y + wv.y) + n.y) + s.y) + c2v * (d1.y + d2.y);
    return r;
}

// The same on a tile whose rows carry zeros beside and around the box (pitch elements a row): p is
// the centre node, no bounds to check.
template <typename R, bool IMP>
__device__ __forceinline__ c2<R> stencil_padded(const Stencil &st, R c0, R c1, R c2v, const c2<R> *p, int pitch,
                                                int gx, int gy) {
    const int dd = st.diag == 0 ? pitch + 1 : 1 - pitch;
    const c2<R> cc = p[0], e = p[1], wv = p[-1], n = p[pitch], s = p[-pitch], d1 = p[dd], d2 = p[-dd];
    if (IMP) {
        const int cls = node_class(st.N, gx, gy);
        if (cls != 4) return boundary_row<R>(st.bcoef + cls * 7, cc, e, wv, n, s, d1, d2);
    }
    c2<R> r;
    r.x = c0 * cc.x + c1 * (((e.x + wv.x) + n.x) + s.x) + c2v * (d1.x + d2.x);
    r.y = c0 * cc.y + c1 * (((e.y + wv.y) + n.y) + s.y) + c2v * (d1.y + d2.y);
    return r;
}

// Block reduction of `nv` complex partial sums held by every thread (acc computed per l by
// the caller through `get`), written to out[0..nv).
template <typename R, typename F>
__device__ void block_reduce_many(int nv, F get, c2<R> *red /*[NWARP][LDP]*/, c2<R> *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int l = 0; l < nv; l++) {
        c2<R> a = get(l);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { a.x += shfl_xor(a.x, o); a.y += shfl_xor(a.y, o); }
        if (lane == 0) red[warp * LDP + l] = a;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < nv; l += blockDim.x) {
        c2<R> s = mk<R>(0, 0);
        for (int q = 0; q < NWARP; q++) s = cadd<R>(s, red[q * LDP + l]);
        out[l] = s;
    }
}

template <typename R> __device__ R block_sum(R v, R *red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    R s = 0;
    if (threadIdx.x == 0)
        for (int q = 0; q < NWARP; q++) s += red[q];
    return s;
}

// ------------------------------------------------------------------------------------------
// restriction f̃_j = R_j v (Eq. 3), global complex128 → packed local precision R
// ------------------------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_restrict(LocalArgs<R> a, int gw, long long nglob, const double2 *__restrict__ glob,
           c2<R> *__restrict__ out, const int *__restrict__ flag) {
    const Tile tl = a.ftiles[blockIdx.x];
    const Task T = a.tasks[tl.task];
    CHAIN_ENTER();
    LAUNDER(glob); LAUNDER(flag);
    if (flag && !flag[tl.task]) return;
    const int cnt = tl.nr * T.nx;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        int y = tl.r0 + e / T.nx, x = e % T.nx;
        long long gi = (long long)(T.ix0 + x - a.glo) + (long long)(T.iy0 + y - a.glo) * gw +
                       (long long)T.rhs * nglob;
        double2 v = glob[gi];
        out[T.foff + (long long)y * T.nx + x] = mk<R>((R)v.x, (R)v.y);
    }
}

// z = Σ_j R_jᵀ D_j x_j: every owned node is written by exactly one task (no atomics).
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_scatter(LocalArgs<R> a, int gw, long long nglob, const c2<R> *__restrict__ x,
          double2 *__restrict__ glob, const int *__restrict__ flag) {
    const Tile tl = a.ftiles[blockIdx.x];
    if (flag && !flag[tl.task]) return;
    const Task T = a.tasks[tl.task];
    const int cnt = tl.nr * T.nx;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        int y = tl.r0 + e / T.nx, xx = e % T.nx;
        int gx = T.ix0 + xx, gy = T.iy0 + y;
        if (gx < T.ox0 || gx > T.ox1 || gy < T.oy0 || gy > T.oy1) continue;
        c2<R> v = x[T.foff + (long long)y * T.nx + xx];
        glob[(long long)(gx - a.glo) + (long long)(gy - a.glo) * gw + (long long)T.rhs * nglob] =
            make_double2((double)v.x, (double)v.y);
    }
}

// out = A_j in   or   out = f - A_j in   (fine tiles, neighbours read through L1)
template <typename R, bool IMP>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_local_A(LocalArgs<R> a, const c2<R> *__restrict__ in, c2<R> *__restrict__ out,
          const c2<R> *__restrict__ f, const int *__restrict__ flag) {
    extern __shared__ unsigned char smem_raw[];
    c2<R> *u = reinterpret_cast<c2<R> *>(smem_raw);
    const Tile tl = a.ftiles[blockIdx.x];
    if (flag && !flag[tl.task]) return;
    const Task T = a.tasks[tl.task];
    const int y0 = tl.r0 - 1, nrows = tl.nr + 2;
    for (int e = threadIdx.x; e < nrows * T.nx; e += blockDim.x) {
        int yy = y0 + e / T.nx, xx = e % T.nx;
        u[e] = (yy >= 0 && yy < T.ny) ? in[T.foff + (long long)yy * T.nx + xx] : mk<R>(0, 0);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < tl.nr * T.nx; e += blockDim.x) {
        int y = tl.r0 + e / T.nx, x = e % T.nx;
        c2<R> w = stencil_smem<R, IMP>(a.st, u, y0, nrows, T.nx, T.ny, x, y, T.ix0, T.iy0);
        long long gi = T.foff + (long long)y * T.nx + x;
        if (f) w = csub<R>(f[gi], w);
        out[gi] = w;
    }
}

// y = Z_jᵀ t (coarse tiles), with t = A_j in (apply_A) or t = in; y in FP64.
template <typename R, bool IMP>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_zt(LocalArgs<R> a, const c2<R> *__restrict__ in, double2 *__restrict__ yout, int apply_A,
     const int *__restrict__ flag) {
    extern __shared__ unsigned char smem_raw[];
    const Tile tl = a.ctiles[blockIdx.x];
    const Task T = a.tasks[tl.task];
    CHAIN_ENTER();
    LAUNDER(in); LAUNDER(flag);
    if (flag && !flag[tl.task]) return;
    const int nx = T.nx, ny = T.ny, mx = T.mx;
    // fine rows feeding coarse rows [r0, r0+nr): 2c-1 .. 2c+3
    const int F0 = 2 * tl.r0 - 1, F1 = 2 * (tl.r0 + tl.nr - 1) + 3;
    const int nF = F1 - F0 + 1;                    // 2*nr + 3
    const int V0 = F0 - 1, nV = nF + 2;            // input rows for the stencil
    c2<R> *vin = reinterpret_cast<c2<R> *>(smem_raw);
    c2<R> *t = vin + (apply_A ? nV * nx : 0);
    c2<R> *sx = t + nF * nx;
    if (apply_A) {
        for (int e = threadIdx.x; e < nV * nx; e += blockDim.x) {
            int yy = V0 + e / nx, xx = e % nx;
            vin[e] = (yy >= 0 && yy < ny) ? in[T.foff + (long long)yy * nx + xx] : mk<R>(0, 0);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < nF * nx; e += blockDim.x) {
            int yy = F0 + e / nx, xx = e % nx;
            t[e] = (yy >= 0 && yy < ny) ? stencil_smem<R, IMP>(a.st, vin, V0, nV, nx, ny, xx, yy, T.ix0, T.iy0)
                                        : mk<R>(0, 0);
        }
    } else {
        for (int e = threadIdx.x; e < nF * nx; e += blockDim.x) {
            int yy = F0 + e / nx, xx = e % nx;
            t[e] = (yy >= 0 && yy < ny) ? in[T.foff + (long long)yy * nx + xx] : mk<R>(0, 0);
        }
    }
    __syncthreads();
    // x-direction: sx[f][cx] = Σ_a w_a t[f][2cx-1+a]
    for (int e = threadIdx.x; e < nF * mx; e += blockDim.x) {
        int fr = e / mx, cx = e % mx;
        c2<R> s = mk<R>(0, 0);
#pragma unroll
        for (int q = 0; q < 5; q++) {
            int fx = 2 * cx - 1 + q;
            if (fx >= 0 && fx < nx) {
                c2<R> v = t[fr * nx + fx];
                s.x = fma(zw<R>(q), v.x, s.x);
                s.y = fma(zw<R>(q), v.y, s.y);
            }
        }
        sx[e] = s;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < tl.nr * mx; e += blockDim.x) {
        int cy = tl.r0 + e / mx, cx = e % mx;
        c2<R> s = mk<R>(0, 0);
#pragma unroll
        for (int q = 0; q < 5; q++) {
            int fy = 2 * cy - 1 + q;
            if (fy >= 0 && fy < ny) {
                c2<R> v = sx[(fy - F0) * mx + cx];
                s.x = fma(zw<R>(q), v.x, s.x);
                s.y = fma(zw<R>(q), v.y, s.y);
            }
        }
        yout[T.coff + (long long)cy * mx + cx] = make_double2((double)s.x, (double)s.y);
    }
}

// Z s for box rows [F0, F0+nF): s (FP64 coarse) → px (x-interpolated coarse rows) → out(row - F0,
// column, value) for the rows inside the box.  Fine indices go in pairs (2m, 2m + 1), which take the
// coarse entries m-1, m, m+1 with the weights (1/2, 1/2, 0) and (1/8, 3/4, 1/8): a thread makes both
// from three loads, and entries outside the coarse box are staged as zeros, so nothing is selected
// or checked per tap (the sums in the order of the taps).  Shared buffers: sc[rows·((nx+1)/2 + 2)],
// px[rows·nx], rows = prolong_max_cy(nF).  Waits for the thread's asynchronous copies before the
// last barrier; ends without one.
__host__ __device__ inline int prolong_max_cy(int nrows_fine) { return nrows_fine / 2 + 3; }
__host__ __device__ inline int prolong_pitch(int nx) { return (nx + 1) / 2 + 2; }

__device__ __forceinline__ void async_copy(float2 *dst, const float2 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_copy(double2 *dst, const double2 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <typename R, typename Out>
__device__ __forceinline__ void prolong_rows(const Task &T, const double2 *__restrict__ s, int F0, int nF,
                                             c2<R> *sc, c2<R> *px, Out out) {
    const int nx = T.nx, ny = T.ny, mx = T.mx, my = T.my;
    const int hx = (nx + 1) / 2, P = prolong_pitch(nx);
    const int M0 = max(F0, 0) >> 1, M1 = (min(F0 + nF, ny) - 1) >> 1, nm = M1 - M0 + 1;
    const BoxDiv dP(P), dhx(hx), dnx(nx);
    auto mix2 = [](c2<R> p, c2<R> q) {
        return mk<R>(fma((R)0.5, q.x, (R)0.5 * p.x), fma((R)0.5, q.y, (R)0.5 * p.y));
    };
    auto mix3 = [](c2<R> p, c2<R> q, c2<R> r) {
        return mk<R>(fma((R)0.125, r.x, fma((R)0.75, q.x, (R)0.125 * p.x)),
                     fma((R)0.125, r.y, fma((R)0.75, q.y, (R)0.125 * p.y)));
    };
#pragma unroll 2
    for (int e = threadIdx.x; e < (nm + 2) * P; e += blockDim.x) {
        const int rr = dP.q(e), cx = e - rr * P - 1, cy = M0 - 1 + rr;
        c2<R> v = mk<R>(0, 0);
        if ((unsigned)cx < (unsigned)mx && (unsigned)cy < (unsigned)my)
            v = narrow_c<R>(s[T.coff + (long long)cy * mx + cx]);
        sc[e] = v;
    }
    __syncthreads();
#pragma unroll 1
    for (int e = threadIdx.x; e < (nm + 2) * hx; e += blockDim.x) {
        const int r = dhx.q(e), q = e - r * hx;
        const c2<R> *p = sc + r * P + q;
        const c2<R> va = p[0], vb = p[1], vc = p[2];
        c2<R> *o = px + r * nx + 2 * q;
        o[0] = mix2(va, vb);
        if (2 * q + 1 < nx) o[1] = mix3(va, vb, vc);
    }
    async_wait();
    __syncthreads();
#pragma unroll 1
    for (int e = threadIdx.x; e < nm * nx; e += blockDim.x) {
        const int m = dnx.q(e), fx = e - m * nx, f = 2 * (M0 + m) - F0;
        const c2<R> *p = px + m * nx + fx;
        const c2<R> va = p[0], vb = p[nx], vc = p[2 * nx];
        if (f >= 0) out(f, fx, mix2(va, vb));
        if (f + 1 < nF && f + 1 + F0 < ny) out(f + 1, fx, mix3(va, vb, vc));
    }
}

// out = add + Z s on fine tiles (add may be null)
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_z(LocalArgs<R> a, const double2 *__restrict__ s, const c2<R> *__restrict__ add,
    c2<R> *__restrict__ out, const int *__restrict__ flag, R sign) {
    extern __shared__ unsigned char smem_raw[];
    const Tile tl = a.ftiles[blockIdx.x];
    if (flag && !flag[tl.task]) return;
    const Task T = a.tasks[tl.task];
    const int maxc = prolong_max_cy(tl.nr);
    c2<R> *sc = reinterpret_cast<c2<R> *>(smem_raw);
    c2<R> *px = sc + maxc * prolong_pitch(T.nx);
    c2<R> *zs = px + maxc * T.nx;
    prolong_rows<R>(T, s, tl.r0, tl.nr, sc, px, [&](int r, int fx, c2<R> v) { zs[r * T.nx + fx] = v; });
    __syncthreads();
    for (int e = threadIdx.x; e < tl.nr * T.nx; e += blockDim.x) {
        long long gi = T.foff + (long long)tl.r0 * T.nx + e;
        c2<R> v = cscale<R>(sign, zs[e]);
        if (add) v = cadd<R>(add[gi], v);
        out[gi] = v;
    }
}

// Arnoldi (mode 0): out = A (in - Z s), partial dots V_l^H out (l < nv);
// residual (mode 1): out = in - A (Z s), partial ||out||².
template <typename R, bool IMP>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_prolong_stencil(LocalArgs<R> a, int mode, const c2<R> *__restrict__ in,
                  const double2 *__restrict__ s, c2<R> *__restrict__ out,
                  const c2<R> *__restrict__ V, int nv, c2<R> *__restrict__ part,
                  const int *__restrict__ flag) {
    extern __shared__ unsigned char smem_raw[];
    const Tile tl = a.ftiles[blockIdx.x];
    const Task T = a.tasks[tl.task];
    CHAIN_ENTER();
    LAUNDER(in); LAUNDER(s); LAUNDER(V); LAUNDER(flag);
    if (flag && !flag[tl.task]) return;
    const int nx = T.nx, ny = T.ny;
    const int F0 = tl.r0 - 1, nF = tl.nr + 2;
    const int maxc = prolong_max_cy(nF);
    c2<R> *sc = reinterpret_cast<c2<R> *>(smem_raw);
    c2<R> *px = sc + maxc * prolong_pitch(nx);
    c2<R> *u = px + maxc * nx;                     // nF*nx
    c2<R> *red = u + nF * nx;                      // NWARP*LDP
    prolong_rows<R>(T, s, F0, nF, sc, px,          // u = Z s on the box's rows of F0..F0+nF-1
                    [&](int r, int fx, c2<R> v) { u[r * nx + fx] = v; });
    __syncthreads();
    if (mode == 0) {
        for (int e = threadIdx.x; e < nF * nx; e += blockDim.x) {
            int yy = F0 + e / nx;
            if (yy >= 0 && yy < ny) u[e] = csub<R>(in[T.foff + (long long)yy * nx + e % nx], u[e]);
        }
        __syncthreads();
    }
    c2<R> wv[EPT];
    const int cnt = tl.nr * nx;
    R nrm = 0;
#pragma unroll
    for (int k = 0; k < EPT; k++) {
        int e = threadIdx.x + k * LOCAL_THREADS;
        wv[k] = mk<R>(0, 0);
        if (e < cnt) {
            int y = tl.r0 + e / nx, x = e % nx;
            c2<R> w = stencil_smem<R, IMP>(a.st, u, F0, nF, nx, ny, x, y, T.ix0, T.iy0);
            long long gi = T.foff + (long long)y * nx + x;
            if (mode == 1) w = csub<R>(in[gi], w);
            out[gi] = w;
            wv[k] = w;
            nrm = fma(w.x, w.x, fma(w.y, w.y, nrm));
        }
    }
    c2<R> *mypart = part + (long long)blockIdx.x * LDP;
    if (mode == 0) {
        const long long base = T.foff + (long long)tl.r0 * nx;
        block_reduce_many<R>(nv, [&](int l) {
            c2<R> acc = mk<R>(0, 0);
            const c2<R> *vl = V + (long long)l * a.ld + base;
#pragma unroll
            for (int k = 0; k < EPT; k++) {
                int e = threadIdx.x + k * LOCAL_THREADS;
                if (e < cnt) cdotc_acc<R>(acc, vl[e], wv[k]);
            }
            return acc;
        }, red, mypart);
    } else {
        R *redr = reinterpret_cast<R *>(red);
        R tot = block_sum<R>(nrm, redr);
        if (threadIdx.x == 0) mypart[LDP - 1] = mk<R>(tot, 0);
    }
}

// Sum over the task's tiles of the squared-norm slot (LDP-1), by one warp: lane q adds tiles
// q, q+32, ..., then a fixed shuffle tree (deterministic); every lane returns the total.
template <typename R>
__device__ __forceinline__ R task_norm2_warp(const c2<R> *part, const Task &T) {
    const int lane = threadIdx.x & 31;
    R s = 0;
    for (int q = lane; q < T.ntiles; q += 32) s += part[(long long)(T.tile0 + q) * LDP + LDP - 1].x;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Task sums of partial slots l < nv (and, if part2, plus the same slots of part2) into out[l]:
// warp w takes l = w, w + NWARP, ...; its lane q adds tiles q, q+32, ..., then a fixed shuffle
// tree (deterministic).  All tile partials of a slot are loaded at once instead of one after
// another.
template <typename R>
__device__ __forceinline__ void task_sums_warp(const c2<R> *part, const c2<R> *part2, const Task &T, int nv,
                                               c2<R> *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int l = warp; l < nv; l += NWARP) {
        c2<R> s = mk<R>(0, 0);
        for (int q = lane; q < T.ntiles; q += 32) {
            s = cadd<R>(s, part[(long long)(T.tile0 + q) * LDP + l]);
            if (part2) s = cadd<R>(s, part2[(long long)(T.tile0 + q) * LDP + l]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { s.x += shfl_xor(s.x, o); s.y += shfl_xor(s.y, o); }
        if (lane == 0) out[l] = s;
    }
}

// Classical Gram-Schmidt passes 2 and 3 (CGS2): w -= V h (h = task sum of part_in);
// pass 2 also forms the partial dots V^H w, pass 3 the partial ||w||².
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_cgs_update(LocalArgs<R> a, int pass, c2<R> *__restrict__ w, const c2<R> *__restrict__ V, int nv,
             const c2<R> *__restrict__ part_in, c2<R> *__restrict__ part_out,
             const int *__restrict__ flag) {
    __shared__ c2<R> hv[LDP];
    __shared__ c2<R> red[NWARP * LDP];
    const Tile tl = a.ftiles[blockIdx.x];
    if (flag && !flag[tl.task]) return;
    const Task T = a.tasks[tl.task];
    task_sums_warp<R>(part_in, nullptr, T, nv, hv);
    __syncthreads();
    const int cnt = tl.nr * T.nx;
    const long long base = T.foff + (long long)tl.r0 * T.nx;
    c2<R> wv[EPT];
    R nrm = 0;
#pragma unroll
    for (int k = 0; k < EPT; k++) {
        int e = threadIdx.x + k * LOCAL_THREADS;
        wv[k] = mk<R>(0, 0);
        if (e < cnt) {
            c2<R> x = w[base + e];
            for (int l = 0; l < nv; l++) caxpy_neg<R>(x, hv[l], V[(long long)l * a.ld + base + e]);
            w[base + e] = x;
            wv[k] = x;
            nrm = fma(x.x, x.x, fma(x.y, x.y, nrm));
        }
    }
    c2<R> *mypart = part_out + (long long)blockIdx.x * LDP;
    if (pass == 2) {
        block_reduce_many<R>(nv, [&](int l) {
            c2<R> acc = mk<R>(0, 0);
            const c2<R> *vl = V + (long long)l * a.ld + base;
#pragma unroll
            for (int k = 0; k < EPT; k++) {
                int e = threadIdx.x + k * LOCAL_THREADS;
                if (e < cnt) cdotc_acc<R>(acc, vl[e], wv[k]);
            }
            return acc;
        }, red, mypart);
    } else {
        R tot = block_sum<R>(nrm, reinterpret_cast<R *>(red));
        if (threadIdx.x == 0) mypart[LDP - 1] = mk<R>(tot, 0);
    }
}

// Complex Givens rotation G = [c s; -conj(s) c], c real, with G [a; b] = [r; 0] (the standard
// complex form, cf. Bindel, Demmel, Kahan & Marques, ACM TOMS 2002), magnitudes by hypot.
template <typename R>
__device__ void givens(c2<R> a, c2<R> b, R &c, c2<R> &s, c2<R> &r) {
    R aa = hypot(a.x, a.y), bb = hypot(b.x, b.y);
    if (bb == (R)0) { c = 1; s = mk<R>(0, 0); r = a; return; }
    if (aa == (R)0) { c = 0; s = mk<R>(b.x / bb, -b.y / bb); r = mk<R>(bb, 0); return; }
    R t = hypot(aa, bb);
    c2<R> ph = mk<R>(a.x / aa, a.y / aa);
    c = aa / t;
    c2<R> cb = mk<R>(b.x / t, -b.y / t);       // conj(b)/t
    s = cmul<R>(ph, cb);
    r = mk<R>(ph.x * t, ph.y * t);
}

// End of Arnoldi step i: normalise v_{i+1} = w/||w|| (every tile of the task) and, on the
// task's first tile, rotate the new Hessenberg column, update g and test |g_{i+1}| <= tol·ref.
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_givens_normalize(LocalArgs<R> a, InnerState<R> S, int restart, int i, c2<R> *__restrict__ w,
                   const c2<R> *__restrict__ p1, const c2<R> *__restrict__ p2,
                   const c2<R> *__restrict__ p3, const int *__restrict__ act_in,
                   int *__restrict__ act_out, Progress pr, R tol, int maxit) {
    __shared__ R hn_s;
    __shared__ c2<R> hsum[LDP];
    const Tile tl = a.ftiles[blockIdx.x];
    const Task T = a.tasks[tl.task];
    const bool first = blockIdx.x == T.tile0;          // this tile also updates the task's rotations
    if (!act_in[tl.task]) {
        if (first && threadIdx.x == 0) publish(pr, i + 1, 0);
        return;
    }
    if (threadIdx.x < 32) {
        const R s = task_norm2_warp<R>(p3, T);
        if (threadIdx.x == 0) hn_s = sqrt(s);
    }
    // Hessenberg column entries h_l = (pass 1 + pass 2 dots), one task sum per thread
    if (first) task_sums_warp<R>(p1, p2, T, i + 1, hsum);
    __syncthreads();
    const R hn = hn_s;
    if (hn > (R)0) {
        const R inv = (R)1 / hn;
        const long long base = T.foff + (long long)tl.r0 * T.nx;
        for (int e = threadIdx.x; e < tl.nr * T.nx; e += blockDim.x) {
            c2<R> v = w[base + e];
            w[base + e] = mk<R>(v.x * inv, v.y * inv);
        }
    }
    if (!first || threadIdx.x != 0) return;
    const int t = tl.task;
    c2<R> *H = S.H + (long long)t * (restart + 1) * restart;
    c2<R> *hc = H + (long long)i * (restart + 1);
    R *cs = S.cs + (long long)t * restart;
    c2<R> *sn = S.sn + (long long)t * restart;
    c2<R> *g = S.g + (long long)t * (restart + 1);
    for (int l = 0; l <= i; l++) hc[l] = hsum[l];
    for (int l = 0; l < i; l++) {
        c2<R> x = hc[l], y = hc[l + 1];
        c2<R> sx = sn[l];
        // [c s; -conj(s) c] [x; y]
        hc[l] = cadd<R>(cscale<R>(cs[l], x), cmul<R>(sx, y));
        hc[l + 1] = csub<R>(cscale<R>(cs[l], y), cmul<R>(mk<R>(sx.x, -sx.y), x));
    }
    R c; c2<R> s, r;
    givens<R>(hc[i], mk<R>(hn, 0), c, s, r);
    cs[i] = c; sn[i] = s;
    hc[i] = r;
    hc[i + 1] = mk<R>(0, 0);
    c2<R> gi = g[i];
    g[i + 1] = mk<R>(-(s.x * gi.x + s.y * gi.y), -(s.x * gi.y - s.y * gi.x));   // -conj(s) g_i
    g[i] = cscale<R>(c, gi);
    const int its = S.its[t] + 1;
    S.its[t] = its;
    S.kcols[t] = i + 1;
    const R res = hypot(g[i + 1].x, g[i + 1].y);
    const bool conv = res <= tol * S.ref[t] || !(hn > (R)0);
    const bool stop = conv || its >= maxit || i + 1 >= restart;
    if (conv || its >= maxit) S.conv[t] = 1;
    act_out[t] = stop ? 0 : 1;
    publish(pr, i + 1, stop ? 0 : 1);
}

// Start of a cycle: r = P(f̃ - A u) was written into v0 by k_prolong_stencil (mode 1) with its
// partial norms in p3; normalise, set g = [β, 0, ...] and decide whether Arnoldi is needed.
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_init_cycle(LocalArgs<R> a, InnerState<R> S, int restart, c2<R> *__restrict__ v0,
             const c2<R> *__restrict__ p3, const int *__restrict__ flag, int *__restrict__ act_out,
             Progress pr, R tol, int maxit, int set_ref) {
    __shared__ R beta_s;
    const Tile tl = a.ftiles[blockIdx.x];
    const Task T = a.tasks[tl.task];
    CHAIN_ENTER();
    LAUNDER(p3); LAUNDER(flag);
    if (!flag[tl.task]) {
        if (blockIdx.x == T.tile0 && threadIdx.x == 0) publish(pr, 0, 0);
        return;
    }
    if (threadIdx.x < 32) {
        const R s = task_norm2_warp<R>(p3, T);
        if (threadIdx.x == 0) beta_s = sqrt(s);
    }
    __syncthreads();
    const R beta = beta_s;
    if (beta > (R)0) {
        const R inv = (R)1 / beta;
        const long long base = T.foff + (long long)tl.r0 * T.nx;
        for (int e = threadIdx.x; e < tl.nr * T.nx; e += blockDim.x) {
            c2<R> v = v0[base + e];
            v0[base + e] = mk<R>(v.x * inv, v.y * inv);
        }
    }
    if (blockIdx.x != T.tile0 || threadIdx.x != 0) return;
    const int t = tl.task;
    if (set_ref) S.ref[t] = beta;
    c2<R> *g = S.g + (long long)t * (restart + 1);
    g[0] = mk<R>(beta, 0);
    for (int l = 1; l <= restart; l++) g[l] = mk<R>(0, 0);
    S.kcols[t] = 0;
    const bool done = !(beta > tol * S.ref[t]) || S.its[t] >= maxit;
    if (done) S.conv[t] = 1;
    act_out[t] = done ? 0 : 1;
    publish(pr, 0, done ? 0 : 1);
}

// y = H(0:k,0:k)⁻¹ g(0:k) for task t (k <= restart <= 64), by one warp.  Up to 16 columns: H through
// shared memory in one round of loads, lane 2r + c keeps component c of row r, and a step back
// substitutes one entry for all rows above at once (one thread with its loads in a chain took 5 us).
constexpr int SMALL_K = 16;
template <typename R>
__device__ void solve_small(const InnerState<R> &S, int restart, int t, int k, c2<R> *y) {
    __shared__ c2<R> hs[SMALL_K * SMALL_K];
    const c2<R> *H = S.H + (long long)t * (restart + 1) * restart;
    const c2<R> *g = S.g + (long long)t * (restart + 1);
    const int lane = threadIdx.x & 31;
    if (k <= SMALL_K) {
        const int row = lane >> 1, im = lane & 1;
        R acc = row < k ? reinterpret_cast<const R *>(g)[lane] : (R)0;
        for (int e = lane; e < k * SMALL_K; e += 32) {
            const int l = e / SMALL_K, r = e % SMALL_K;
            if (r <= l) hs[e] = H[(long long)l * (restart + 1) + r];
        }
        __syncwarp();
        // row r's lanes divide by its diagonal: q = num·(1/den), once corrected by its remainder
        const c2<R> d = row < k ? hs[row * SMALL_K + row] : mk<R>(1, 0);
        const R den = d.x * d.x + d.y * d.y, rden = (R)1 / den, di = im ? -d.y : d.y;
        for (int r = k - 1; r >= 0; r--) {
            const R num = fma(acc, d.x, shfl_xor(acc, 1) * di);
            R v = num * rden;
            v = fma(fma(-v, den, num), rden, v);
            const R yx = shfl(v, 2 * r), yy = shfl(v, 2 * r + 1);
            if (lane == 0) y[r] = mk<R>(yx, yy);
            if (row < r) {
                const c2<R> h = hs[r * SMALL_K + row];
                acc = fma(-h.x, im ? yy : yx, fma(im ? -h.y : h.y, im ? yx : yy, acc));
            }
        }
        return;
    }
    if (lane) return;
    for (int r = k - 1; r >= 0; r--) {
        c2<R> sacc = g[r];
        for (int l = r + 1; l < k; l++) sacc = csub<R>(sacc, cmul<R>(H[(long long)l * (restart + 1) + r], y[l]));
        c2<R> d = H[(long long)r * (restart + 1) + r];
        R den = d.x * d.x + d.y * d.y;
        y[r] = mk<R>((sacc.x * d.x + sacc.y * d.y) / den, (sacc.y * d.x - sacc.x * d.y) / den);
    }
}

// Coarse part of the completion x = ũ + Z E⁻¹ Zᵀ(f̃ - A ũ): with ũ = ũ₀ + V y, linearity gives
// E⁻¹ Zᵀ(f̃ - A ũ) = s₀ - Σ_i y_i s_{i+1}, where s₀ = E⁻¹ Zᵀ(f̃ - A ũ₀) was solved at the start of
// the cycle and s_{i+1} = E⁻¹ Zᵀ A v_i in Arnoldi step i (slots of sbuf, stride ldc).
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_coarse_combine(LocalArgs<R> a, InnerState<R> S, int restart, const double2 *__restrict__ sbuf,
                 double2 *__restrict__ sc, const int *__restrict__ flag) {
    __shared__ double2 yd[MAX_RESTART];
    __shared__ c2<R> y[MAX_RESTART];
    const Tile tl = a.ctiles[blockIdx.x];
    const Task T = a.tasks[tl.task];
    CHAIN_ENTER();
    LAUNDER(sbuf); LAUNDER(flag);
    if (flag && !flag[tl.task]) return;
    const int k = S.kcols[tl.task];
    if (threadIdx.x < 32) solve_small<R>(S, restart, tl.task, k, y);
    __syncthreads();
    if (threadIdx.x < k) yd[threadIdx.x] = widen_c(y[threadIdx.x]);
    __syncthreads();
    for (int e = threadIdx.x; e < tl.nr * T.mx; e += blockDim.x) {
        const long long idx = T.coff + (long long)tl.r0 * T.mx + e;
        double2 acc = sbuf[idx];
#pragma unroll 4
        for (int l = 0; l < k; l++) {
            const double2 sv = sbuf[(long long)(l + 1) * a.ldc + idx];
            const double yr = yd[l].x, yi = yd[l].y;
            acc.x = fma(-yr, sv.x, fma(yi, sv.y, acc.x));
            acc.y = fma(-yr, sv.y, fma(-yi, sv.x, acc.y));
        }
        sc[idx] = acc;
    }
}

// End of a cycle for its tasks: ũ += V y with y = H⁻¹ g (each tile solves the small triangle
// itself; first: ũ was zero and is not read), and for a task that is done the completed solution
// ũ + Z s straight into the owned nodes of the global vector, z = Σ_j R_jᵀ D_j x_j (every owned
// node is written by exactly one task, no atomics).  A task that neither converged nor ran out of
// iterations keeps ũ and is flagged for another cycle.  One pass over V and z where the update,
// the prolongation and the scatter made three, with ũ and x through memory in between: 13 us
// for the three kernels' 26 at k=200.
template <typename R>
__global__ void __launch_bounds__(LOCAL_THREADS)
k_finish(LocalArgs<R> a, InnerState<R> S, int restart, int first, c2<R> *__restrict__ u, const c2<R> *__restrict__ V,
         const double2 *__restrict__ s, const int *__restrict__ flag, int *__restrict__ rs_out,
         int *__restrict__ its_out, int maxit, long long nglob, double2 *__restrict__ glob) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ c2<R> y[MAX_RESTART];
    const Tile tl = a.ftiles[blockIdx.x];
    const int t = tl.task;
    const Task T = a.tasks[t];
    CHAIN_ENTER();
    LAUNDER(V); LAUNDER(s); LAUNDER(flag);
    if (!flag[t]) return;
    const int k = S.kcols[t];
    const bool again = !S.conv[t] && S.its[t] < maxit;
    if (threadIdx.x < 32) solve_small<R>(S, restart, t, k, y);
    if (threadIdx.x == 32 && blockIdx.x == T.tile0) {
        rs_out[t] = again ? 1 : 0;
        its_out[t] = again ? ~S.its[t] : S.its[t];        // (the host's pinned memory)
    }
    const int maxc = prolong_max_cy(tl.nr);
    c2<R> *sc = reinterpret_cast<c2<R> *>(smem_raw);
    c2<R> *px = sc + maxc * prolong_pitch(T.nx);
    c2<R> *zs = px + maxc * T.nx;
    if (!again) prolong_rows<R>(T, s, tl.r0, tl.nr, sc, px, [&](int r, int fx, c2<R> v) { zs[r * T.nx + fx] = v; });
    __syncthreads();
    const BoxDiv dnx(T.nx);
    const long long base = T.foff + (long long)tl.r0 * T.nx;
    for (int e = threadIdx.x; e < tl.nr * T.nx; e += blockDim.x) {
        const int yy = dnx.q(e), gx = T.ix0 + e - yy * T.nx, gy = T.iy0 + tl.r0 + yy;
        const bool own = gx >= T.ox0 && gx <= T.ox1 && gy >= T.oy0 && gy <= T.oy1;
        if (!again && !own) continue;
        c2<R> x = first ? mk<R>(0, 0) : u[base + e];
#pragma unroll 4
        for (int l = 0; l < k; l++) caxpy<R>(x, y[l], V[(long long)l * a.ld + base + e]);
        if (again) {
            u[base + e] = x;
        } else {
            x = cadd<R>(x, zs[e]);
            glob[(long long)(gx - a.glo) + (long long)(gy - a.glo) * a.gw + (long long)T.rhs * nglob] =
                widen_c(x);
        }
    }
}

// ref_t = ||P f̃_t|| from the per-tile partial norms of P f̃ (one thread per task); used when
// the cycle starts from a non-zero initial guess.
template <typename R>
__global__ void k_set_ref(LocalArgs<R> a, InnerState<R> S, const c2<R> *__restrict__ p3,
                          const int *__restrict__ flag) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.ntasks || (flag && !flag[t])) return;
    const Task T = a.tasks[t];
    R s = 0;
    for (int q = 0; q < T.ntiles; q++) s += p3[(long long)(T.tile0 + q) * LDP + LDP - 1].x;
    S.ref[t] = sqrt(s);
}

template <typename RI, typename RO>
__global__ void k_cast(long long n, const c2<RI> *__restrict__ in, c2<RO> *__restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        out[i] = mk<RO>((RO)in[i].x, (RO)in[i].y);
}

// ------------------------------------------------------------------------------------------
// One inner Arnoldi step in one launch (every phase between two coarse solves), one cluster of
// C CTAs per task: CTA `rank` holds box rows [rank·ny/C, (rank+1)·ny/C) and coarse rows
// [rank·my/C, (rank+1)·my/C).  The new vector w stays in shared memory from the stencil to
// the normalisation; the two sets of task-wide sums (first CGS dots; second CGS dots and ||w||²) are
// all-gathered through distributed shared memory, one cluster barrier each, and every CTA adds
// the C partials in rank order (deterministic, bitwise the same in every CTA).  Steps:
//   A  w = A_j(v_i - Z_j s_{i+1}) (s_{i+1} = E_j⁻¹ Z_jᵀ A_j v_i from the coarse solve), h1 = V^H w
//   B  w -= V h1, h2 = V^H w          (CGS2, both passes against V_0..V_i)
//   C  w -= V h2, ||w||
//   D  v_{i+1} = w/||w||; Hessenberg column h1 + h2, Givens rotation, stop test (every CTA
//      computes the same decision; rank 0 writes the state)
//   E  if the task goes on: y = Z_jᵀ A_j v_{i+1} for the next step's coarse solve (after a
//      cluster barrier that publishes v_{i+1})
// ------------------------------------------------------------------------------------------
constexpr int STEP_CMAX = 8;                       // largest cluster (portable size)

template <typename R> struct StepArgs {
    const Task *tasks;
    Stencil st;
    long long ld;
    int C;                  // CTAs per task (cluster size)
    int i;                  // Arnoldi index
    int restart;
    c2<R> *V;               // basis, vector l at V + l·ld
    const double2 *s;       // s_{i+1} (coarse, FP64)
    double2 *y;             // out: Zᵀ A v_{i+1}
    InnerState<R> S;
    const int *act_in;
    int *act_out;
    Progress pr;
    R tol;
    int maxit;
    R c0, c1, c2v;          // the interior stencil in the inner precision
};

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// generic address of the same shared-memory object in CTA `rank` of the cluster
template <typename T> __device__ __forceinline__ T *cluster_map(T *p, unsigned rank) {
    uint64_t out;
    asm volatile("mapa.u64 %0, %1, %2;\n" : "=l"(out) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
    return reinterpret_cast<T *>(out);
}

size_t step_smem_bytes(int max_nx, int max_ny, int C, int bytes_per_c) {
    const int nr = (max_ny + C - 1) / C, nF = nr + 2, maxc = prolong_max_cy(nF);
    const int my = max_ny / 2, ncy = (my + C - 1) / C, nFz = 2 * ncy + 3, nVz = nFz + 2;
    const size_t px = (size_t)maxc * prolong_pitch(max_nx) + (size_t)maxc * max_nx, w = (size_t)nr * max_nx;
    const size_t a = (px > w ? px : w) + (size_t)nF * (max_nx + 3);
    const size_t e = (size_t)(nVz + nFz) * (max_nx + 3);
    return (a > e ? a : e) * bytes_per_c;
}

// Bound: with FP64 vectors by the FP64 pipe (64 clocks a warp instruction, whatever its lanes do),
// with FP32 by the chain of phases and by fetching instructions that run once or twice each.  So w is
// kept in shared memory, where loops over a thread's elements need no unrolling and end with the box
// (70 KB of code; with w in registers and every loop unrolled 126 KB and 23 us for 17 at k=100); up
// to four basis vectors go through a pass together (w read and written once, the second dots in the
// pass of the first update); the eight sums of four vectors are reduced by halves across the lanes
// (9 additions for 40); ||w||² after the second pass is ||w'||² - ||h2||², both known from the second
// all-gather (V is orthonormal; where h2 is not small against w' and the difference could cancel, it
// is summed directly); tiles in shared memory carry a frame of zeros instead of bounds checks; the
// column's rotations run in one warp, real components, divisions and products spread over its lanes,
// beside the other warps' scaling of v.  Per step: k=100 FP32 21.2 -> 17.0 us, k=200 25 -> 19.8,
// 8192 boxes of 84 x 84 2392 -> 1329; FP64 k=20 49 -> 19.3, k=100 82 -> 60.
template <typename R, bool IMP>
__global__ void __launch_bounds__(LOCAL_THREADS, sizeof(R) == 4 ? 4 : 2)
k_arnoldi_step(StepArgs<R> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ R red[NWARP][2 * LDP];                // per-warp partials (real components)
    __shared__ R gat[2][STEP_CMAX][2 * LDP];         // cluster all-gather slots (written remotely)
    __shared__ c2<R> h1s[LDP], h2s[LDP], hcs[LDP];   // task sums of the two CGS passes, the column
    __shared__ R cs_s[MAX_RESTART];
    __shared__ c2<R> sn_s[MAX_RESTART];
    __shared__ c2<R> g_s;
    __shared__ R ref_s, hn_s, inv_s;
    __shared__ int its_s, stop_s, direct_s;
    const int C = a.C;
    const int t = (int)blockIdx.x / C;
    const unsigned rank = cluster_rank();
    const Task T = a.tasks[t];
    CHAIN_ENTER();
    if (!a.act_in[t]) {                              // the same flag for every CTA of the cluster
        if (rank == 0 && threadIdx.x == 0) {
            a.act_out[t] = 0;
            publish(a.pr, a.i + 1, 0);
        }
        return;
    }
    const int nx = T.nx, ny = T.ny, mx = T.mx, my = T.my;
    const BoxDiv dnx(nx);
    const int i = a.i, nv = i + 1;
    const int r0 = (int)(rank * ny) / C, r1 = (int)((rank + 1) * ny) / C, nr = r1 - r0;
    const int cnt = nr * nx;
    const long long base = T.foff + (long long)r0 * nx;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // ---- A: u = v_i - Z s on rows [r0-1, r1], w = A u on own rows ----
    c2<R> *sc = reinterpret_cast<c2<R> *>(smem_raw);
    const int F0 = r0 - 1, nF = nr + 2, maxc = prolong_max_cy(nF), PU = nx + 2;
    c2<R> *px = sc + maxc * prolong_pitch(nx);
    c2<R> *u = sc + max(maxc * (prolong_pitch(nx) + nx), cnt);   // nF rows of nx + 2, a zero on each side
    c2<R> *const ws = sc;                            // w on own rows, once sc and px are used up
    // rows [y0, y0 + n) of vector v into a framed tile (asynchronously)
    auto stage = [&](const c2<R> *v, c2<R> *tile, int y0, int n, int pitch) {
        const BoxDiv dp(pitch);
#pragma unroll 2
        for (int e = tid; e < n * pitch; e += LOCAL_THREADS) {
            const int q = dp.q(e), x = e - q * pitch - 1, yy = y0 + q;
            if ((unsigned)x < (unsigned)nx && (unsigned)yy < (unsigned)ny) async_copy(tile + e, v + (long long)yy * nx + x);
            else tile[e] = mk<R>(0, 0);
        }
    };
    const c2<R> *const Vt = a.V + T.foff;
    if (nr > 0) stage(Vt + (long long)i * a.ld, u, F0, nF, PU);
    // Givens state of earlier steps (written by earlier launches; rank 0 rewrites it below, after
    // every CTA has passed the first cluster barrier)
    if (tid < i) {
        cs_s[tid] = a.S.cs[(long long)t * a.restart + tid];
        sn_s[tid] = a.S.sn[(long long)t * a.restart + tid];
    }
    if (tid == LOCAL_THREADS - 1) {
        g_s = a.S.g[(long long)t * (a.restart + 1) + i];
        ref_s = a.S.ref[t];
        its_s = a.S.its[t];
    }
    const int nw = min(NWARP, (cnt + 31) / 32);      // warps that hold any of the elements tid + 256 k
    if (nr > 0) {
        prolong_rows<R>(T, a.s, F0, nF, sc, px, [&](int r, int fx, c2<R> z) {
            c2<R> *p = u + r * PU + 1 + fx;
            *p = csub<R>(*p, z);
        });
        __syncthreads();
#pragma unroll 1
        for (int e = tid; e < cnt; e += LOCAL_THREADS) {
            const int qy = dnx.q(e), xx = e - qy * nx;
            ws[e] = stencil_padded<R, IMP>(a.st, a.c0, a.c1, a.c2v, u + (qy + 1) * PU + 1 + xx, PU, T.ix0 + xx,
                                           T.iy0 + r0 + qy);
        }
    }
    // task-wide sums of n real values: the warps' partials red[warp][j] are added per CTA and sent to
    // slot gat[b][rank][j] of every CTA, then one cluster barrier, then each CTA adds the C slots in
    // rank order: get(j, sum)
    auto gather = [&](int b, int n, auto get) {
        __syncthreads();
        for (int j = lane; j < n; j += 32)
            for (int dst = warp; dst < C; dst += NWARP) {
                R sum = 0;
#pragma unroll 1
                for (int q = 0; q < nw; q++) sum += red[q][j];
                *cluster_map(&gat[b][rank][j], (unsigned)dst) = sum;
            }
        cluster_barrier();
        for (int j = tid; j < n; j += LOCAL_THREADS) {
            R sum = gat[b][0][j];
#pragma unroll 1
            for (int q = 1; q < C; q++) sum += gat[b][q][j];
            get(j, sum);
        }
        __syncthreads();
    };
    // one pass of basis vectors l0 .. l0 + 3 over the thread's elements: UPD subtracts h_l v_l from w,
    // DOT adds conj(v_l)·w to acc[l]; both: also |w|² to nrm
    const c2<R> *const Vb = a.V + base;
    R nrm = 0;
    c2<R> acc[4];
    auto pass = [&](auto upd, auto dot, int l0, const c2<R> *h) {
        constexpr bool UPD = decltype(upd)::value, DOT = decltype(dot)::value;
        const int nl = min(4, nv - l0);
        const c2<R> *const vp = Vb + (long long)l0 * a.ld;
        c2<R> hl[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (UPD) hl[q] = h[l0 + min(q, nl - 1)];
            if (DOT) acc[q] = mk<R>(0, 0);
        }
#pragma unroll 2
        for (int e = tid; e < cnt; e += LOCAL_THREADS) {
            c2<R> v[4], w = ws[e];
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (q == 0 || q < nl) v[q] = vp[q * a.ld + e];
            if (UPD) {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (q == 0 || q < nl) caxpy_neg<R>(w, hl[q], v[q]);
                ws[e] = w;
            }
            if (DOT) {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (q == 0 || q < nl) cdotc_acc<R>(acc[q], v[q], w);
            }
            if (UPD && DOT) nrm = fma(w.x, w.x, fma(w.y, w.y, nrm));
        }
    };
    // the eight sums of four vectors over the warp: lanes 16, 8, 4 apart keep one half each
    auto reduce4 = [&](int l0) {
        R v[8];
#pragma unroll
        for (int q = 0; q < 4; q++) { v[2 * q] = acc[q].x; v[2 * q + 1] = acc[q].y; }
#pragma unroll
        for (int half = 4; half > 0; half >>= 1) {
            const bool up = (lane & (4 * half)) != 0;
#pragma unroll
            for (int q = 0; q < half; q++) {
                const R x = shfl_xor(up ? v[q] : v[q + half], 4 * half);
                v[q] = (up ? v[q + half] : v[q]) + x;
            }
        }
        v[0] += shfl_xor(v[0], 2);
        v[0] += shfl_xor(v[0], 1);
        const int j = 2 * l0 + (lane >> 2);
        if ((lane & 3) == 0 && j < 2 * LDP) red[warp][j] = v[0];
    };
    using yes = std::true_type;
    using no = std::false_type;
    // h1 = V^H w
    if (warp < nw)
#pragma unroll 1
        for (int l0 = 0; l0 < nv; l0 += 4) {
            pass(no(), yes(), l0, nullptr);
            reduce4(l0);
        }
    gather(0, 2 * nv, [&](int j, R v) { reinterpret_cast<R *>(h1s)[j] = v; });
    // ---- B: w -= V h1 and, in the pass of the last vectors, h2 = V^H w; slot nv of the sums: ||w||² ----
    if (warp < nw) {
        const int ll = (nv - 1) & ~3;
#pragma unroll 1
        for (int l0 = 0; l0 < ll; l0 += 4) pass(yes(), no(), l0, h1s);
        pass(yes(), yes(), ll, h1s);
        // (in a free place among the last four)
#pragma unroll 1
        for (int l0 = ll; l0 <= nv; l0 += 4) {
            if (l0 > ll) acc[0] = acc[1] = acc[2] = acc[3] = mk<R>(0, 0);
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (l0 + q == nv) acc[q] = mk<R>(nrm, 0);
            reduce4(l0);
        }
#pragma unroll 1
        for (int l0 = 0; l0 < ll; l0 += 4) {
            pass(no(), yes(), l0, nullptr);
            reduce4(l0);
        }
    }
    gather(1, 2 * nv + 1, [&](int j, R v) { reinterpret_cast<R *>(h2s)[j] = v; });
    // ---- C: w -= V h2; the last warp first forms ||w|| ----
    if (warp == NWARP - 1) {
        R hh = 0;
        for (int j = lane; j < 2 * nv; j += 32) { const R x = reinterpret_cast<const R *>(h2s)[j]; hh = fma(x, x, hh); }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) hh += shfl_xor(hh, o);
        const R n2 = h2s[nv].x, hn = sqrt(n2 - hh);
        if (lane == 0) {
            direct_s = hh > (R)0.0625 * n2;
            hn_s = hn;
            inv_s = (R)1 / hn;
        }
    }
    if (warp < nw)
#pragma unroll 1
        for (int l0 = 0; l0 < nv; l0 += 4) pass(yes(), no(), l0, h2s);
    __syncthreads();
    if (direct_s) {                                  // (the same decision in every CTA)
        nrm = 0;
        for (int e = tid; e < cnt; e += LOCAL_THREADS) nrm = fma(ws[e].x, ws[e].x, fma(ws[e].y, ws[e].y, nrm));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nrm += shfl_xor(nrm, o);
        if (lane == 0) red[warp][0] = nrm;
        gather(0, 1, [&](int, R v) { hn_s = sqrt(v); inv_s = (R)1 / sqrt(v); });
    }
    const R hn = hn_s;
    // ---- D: v_{i+1} = w/||w||; Givens rotation and stop test ----
    if (hn > (R)0) {
        const R inv = inv_s;
        c2<R> *vn = a.V + (long long)(i + 1) * a.ld + base;
#pragma unroll 1
        for (int e = tid; e < cnt; e += LOCAL_THREADS) vn[e] = mk<R>(ws[e].x * inv, ws[e].y * inv);
    }
    if (warp == NWARP - 1) {
        for (int l = lane; l <= i; l += 32) hcs[l] = cadd<R>(h1s[l], h2s[l]);
        __syncwarp();
        // earlier rotations: lanes 0, 1 form c x + s y, lanes 2, 3 c y - conj(s) x
        c2<R> x = hcs[0];
        __syncwarp();
        const bool second = (lane & 2) != 0, im = (lane & 1) != 0;
        for (int l = 0; l < i; l++) {
            const c2<R> yv = hcs[l + 1], sx = sn_s[l];
            const R p = second ? (im ? yv.y : yv.x) : (im ? x.y : x.x);
            const R q = second ? (im ? -x.y : -x.x) : (im ? yv.y : yv.x);
            const R r = second ? (im ? x.x : -x.y) : (im ? yv.x : -yv.y);
            const R o = fma(cs_s[l], p, fma(sx.x, q, sx.y * r));
            if (lane < 2) reinterpret_cast<R *>(hcs)[2 * l + lane] = o;
            x = mk<R>(shfl(o, 2), shfl(o, 3));
        }
        R c;
        c2<R> sv, rr;
        rotation_warp<R>(x, hn, c, sv, rr);
        const c2<R> gi = g_s;
        const c2<R> gn = mk<R>(-(sv.x * gi.x + sv.y * gi.y), -(sv.x * gi.y - sv.y * gi.x));   // -conj(s) g_i
        const int its = its_s + 1;
        const R res = hyp(gn.x, gn.y);
        const bool conv = res <= a.tol * ref_s || !(hn > (R)0);
        const bool stop = conv || its >= a.maxit || i + 1 >= a.restart;
        if (lane == 0) {
            stop_s = stop ? 1 : 0;
            hcs[i] = rr;
            hcs[i + 1] = mk<R>(0, 0);
        }
        __syncwarp();
        if (rank == 0) {
            c2<R> *Hc = a.S.H + (long long)t * (a.restart + 1) * a.restart + (long long)i * (a.restart + 1);
            for (int l = lane; l <= i + 1; l += 32) Hc[l] = hcs[l];
            if (lane == 0) {
                a.S.cs[(long long)t * a.restart + i] = c;
                a.S.sn[(long long)t * a.restart + i] = sv;
                c2<R> *g = a.S.g + (long long)t * (a.restart + 1);
                g[i] = cscale<R>(c, gi);
                g[i + 1] = gn;
                a.S.its[t] = its;
                a.S.kcols[t] = i + 1;
                if (conv || its >= a.maxit) a.S.conv[t] = 1;
                a.act_out[t] = stop ? 0 : 1;
            }
        }
    }
    __syncthreads();
    const bool counts = rank == 0 && tid == 0;    // (the count's round trip overlaps what follows)
    if (stop_s) {                                 // the same decision in every CTA
        if (counts) publish(a.pr, i + 1, 0);
        return;
    }
    // ---- E: y = Zᵀ A v_{i+1} on coarse rows [c0, c1) ----
    cluster_barrier();                            // v_{i+1} of every CTA written and visible
    const int c0 = (int)(rank * my) / C, c1 = (int)((rank + 1) * my) / C;
    if (counts && c1 <= c0) publish(a.pr, i + 1, 1);
    if (c1 <= c0) return;
    const int G0 = 2 * c0 - 1, G1 = 2 * (c1 - 1) + 3, nG = G1 - G0 + 1, nW = nG + 2, PE = nx + 3;
    c2<R> *vin = reinterpret_cast<c2<R> *>(smem_raw);                 // rows G0 - 1 .. G1 + 1
    c2<R> *tt = vin + nW * PE;
    stage(Vt + (long long)(i + 1) * a.ld, vin, G0 - 1, nW, PE);
#pragma unroll 1
    for (int e = tid; e < 3 * nG; e += LOCAL_THREADS) {               // columns -1, nx, nx + 1 of A v
        const int q = e / 3, b = e - 3 * q;
        tt[q * PE + (b ? nx + b : 0)] = mk<R>(0, 0);
    }
    if (counts) publish(a.pr, i + 1, 1);
    async_wait();
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < nG * nx; e += LOCAL_THREADS) {
        const int q = dnx.q(e), yy = G0 + q, xx = e - q * nx;
        c2<R> v = mk<R>(0, 0);
        if ((unsigned)yy < (unsigned)ny)
            v = stencil_padded<R, IMP>(a.st, a.c0, a.c1, a.c2v, vin + (q + 1) * PE + 1 + xx, PE, T.ix0 + xx, T.iy0 + yy);
        tt[q * PE + 1 + xx] = v;
    }
    __syncthreads();
    auto five = [](const c2<R> *p, int step) {    // Σ (1,4,6,4,1)/8 · p[q·step]
        c2<R> s = mk<R>(0, 0);
#pragma unroll
        for (int q = 0; q < 5; q++) {
            const c2<R> v = p[q * step];
            s.x = fma(zw<R>(q), v.x, s.x);
            s.y = fma(zw<R>(q), v.y, s.y);
        }
        return s;
    };
    const BoxDiv dmx(mx);
    c2<R> *sx = vin;                              // (A v is done with v)
#pragma unroll 1
    for (int e = tid; e < nG * mx; e += LOCAL_THREADS) {
        const int fr = dmx.q(e), cx = e - fr * mx;
        sx[e] = five(tt + fr * PE + 2 * cx, 1);
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < (c1 - c0) * mx; e += LOCAL_THREADS) {
        const int qc = dmx.q(e), cx = e - qc * mx;
        a.y[T.coff + (long long)c0 * mx + e] = widen_c(five(sx + 2 * qc * mx + cx, mx));
    }
}

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------
template <typename R> static size_t csz() { return sizeof(c2<R>); }

template <typename R>
void launch_restrict(const LocalArgs<R> &a, const double2 *glob, long long nglob, c2<R> *out,
                     const int *flag, cudaStream_t s) {
    launch_chained(k_restrict<R>, a.nftiles, LOCAL_THREADS, 0, s, a, a.gw, nglob, glob, out, flag);
}
template <typename R>
void launch_scatter(const LocalArgs<R> &a, const c2<R> *x, double2 *glob, long long nglob,
                    const int *flag, cudaStream_t s) {
    k_scatter<R><<<a.nftiles, LOCAL_THREADS, 0, s>>>(a, a.gw, nglob, x, glob, flag);
}
template <typename R>
void launch_local_A(const LocalArgs<R> &a, const c2<R> *in, c2<R> *out, const c2<R> *f,
                    const int *flag, cudaStream_t s) {
    size_t sm = (size_t)(a.frows + 2) * a.max_nx * csz<R>();
    if (a.st.bc) k_local_A<R, true><<<a.nftiles, LOCAL_THREADS, sm, s>>>(a, in, out, f, flag);
    else k_local_A<R, false><<<a.nftiles, LOCAL_THREADS, sm, s>>>(a, in, out, f, flag);
}
template <typename R>
size_t zt_smem(const LocalArgs<R> &a, int apply_A) {
    int nF = 2 * a.crows + 3, nV = nF + 2;
    return ((size_t)(apply_A ? nV : 0) * a.max_nx + (size_t)nF * a.max_nx + (size_t)nF * (a.max_nx / 2 + 1)) * csz<R>();
}
template <typename R>
void launch_zt(const LocalArgs<R> &a, const c2<R> *in, double2 *y, int apply_A, const int *flag,
               cudaStream_t s) {
    if (a.st.bc) launch_chained(k_zt<R, true>, a.nctiles, LOCAL_THREADS, zt_smem(a, apply_A), s, a, in, y, apply_A, flag);
    else launch_chained(k_zt<R, false>, a.nctiles, LOCAL_THREADS, zt_smem(a, apply_A), s, a, in, y, apply_A, flag);
}
template <typename R>
size_t z_smem(const LocalArgs<R> &a) {
    const int maxc = prolong_max_cy(a.frows);
    return ((size_t)maxc * prolong_pitch(a.max_nx) + (size_t)maxc * a.max_nx + (size_t)a.frows * a.max_nx) * csz<R>();
}
template <typename R>
void launch_z(const LocalArgs<R> &a, const double2 *sc, const c2<R> *add, c2<R> *out,
              const int *flag, cudaStream_t s, R sign) {
    k_z<R><<<a.nftiles, LOCAL_THREADS, z_smem(a), s>>>(a, sc, add, out, flag, sign);
}
template <typename R>
size_t ps_smem(const LocalArgs<R> &a) {
    int nF = a.frows + 2, maxc = prolong_max_cy(nF);
    return ((size_t)maxc * prolong_pitch(a.max_nx) + (size_t)maxc * a.max_nx + (size_t)nF * a.max_nx +
            (size_t)NWARP * LDP) * csz<R>();
}
template <typename R>
void launch_prolong_stencil(const LocalArgs<R> &a, int mode, const c2<R> *in, const double2 *sc,
                            c2<R> *out, const c2<R> *V, int nv, c2<R> *part, const int *flag,
                            cudaStream_t s) {
    if (a.st.bc)
        launch_chained(k_prolong_stencil<R, true>, a.nftiles, LOCAL_THREADS, ps_smem(a), s, a, mode, in, sc, out, V, nv, part,
                       flag);
    else
        launch_chained(k_prolong_stencil<R, false>, a.nftiles, LOCAL_THREADS, ps_smem(a), s, a, mode, in, sc, out, V, nv, part,
                       flag);
}
template <typename R>
void launch_cgs_update(const LocalArgs<R> &a, int pass, c2<R> *w, const c2<R> *V, int nv,
                       const c2<R> *part_in, c2<R> *part_out, const int *flag, cudaStream_t s) {
    k_cgs_update<R><<<a.nftiles, LOCAL_THREADS, 0, s>>>(a, pass, w, V, nv, part_in, part_out, flag);
}
template <typename R>
void launch_givens_normalize(const LocalArgs<R> &a, const InnerState<R> &S, int restart, int i,
                             c2<R> *w, const c2<R> *p1, const c2<R> *p2, const c2<R> *p3,
                             const int *act_in, int *act_out, const Progress &pr, R tol, int maxit,
                             cudaStream_t s) {
    k_givens_normalize<R><<<a.nftiles, LOCAL_THREADS, 0, s>>>(a, S, restart, i, w, p1, p2, p3, act_in,
                                                               act_out, pr, tol, maxit);
}
template <typename R>
void launch_init_cycle(const LocalArgs<R> &a, const InnerState<R> &S, int restart, c2<R> *v0,
                       const c2<R> *p3, const int *flag, int *act_out, const Progress &pr, R tol,
                       int maxit, int set_ref, cudaStream_t s) {
    launch_chained(k_init_cycle<R>, a.nftiles, LOCAL_THREADS, 0, s, a, S, restart, v0, p3, flag, act_out, pr, tol, maxit,
                   set_ref);
}
template <typename R>
void launch_finish(const LocalArgs<R> &a, const InnerState<R> &S, int restart, int first, c2<R> *u, const c2<R> *V,
                   const double2 *sc, const int *flag, int *rs_out, int *its_out, int maxit, long long nglob,
                   double2 *glob, cudaStream_t s) {
    launch_chained(k_finish<R>, a.nftiles, LOCAL_THREADS, z_smem(a), s, a, S, restart, first, u, V, sc, flag, rs_out, its_out,
                   maxit, nglob, glob);
}
template <typename R>
void launch_set_ref(const LocalArgs<R> &a, const InnerState<R> &S, const c2<R> *p3, const int *flag,
                    cudaStream_t s) {
    k_set_ref<R><<<(a.ntasks + 127) / 128, 128, 0, s>>>(a, S, p3, flag);
}
template <typename R>
void launch_coarse_combine(const LocalArgs<R> &a, const InnerState<R> &S, int restart,
                           const double2 *sbuf, double2 *sc, const int *flag, cudaStream_t s) {
    launch_chained(k_coarse_combine<R>, a.nctiles, LOCAL_THREADS, 0, s, a, S, restart, sbuf, sc, flag);
}
template <typename R>
cudaError_t launch_arnoldi_step(const LocalArgs<R> &la, int C, int i, int restart, c2<R> *V, const double2 *sc,
                                double2 *y, const InnerState<R> &S, const int *act_in, int *act_out,
                                const Progress &pr, R tol, int maxit, size_t smem, cudaStream_t s) {
    StepArgs<R> a;
    a.tasks = la.tasks; a.st = la.st; a.ld = la.ld; a.C = C; a.i = i; a.restart = restart;
    a.V = V; a.s = sc; a.y = y; a.S = S; a.act_in = act_in; a.act_out = act_out; a.pr = pr;
    a.tol = tol; a.maxit = maxit;
    a.c0 = (R)la.st.c0; a.c1 = (R)la.st.c1; a.c2v = (R)la.st.c2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(la.ntasks * C));
    cfg.blockDim = dim3(LOCAL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (la.st.bc) return cudaLaunchKernelEx(&cfg, k_arnoldi_step<R, true>, a);
    return cudaLaunchKernelEx(&cfg, k_arnoldi_step<R, false>, a);
}

// Largest cluster of CTAs holding `smem` bytes of dynamic shared memory each that the device can
// co-schedule (0 on error); sets the kernels' dynamic shared-memory limit to `smem` first.
template <typename R> int arnoldi_step_max_cluster(size_t smem, int C) {
    cudaError_t e;
    if ((e = allow_smem(k_arnoldi_step<R, false>)) != cudaSuccess)
        return 0;
    if ((e = allow_smem(k_arnoldi_step<R, true>)) != cudaSuccess)
        return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(LOCAL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_arnoldi_step<R, false>, &cfg) != cudaSuccess) return 0;
    return n;
}

void launch_cast(long long n, const void *in, int in_double, void *out, int out_double,
                 cudaStream_t s) {
    int grid = (int)((n + 255) / 256);
    if (grid > 4096) grid = 4096;
    if (grid < 1) grid = 1;
    if (in_double && out_double)
        k_cast<double, double><<<grid, 256, 0, s>>>(n, (const double2 *)in, (double2 *)out);
    else if (in_double)
        k_cast<double, float><<<grid, 256, 0, s>>>(n, (const double2 *)in, (float2 *)out);
    else if (out_double)
        k_cast<float, double><<<grid, 256, 0, s>>>(n, (const float2 *)in, (double2 *)out);
    else
        k_cast<float, float><<<grid, 256, 0, s>>>(n, (const float2 *)in, (float2 *)out);
}

size_t local_max_dynamic_smem(int max_nx, int bytes_per_c, int frows, int crows) {
    int nF = frows + 2, maxc = prolong_max_cy(nF);
    size_t ps = ((size_t)maxc * prolong_pitch(max_nx) + (size_t)maxc * max_nx + (size_t)nF * max_nx +
                 (size_t)NWARP * LDP) * bytes_per_c;
    int cF = 2 * crows + 3;
    size_t zt = ((size_t)(cF + 2) * max_nx + (size_t)cF * max_nx + (size_t)cF * (max_nx / 2 + 1)) * bytes_per_c;
    return ps > zt ? ps : zt;
}

template <typename R> cudaError_t set_local_smem_limits() {
    cudaError_t e;
    if ((e = allow_smem(k_prolong_stencil<R, false>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_prolong_stencil<R, true>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_zt<R, false>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_zt<R, true>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_z<R>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_finish<R>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_local_A<R, false>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_local_A<R, true>)) != cudaSuccess) return e;
    return cudaSuccess;
}

#define INST(R)                                                                                         \
    template void launch_restrict<R>(const LocalArgs<R> &, const double2 *, long long, c2<R> *, const int *, cudaStream_t); \
    template void launch_scatter<R>(const LocalArgs<R> &, const c2<R> *, double2 *, long long, const int *, cudaStream_t); \
    template void launch_local_A<R>(const LocalArgs<R> &, const c2<R> *, c2<R> *, const c2<R> *, const int *, cudaStream_t); \
    template void launch_zt<R>(const LocalArgs<R> &, const c2<R> *, double2 *, int, const int *, cudaStream_t); \
    template void launch_z<R>(const LocalArgs<R> &, const double2 *, const c2<R> *, c2<R> *, const int *, cudaStream_t, R); \
    template void launch_prolong_stencil<R>(const LocalArgs<R> &, int, const c2<R> *, const double2 *, c2<R> *, const c2<R> *, int, c2<R> *, const int *, cudaStream_t); \
    template void launch_cgs_update<R>(const LocalArgs<R> &, int, c2<R> *, const c2<R> *, int, const c2<R> *, c2<R> *, const int *, cudaStream_t); \
    template void launch_givens_normalize<R>(const LocalArgs<R> &, const InnerState<R> &, int, int, c2<R> *, const c2<R> *, const c2<R> *, const c2<R> *, const int *, int *, const Progress &, R, int, cudaStream_t); \
    template void launch_init_cycle<R>(const LocalArgs<R> &, const InnerState<R> &, int, c2<R> *, const c2<R> *, const int *, int *, const Progress &, R, int, int, cudaStream_t); \
    template void launch_finish<R>(const LocalArgs<R> &, const InnerState<R> &, int, int, c2<R> *, const c2<R> *, const double2 *, const int *, int *, int *, int, long long, double2 *, cudaStream_t); \
    template cudaError_t set_local_smem_limits<R>(); \
    template void launch_coarse_combine<R>(const LocalArgs<R> &, const InnerState<R> &, int, const double2 *, double2 *, const int *, cudaStream_t); \
    template void launch_set_ref<R>(const LocalArgs<R> &, const InnerState<R> &, const c2<R> *, const int *, cudaStream_t); \
    template cudaError_t launch_arnoldi_step<R>(const LocalArgs<R> &, int, int, int, c2<R> *, const double2 *, double2 *, const InnerState<R> &, const int *, int *, const Progress &, R, int, size_t, cudaStream_t); \
    template int arnoldi_step_max_cluster<R>(size_t, int);

INST(float)
INST(double)

}  // namespace hdd
