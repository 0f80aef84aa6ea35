// kernels_dense.cu — the coarse solve E_j⁻¹ y as a matrix product on the 5th-generation tensor
// cores, with the explicit inverse of every distinct E_j formed at set-up.
//
// The banded substitutions (kernels_coarse.cu) are one dependent chain per vector: 164 us per
// launch at k=200 however few bytes they read.  E_j⁻¹ y has no chain.  It reads more (m² entries
// per shape, 170 MB for the four shapes of k=200), all shapes' tiles spread over all SMs, and
// every task of a shape is one more column of the same product.
//
// Arithmetic: integers, exact.  Row i of E_j⁻¹ is scaled by a power of two 2^ea and rounded to
// multiples of 2^(ea-55); each column of y likewise (2^eb).  The 56-bit integers are written in
// base 256 with DSL = 7 signed digits of at most 128, which BF16 holds exactly.  A product of two
// digits has at most 14 bits, so the FP32 accumulators of the tensor cores hold the sums of
// products of equal weight exactly up to 2^24.  On smooth data the leading digits add up instead of
// cancelling (a constant against E⁻¹ at k = 4 reaches 1.45·2^24 over 4096 columns, where whole rows
// in one sum then cost 1e-10 to 4e-8 of the solution), so a sum runs over at most dense_seg() chunks
// before it moves to integers: 64 chunks of 16 columns, where the products of the leading digits stay
// within 2^24 whatever the data (0.64·2^24 at most was seen for all of them together: constants,
// half-sines, rows of E⁻¹ itself), 32 for complex E, whose rows can be constant to more
// than a digit (impedance condition, small k).  Sums of weight p + q < DS are kept, the rest
// lies below a 2^-8DS part of a column's and a row's largest entries: DS = 7 for the complex128
// iteration, DS = 6 (48 bits, what the double-FP32 banded solve carries) for the complex64 one.
// The DS sums are put together in 64-bit integers, in units of 2^13 of the last one's: a part of a
// tile rounds its two last sums to such a unit (2^-60 of a full product), and the parts add up to
// the same bits in whatever order they come.
#include "hdd_common.cuh"
#include "umma.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

namespace hdd {

constexpr int DE_G = 3;                          // groups of four widening warps
__host__ __device__ constexpr int de_threads(bool by) { return 320 + (by ? 128 * DE_G : 0); }   // 8 epilogue warps, a copy warp, an MMA warp, the widening warps
constexpr unsigned long long DE_LIMIT = 2000000000ull;   // ns after which a device wait gives up

// v·2^(F-e) rounded to an integer, |v| < 2^e: at most 2^F (F <= 55).  On the significand, in
// integer instructions: the FP64 pipe does two operations a clock.
template <int F>
__device__ __forceinline__ long long fixed_point(double v, int e) {
    const long long b = __double_as_longlong(v);
    const int E = (int)((b >> 52) & 0x7ff);
    long long m = (b & 0xfffffffffffffll) | (E ? 1ll << 52 : 0);
    const int sh = (E ? E : 1) - 1075 + F - e;              // m·2^sh, sh <= F - 53
    if (sh >= 0) m <<= sh;
    else m = sh < -54 ? 0 : (m + (1ll << (-sh - 1))) >> -sh;
    return b < 0 ? -m : m;
}
// lowest signed digit of q in base 256; q becomes the rest
__device__ __forceinline__ int digit256(long long &q) {
    const int d = (int)(signed char)(q & 255);   // -128..127
    q = (q - d) >> 8;
    return d;
}
__device__ __forceinline__ uint32_t bf16_pair(int a, int b) {
    __nv_bfloat162 v = __floats2bfloat162_rn((float)a, (float)b);
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
// exponent e with |v| < 2^e from the bits of the largest |v|
__device__ __forceinline__ int exp_of(unsigned long long bits) { return (int)(bits >> 52) - 1022; }
constexpr unsigned long long INF_BITS = 0x7ff0000000000000ull;
constexpr int EXP_NAN = 1 << 20;                 // exponent of a row or column that is not finite

// v·2^e rounded to FP64, in integer instructions (the FP64 pipe would take 15 k clocks for the
// outputs of one tile); NaN for an exponent that holds EXP_NAN.
__device__ __forceinline__ double from_fixed(long long v, int e) {
    if (v == 0 && e < EXP_NAN / 2) return 0.0;
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);
    const unsigned long long m = ((a << lz) >> 1) + (1ull << 9);     // top bit at 62, rounded at bit 10
    const int x = e + 63 - lz + 1023;                                // biased exponent of the top bit
    if (x < 2 || x > 2045)                                           // near the ends of the range
        return e >= EXP_NAN / 2 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)v, e);
    // the significand's top bit (and a carry of the rounding) add to the exponent field
    return __longlong_as_double((long long)(((unsigned long long)(x - 1) << 52) + (m >> 10)) | (v & (1ll << 63)));
}

// ------------------------------------------------------------------------------------------
// Set-up: columns of E⁻¹ by the blocked substitutions of every unit vector
// ------------------------------------------------------------------------------------------

// One CTA solves 16 unit vectors (columns 16·Jc .. of E⁻¹; of a real-equivalent factor the unit
// vectors of 16 real parts) with the shape's block operators, thread (r, c) row r of a block and
// column c.  E⁻¹ is symmetric (complex symmetric under the impedance condition), so the backward
// sweep stops at the columns' own block and only rows from there on are kept.  The forward sweep
// starts at the first block the permuted unit vectors reach.  Bound by the FP64 pipe (2 FMA per
// clock and SM): about m²·(w_l + w_u)/2 FMAs per shape, 0.35 G at m = 1681.
// W: job's columns row-major, 16 doubles per row, rows 0 .. 16·nblk.
template <bool RE2>
__global__ void __launch_bounds__(256)
k_inv_cols(const InvJob *__restrict__ jobs, const BlockFactor *__restrict__ shapes, const double *__restrict__ Mall,
           const int *__restrict__ Pall, const int4 *__restrict__ Meta, double *__restrict__ Wall, int maxK, int cw) {
    extern __shared__ __align__(16) double dsm[];
    double *Mb[2] = {dsm, dsm + (size_t)BNB * maxK};
    double *win = dsm + 2 * (size_t)BNB * maxK;       // cw x 16
    double *yb = win + (size_t)cw * 16;               // 16 x 16
    __shared__ int pos[16];
    const InvJob jb = jobs[blockIdx.x];
    const BlockFactor F = shapes[jb.shape];
    const double *M = Mall;
    const int4 *meta = Meta + F.meta_off;
    const int *perm = Pall + F.perm_off;
    const int tid = threadIdx.x, r = tid >> 4, c = tid & 15, mask = cw - 1, nb = F.nblk;
    double *W = Wall + jb.woff;
    auto unit = [&](int col) { return RE2 ? 2 * (16 * jb.jc + col) : 16 * jb.jc + col; };
    if (tid < 16) pos[tid] = 0x7fffffff;
    __syncthreads();
    {   // row of the permuted unit vector: perm[i] = unit
        const int u0 = unit(0), u1 = unit(15);
        for (int i = tid; i < F.m; i += 256) {
            const int u = perm[i];
            if (u < u0 || u > u1) continue;
            if (RE2 && (u & 1)) continue;
            pos[RE2 ? (u - u0) >> 1 : u - u0] = i;
        }
    }
    for (int e = tid; e < cw * 16; e += 256) win[e] = 0.0;
    __syncthreads();
    int Js = nb;
    for (int q = 0; q < 16; q++) Js = min(Js, pos[q] == 0x7fffffff ? nb : pos[q] / BNB);
    const int Jstop = RE2 ? 2 * jb.jc : jb.jc;
    const int mypos = pos[c];
    auto fetch = [&](int off, int w, int b) {
        const double *src = M + off;
        const int n = BNB * op_stride(w);
        for (int e = 2 * tid; e < n; e += 512) {
            const unsigned d = (unsigned)__cvta_generic_to_shared(Mb[b] + e);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src + e) : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    auto arrived = [&]() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); __syncthreads(); };
    // forward: y_J = M_J [b_J; y of the w rows before block J]
    if (Js < nb) fetch(meta[Js].x, meta[Js].y, 0);
    for (int J = Js; J < nb; J++) {
        const int b = (J - Js) & 1, w = meta[J].y, K = op_stride(w);
        arrived();
        if (J + 1 < nb) fetch(meta[J + 1].x, meta[J + 1].y, b ^ 1);
        const double *row = Mb[b] + (size_t)r * K;
        double s0 = 0.0, s1 = 0.0;
        if (mypos / BNB == J) s0 = row[mypos & (BNB - 1)];
        const int base = J * BNB - w;
        int k = max(0, Js * BNB - base);
        for (; k + 1 < w; k += 2) {
            s0 = fma(row[BNB + k], win[((base + k) & mask) * 16 + c], s0);
            s1 = fma(row[BNB + k + 1], win[((base + k + 1) & mask) * 16 + c], s1);
        }
        if (k < w) s0 = fma(row[BNB + k], win[((base + k) & mask) * 16 + c], s0);
        s0 += s1;
        win[((J * BNB + r) & mask) * 16 + c] = s0;
        W[(size_t)(J * BNB + r) * 16 + c] = s0;
    }
    __syncthreads();
    for (int e = tid; e < cw * 16; e += 256) win[e] = 0.0;
    // backward: x_J = M_J [y_J; x of the w rows after block J]
    fetch(meta[nb - 1].z, meta[nb - 1].w, 0);
    for (int J = nb - 1; J >= Jstop; J--) {
        const int b = (nb - 1 - J) & 1, w = meta[J].w, K = op_stride(w);
        const double yv = J >= Js ? W[(size_t)(J * BNB + r) * 16 + c] : 0.0;
        __syncthreads();                                 // the previous step's reads of yb are done
        yb[r * 16 + c] = yv;
        arrived();
        if (J > Jstop) fetch(meta[J - 1].z, meta[J - 1].w, b ^ 1);
        const double *row = Mb[b] + (size_t)r * K;
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int k = 0; k < BNB; k += 2) {
            s0 = fma(row[k], yb[k * 16 + c], s0);
            s1 = fma(row[k + 1], yb[(k + 1) * 16 + c], s1);
        }
        const int base = (J + 1) * BNB, wr = min(w, nb * BNB - base);
        int k = 0;
        for (; k + 1 < wr; k += 2) {
            s0 = fma(row[BNB + k], win[((base + k) & mask) * 16 + c], s0);
            s1 = fma(row[BNB + k + 1], win[((base + k + 1) & mask) * 16 + c], s1);
        }
        if (k < wr) s0 = fma(row[BNB + k], win[((base + k) & mask) * 16 + c], s0);
        s0 += s1;
        win[((J * BNB + r) & mask) * 16 + c] = s0;
        W[(size_t)(J * BNB + r) * 16 + c] = s0;
    }
}

// Entry (i, j) of E⁻¹ (its part 0 real, 1 imaginary) from the kept lower blocks.
__device__ __forceinline__ double inv_entry(const double *__restrict__ W, size_t rows, int re2, int part, int i, int j) {
    if ((i >> 4) < (j >> 4)) { const int t = i; i = j; j = t; }
    const size_t row = re2 ? 2 * (size_t)i + part : (size_t)i;
    return W[((size_t)(j >> 4) * rows + row) * 16 + (j & 15)];
}

// rmax[i] = bits of the largest |entry| of row i (zeroed before): CTA (chunk of 128 rows, column
// block, shape); every kept entry below the diagonal block serves its row and, mirrored, its column.
__global__ void __launch_bounds__(128)
k_inv_rowmax(const InvShape *__restrict__ sh, const double *__restrict__ Wall, unsigned long long *__restrict__ rmax) {
    const InvShape S = sh[blockIdx.z];
    const int jc = blockIdx.y, i = blockIdx.x * 128 + threadIdx.x;
    if (jc * 16 >= S.m || (int)blockIdx.x * 128 + 127 < jc * 16 || (int)blockIdx.x * 128 >= S.m) return;
    const double *W = Wall + S.woff;
    const bool in = i < S.m && (i >> 4) >= jc;
    unsigned long long mine = 0;
    for (int c = 0; c < 16; c++) {
        const int j = jc * 16 + c;
        unsigned long long v = 0;
        if (in && j < S.m) {
            const size_t row = S.re2 ? 2 * (size_t)i : (size_t)i;
            v = abs_bits(W[((size_t)jc * S.rows + row) * 16 + c]);
            if (S.re2) v = max(v, abs_bits(W[((size_t)jc * S.rows + row + 1) * 16 + c]));
        }
        mine = max(mine, v);
        unsigned long long cv = (i >> 4) > jc ? v : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cv = max(cv, __shfl_xor_sync(0xffffffffu, cv, o));
        if ((threadIdx.x & 31) == 0 && cv) atomicMax(&rmax[S.roff + j], cv);
    }
    if (in) atomicMax(&rmax[S.roff + i], mine);
}

// The digits of E⁻¹: CTA (16 columns, 128 rows, shape), thread = row.  Operand layout per tile of
// 128 rows and chunk of 16 columns: DSL slices of 2 x 128 records of 8 BF16 (K-major, unswizzled).
__global__ void __launch_bounds__(128)
k_inv_slice(const InvShape *__restrict__ sh, const double *__restrict__ Wall,
            const unsigned long long *__restrict__ rmax, int *__restrict__ rexp, uint4 *__restrict__ A) {
    const InvShape S = sh[blockIdx.z];
    const int k = blockIdx.x, rt = blockIdx.y;
    if (k >= S.kseg || rt >= S.mt) return;
    const double *W = Wall + S.woff;
    const int i = rt * 128 + threadIdx.x;
    const unsigned long long mx = i < S.m ? rmax[S.roff + i] : 0;
    const int e = exp_of(mx);
    const bool ok = i < S.m && mx < INF_BITS;
    if (k == 0) rexp[S.soff + i] = mx < INF_BITS ? e : EXP_NAN;
    for (int part = 0; part <= S.re2; part++) {
        uint4 *dst = A + S.aoff / 16 + ((size_t)rt * S.kc + part * S.kseg + k) * (dense_abytes(false) / 16);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            long long q[8];
#pragma unroll
            for (int x = 0; x < 8; x++) {
                const int j = k * 16 + 8 * h + x;
                q[x] = ok && j < S.m ? fixed_point<55>(inv_entry(W, S.rows, S.re2, part, i, j), e) : 0;
            }
#pragma unroll
            for (int p = DSL - 1; p >= 0; p--) {
                int d[8];
#pragma unroll
                for (int x = 0; x < 8; x++) d[x] = p > 0 ? digit256(q[x]) : (int)q[x];
                dst[(p * 2 + h) * 128 + threadIdx.x] = make_uint4(bf16_pair(d[0], d[1]), bf16_pair(d[2], d[3]),
                                                                  bf16_pair(d[4], d[5]), bf16_pair(d[6], d[7]));
            }
        }
    }
}

// The same as bytes: DSL slices of 128 records of 16 signed bytes.  The leading digit
// of an entry at 0.996 of the row's power of two or above would be 128: such a row takes the next
// power (its entries then still have 54 bits below the largest, as a row just above a power has).
__global__ void __launch_bounds__(128)
k_inv_slice_bytes(const InvShape *__restrict__ sh, const double *__restrict__ Wall,
            const unsigned long long *__restrict__ rmax, int *__restrict__ rexp, uint4 *__restrict__ A) {
    const InvShape S = sh[blockIdx.z];
    const int k = blockIdx.x, rt = blockIdx.y;
    if (k >= S.kseg || rt >= S.mt) return;
    const double *W = Wall + S.woff;
    const int i = rt * 128 + threadIdx.x;
    const unsigned long long mx = i < S.m ? rmax[S.roff + i] : 0;
    const int e = exp_of(mx) + (((mx >> 44) & 0xff) >= 0xfd ? 1 : 0);
    const bool ok = i < S.m && mx < INF_BITS;
    if (k == 0) rexp[S.soff + i] = mx < INF_BITS ? e : EXP_NAN;
    for (int part = 0; part <= S.re2; part++) {
        uint4 *dst = A + S.aoff / 16 + ((size_t)rt * S.kc + part * S.kseg + k) * (dense_abytes(true) / 16);
        uint32_t w[DSL][4];
#pragma unroll
        for (int h = 0; h < 4; h++) {
            long long q[4];
#pragma unroll
            for (int x = 0; x < 4; x++) {
                const int j = k * 16 + 4 * h + x;
                q[x] = ok && j < S.m ? fixed_point<55>(inv_entry(W, S.rows, S.re2, part, i, j), e) : 0;
            }
#pragma unroll
            for (int p = DSL - 1; p >= 0; p--) {
                uint32_t v = 0;
#pragma unroll
                for (int x = 0; x < 4; x++) v |= (uint32_t)((p > 0 ? digit256(q[x]) : (int)q[x]) & 255) << (8 * x);
                w[p][h] = v;
            }
        }
#pragma unroll
        for (int p = 0; p < DSL; p++) dst[p * 128 + threadIdx.x] = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    }
}

// ------------------------------------------------------------------------------------------
// Small orders: E⁻¹ in FP64, column by column, and its product in one launch
// ------------------------------------------------------------------------------------------
// inv[off + c·ld + r] (or its complex entry): CTA (16 columns, 128 rows, shape), thread = row
__global__ void __launch_bounds__(128)
k_small_pack(const InvShape *__restrict__ sh, const SmallShape *__restrict__ ss, const double *__restrict__ Wall,
             double *__restrict__ inv) {
    const InvShape S = sh[blockIdx.z];
    const SmallShape Q = ss[blockIdx.z];
    const int i = blockIdx.y * 128 + threadIdx.x;
    if (i >= Q.ld) return;
    const double *W = Wall + S.woff;
    for (int c = 0; c < 16; c++) {
        const int j = blockIdx.x * 16 + c;
        if (j >= S.m) break;
        for (int part = 0; part <= S.re2; part++)
            inv[((Q.off + (long long)j * Q.ld + i) << S.re2) + part] = i < S.m ? inv_entry(W, S.rows, S.re2, part, i, j) : 0.0;
    }
}

// out = E⁻¹ in of a task's SM_R rows: lane = row x one of four columns, warps share the columns.
// Bound by the FP64 pipe (a warp instruction is 64 clocks of its scheduler): m² · 2 products a task
// (4 for complex E) over as many CTAs as there are blocks of rows; the matrix comes from L2, and the
// first entries are loaded before the wait for the kernel in front.  m = 64, 4
// tasks: 7 us by events around it where the banded sweeps take 13 and the three kernels of the
// digits 15; m = 576: 11 us (62, 16).  CTA task·nb + block of rows: in the grid's first dimension, as
// a batch may have more tasks than the others hold.
constexpr int SM_R = 8, SM_T = 256, SM_PRE = 4;
template <bool RE2>
__global__ void __launch_bounds__(SM_T)
k_small_solve(const Task *__restrict__ tasks, const SmallShape *__restrict__ ss, const double *__restrict__ inv,
              const double2 *__restrict__ in, double2 *__restrict__ out, const int *__restrict__ flag, int nb) {
    using A = typename std::conditional<RE2, double2, double>::type;
    extern __shared__ double2 xs[];
    __shared__ double red[2 * SM_R][SM_T / 32];
    const int t = blockIdx.x / nb, rb = blockIdx.x - t * nb, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Task T = tasks[t];
    const SmallShape S = ss[T.shape];
    const int r0 = rb * SM_R, c0 = warp * 4 + (lane >> 3);
    const bool mine = r0 < S.m;
    const A *M = reinterpret_cast<const A *>(inv) + S.off + r0 + (lane & 7);
    A pre[SM_PRE];
    if (mine)
#pragma unroll
        for (int q = 0; q < SM_PRE; q++)
            if (c0 + 32 * q < S.m) pre[q] = M[(long long)(c0 + 32 * q) * S.ld];
    CHAIN_ENTER();
    LAUNDER(in); LAUNDER(flag);
    if (!mine || (flag && !flag[t])) return;
    for (int i = tid; i < S.m; i += SM_T) xs[i] = in[T.coff + i];
    __syncthreads();
    double ax = 0.0, ay = 0.0;
    auto add = [&](A a, double2 x) {
        if constexpr (RE2) {
            ax = fma(a.x, x.x, fma(-a.y, x.y, ax));
            ay = fma(a.x, x.y, fma(a.y, x.x, ay));
        } else {
            ax = fma(a, x.x, ax);
            ay = fma(a, x.y, ay);
        }
    };
#pragma unroll
    for (int q = 0; q < SM_PRE; q++)
        if (c0 + 32 * q < S.m) add(pre[q], xs[c0 + 32 * q]);
#pragma unroll 4
    for (int c = c0 + 32 * SM_PRE; c < S.m; c += 32) add(M[(long long)c * S.ld], xs[c]);
    const bool im = (lane & 8) != 0;                      // one component each after the first exchange
    double v = (im ? ay : ax) + shfl_xor(im ? ax : ay, 8);
    v += shfl_xor(v, 16);
    if (lane < 16) red[lane][warp] = v;                   // lane = 8·component + row
    __syncthreads();
    if (tid < 16 * (SM_T / 32)) {
        const int k = tid >> 3;
        double s = red[k][tid & 7];
        s += shfl_xor(s, 4);
        s += shfl_xor(s, 2);
        s += shfl_xor(s, 1);
        const int r = r0 + (k & 7);
        if ((tid & 7) == 0 && r < S.m) reinterpret_cast<double *>(out + T.coff + r)[k >> 3] = s;
    }
}
void launch_small_solve(const Task *tasks, int ntask, const SmallShape *ss, int mmax, int re2, const double *inv,
                        const double2 *in, double2 *out, const int *flag, cudaStream_t s) {
    const int nb = (mmax + SM_R - 1) / SM_R;
    const dim3 grid((unsigned)nb * (unsigned)ntask);
    const size_t sm = (size_t)mmax * sizeof(double2);
    if (re2) launch_chained(k_small_solve<true>, grid, SM_T, sm, s, tasks, ss, inv, in, out, flag, nb);
    else launch_chained(k_small_solve<false>, grid, SM_T, sm, s, tasks, ss, inv, in, out, flag, nb);
}

// ------------------------------------------------------------------------------------------
// The solve
// ------------------------------------------------------------------------------------------

// Digits of the right-hand sides: CTA 1 + DSPLIT·task + share of its rows, the task's Re and Im columns of
// the shape's product, each scaled by its own power of two (real factors), or both by one
// (complex: columns [Re; -Im] and [Im; Re] against [Re E⁻¹ | Im E⁻¹]).  Layout per column tile and
// chunk of 16 rows: 2 x DS x nt records of 8 BF16.  cexp: the column's exponent (EXP_NAN for a
// column that is not finite, so that it stays visible).  Tasks not
// flagged are left as they are: their columns are computed from whatever is there and not written
// out.  Bound by latency (a column maximum, then one record per thread): four shares per task.
// CTA 0 instead forms the table of units that k_dense_mma splits its work by, from the flags: those come from
// the kernel in front of this one, whose results a kernel may read behind its own wait only, and
// k_dense_mma's wait is for this one.
constexpr int DSPLIT = 4;

// part[q] = {units, weight} of the shapes before q that have a flagged task, q = 0..ns; part[ns + 1].x:
// the CTAs that share them.  A unit weighs the bytes it streams, in KB, and a tile DENSE_TILEW units
// more (the sums of the tile before it leave TMEM meanwhile).
__device__ __forceinline__ void dense_units(int ns, const int4 *__restrict__ sunits, const int *__restrict__ tshape, int ntask,
                                            const int *flag, int grid, int2 *__restrict__ part) {
    __shared__ unsigned on[DENSE_MAXNS / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int q = tid; q < DENSE_MAXNS / 32; q += blockDim.x) on[q] = flag ? 0u : ~0u;
    __syncthreads();
    if (flag)
#pragma unroll 4
        for (int t = tid; t < ntask; t += blockDim.x) {
            const int q = tshape[t];
            if (flag[t]) atomicOr(&on[q >> 5], 1u << (q & 31));
        }
    __syncthreads();
    if (tid >= 32) return;
    int carry = 0, carryw = 0;
    for (int q0 = 0; q0 <= ns; q0 += 32) {
        const int q = q0 + lane;
        const int4 n = q < ns ? sunits[q] : make_int4(0, 0, 1, 0);      // tiles, chunks, weight of a unit
        const int has = q < ns && (on[q0 >> 5] >> lane & 1u), u = has ? n.x * n.y : 0, w = has ? n.x * (n.y + DENSE_TILEW) * n.z : 0;
        int s = u, z = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, s, o), x = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) { s += v; z += x; }
        }
        if (q <= ns) part[q] = make_int2(carry + s - u, carryw + z - w);
        carry += __shfl_sync(0xffffffffu, s, 31);
        carryw += __shfl_sync(0xffffffffu, z, 31);
    }
    if (lane == 0) part[ns + 1] = make_int2(min(grid, max(1, carry / DENSE_MINU)), 0);
}

template <int DS>
__global__ void __launch_bounds__(128)
k_dense_slice(const DenseTask *__restrict__ recs, const double2 *__restrict__ in, uint4 *__restrict__ B, int *__restrict__ cexp,
              const int *__restrict__ flag, int ns, const int4 *__restrict__ sunits, const int *__restrict__ tshape, int ntask,
              int grid, int2 *__restrict__ part) {
    const int tid = threadIdx.x;
    if (blockIdx.x == 0) {
        CHAIN_ENTER();
        LAUNDER(flag);
        dense_units(ns, sunits, tshape, ntask, flag, grid, part);
        return;
    }
    const int t = (blockIdx.x - 1) / DSPLIT, share = (blockIdx.x - 1) % DSPLIT;
    const DenseTask S = recs[t];
    CHAIN_ENTER();
    LAUNDER(in); LAUNDER(flag);
    if (flag && !flag[t]) return;
    const double2 *y = in + S.coff;
    __shared__ unsigned long long red[2][4];
    unsigned long long mx = 0, my = 0;
#pragma unroll 8
    for (int i = tid; i < S.m; i += 128) {
        const double2 v = y[i];
        mx = max(mx, abs_bits(v.x));
        my = max(my, abs_bits(v.y));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        my = max(my, __shfl_xor_sync(0xffffffffu, my, o));
    }
    if ((tid & 31) == 0) { red[0][tid >> 5] = mx; red[1][tid >> 5] = my; }
    __syncthreads();
    mx = max(max(red[0][0], red[0][1]), max(red[0][2], red[0][3]));
    my = max(max(red[1][0], red[1][1]), max(red[1][2], red[1][3]));
    if (S.re2) mx = my = max(mx, my);
    const int ex = exp_of(mx), ey = exp_of(my);
    const bool okx = mx < INF_BITS, oky = my < INF_BITS;
    if (tid == 0 && share == 0) {
        cexp[2 * t] = okx ? ex - 49 : EXP_NAN;
        cexp[2 * t + 1] = oky ? ey - 49 : EXP_NAN;
    }
    uint4 *Bt = B + S.b0;
    // items: records of 8 rows x {Re, Im}
    for (int it = share * 128 + tid; it < 4 * S.kseg; it += DSPLIT * 128) {
        const int o = it >> 1, im = it & 1;
        const bool ok = im ? oky : okx;
        const int e = im ? ey : ex;
        long long q[8];
#pragma unroll
        for (int x = 0; x < 8; x++) {
            const int i = 8 * o + x;
            const double v = i < S.m ? reinterpret_cast<const double *>(y + i)[im] : 0.0;
            q[x] = ok ? fixed_point<8 * DS - 1>(v, e) : 0;
        }
        uint4 *d0 = Bt + (size_t)(o >> 1) * (2 * DS * S.nt) + (size_t)(o & 1) * DS * S.nt;
        uint4 *d1 = d0 + (size_t)S.kseg * (2 * DS * S.nt);        // the imaginary half (complex)
#pragma unroll
        for (int p = DS - 1; p >= 0; p--) {
            int a[8];
#pragma unroll
            for (int x = 0; x < 8; x++) a[x] = p > 0 ? digit256(q[x]) : (int)q[x];
            const uint4 r = make_uint4(bf16_pair(a[0], a[1]), bf16_pair(a[2], a[3]), bf16_pair(a[4], a[5]), bf16_pair(a[6], a[7]));
            d0[p * S.nt + im] = r;
            if (S.re2)      // Re to the second column of the imaginary half, -Im to the first
                d1[p * S.nt + (im ^ 1)] = im ? make_uint4(r.x ^ 0x80008000u, r.y ^ 0x80008000u, r.z ^ 0x80008000u, r.w ^ 0x80008000u) : r;
        }
    }
}

// 32 lanes x 8 columns of TMEM, without the wait
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// Barrier 1 over the 256 epilogue threads; true if ok holds in all of them.
__device__ __forceinline__ bool epilogue_all(bool ok) {
    int r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %1, 0;\n"
        "barrier.cta.red.and.pred q, 1, 256, p;\n"
        "selp.b32 %0, 1, 0, q;\n"
        "}\n" : "=r"(r) : "r"((int)ok) : "memory");
    return r != 0;
}

// Four signed bytes to BF16: 128 + (b & 127) and 128 or 256 share their upper byte 0x43, and their
// difference is b, exactly.
__device__ __forceinline__ uint2 widen_digits(uint32_t b) {
    auto two = [](uint32_t w) {
        const uint32_t lo = w & 0xff7fff7fu, hi = w & 0xff80ff80u;
        const __nv_bfloat162 r = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&lo),
                                         *reinterpret_cast<const __nv_bfloat162 *>(&hi));
        return *reinterpret_cast<const uint32_t *>(&r);
    };
    return make_uint2(two(__byte_perm(b, 0x43434343u, 0x4140)), two(__byte_perm(b, 0x43434343u, 0x4342)));
}

// out = E⁻¹ in for the flagged tasks.  Persistent, one CTA per SM.  The work is the list of
// (tile of 128 rows, column tile, chunk of 16 operator columns) units of the shapes with a flagged
// task, cut into gridDim.x ranges of equal bytes: a CTA's range is a few tiles, the first and last of them
// shared with its neighbours.  One warp streams the operator's and the right-hand sides' digits
// through a ring of shared-memory stages with bulk copies, one warp issues the MMAs, eight warps
// put the DS sums together.  Byte digits (BY): three groups of four warps take the stages in turn and
// widen the operator's digits to BF16 in a second ring, a thread a row, 2 instructions a digit; half
// the bytes are read, and a stage holds two chunks (k=100, 16 columns a tile, with the kernels around
// it 33.9 -> 31.6 us; k=160 50.8 -> 45.0).  MMAs: the sums of weight s lie in TMEM columns
// s·nt.., the digits of
// the right-hand sides side by side in the operand, so operator digit p against digits 0..DS-1-p
// is one product of (DS - p)·nt columns into the columns from p·nt on (cut at 256, the widest
// MMA): the operator digit is read once for all of them.  The issuing loop is walked by a whole
// warp with one elected lane: from a single divergent lane the descriptors went through ordinary
// registers and an MMA took 228 clocks to issue, twice what a 240-column one runs (120).
// A tile that is not whole in one segment (a CTA's part of it, at most dense_seg() chunks) is added to
// 64-bit integers in L2 (atomics; the order does not matter) and written out by k_dense_finish.
// No CTA waits for another.
// Every mbarrier wait is bounded; on a timeout the CTA sets *err and leaves (1; 2 if work it had
// issued did not finish either, see kernels_cnn_tc.cu).
template <int DS, bool BY>
__global__ void __launch_bounds__(de_threads(BY), 1)
k_dense_mma(const DenseShape *__restrict__ sh, int ns, const int4 *__restrict__ sunits,
            const int *__restrict__ tlist, const long long *__restrict__ tcoff,
            const int *__restrict__ flag, const uint8_t *__restrict__ A, const int *__restrict__ rexp,
            const uint8_t *__restrict__ B, const int *__restrict__ cexp, double2 *__restrict__ out,
            unsigned long long *__restrict__ ws, const int2 *__restrict__ part, int ntmax, int nst, int kbs, int *__restrict__ err) {
    constexpr int T = de_threads(BY);
    const int kb = BY ? kbs : 1;
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ uint64_t full[DENSE_MAXST], empty[DENSE_MAXST], xfull[DENSE_NX], accf, acce, drain;
    __shared__ uint32_t tbase;
    __shared__ volatile int bad;
    __shared__ long long ccoff[2][40];               // per column pair of a segment: its task's output, -1: none,
    __shared__ int2 ccexp[2][40];                    // and its columns' exponents
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int2 *pre = reinterpret_cast<int2 *>(sm);                  // ns + 1 offsets {units, weight}
    uint8_t *wide = sm + (((size_t)(ns + 1) * 8 + 127) & ~(size_t)127);       // BF16 operator digits
    constexpr uint32_t AB = DS * (BY ? 2048u : 4096u), XB = DS * 4096u;       // operator bytes per chunk used, and widened
    const int nx = kb == 2 ? 2 : DENSE_NX;                        // (at most nst)
    uint8_t *ring = wide + (BY ? (size_t)nx * kb * XB : 0);
    const uint32_t stage = (uint32_t)kb * (AB + 2u * DS * 16u * (uint32_t)ntmax);
    if (warp == 0) umma::tmem_alloc(&tbase, 512);
    if (tid == 0) {
        for (int s = 0; s < nst; s++) { umma::mbar_init(&full[s], 1); umma::mbar_init(&empty[s], 1); }
        if (BY)
            for (int s = 0; s < nx; s++) umma::mbar_init(&xfull[s], 4);
        umma::mbar_init(&accf, 1);
        umma::mbar_init(&acce, 8);
        umma::mbar_init(&drain, 1);
        bad = 0;
    }
    // units and weight of the shapes with work (dense_units)
    CHAIN_ENTER();
    LAUNDER(part); LAUNDER(cexp); LAUNDER(flag);
    for (int q = tid; q <= ns; q += T) pre[q] = part[q];
    const long long G = part[ns + 1].x;
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t td = tbase;
    const int U = pre[ns].x;
    const long long Wt = pre[ns].y;
    // CTA b takes the units that start in [Wt·b/G, Wt·(b+1)/G) of the total weight
    auto shape_of = [&](int v, bool wt) {            // the last shape whose offset is at most v
        int lo = 0, hi = ns;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if ((wt ? pre[mid].y : pre[mid].x) <= v) lo = mid; else hi = mid;
        }
        return lo;
    };
    auto unit_from = [&](long long b) {
        const int p = (int)(Wt * b / G);
        if (p >= Wt) return U;
        const int q = shape_of(p, true);
        const int4 n = sunits[q];
        const int tw = (n.y + DENSE_TILEW) * n.z, r = p - pre[q].y, t = r / tw, k = r - t * tw - DENSE_TILEW * n.z;
        return pre[q].x + t * n.y + (k > 0 ? (k + n.z - 1) / n.z : 0);
    };
    const int ub = unit_from(blockIdx.x), ue = unit_from(blockIdx.x + 1);
    struct Seg { int q, rt, ct, k0, k1; };
    auto seg_at = [&](int u) {
        const int lo = shape_of(u, false);
        const int kc = sh[lo].kc, nct = sh[lo].nct;
        const int l = u - pre[lo].x, tile = l / kc;
        Seg g;
        g.q = lo; g.rt = tile / nct; g.ct = tile - g.rt * nct; g.k0 = l - tile * kc;
        int n = min(kc - g.k0, ue - u);
        const int cap = dense_seg(sh[lo].re2);
        if (n > cap) {                               // in equal parts, of whole stages
            const int parts = (n + cap - 1) / cap;
            n = ((n + parts - 1) / parts + kb - 1) / kb * kb;
        }
        g.k1 = g.k0 + n;
        return g;
    };
    auto wait = [&](uint64_t *b, uint32_t par) {
        if (umma::mbar_wait_ns(b, par, DE_LIMIT, &bad)) return true;
        bad = 1;
        return false;
    };
    int issued = 0;
    if (warp == 8) {
        if (lane == 0) {
            bool ok = true;
            int it = 0;
            for (int u = ub; ok && u < ue;) {
                const Seg g = seg_at(u);
                const DenseShape S = sh[g.q];
                const uint32_t bb = 2u * DS * 16u * (uint32_t)S.nt;
                const uint8_t *a = A + S.aoff + ((size_t)g.rt * S.kc + g.k0) * dense_abytes(BY);
                const uint8_t *b = B + S.boff + ((size_t)g.ct * S.kc + g.k0) * bb;
                for (int k = g.k0; k < g.k1; k += kb, it++) {
                    const int st = it % nst, use = it / nst, n = min(kb, g.k1 - k);
                    uint8_t *d = ring + (size_t)st * stage;
                    if (use > 0 && !(ok = wait(&empty[st], (use - 1) & 1))) break;
                    umma::mbar_expect_tx(&full[st], (uint32_t)n * (AB + bb));
                    for (int j = 0; j < n; j++) umma::bulk_g2s(d + j * AB, a + (size_t)j * dense_abytes(BY), AB, &full[st]);
                    umma::bulk_g2s(d + kb * AB, b, (uint32_t)n * bb, &full[st]);
                    issued++;
                    a += (size_t)n * dense_abytes(BY);
                    b += (size_t)n * bb;
                }
                u += g.k1 - g.k0;
            }
        }
    } else if (warp == 9) {
        // the whole warp walks the loop, so that addresses stay in uniform registers; one lane issues
        const bool leader = umma::elect_one();
        const uint32_t ring0 = umma::smem_u32(ring) >> 4, st16 = stage >> 4, wide0 = umma::smem_u32(wide) >> 4;
        const uint32_t ahi = (128u >> 4) | 0x4000u, alb = (2048u >> 4) << 16;
        bool ok = true;
        int seg = 0, st = 0, sx = 0;
        uint32_t par = 0, parx = 0;
        for (int u = ub; ok && u < ue; seg++) {
            const Seg g = seg_at(u);
            const uint32_t nt = (uint32_t)__shfl_sync(0xffffffffu, sh[g.q].nt, 0);
            const int nk = __shfl_sync(0xffffffffu, g.k1 - g.k0, 0);
            const uint32_t blb = (DS * nt) << 16;
            if (seg > 0 && !(ok = __all_sync(0xffffffffu, wait(&acce, (seg - 1) & 1)))) break;
            umma::fence_after_sync();
            for (int k = 0; k < nk; k += kb) {
                const int n = min(kb, nk - k);
                ok = __all_sync(0xffffffffu, BY ? wait(&xfull[sx], parx) : wait(&full[st], par));   // (widened: the stage had arrived)
                if (!ok) break;
                umma::fence_after_sync();
                if (leader) {
                    for (int j = 0; j < n; j++) {
                        const uint32_t r = ring0 + (uint32_t)st * st16;
                        const uint32_t al = alb | (BY ? wide0 + (uint32_t)(sx * kb + j) * (XB >> 4) : r + (uint32_t)j * (AB >> 4));
                        const uint32_t bl = blb | (r + (uint32_t)kb * (AB >> 4) + (uint32_t)j * (2u * DS) * nt);
#pragma unroll
                        for (uint32_t p = 0; p < DS; p++) {
                            const uint32_t cols = (DS - p) * nt, n0 = min(256u, cols), d = td + p * nt, acc = p > 0 || k + j > 0;
                            umma::mma_bf16_lohi(d, al + p * 256u, bl, ahi, umma::idesc_bf16_f32(128, (int)n0), acc);
                            if (cols > 256)
                                umma::mma_bf16_lohi(d + 256u, al + p * 256u, bl + 256u, ahi,
                                                    umma::idesc_bf16_f32(128, (int)(cols - 256u)), acc);
                        }
                    }
                    umma::commit(&empty[st]);
                }
                __syncwarp();
                if (++st == nst) { st = 0; par ^= 1u; }
                if (++sx == nx) { sx = 0; parx ^= 1u; }
            }
            if (ok && leader) umma::commit(&accf);
            __syncwarp();
            u += g.k1 - g.k0;
        }
    } else if (BY && warp >= 10) {
        const int row = ((warp - 10) & 3) * 32 + lane, grp = (warp - 10) >> 2;
        int it = 0;
        bool ok = true;
        for (int u = ub; ok && u < ue;) {
            const Seg g = seg_at(u);
            for (int k = g.k0; k < g.k1; k += kb, it++) {
                if (it % DE_G != grp) continue;
                const int st = it % nst, sx = it % nx, old = it - nx, n = min(kb, g.k1 - k);
                if (old >= 0) ok = wait(&empty[old % nst], (old / nst) & 1);       // its place in the second ring is free
                if (ok) ok = wait(&full[st], (it / nst) & 1);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                for (int j = 0; j < n; j++) {
                    const uint4 *s = reinterpret_cast<const uint4 *>(ring + (size_t)st * stage + (size_t)j * AB) + row;
                    uint4 *d = reinterpret_cast<uint4 *>(wide + (size_t)(sx * kb + j) * XB) + row;
                    uint4 v[DS];
#pragma unroll
                    for (int p = 0; p < DS; p++) v[p] = s[p * 128];
#pragma unroll
                    for (int p = 0; p < DS; p++) {
                        const uint2 a = widen_digits(v[p].x), b = widen_digits(v[p].y), c = widen_digits(v[p].z), e = widen_digits(v[p].w);
                        d[(2 * p) * 128] = make_uint4(a.x, a.y, b.x, b.y);
                        d[(2 * p + 1) * 128] = make_uint4(c.x, c.y, e.x, e.y);
                    }
                }
                umma::fence_async_smem();
                __syncwarp();
                if (lane == 0) umma::mbar_arrive(&xfull[sx]);
            }
            u += g.k1 - g.k0;
        }
    } else {
        int seg = 0;
        for (int u = ub; u < ue; seg++) {
            const Seg g = seg_at(u);
            const DenseShape S = sh[g.q];
            // what the columns' outputs need, ahead of the sums (a chain of loads per column otherwise)
            const int pair0 = g.ct * (S.nt / 2), npair = min(S.nt / 2, S.ntask - pair0);   // tasks of this column tile
            long long *co = ccoff[seg & 1];
            int2 *ce = ccexp[seg & 1];
            if (tid < S.nt / 2) {
                co[tid] = -1;
                if (tid < npair) {
                    const int t = tlist[S.t0 + pair0 + tid];
                    if (!flag || flag[t]) {
                        co[tid] = tcoff[t];
                        ce[tid] = make_int2(cexp[2 * t], cexp[2 * t + 1]);
                    }
                }
            }
            bool ok = true;
            if (lane == 0) ok = wait(&accf, seg & 1);
            if (!epilogue_all(ok)) break;                    // all eight warps leave, or none
            umma::fence_after_sync();
            const bool whole = g.k0 == 0 && g.k1 == S.kc;
            const int row = (warp & 3) * 32 + lane, i = g.rt * 128 + row;
            const int c0 = (warp >> 2) * (S.nt / 2), c1 = c0 + S.nt / 2;
            const int re = i < S.m ? rexp[S.soff + i] : 0;
            auto emit = [&](int c, long long vx, long long vy) {        // columns c, c + 1: one task
                const long long o = co[c / 2];
                if (i >= S.m || o < 0) return;
                const int2 e = ce[c / 2];
                out[o + i] = make_double2(from_fixed(vx, re + e.x), from_fixed(vy, re + e.y));
            };
            unsigned long long *acc = ws + S.acc0 + ((size_t)g.rt * S.nct + g.ct) * 128 * S.nt + row;
            for (int c = c0; c < c1; c += 8) {
                uint32_t v[DS][8];
#pragma unroll
                for (int s = 0; s < DS; s++)
                    tmem_ld8_nowait(td + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(s * S.nt + c), v[s]);
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                long long x[8];
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    // Σ a_s 2^(48-8s) in units of 2^13 (|Σ| < 2^63 up to 8192 operator columns).  The last
                    // two sums join in FP32, whose rounding of them is below the digits left out
                    // (conversions to integers are 16 a clock: one less of DS)
                    long long a[DS - 1];
#pragma unroll
                    for (int s = 0; s < DS - 2; s++) a[s] = __float2int_rn(__uint_as_float(v[s][e]));
                    const float lo = __uint_as_float(v[DS - 2][e]), ll = __uint_as_float(v[DS - 1][e]);
                    a[DS - 2] = __float2int_rn(DS == 6 ? fmaf(ll, 0x1p-5f, lo * 8.0f) : fmaf(ll, 0x1p-13f, lo * 0x1p-5f));
                    x[e] = (a[0] << 35) + (a[1] << 27) + (a[2] << 19) + (a[3] << 11) + a[DS - 2];
                    if (DS == 7) x[e] += a[4] << 3;
                }
                if (whole) {
#pragma unroll
                    for (int e = 0; e < 8; e += 2) emit(c + e, x[e], x[e + 1]);
                } else {
#pragma unroll
                    for (int e = 0; e < 8; e++) atomicAdd(acc + (size_t)(c + e) * 128, (unsigned long long)x[e]);
                }
            }
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&acce);
            u += g.k1 - g.k0;
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    if (bad) {
        bool drained = true;
        if (warp == 8 && lane == 0)                              // copies issued and not yet seen complete
            for (int st = 0; st < nst; st++) {
                const int n = issued / nst + (st < issued % nst ? 1 : 0);
                if (n > 0) drained &= umma::mbar_wait_ns(&full[st], (n - 1) & 1, DE_LIMIT, nullptr);
            }
        if (warp == 9) {
            if (umma::elect_one()) umma::commit(&drain);         // the lane that issued the MMAs
            __syncwarp();
            drained = umma::mbar_wait_ns(&drain, 0, DE_LIMIT, nullptr);
        }
        drained = __syncthreads_and(drained);
        if (tid == 0) atomicMax(err, drained ? 1 : 2);
    }
    umma::fence_after_sync();
    if (warp == 0) umma::tmem_dealloc(td, 512);
}

// The outputs of the tiles that were shared between CTAs, and their sums back to zero.  Item: 8
// column pairs of one tile; its shape's offsets and the number of CTAs come from k_dense_slice.  In
// the CTA that added a tile's last part this took 12 k clocks with the other SMs idle (6 us at
// k=200); over all SMs, launched ahead and waiting, about 2 us.
__global__ void __launch_bounds__(256)
k_dense_finish(const DenseShape *__restrict__ sh, int ns, const int4 *__restrict__ sunits, const int4 *__restrict__ items,
               int nitem, const int *__restrict__ tlist, const long long *__restrict__ tcoff, const int *__restrict__ flag,
               const int *__restrict__ rexp, const int *__restrict__ cexp, double2 *__restrict__ out,
               unsigned long long *__restrict__ ws, const int2 *__restrict__ part) {
    const int tid = threadIdx.x, row = tid & 127;
    bool waited = false;
    for (int b = blockIdx.x; b < nitem; b += gridDim.x) {
        // everything but the flags, sums and exponents is there before the products are done
        const int4 it = items[b];                                                // shape, tile (rt·nct + ct), first pair
        const DenseShape S = sh[it.x];
        const int4 n = sunits[it.x];
        const int rt = it.y / S.nct, ct = it.y - rt * S.nct, i = rt * 128 + row;
        const int re = i < S.m ? rexp[S.soff + i] : 0;
        int t[4];
        long long o[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int task = ct * (S.nt / 2) + it.z + (tid >> 7) + 2 * e;
            t[e] = task < S.ntask && i < S.m ? tlist[S.t0 + task] : -1;
            o[e] = t[e] >= 0 ? tcoff[t[e]] + i : 0;
        }
        if (!waited) {
            CHAIN_ENTER();
            LAUNDER(flag); LAUNDER(cexp); LAUNDER(part);
            waited = true;
        }
        unsigned long long *acc = ws + S.acc0 + (size_t)it.y * 128 * S.nt + row;
        unsigned long long x[8];
        int2 ce[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int pr = it.z + (tid >> 7) + 2 * e;
            x[2 * e] = __ldcg(acc + (size_t)(2 * pr) * 128);
            x[2 * e + 1] = __ldcg(acc + (size_t)(2 * pr + 1) * 128);
            ce[e] = t[e] >= 0 ? make_int2(cexp[2 * t[e]], cexp[2 * t[e] + 1]) : make_int2(0, 0);
            if (t[e] >= 0 && flag && !flag[t[e]]) t[e] = -1;
        }
        const int2 p0 = part[it.x], p1 = part[it.x + 1];
        const unsigned G = (unsigned)part[ns + 1].x, Wt = (unsigned)part[ns].y;
        if (p1.x == p0.x) continue;                                              // no task of this shape
        // the CTAs that hold the tile's first and last unit: one and the same wrote a tile of one segment out itself
        const unsigned long long w0 = (unsigned)(p0.y + it.y * (n.y + DENSE_TILEW) * n.z + DENSE_TILEW * n.z),
                                 w1 = w0 + (unsigned)((n.y - 1) * n.z);
        if (n.y <= dense_seg(S.re2) && ((w0 + 1) * G - 1) / Wt == ((w1 + 1) * G - 1) / Wt) continue;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int pr = it.z + (tid >> 7) + 2 * e;
            __stcg(acc + (size_t)(2 * pr) * 128, 0ull);
            __stcg(acc + (size_t)(2 * pr + 1) * 128, 0ull);
            if (t[e] < 0) continue;
            out[o[e]] = make_double2(from_fixed((long long)x[2 * e], re + ce[e].x), from_fixed((long long)x[2 * e + 1], re + ce[e].y));
        }
    }
    if (!waited) asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// ------------------------------------------------------------------------------------------
size_t inv_cols_smem(int maxK, int cw) { return ((size_t)2 * BNB * maxK + (size_t)cw * 16 + 256) * sizeof(double); }

cudaError_t launch_inv(const InvJob *jobs, int njobs, const InvShape *sh, int ns, int mmax, int ksegmax, int mtmax,
                       const BlockFactor *shapes, const double *Mall, const int *Pall, const int4 *Meta, double *W,
                       int maxK, int cw, int re2, unsigned long long *rmax, int *rexp, uint8_t *A, bool by,
                       const SmallShape *ss, double *inv, cudaStream_t s) {
    const size_t smem = inv_cols_smem(maxK, cw);
    const cudaError_t e = re2 ? allow_smem(k_inv_cols<true>) : allow_smem(k_inv_cols<false>);
    if (e != cudaSuccess) return e;
    if (re2) k_inv_cols<true><<<njobs, 256, smem, s>>>(jobs, shapes, Mall, Pall, Meta, W, maxK, cw);
    else k_inv_cols<false><<<njobs, 256, smem, s>>>(jobs, shapes, Mall, Pall, Meta, W, maxK, cw);
    if (ss) {
        k_small_pack<<<dim3(ksegmax, (mmax + 127 + SM_R) / 128, ns), 128, 0, s>>>(sh, ss, W, inv);
        return cudaGetLastError();
    }
    k_inv_rowmax<<<dim3((mmax + 127) / 128, (mmax + 15) / 16, ns), 128, 0, s>>>(sh, W, rmax);
    if (by) k_inv_slice_bytes<<<dim3(ksegmax, mtmax, ns), 128, 0, s>>>(sh, W, rmax, rexp, reinterpret_cast<uint4 *>(A));
    else k_inv_slice<<<dim3(ksegmax, mtmax, ns), 128, 0, s>>>(sh, W, rmax, rexp, reinterpret_cast<uint4 *>(A));
    return cudaGetLastError();
}

static size_t dense_smem(int ds, bool by, int ns, int ntmax, int kb, int nst) {
    return (((size_t)(ns + 1) * 8 + 127) & ~(size_t)127) +
           (size_t)kb * ((by ? (kb == 2 ? 2 : DENSE_NX) * (size_t)ds * 4096 : 0) +
                         (size_t)nst * ((size_t)ds * (by ? 2048 : 4096) + 2 * (size_t)ds * 16 * ntmax));
}
// Chunks per stage and stages.  A stage costs the issuing warp a wait and a commit, some 220 clocks
// each, and the widening warps their waits and a proxy fence, where a chunk of 16 columns is 315
// clocks of MMAs at nt = 16: two chunks a stage with byte digits where three such stages fit (up to 32
// columns a tile).  With BF16 digits two a stage gave 1 % there and lost 1 % at 80 columns: one.
void dense_stages(int ds, bool by, int ns, int ntmax, int &kb, int &nst) {
    for (kb = by ? 2 : 1;; kb--) {
        nst = by ? DENSE_MAXST : 7;
        while (nst > (by ? 3 : 2) && dense_smem(ds, by, ns, ntmax, kb, nst) > 223 * 1024) nst--;
        if (kb == 1 || dense_smem(ds, by, ns, ntmax, kb, nst) <= 223 * 1024) return;
    }
}
cudaError_t dense_set_smem() {
    cudaError_t e;
    if ((e = allow_smem(k_dense_mma<6, false>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_dense_mma<7, false>)) != cudaSuccess) return e;
    if ((e = allow_smem(k_dense_mma<6, true>)) != cudaSuccess) return e;
    return allow_smem(k_dense_mma<7, true>);
}
template <int DS>
static void dense_launch(const DensePlanArgs &p, const double2 *in, double2 *out, const int *flag, cudaStream_t s) {
    launch_chained(k_dense_slice<DS>, dim3(1 + p.ntask * DSPLIT), 128, 0, s, p.recs, in, reinterpret_cast<uint4 *>(p.B), p.cexp,
                   flag, p.ns, p.sunits, p.tshape, p.ntask, p.grid, p.part);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.grid);
    cfg.blockDim = dim3(de_threads(p.by));
    cfg.dynamicSmemBytes = dense_smem(DS, p.by, p.ns, p.ntmax, p.kb, p.nst);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    auto mma = p.by ? k_dense_mma<DS, true> : k_dense_mma<DS, false>;
    cudaLaunchKernelEx(&cfg, mma, p.sh, p.ns, p.sunits, p.tlist, p.tcoff, flag, p.A, p.rexp,
                       (const uint8_t *)p.B, (const int *)p.cexp, out, p.ws, (const int2 *)p.part, p.ntmax, p.nst, p.kb, p.err);
    cfg.gridDim = dim3(std::min(p.nitem, 2 * p.grid));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    cudaLaunchKernelEx(&cfg, k_dense_finish, p.sh, p.ns, p.sunits, p.items, p.nitem, p.tlist, p.tcoff, flag, p.rexp,
                       (const int *)p.cexp, out, p.ws, (const int2 *)p.part);
}
void launch_dense_solve(int ds, const DensePlanArgs &p, const double2 *in, double2 *out, const int *flag, cudaStream_t s) {
    if (ds == 6) dense_launch<6>(p, in, out, flag, s);
    else dense_launch<7>(p, in, out, flag, s);
}

}  // namespace hdd
