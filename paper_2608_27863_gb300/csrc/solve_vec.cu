// FP64 vector kernels for the trace-space Krylov solver.  Reductions use a
// fixed grid and a fixed combination order, so results are bitwise
// reproducible from run to run.
#include <algorithm>

#include "solve.cuh"

namespace hdg {

__global__ void k_dot_part(const double* x, const double* y, int64_t n, double* part) {
    __shared__ double red[32];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s = fma(x[i], y[i], s);
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// sum of part[0 .. nparts) by one warp: lane l adds parts l, l + 32, ... in
// order, then a fixed shuffle tree
__device__ __forceinline__ double warp_sum_parts(const double* part, int nparts) {
    const int lane = threadIdx.x & 31;
    double t = 0.0;
    for (int b = lane; b < nparts; b += 32) t += part[b];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
    return t;
}

__global__ void k_dot_final(const double* part, int nparts, double* out, int take_sqrt) {
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        const double t = warp_sum_parts(part, nparts);
        if (threadIdx.x == 0) *out = take_sqrt ? sqrt(t) : t;
    }
}

// The eight sums over a warp of acc[0..7]: lane l returns the sum of acc[l >> 2].  Lanes
// exchange halves of the set, so 9 additions replace the 40 of eight separate trees (an FP64
// addition of a warp takes 16 cycles of an SM here, and they were most of the dot kernel's time).
__device__ __forceinline__ double warp_sum8(const double (&acc)[8]) {
    const int lane = threadIdx.x & 31;
    double v4[4], v2[2], v;
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        v4[q] = (h16 ? acc[q + 4] : acc[q]) + __shfl_xor_sync(0xffffffffu, h16 ? acc[q] : acc[q + 4], 16);
#pragma unroll
    for (int q = 0; q < 2; ++q)
        v2[q] = (h8 ? v4[q + 2] : v4[q]) + __shfl_xor_sync(0xffffffffu, h8 ? v4[q] : v4[q + 2], 8);
    v = (h4 ? v2[1] : v2[0]) + __shfl_xor_sync(0xffffffffu, h4 ? v2[0] : v2[1], 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// Apply the previous rotations to column j of the Hessenberg matrix, form rotation j and rotate
// the right-hand side; R [m][m] upper triangle, cs / sn rotations, gv the rotated rhs.  Called by
// the whole block with col[0..j+1], c[0..j) and s[0..j) staged in shared memory.
__device__ void givens_column(double* col, const double* c, const double* s, int j, const Givens& G) {
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 0; i < j; ++i) {
            const double t = c[i] * col[i] + s[i] * col[i + 1];
            col[i + 1] = -s[i] * col[i] + c[i] * col[i + 1];
            col[i] = t;
        }
        const double h0 = col[j], h1 = col[j + 1], den = hypot(h0, h1);
        const double cj = den > 0.0 ? h0 / den : 1.0, sj = den > 0.0 ? h1 / den : 0.0;
        G.cs[j] = cj;
        G.sn[j] = sj;
        col[j] = den;
        const double g = G.gv[j];
        G.gv[j + 1] = -sj * g;
        G.gv[j] = cj * g;
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= j; i += blockDim.x) G.R[(size_t)i * G.m + j] = col[i];
}

// One pass of the classical Gram-Schmidt process of w against V_0 .. V_{k-1}:
//   MODE 0  out[j] = V_j . w
//   MODE 1  w -= sum_j coef[j] V_j, out[j] = V_j . w (the new w), add[j] += out[j]
//   MODE 2  w -= sum_j coef[j] V_j, *out = ||w||_2 (the new w), then the Givens step of column
//           k - 1 when G.R is given (hcol = G.col, *out its last entry)
// The last block to finish sums the blocks' partials in block order, so that no launch
// follows for the sums: an orthogonalisation with its norm and Givens step is three launches
// instead of nine, which is what sets the time of small systems (one SDIRK3 step on 64 quads,
// 1,536 unknowns, 480 GMRES iterations in a graph: 42.3 -> 26.1 ms, with the back substitution by a
// warp instead of a thread).  Large systems are bound by the FP64 pipe, 629e9 multiply-adds per second:
// k n of them in MODE 0 and 2, 2 k n in MODE 1 (2.7e5 unknowns, k ~ 78: 34 and 67 us; measured MODE 0
// 62, MODE 1 90, MODE 2 38 us).
// Tried for MODE 0: 256 threads with four rows in flight 69 us (MODE 1 116: too few loads in
// flight for its first part), no barrier between the groups 102 us (the warps drift over all k
// streams).  part: [k][gridDim.x]; ticket: zero between launches.
template <int MODE, int NTHR>
__global__ void __launch_bounds__(NTHR) k_orth(const double* __restrict__ V, int64_t ldv, int k, double* w, int64_t n,
                                               const double* coef, double* part, unsigned* ticket, double* out,
                                               double* add, Givens G) {
    constexpr int NW = NTHR / 32;
    extern __shared__ double wsum[];                    // [k][NW] the warps' sums (MODE 0, 1)
    __shared__ double cf[kMaxBasis];
    __shared__ double red[NW];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = gridDim.x;
    const int64_t i0 = (int64_t)blockIdx.x * NTHR + tid, step = (int64_t)nb * NTHR;
    double nrm = 0.0;
    if (MODE > 0) {
        for (int j = tid; j < k; j += NTHR) cf[j] = coef[j];
        __syncthreads();
        for (int64_t i = i0; i < n; i += step) {
            double s = w[i];
            int j = 0;
            for (; j + 8 <= k; j += 8) {
                double v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = V[(size_t)(j + q) * ldv + i];
#pragma unroll
                for (int q = 0; q < 8; ++q) s = fma(-cf[j + q], v[q], s);
            }
            for (; j < k; ++j) s = fma(-cf[j], V[(size_t)j * ldv + i], s);
            w[i] = s;
            if (MODE == 2) nrm = fma(s, s, nrm);
        }
    }
    if (MODE == 2) {
        for (int off = 16; off > 0; off >>= 1) nrm += __shfl_down_sync(0xffffffffu, nrm, off);
        if (lane == 0) red[warp] = nrm;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int q = 0; q < NW; ++q) t += red[q];
            part[blockIdx.x] = t;
        }
    } else {
        // steps of (eight vectors, RU rows per thread), the next step's values loaded before the current
        // ones are used; a barrier per group keeps the block's warps on the same eight streams
        constexpr int RU = NTHR > 128 ? 2 : 1;
        const int nst = (int)((n + step * RU - 1) / (step * RU)), total = ((k + 7) / 8) * nst;
        double cur[RU][8], cw[RU], acc[8];
        auto load = [&](int it, double (&v)[RU][8], double (&wv)[RU]) {
            const int j0 = 8 * (it / nst), st = it % nst;
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                const int64_t i = i0 + (int64_t)(st * RU + r) * step;
                const bool in = i < n;
                wv[r] = in ? w[i] : 0.0;                // written above by this thread
#pragma unroll
                for (int q = 0; q < 8; ++q) v[r][q] = in && j0 + q < k ? V[(size_t)(j0 + q) * ldv + i] : 0.0;
            }
        };
        load(0, cur, cw);
        for (int it = 0; it < total; ++it) {
            const int j0 = 8 * (it / nst), st = it % nst;
            double nxt[RU][8], nw[RU];
            if (it + 1 < total) load(it + 1, nxt, nw);
            if (st == 0) {
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] = 0.0;
            }
#pragma unroll
            for (int r = 0; r < RU; ++r)
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] = fma(cur[r][q], cw[r], acc[q]);
            if (st == nst - 1) {
                const double v = warp_sum8(acc);
                if ((lane & 3) == 0 && j0 + (lane >> 2) < k) wsum[(j0 + (lane >> 2)) * NW + warp] = v;
                if (NTHR > 128) __syncthreads();
            }
#pragma unroll
            for (int r = 0; r < RU; ++r) {
                cw[r] = nw[r];
#pragma unroll
                for (int q = 0; q < 8; ++q) cur[r][q] = nxt[r][q];
            }
        }
        __syncthreads();
        for (int j = tid; j < k; j += NTHR) {
            double t = 0.0;
#pragma unroll
            for (int q = 0; q < NW; ++q) t += wsum[j * NW + q];
            part[(size_t)j * nb + blockIdx.x] = t;
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(ticket, 1u) == (unsigned)nb - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) *ticket = 0u;
    if (MODE == 2) {
        if (warp == 0) {
            const double t = warp_sum_parts(part, nb);
            if (lane == 0) red[0] = sqrt(t);
        }
        __syncthreads();
        const double h = red[0];
        if (tid == 0) *out = h;
        if (G.R) {
            __shared__ double gc[kMaxBasis], gs[kMaxBasis];
            for (int i = tid; i < k; i += NTHR) cf[i] = G.col[i];
            for (int i = tid; i < k - 1; i += NTHR) { gc[i] = G.cs[i]; gs[i] = G.sn[i]; }
            if (tid == 0) cf[k] = h;
            givens_column(cf, gc, gs, k - 1, G);
        }
    } else {
        for (int j = warp; j < k; j += NW) {
            const double t = warp_sum_parts(part + (size_t)j * nb, nb);
            if (lane == 0) {
                out[j] = t;
                if (MODE == 1) add[j] += t;
            }
        }
    }
}

cudaError_t orthogonalise_init() {
    constexpr int sm = (int)sizeof(double) * kMaxBasis * 16;
    const cudaError_t e = cudaFuncSetAttribute(k_orth<0, 512>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k_orth<1, 512>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

void orthogonalise(cudaStream_t st, const double* V, int64_t n, int k, double* w, double* hcol, double* htmp,
                   double* part, unsigned* ticket, const Givens& G) {
    // One block per SM.  Narrow blocks, which leave no SM idle, up to two rows a thread; wide ones keep more loads in
    // flight from there on.  A GMRES iteration with bases up to 100, narrow / wide, in us: 2,400 unknowns 89 / 128,
    // 18,816 105 / 136, 24,576 122 / 140, 38,400 130 / 145, 48,600 149 / 153, 60,000 167 / 161, 101,400 230 / 198;
    // with bases up to 300 the sides meet between 38,400 (254 / 297) and 48,600 (315 / 306).
    const Givens none{};
    if (n <= 2 * (int64_t)kOrthBlocks * 128) {
        const unsigned nb = (unsigned)std::min<int64_t>(kOrthBlocks, (n + 127) / 128);
        const size_t sm = sizeof(double) * k * 4;
        k_orth<0, 128><<<nb, 128, sm, st>>>(V, n, k, w, n, nullptr, part, ticket, hcol, nullptr, none);
        k_orth<1, 128><<<nb, 128, sm, st>>>(V, n, k, w, n, hcol, part, ticket, htmp, hcol, none);
        k_orth<2, 128><<<nb, 128, 0, st>>>(V, n, k, w, n, htmp, part, ticket, hcol + k, nullptr, G);
    } else {
        const unsigned nb = (unsigned)std::min<int64_t>(kOrthBlocks, (n + 511) / 512);
        const size_t sm = sizeof(double) * k * 16;
        k_orth<0, 512><<<nb, 512, sm, st>>>(V, n, k, w, n, nullptr, part, ticket, hcol, nullptr, none);
        k_orth<1, 512><<<nb, 512, sm, st>>>(V, n, k, w, n, hcol, part, ticket, htmp, hcol, none);
        k_orth<2, 512><<<nb, 512, 0, st>>>(V, n, k, w, n, htmp, part, ticket, hcol + k, nullptr, G);
    }
}

__global__ void k_axpy_dev(const double* coef, double sign, const double* x, double* y, int64_t n) {
    const double a = sign * (*coef);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = fma(a, x[i], y[i]);
}

__global__ void k_scale_dev(const double* x, const double* div, double* y, int64_t n) {
    const double s = 1.0 / (*div);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = x[i] * s;
}

__global__ void k_axpby(double a, const double* x, double b, double* y, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = a * x[i] + b * y[i];
}

__global__ void k_combine(const double* V, int64_t ldv, const double* coef, int k, double* x, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double s = x[i];
        for (int j = 0; j < k; ++j) s = fma(coef[j], V[(size_t)j * ldv + i], s);
        x[i] = s;
    }
}

__global__ void k_sum_parts(const double* p1, int64_t n1, const double* p2, int64_t n2, double* out) {
    __shared__ double red[2][32];
    double a = 0.0, b = 0.0;
    for (int64_t i = threadIdx.x; i < n1; i += blockDim.x) a += p1[i];
    for (int64_t i = threadIdx.x; i < n2; i += blockDim.x) b += p2[i];
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
    }
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = a; red[1][threadIdx.x >> 5] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s1 = 0.0, s2 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { s1 += red[0][w]; s2 += red[1][w]; }
        out[0] = sqrt(s1 + s2);
        out[1] = sqrt(s1);
        out[2] = sqrt(s2);
    }
}

// y = x / div, or 0 when div is zero (lucky breakdown of the Arnoldi process)
__global__ void k_scale_safe(const double* x, const double* div, double* y, int64_t n) {
    const double d = *div;
    const double s = d != 0.0 ? 1.0 / d : 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = x[i] * s;
}

// y = R^{-1} gv (k x k upper triangle, zero diagonals skipped), one warp: the solved entry
// updates the entries above it, lanes over the rows
__global__ void k_backsolve(const double* R, const double* gv, int k, int m, double* y) {
    __shared__ double g[kMaxBasis];
    const int lane = threadIdx.x;
    for (int i = lane; i < k; i += 32) g[i] = gv[i];
    __syncwarp();
    for (int i = k - 1; i >= 0; --i) {
        const double d = R[(size_t)i * m + i];
        const double yi = d != 0.0 ? g[i] / d : 0.0;
        for (int l = lane; l < i; l += 32) g[l] -= R[(size_t)l * m + i] * yi;
        if (lane == 0) y[i] = yi;
        __syncwarp();
    }
}

__global__ void k_set_first(const double* beta, double* gv, int m) {
    for (int i = threadIdx.x; i <= m; i += blockDim.x) gv[i] = (i == 0) ? *beta : 0.0;
}

// append the residual norm to a device-side history
__global__ void k_hist_push(const double* norms, double* hist, int* counter, int cap) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        int k = *counter;
        if (k < cap) hist[k] = norms[0];
        *counter = k + 1;
    }
}

// z = a x + b y + c z
__global__ void k_lincomb3(double a, const double* x, double b, const double* y, double c, double* z, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        z[i] = a * x[i] + b * y[i] + c * z[i];
}

// Reduced-basis window: partial sums of the Gram matrix Z^T Z (pairs k <= l)
// and of Z^T g over row tiles; thread t of a block owns quantity t.
__global__ void k_rb_gram_part(const double* Z, int nb, const double* g, int64_t n, double* part) {
    constexpr int TR = 128;
    __shared__ double zs[kRbMax][TR];
    __shared__ double gs[TR];
    const int t = threadIdx.x;
    const int npair = nb * (nb + 1) / 2;
    int k = -1, l = -1;                     // quantity t: pair (k, l) with k <= l, or (k, g) when l == nb
    if (t < npair) {
        int r = t;
        k = 0;
        while (r >= nb - k) { r -= nb - k; ++k; }
        l = k + r;
    } else if (t < npair + nb) {
        k = t - npair;
        l = nb;
    }
    double acc = 0.0;
    for (int64_t r0 = (int64_t)blockIdx.x * TR; r0 < n; r0 += (int64_t)gridDim.x * TR) {
        __syncthreads();
        for (int idx = t; idx < (nb + 1) * TR; idx += blockDim.x) {
            const int c = idx / TR, i = idx - c * TR;
            const int64_t row = r0 + i;
            const double v = row < n ? (c < nb ? Z[(size_t)c * n + row] : g[row]) : 0.0;
            if (c < nb) zs[c][i] = v; else gs[i] = v;
        }
        __syncthreads();
        if (k >= 0) {
            const double* b = (l < nb) ? zs[l] : gs;
            for (int i = 0; i < TR; ++i) acc = fma(zs[k][i], b[i], acc);
        }
    }
    part[(size_t)blockIdx.x * blockDim.x + t] = acc;
}

// Sums the partials in block order, then solves the normal equations
// (Z^T Z) c = Z^T g by Cholesky with diagonal pivoting; pivots below
// 1e-13 of the largest diagonal are dropped (their coefficients are zero), so
// an empty or rank-deficient window gives a finite least-squares solution.
__global__ void k_rb_solve(const double* part, int nparts, int nb, double* c) {
    __shared__ double q[kRbMax * (kRbMax + 1) / 2 + kRbMax];
    const int t = threadIdx.x;
    const int nq = nb * (nb + 1) / 2 + nb;
    if (t < nq) {
        double s = 0.0;
        for (int b = 0; b < nparts; ++b) s += part[(size_t)b * blockDim.x + t];
        q[t] = s;
    }
    __syncthreads();
    if (t != 0) return;
    double G[kRbMax][kRbMax], rhs[kRbMax], y[kRbMax];
    int pidx[kRbMax];
    int idx = 0;
    for (int k = 0; k < nb; ++k)
        for (int l = k; l < nb; ++l) { G[k][l] = q[idx]; G[l][k] = q[idx]; ++idx; }
    for (int k = 0; k < nb; ++k) { rhs[k] = q[idx + k]; pidx[k] = k; c[k] = 0.0; }
    double dmax = 0.0;
    for (int k = 0; k < nb; ++k) dmax = fmax(dmax, G[k][k]);
    int r = 0;                               // accepted pivots
    for (; r < nb; ++r) {
        int best = r;
        for (int i = r + 1; i < nb; ++i)
            if (G[pidx[i]][pidx[i]] > G[pidx[best]][pidx[best]]) best = i;
        const int tmp = pidx[r]; pidx[r] = pidx[best]; pidx[best] = tmp;
        const int pr = pidx[r];
        const double d = G[pr][pr];
        if (!(d > 1e-13 * dmax)) break;
        const double ld = sqrt(d);
        G[pr][pr] = ld;
        for (int i = r + 1; i < nb; ++i) G[pidx[i]][pr] /= ld;     // column r of L, stored at (pidx[i], pr)
        for (int i = r + 1; i < nb; ++i)
            for (int j = r + 1; j <= i; ++j) {
                const double v = G[pidx[i]][pidx[j]] - G[pidx[i]][pr] * G[pidx[j]][pr];
                G[pidx[i]][pidx[j]] = v;
                G[pidx[j]][pidx[i]] = v;
            }
    }
    for (int i = 0; i < r; ++i) {            // L y = P rhs
        double s = rhs[pidx[i]];
        for (int j = 0; j < i; ++j) s -= G[pidx[i]][pidx[j]] * y[j];
        y[i] = s / G[pidx[i]][pidx[i]];
    }
    for (int i = r - 1; i >= 0; --i) {       // L^T x = y
        double s = y[i];
        for (int j = i + 1; j < r; ++j) s -= G[pidx[j]][pidx[i]] * y[j];
        y[i] = s / G[pidx[i]][pidx[i]];
    }
    for (int i = 0; i < r; ++i) c[pidx[i]] = y[i];
}

// insert (w, z) into slot head[0] of the window
__global__ void k_rb_store(const double* w, const double* z, double* W, double* Z, const int* head, int64_t n) {
    const int slot = head[0];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        W[(size_t)slot * n + i] = w[i];
        Z[(size_t)slot * n + i] = z[i];
    }
}

__global__ void k_rb_advance(int* head, int nb) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        head[0] = (head[0] + 1) % nb;
        head[1] = min(head[1] + 1, nb);
    }
}

__global__ void k_av_vertex(const double* __restrict__ fe, const int32_t* __restrict__ vrow,
                            const int32_t* __restrict__ vcol, double* __restrict__ fv, int64_t V) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    double s = 0.0;
    for (int32_t k = vrow[v]; k < vrow[v + 1]; ++k) s += fe[vcol[k]];
    const int32_t n = vrow[v + 1] - vrow[v];
    fv[v] = n > 0 ? s / n : 0.0;
}

__global__ void k_av_emean(const double* __restrict__ fv, const int32_t* __restrict__ ev, int nc,
                           double* __restrict__ fe, int64_t E) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    double s = 0.0;
    for (int c = 0; c < nc; ++c) s += fv[ev[e * nc + c]];
    fe[e] = s / nc;
}

__global__ void k_diag_sum(const double* __restrict__ part, int64_t E, double* __restrict__ out) {
    __shared__ double red[4][256];
    const int t = threadIdx.x;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t e = t; e < E; e += blockDim.x)
        for (int k = 0; k < 4; ++k) a[k] += part[e * 4 + k];
    for (int k = 0; k < 4; ++k) red[k][t] = a[k];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (t < w)
            for (int k = 0; k < 4; ++k) red[k][t] += red[k][t + w];
        __syncthreads();
    }
    if (t < 4) out[t] = red[t][0];
}

__global__ void k_to_f32(const double* x, float* y, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

}  // namespace hdg
