// Mixed-precision condensation.  The interior block At and both right-hand
// sides stay in FP64 and At is factored with partial pivoting in FP64; the
// blocks Bt, Ct, Dt and the condensed trace blocks are FP32.
//
// k_elim_mixed runs the bordered elimination of k_elim on the FP64 part and
// the two FP32 off-diagonal regions, but does not touch Dt: after the last
// panel the interior rows hold [U | Z = L^{-1} P Bt | z = L^{-1} P Rt] and the
// trace rows' multipliers W = Ct U^{-1}, so that the Schur complement is one
// product S^K = Dt - W Z (K = n_u) and -g^K = Rh - W z, left to k_schur_*.
// The default is the same in pieces: the FP64 LU of At alone (k_lu_small in
// shared memory, k_lu_mixed above n_u = 135), then Z and W by k_trsm in FP32.
#pragma once

#include "kernels.cuh"

namespace hdg {

// one (up to) 64 x 64 tile of A22 -= L21 U12 in type T; rows/cols >= r_end/c_end skipped
template <int NII, int NJJ, int NB, int TCW, class T, class RowP>
__device__ __forceinline__ void trail_tile_t(RowP rowp, const T* pan, const T* ust, int rb, int ct, int lrow0,
                                             int kb, int tx, int ty, int r_end, int c_end) {
    T acc[NII][NJJ];
    T* rp[NII];
#pragma unroll
    for (int ii = 0; ii < NII; ++ii) {
        int r = rb + ty + 16 * ii;
        rp[ii] = (r < r_end) ? rowp(r) : nullptr;
#pragma unroll
        for (int jj = 0; jj < NJJ; ++jj) {
            int c = ct + tx + 16 * jj;
            acc[ii][jj] = (rp[ii] && c < c_end) ? rp[ii][c] : T(0);
        }
    }
    for (int j = 0; j < kb; ++j) {
        T lv[NII], uv[NJJ];
#pragma unroll
        for (int ii = 0; ii < NII; ++ii) {
            int r = rb + ty + 16 * ii;
            lv[ii] = (r < r_end) ? pan[(size_t)(r - lrow0) * NB + j] : T(0);
        }
#pragma unroll
        for (int jj = 0; jj < NJJ; ++jj) uv[jj] = ust[j * TCW + tx + 16 * jj];
#pragma unroll
        for (int ii = 0; ii < NII; ++ii)
#pragma unroll
            for (int jj = 0; jj < NJJ; ++jj) acc[ii][jj] = fma(-lv[ii], uv[jj], acc[ii][jj]);
    }
#pragma unroll
    for (int ii = 0; ii < NII; ++ii) {
        if (!rp[ii]) continue;
#pragma unroll
        for (int jj = 0; jj < NJJ; ++jj) {
            int c = ct + tx + 16 * jj;
            if (c < c_end) rp[ii][c] = acc[ii][jj];
        }
    }
}

// trailing update of one storage region: rows [r_begin, r_end) (absolute bordered
// rows, rowp(r) gives the region row), columns [0, c_end) of the region with U12
// row j at urow(j)
template <class T, int NB, int NTH, class RowP, class URow>
__device__ void trailing_region(RowP rowp, URow urow, int r_begin, int r_end, int c_begin, int c_end,
                                const T* pan, int lrow0, int kb, T* ust) {
    constexpr int TCW = 64;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll 1
    for (int ct = c_begin; ct < c_end; ct += TCW) {
        for (int idx = tid; idx < kb * TCW; idx += NTH) {
            int j = idx / TCW, cc = idx - j * TCW;
            ust[j * TCW + cc] = (ct + cc < c_end) ? (T)urow(j)[ct + cc] : T(0);
        }
        __syncthreads();
        int njj = 0;
        while (njj < 4 && ct + 16 * njj < c_end) ++njj;
#pragma unroll 1
        for (int rb = r_begin; rb < r_end; rb += 64) {
            int nii = 0;
            while (nii < 4 && rb + 16 * nii < r_end) ++nii;
            switch (nii * 4 + njj - 5) {
#define HDG_TT(I, J) case (I) * 4 + (J) - 5: trail_tile_t<I, J, NB, TCW, T>(rowp, pan, ust, rb, ct, lrow0, kb, tx, ty, r_end, c_end); break;
                HDG_TT(1, 1) HDG_TT(1, 2) HDG_TT(1, 3) HDG_TT(1, 4)
                HDG_TT(2, 1) HDG_TT(2, 2) HDG_TT(2, 3) HDG_TT(2, 4)
                HDG_TT(3, 1) HDG_TT(3, 2) HDG_TT(3, 3) HDG_TT(3, 4)
                HDG_TT(4, 1) HDG_TT(4, 2) HDG_TT(4, 3) HDG_TT(4, 4)
#undef HDG_TT
                default: break;
            }
        }
        __syncthreads();
    }
}

template <class C, int NB>
constexpr int elim_mixed_smem_bytes() {
    return C::NU * NB * 8 + NB * 64 * 8 +                     // top panel (FP64), U12 staging (FP64)
           (C::NT * NB + C::NU * NB + NB * 64 + NB) * 4;      // bottom panel, top panel copy, staging, pivot row (FP32)
}

template <class C, int NB, int NTH, int MINB = 2>
__global__ void __launch_bounds__(NTH, MINB) k_elim_mixed(Regions<float> R, int64_t e0, int32_t* status) {
    constexpr int NU = C::NU, NT = C::NT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t el = blockIdx.x, e = e0 + el;
    double* A11 = R.a11 + e * R.a11_es;
    float* A12 = R.a12 + e * R.a12_es;
    float* A21 = R.a21 + el * R.a21_es;
    double* rt = R.rt + e * R.rt_es;
    const int64_t s11 = R.a11_rs, s12 = R.a12_rs, s21 = R.a21_rs, srt = R.rt_rs;
    extern __shared__ double sm[];
    double* pan = sm;                                        // [NU][NB]  rows of At (FP64), relative to k0
    double* ust64 = pan + NU * NB;                           // [NB][64]
    float* panb = reinterpret_cast<float*>(ust64 + NB * 64); // [NT][NB]  rows of Ct (FP32)
    float* pant = panb + NT * NB;                            // [NU][NB]  FP32 copy of pan
    float* ust32 = pant + NU * NB;                           // [NB][64]
    float* prow = ust32 + NB * 64;                           // [NB]      pivot row (FP32)
    __shared__ int piv[NB];
    __shared__ int sflag;
    __shared__ double s_inv;
    if (tid == 0) sflag = 0;

    for (int k0 = 0; k0 < NU; k0 += NB) {
        const int kb = min(NB, NU - k0), ntop = NU - k0;
#pragma unroll 1
        for (int idx = tid; idx < ntop * kb; idx += NTH) {
            int rr = idx / kb, c = idx - rr * kb;
            pan[rr * NB + c] = A11[(k0 + rr) * s11 + k0 + c];
        }
#pragma unroll 1
        for (int idx = tid; idx < NT * kb; idx += NTH) {
            int rr = idx / kb, c = idx - rr * kb;
            panb[rr * NB + c] = A21[rr * s21 + k0 + c];
        }
        __syncthreads();
        for (int j = 0; j < kb; ++j) {
            // warp 0 alone: pivot search (largest magnitude, lowest row on ties), row
            // interchange inside the panel and the FP32 pivot row; one barrier per step
            if (warp == 0) {
                int pr = warp_pivot(j, ntop, [&](int r) { return pan[r * NB + j]; });
                if (pr == INT_MAX) {
                    pr = j;
                    if (lane == 0) sflag |= 2;
                }
                if (lane < kb && pr != j) {
                    const double t = pan[j * NB + lane];
                    pan[j * NB + lane] = pan[pr * NB + lane];
                    pan[pr * NB + lane] = t;
                }
                __syncwarp();
                if (lane < kb) prow[lane] = (float)pan[j * NB + lane];
                __syncwarp();
                if (lane == 0) {
                    piv[j] = pr;
                    int fl = 0;
                    s_inv = pivot_reciprocal(pan[j * NB + j], fl);
                    if (fl) sflag |= fl;
                }
            }
            __syncthreads();
            const double inv = s_inv;
            const float invf = (float)inv;
#pragma unroll 1
            for (int rr = j + 1 + tid; rr < ntop; rr += NTH) {       // rows of At: FP64
                double l = pan[rr * NB + j] * inv;
                pan[rr * NB + j] = l;
                for (int c = j + 1; c < kb; ++c) pan[rr * NB + c] = fma(-l, pan[j * NB + c], pan[rr * NB + c]);
            }
#pragma unroll 1
            for (int rr = tid; rr < NT; rr += NTH) {                 // rows of Ct: FP32 multipliers
                float l = panb[rr * NB + j] * invf;
                panb[rr * NB + j] = l;
                for (int c = j + 1; c < kb; ++c) panb[rr * NB + c] = fmaf(-l, prow[c], panb[rr * NB + c]);
            }
            __syncthreads();
        }
#pragma unroll 1
        for (int idx = tid; idx < ntop * kb; idx += NTH) {
            int rr = idx / kb, c = idx - rr * kb;
            A11[(k0 + rr) * s11 + k0 + c] = pan[rr * NB + c];
            pant[rr * NB + c] = (float)pan[rr * NB + c];
        }
#pragma unroll 1
        for (int idx = tid; idx < NT * kb; idx += NTH) {
            int rr = idx / kb, c = idx - rr * kb;
            A21[rr * s21 + k0 + c] = panb[rr * NB + c];
        }
        __syncthreads();
        // interior rows of the trailing columns: swaps, then U12 = L11^{-1} A12
        const int c0 = k0 + kb;
        const int nd = NU - c0 + 1;                               // FP64 columns: At [c0, NU) and Rt
#pragma unroll 1
        for (int cc = tid; cc < nd + NT; cc += NTH) {
            if (cc < nd) {
                double* col = cc < nd - 1 ? A11 + c0 + cc : rt;
                const int64_t st = cc < nd - 1 ? s11 : srt;
                for (int j = 0; j < kb; ++j) {
                    int pr = piv[j];
                    if (pr != j) { double t = col[(k0 + j) * st]; col[(k0 + j) * st] = col[(k0 + pr) * st]; col[(k0 + pr) * st] = t; }
                }
                double xv[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    if (j < kb) {
                        double s = col[(k0 + j) * st];
#pragma unroll
                        for (int i = 0; i < NB; ++i)
                            if (i < j) s = fma(-pan[j * NB + i], xv[i], s);
                        xv[j] = s;
                        col[(k0 + j) * st] = s;
                    }
                }
            } else {
                float* col = A12 + (cc - nd);
                for (int j = 0; j < kb; ++j) {
                    int pr = piv[j];
                    if (pr != j) { float t = col[(k0 + j) * s12]; col[(k0 + j) * s12] = col[(k0 + pr) * s12]; col[(k0 + pr) * s12] = t; }
                }
                float xv[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    if (j < kb) {
                        float s = col[(k0 + j) * s12];
#pragma unroll
                        for (int i = 0; i < NB; ++i)
                            if (i < j) s = fmaf(-pant[j * NB + i], xv[i], s);
                        xv[j] = s;
                        col[(k0 + j) * s12] = s;
                    }
                }
            }
        }
        __syncthreads();
        // At (FP64): rows [c0, NU) x cols [c0, NU)
        trailing_region<double, NB, NTH>([&](int r) { return A11 + r * s11; },
                                         [&](int j) { return (const double*)(A11 + (k0 + j) * s11); },
                                         c0, NU, c0, NU, pan, k0, kb, ust64);
        // Ct multipliers (FP32): rows of Ct x cols [c0, NU)
        trailing_region<float, NB, NTH>([&](int r) { return A21 + r * s21; },
                                        [&](int j) { return (const double*)(A11 + (k0 + j) * s11); },
                                        0, NT, c0, NU, panb, 0, kb, ust32);
        // Bt (FP32): rows [c0, NU) x all t columns
        trailing_region<float, NB, NTH>([&](int r) { return A12 + r * s12; },
                                        [&](int j) { return (const float*)(A12 + (k0 + j) * s12); },
                                        c0, NU, 0, NT, pant, k0, kb, ust32);
        // Rt (FP64): rows [c0, NU)
#pragma unroll 1
        for (int r = c0 + tid; r < NU; r += NTH) {
            double s = rt[r * srt];
            for (int j = 0; j < kb; ++j) s = fma(-pan[(r - k0) * NB + j], rt[(k0 + j) * srt], s);
            rt[r * srt] = s;
        }
        __syncthreads();
    }
    if (tid == 0 && sflag) atomicOr(status, sflag);
}

// ----------------------------------------------------------------------------
// A3 + A4 of the mixed form, split by precision.  k_lu_mixed factors the
// interior block in FP64 alone, P At = L U with partial pivoting (blocked
// panels, pivot step in one warp, LAPACK-style full-row interchanges), and
// forms z = L^{-1} P Rt; it stores the interchanges.  The FP32 border then
// needs two triangular solves with many right-hand sides, each independent
// per column (or row) and run by its own kernels:
//   k_trsm<true>:   Z = L^{-1} P Bt   (columns of Bt)
//   k_trsm<false>:  W = Ct U^{-1}     (rows of Ct)
// 32 rows at a time: the solved rows' product, then the diagonal triangle.
// ----------------------------------------------------------------------------
template <class C, int NB>
constexpr int lu_mixed_smem_bytes() { return (C::NU * NB + NB * 64) * 8; }

// The interchange sequence sp (row i exchanged with sp[i], i ascending) as a gather map: row i of P B
// is row out[i] of B.  Whole CTA of NTH threads; sm: NU shared words.
template <int NU, int NTH>
__device__ __forceinline__ void interchanges_to_map(const int* sp, int* sm, int32_t* out) {
    for (int i = threadIdx.x; i < NU; i += NTH) sm[i] = i;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = 0; i < NU; ++i) {
            const int q = sp[i], t = sm[i];
            sm[i] = sm[q];
            sm[q] = t;
        }
    __syncthreads();
    for (int i = threadIdx.x; i < NU; i += NTH) out[i] = sm[i];
}

template <class C, int NB, int NTH>
__global__ void __launch_bounds__(NTH, 2) k_lu_mixed(Regions<float> R, int32_t* __restrict__ perm_out,
                                                     int64_t e0, int32_t* status) {
    constexpr int NU = C::NU;
    static_assert(NTH == 256, "trailing-update layout assumes 256 threads");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t e = e0 + blockIdx.x;
    double* A = R.a11 + e * R.a11_es;
    double* rt = R.rt + e * R.rt_es;
    const int64_t rs = R.a11_rs, srt = R.rt_rs;
    auto rowp = [&](int r) -> double* { return A + (size_t)r * rs; };
    extern __shared__ double sm[];
    double* pan = sm;                    // [NU][NB], row index relative to k0
    double* ust = pan + NU * NB;         // [NB][64]
    __shared__ int piv[NB], spiv[NU], sperm[NU];
    __shared__ int sflag;
    __shared__ double s_inv;
    if (tid == 0) sflag = 0;
    __syncthreads();
#pragma unroll 1
    for (int k0 = 0; k0 < NU; k0 += NB) {
        const int kb = min(NB, NU - k0), nrows = NU - k0;
#pragma unroll 1
        for (int idx = tid; idx < nrows * kb; idx += NTH) {
            const int rr = idx / kb, c = idx - rr * kb;
            pan[rr * NB + c] = rowp(k0 + rr)[k0 + c];
        }
        __syncthreads();
#pragma unroll 1
        for (int j = 0; j < kb; ++j) {
            if (warp == 0) {
                int pr = warp_pivot(j, nrows, [&](int r) { return pan[r * NB + j]; });
                if (pr == INT_MAX) {
                    pr = j;
                    if (lane == 0) sflag |= 2;
                }
                if (lane < kb && pr != j) {
                    const double t = pan[j * NB + lane];
                    pan[j * NB + lane] = pan[pr * NB + lane];
                    pan[pr * NB + lane] = t;
                }
                __syncwarp();
                if (lane == 0) {
                    piv[j] = pr;
                    int fl = 0;
                    s_inv = pivot_reciprocal(pan[j * NB + j], fl);
                    if (fl) sflag |= fl;
                }
            }
            __syncthreads();
            const double inv = s_inv;
#pragma unroll 1
            for (int rr = j + 1 + tid; rr < nrows; rr += NTH) {
                const double l = pan[rr * NB + j] * inv;
                pan[rr * NB + j] = l;
                for (int c = j + 1; c < kb; ++c) pan[rr * NB + c] = fma(-l, pan[j * NB + c], pan[rr * NB + c]);
            }
            __syncthreads();
        }
#pragma unroll 1
        for (int idx = tid; idx < nrows * kb; idx += NTH) {
            const int rr = idx / kb, c = idx - rr * kb;
            rowp(k0 + rr)[k0 + c] = pan[rr * NB + c];
        }
        // interchanges outside the panel (factor columns to the left, trailing columns
        // and the right-hand side), then U12 = L11^{-1} A12 and the same for Rt
        const int c0 = k0 + kb;
#pragma unroll 1
        for (int c = tid; c <= NU; c += NTH) {
            if (c >= k0 && c < c0) continue;
            double* col = c < NU ? A + c : rt;
            const int64_t st = c < NU ? rs : srt;
            for (int j = 0; j < kb; ++j) {
                const int pr = piv[j];
                if (pr != j) {
                    const double t = col[(k0 + j) * st];
                    col[(k0 + j) * st] = col[(k0 + pr) * st];
                    col[(k0 + pr) * st] = t;
                }
            }
            if (c >= c0) {
                double xv[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    if (j < kb) {
                        double s = col[(k0 + j) * st];
#pragma unroll
                        for (int i = 0; i < NB; ++i)
                            if (i < j) s = fma(-pan[j * NB + i], xv[i], s);
                        xv[j] = s;
                        col[(k0 + j) * st] = s;
                    }
                }
            }
        }
        if (tid < kb) spiv[k0 + tid] = k0 + piv[tid];
        __syncthreads();
        trailing_region<double, NB, NTH>(rowp, [&](int j) { return rowp(k0 + j); }, c0, NU, c0, NU, pan, k0, kb, ust);
        // right-hand side: rt[r] -= L21[r] . z1 for the rows below the panel
#pragma unroll 1
        for (int r = c0 + tid; r < NU; r += NTH) {
            double s = rt[r * srt];
            for (int j = 0; j < kb; ++j) s = fma(-pan[(r - k0) * NB + j], rt[(k0 + j) * srt], s);
            rt[r * srt] = s;
        }
        __syncthreads();
    }
    interchanges_to_map<NU, NTH>(spiv, sperm, perm_out + e * NU);
    if (tid == 0 && sflag) atomicOr(status, sflag);
}

// The same factorisation with the whole bordered block [At | Rt] in shared memory, for the sizes
// that fit (n_u <= 135: every element type but the degree-3 hexes), right-looking one column at
// a time.  FP64 multiply-adds take 16 cycles of an SM per warp here, so the shared-memory traffic of
// rank-1 updates is free and no panel is needed; what is left to hide is the pivot chain, and warp 0
// updates the next column first and searches its pivot while the other warps update the rest.  The
// trailing block is walked as one flat range, so that no lane idles at the rows' ends.  4,096 hexes
// p = 2: 10.05 -> 8.7 ms (2/3 n_u^3 at the FP64 pipe's rate: 5.4); 2,867 quads p = 3: 1.65 -> 0.62.
// Threads: a wider CTA shortens an element's chain of columns, a narrower one wastes fewer barrier
// waits when CTAs are many.  LU and triangular solves with 64 / 128 / 256 / 512 threads, in us, on 64
// elements and on many: n_u = 16 36 33 33 35 and 128 135 144 195 (2,916 quads); 36 92 73 67 68 and 424
// 406 413 500; 40 109 82 75 75 and 218 198 201 232 (729 hexes); 64 258 141 115 111 and 1337 1045 968
// 1045; 135 1901 790 506 459 and 7839 3392 2219 2021 (512 hexes).
template <class C>
struct LuShape {
    static constexpr int NU = C::NU;
    static constexpr int LDS = lu_row_stride(NU);        // odd, in doubles: columns without bank conflicts
    static constexpr int NTH = NU > 100 ? 512 : NU > 50 ? 256 : NU > 20 ? 128 : 64;
    static constexpr int smem_bytes = lu_smem_bytes(NU);
    static constexpr bool fits = lu_in_shared_memory(NU);
};

template <class C>
__global__ void __launch_bounds__(LuShape<C>::NTH) k_lu_small(Regions<float> R, int32_t* __restrict__ perm_out,
                                                              int64_t e0, int32_t* status) {
    using S = LuShape<C>;
    constexpr int NU = S::NU, LDS = S::LDS, NTH = S::NTH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t e = e0 + blockIdx.x;
    double* Ag = R.a11 + e * R.a11_es;
    double* rt = R.rt + e * R.rt_es;
    extern __shared__ double sm[];
    double* A = sm;                      // [NU][LDS], column NU the right-hand side
    double* lc = A + NU * LDS;           // [NU] multipliers of the current column
    __shared__ int s_p, sflag, spiv[NU], sperm[NU];
    __shared__ double s_inv;
    if (tid == 0) sflag = 0;
    for (int idx = tid; idx < NU * NU; idx += NTH) {
        const int r = idx / NU, c = idx - r * NU;
        A[r * LDS + c] = Ag[(int64_t)r * R.a11_rs + c];
    }
    for (int r = tid; r < NU; r += NTH) A[r * LDS + NU] = rt[r * R.rt_rs];
    // pivot of column k by warp 0: largest magnitude, lowest row on ties
    auto search = [&](int k) {
        int bi = warp_pivot(k, NU, [&](int r) { return A[r * LDS + k]; });
        if (lane == 0) {
            if (bi == INT_MAX) { bi = k; sflag |= 2; }
            s_p = bi;
            spiv[k] = bi;
        }
    };
    __syncthreads();
    if (warp == 0) search(0);
#pragma unroll 1
    for (int k = 0; k < NU; ++k) {
        __syncthreads();                                 // pivot known, the trailing block updated
        const int p = s_p;
        if (warp == 0) {
            if (lane == 0) {                             // now, while the FP64 pipe is free
                int fl = 0;
                s_inv = pivot_reciprocal(A[p * LDS + k], fl);
                if (fl) sflag |= fl;
            }
        } else if (p != k) {
            for (int c = tid - 32; c <= NU; c += NTH - 32)
                if (c != k) {
                    const double t = A[k * LDS + c];
                    A[k * LDS + c] = A[p * LDS + c];
                    A[p * LDS + c] = t;
                }
        }
        const double pv = A[p * LDS + k];
        __syncthreads();                                 // rows exchanged but for column k
        const double inv = s_inv;
        for (int r = k + 1 + tid; r < NU; r += NTH) lc[r] = A[(r == p ? k : r) * LDS + k] * inv;
        __syncthreads();                                 // row k and the multipliers in place
        if (warp == 0) {
            if (lane == 0) A[k * LDS + k] = pv;
            const double u = k + 1 < NU ? A[k * LDS + k + 1] : 0.0;
            for (int r = k + 1 + lane; r < NU; r += 32) {
                const double l = lc[r];
                A[r * LDS + k] = l;
                A[r * LDS + k + 1] = fma(-l, u, A[r * LDS + k + 1]);
            }
            __syncwarp();
            if (k + 1 < NU) search(k + 1);
        } else {
            // rows k + 1 .. NU - 1, columns k + 2 .. NU as one range
            const int w = NU - 1 - k, st = NTH - 32;
            if (w > 0) {
                const int dr = st / w, dc = st - dr * w;
                int r = (tid - 32) / w, c = (tid - 32) - r * w;
                for (int idx = tid - 32; idx < w * w; idx += st) {
                    double* a = A + (k + 1 + r) * LDS + k + 2 + c;
                    *a = fma(-lc[k + 1 + r], A[k * LDS + k + 2 + c], *a);
                    r += dr;
                    c += dc;
                    if (c >= w) { c -= w; ++r; }
                }
            }
        }
    }
    __syncthreads();
    for (int idx = tid; idx < NU * NU; idx += NTH) {
        const int r = idx / NU, c = idx - r * NU;
        Ag[(int64_t)r * R.a11_rs + c] = A[r * LDS + c];
    }
    for (int r = tid; r < NU; r += NTH) rt[r * R.rt_rs] = A[r * LDS + NU];
    interchanges_to_map<NU, NTH>(spiv, sperm, perm_out + e * NU);
    if (tid == 0 && sflag) atomicOr(status, sflag);
}

template <class C>
struct TrsmShape {
    static constexpr int CW = 64;                           // right-hand sides per CTA
    static constexpr int NTH = 256;
    static constexpr int NBLK = (C::NU + 31) / 32;
    static constexpr int JC = 64;                           // factor columns staged at a time (64 or 32)
    static constexpr int FS = 36;                           // row stride of the staged factor
    static constexpr int smem_floats = NBLK * 32 * CW + JC * FS;
};

// ZS: Z = L^{-1} P Bt for columns [c0, c0 + 64) of Bt; else W = Ct U^{-1} for rows [c0, c0 + 64) of
// Ct (FP32, in place; the factors FP64 in HBM).  X[i][c] holds the block of right-hand sides (W's
// transposed); 32 rows of X at a time: the solved rows' contribution as a product with the staged
// factor (a thread owns 4 rows x 4 columns of one half of the factor's columns: two 16-byte shared
// loads, one of them broadcast, feed sixteen multiply-adds; with 4 x 2 and no halves shared memory
// bound it), then the substitution with the diagonal triangle, four lanes per right-hand
// side with eight rows each, the solved value passed by a shuffle.  4,096 hexes p = 2: Z and W 5.6 ->
// 5.4 ms; 1,320 hexes p = 3: 23.0 -> 9.8 ms (the substitution ran on two warps, and every CTA walked the
// interchange list in global memory).  Inverted diagonal triangles are as fast but lose accuracy
// (error of the right-hand side 0.8e-6 -> 3.5e-6 on quads p = 3).
template <class C, bool ZS>
__global__ void __launch_bounds__(TrsmShape<C>::NTH) k_trsm(Regions<float> R, const int32_t* __restrict__ perm,
                                                            int64_t e0) {
    using S = TrsmShape<C>;
    constexpr int NU = C::NU, NT = C::NT, CW = S::CW, NTH = S::NTH, JC = S::JC, FS = S::FS, NUP = S::NBLK * 32;
    constexpr int NCT = (NT + CW - 1) / CW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t el = blockIdx.x / NCT, e = e0 + el;
    const int c0 = (int)(blockIdx.x % NCT) * CW, cw = min(CW, NT - c0);
    const double* A = R.a11 + e * R.a11_es;
    float* Y = ZS ? R.a12 + e * R.a12_es : R.a21 + el * R.a21_es;
    const int64_t rs = R.a11_rs, ys = ZS ? R.a12_rs : R.a21_rs;
    extern __shared__ __align__(16) float smf[];
    float* X = smf;                       // [NUP][CW]
    float* F = X + NUP * CW;              // [JC][FS] factor columns
    __shared__ float rd[32];              // reciprocal diagonal of U's block
    // the chunk at (i0, j0): F[j][r] = the factor's entry (row i0 + r of L, or column i0 + r of U; column or
    // row j0 + j), 64 or 32 columns left of the diagonal or the 32 of the diagonal block (j0 == i0)
    constexpr int NPRE = 32 * JC / NTH;
    float pre[NPRE];
    auto width = [&](int i0, int j0) { return j0 < i0 ? min(JC, i0 - j0) : 32; };
    auto load = [&](int i0, int j0) {
        const int jc = width(i0, j0), sh = jc == 64 ? 6 : 5;
#pragma unroll
        for (int u = 0; u < NPRE; ++u) {
            const int idx = tid + u * NTH;
            int r, j;
            if (ZS) { r = idx >> sh; j = idx & (jc - 1); } else { j = idx >> 5; r = idx & 31; }
            pre[u] = idx >= 32 * jc || i0 + r >= NU || j0 + j >= NU ? 0.f
                     : (float)(ZS ? A[(int64_t)(i0 + r) * rs + j0 + j] : A[(int64_t)(j0 + j) * rs + i0 + r]);
        }
    };
    load(0, 0);
    if (ZS) {
        for (int idx = tid; idx < NUP * CW; idx += NTH) {
            const int i = idx / CW, c = idx - i * CW;
            X[idx] = i < NU && c < cw ? Y[(int64_t)perm[e * NU + i] * ys + c0 + c] : 0.f;
        }
    } else {
        for (int idx = tid; idx < NUP * CW; idx += NTH) {
            const int c = idx / NUP, i = idx - c * NUP;
            X[i * CW + c] = i < NU && c < cw ? Y[(int64_t)(c0 + c) * ys + i] : 0.f;
        }
    }
    // rows prow.. + 3, columns pcol.. + 3; group 0 the first half of a chunk's factor columns, 1 the second
    const int group = warp >> 2, prow = 8 * (warp & 3) + 4 * (lane >> 4), pcol = 4 * (lane & 15);
    float acc[4][4] = {};
    auto apply = [&](int i0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float4* x = reinterpret_cast<float4*>(X + (i0 + prow + u) * CW + pcol);
            const float4 v = *x;
            *x = make_float4(v.x - acc[u][0], v.y - acc[u][1], v.z - acc[u][2], v.w - acc[u][3]);
            acc[u][0] = acc[u][1] = acc[u][2] = acc[u][3] = 0.f;
        }
    };
    int i0 = 0, j0 = 0;
#pragma unroll 1
    while (i0 < NUP) {
        const int jc = width(i0, j0), sh = jc == 64 ? 6 : 5;
        const bool diag = j0 == i0;
        __syncthreads();                  // X complete, F free
#pragma unroll
        for (int u = 0; u < NPRE; ++u) {
            const int idx = tid + u * NTH;
            if (idx >= 32 * jc) continue;
            int r, j;
            if (ZS) { r = idx >> sh; j = idx & (jc - 1); } else { j = idx >> 5; r = idx & 31; }
            F[j * FS + r] = pre[u];
        }
        if (diag) {
            if (!ZS && tid < 32) {
                const float d = i0 + tid < NU ? (float)A[(int64_t)(i0 + tid) * rs + i0 + tid] : 1.f;
                rd[tid] = d != 0.f ? 1.f / d : 1.f;
            }
            if (i0 > 0) {                 // the first block has no solved rows before it
                if (group == 0) apply(i0);
                __syncthreads();
                if (group == 1) apply(i0);
            }
        }
        __syncthreads();
        const int ni = diag ? i0 + 32 : i0, nj = diag ? 0 : j0 + jc;
        if (ni < NUP) load(ni, nj);       // the next chunk under this one's arithmetic
        if (!diag) {
            const int jb = group * (jc >> 1);
#pragma unroll 8
            for (int j = jb; j < jb + (jc >> 1); ++j) {
                const float4 x = *reinterpret_cast<const float4*>(X + (j0 + j) * CW + pcol);
                const float4 f = *reinterpret_cast<const float4*>(F + j * FS + prow);
                const float fu[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    acc[u][0] = fmaf(fu[u], x.x, acc[u][0]); acc[u][1] = fmaf(fu[u], x.y, acc[u][1]);
                    acc[u][2] = fmaf(fu[u], x.z, acc[u][2]); acc[u][3] = fmaf(fu[u], x.w, acc[u][3]);
                }
            }
        } else {
            const int c = tid >> 2, q = tid & 3;
            float* xc = X + (i0 + 8 * q) * CW + c;
            float x[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) x[m] = xc[m * CW];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                if (!ZS && q == (j >> 3)) x[j & 7] *= rd[j];
                const float xj = __shfl_sync(0xffffffffu, x[j & 7], (lane & ~3) | (j >> 3));
                const float4 f0 = *reinterpret_cast<const float4*>(F + j * FS + 8 * q);
                const float4 f1 = *reinterpret_cast<const float4*>(F + j * FS + 8 * q + 4);
                const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (8 * q + m > j) x[m] = fmaf(-f[m], xj, x[m]);
            }
#pragma unroll
            for (int m = 0; m < 8; ++m) xc[m * CW] = x[m];
        }
        i0 = ni;
        j0 = nj;
    }
    __syncthreads();
    if (ZS) {
        for (int idx = tid; idx < NU * CW; idx += NTH) {
            const int i = idx / CW, c = idx - i * CW;
            if (c < cw) Y[(int64_t)i * ys + c0 + c] = X[idx];
        }
    } else {
        for (int idx = tid; idx < NU * CW; idx += NTH) {
            const int c = idx / NU, i = idx - c * NU;
            if (c < cw) Y[(int64_t)(c0 + c) * ys + i] = X[i * CW + c];
        }
    }
}

// S^K = Dt - W Z (in place over Dt) and Rh <- Rh - W z, FP32 SIMT with FP32
// accumulation (W [t][n_u] = Ct region, Z [n_u][t] = Bt region)
template <class C, int NTH>
__global__ void __launch_bounds__(NTH) k_schur_simt(Regions<float> R, int64_t e0) {
    constexpr int NU = C::NU, NT = C::NT, KC = 32, TW = 64;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t el = blockIdx.x, e = e0 + el;
    const float* W = R.a21 + el * R.a21_es;
    const float* Z = R.a12 + e * R.a12_es;
    float* Dm = R.a22 + el * R.a22_es;
    const double* z = R.rt + e * R.rt_es;
    double* rb = R.rb + el * R.rb_es;
    const int64_t sw = R.a21_rs, sz = R.a12_rs, sd = R.a22_rs;
    __shared__ float Ws[TW][KC + 1];
    __shared__ float Zs[KC][TW];
    // right-hand side: rb -= W z (FP64 accumulation)
    for (int r = tid; r < NT; r += NTH) {
        double s = rb[r * R.rb_rs];
        for (int k = 0; k < NU; ++k) s -= (double)W[r * sw + k] * z[k * R.rt_rs];
        rb[r * R.rb_rs] = s;
    }
    for (int rt0 = 0; rt0 < NT; rt0 += TW)
        for (int ct0 = 0; ct0 < NT; ct0 += TW) {
            float acc[4][4];
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) acc[ii][jj] = 0.f;
            for (int k0 = 0; k0 < NU; k0 += KC) {
                for (int idx = tid; idx < TW * KC; idx += NTH) {
                    int r = idx / KC, k = idx - r * KC;
                    Ws[r][k] = (rt0 + r < NT && k0 + k < NU) ? W[(rt0 + r) * sw + k0 + k] : 0.f;
                    int k2 = idx / TW, c = idx - k2 * TW;
                    Zs[k2][c] = (k0 + k2 < NU && ct0 + c < NT) ? Z[(k0 + k2) * sz + ct0 + c] : 0.f;
                }
                __syncthreads();
#pragma unroll 8
                for (int k = 0; k < KC; ++k) {
                    float a[4], b[4];
#pragma unroll
                    for (int ii = 0; ii < 4; ++ii) a[ii] = Ws[ty + 16 * ii][k];
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) b[jj] = Zs[k][tx + 16 * jj];
#pragma unroll
                    for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) acc[ii][jj] = fmaf(a[ii], b[jj], acc[ii][jj]);
                }
                __syncthreads();
            }
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                int r = rt0 + ty + 16 * ii;
                if (r >= NT) continue;
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    int c = ct0 + tx + 16 * jj;
                    if (c < NT) Dm[r * sd + c] -= acc[ii][jj];
                }
            }
        }
}

// assembly from region views (S^K in Dt, -g^K in Rh) into BSR blocks of type TL
template <class C, class TL>
__global__ void k_assemble_r(Regions<TL> R, int64_t e0, const int32_t* blk, const int32_t* rank,
                             const int32_t* iperm, TL* vals, int pass) {
    constexpr int M = C::M, NF = C::NF, NFP = C::NFP, BS = C::BS;
    const int64_t bid = blockIdx.x;
    const int gl = (int)(bid % NF), fl = (int)((bid / NF) % NF);
    const int64_t el = bid / (NF * NF), e = e0 + el;
    const size_t item = ((size_t)e * NF + fl) * NF + gl;
    if (rank[item] != pass) return;
    TL* out = vals + (size_t)blk[item] * BS * BS;
    const TL* S = R.a22 + el * R.a22_es;
    const int32_t* ipf = iperm + ((size_t)e * NF + fl) * NFP;
    const int32_t* ipg = iperm + ((size_t)e * NF + gl) * NFP;
    for (int idx = threadIdx.x; idx < BS * BS; idx += blockDim.x) {
        int c = idx / BS, r = idx - c * BS;
        int a = r / NFP, k = r - a * NFP, b2 = c / NFP, k2 = c - b2 * NFP;
        int row = (fl * M + a) * NFP + ipf[k];
        int col = (gl * M + b2) * NFP + ipg[k2];
        out[idx] += S[(size_t)row * R.a22_rs + col];
    }
}

template <class C, class TL>
__global__ void k_assemble_g_r(Regions<TL> R, int64_t e0, const int32_t* e2f, const int32_t* frank,
                               const int32_t* iperm, double* g, int pass) {
    constexpr int M = C::M, NF = C::NF, NFP = C::NFP, BS = C::BS;
    const int64_t bid = blockIdx.x;
    const int fl = (int)(bid % NF);
    const int64_t el = bid / NF, e = e0 + el;
    if (frank[e * NF + fl] != pass) return;
    const int64_t F = e2f[e * NF + fl];
    const double* rb = R.rb + el * R.rb_es;
    const int32_t* ipf = iperm + ((size_t)e * NF + fl) * NFP;
    for (int idx = threadIdx.x; idx < BS; idx += blockDim.x) {
        int a = idx / NFP, k = idx - a * NFP;
        int row = (fl * M + a) * NFP + ipf[k];
        g[F * BS + idx] -= rb[row * R.rb_rs];
    }
}

// y = S x with blocks of type TL, FP64 vectors and accumulation
template <class C, class TL>
__global__ void __launch_bounds__(MvShape<C>::NTH) k_matvec_t(const int32_t* rowptr, const int32_t* col,
                                                              const TL* vals, const double* x, double* y) {
    constexpr int BS = C::BS, RB = MvShape<C>::RB, GROUPS = MvShape<C>::GROUPS;
    __shared__ double part[GROUPS][RB];
    const int64_t F = blockIdx.x;
    const int grp = threadIdx.x / RB, r = threadIdx.x - grp * RB;
    double acc0 = 0.0, acc1 = 0.0;
    if (r < BS) {
        for (int b = rowptr[F] + grp; b < rowptr[F + 1]; b += GROUPS) {
            const double* xs = x + (size_t)col[b] * BS;
            const TL* v = vals + (size_t)b * BS * BS + r;
            int c = 0;
#pragma unroll 4
            for (; c + 1 < BS; c += 2) {
                acc0 = fma((double)v[(size_t)c * BS], xs[c], acc0);
                acc1 = fma((double)v[(size_t)(c + 1) * BS], xs[c + 1], acc1);
            }
            if (c < BS) acc0 = fma((double)v[(size_t)c * BS], xs[c], acc0);
        }
    }
    part[grp][r] = acc0 + acc1;
    __syncthreads();
    if (grp == 0 && r < BS) {
        double s = part[0][r];
        for (int g2 = 1; g2 < GROUPS; ++g2) s += part[g2][r];
        y[F * BS + r] = s;
    }
}

// y = S x with FP32 blocks and an FP32 copy of x: products and the sum within
// each block in FP32, the sum over a row's blocks in FP64
__global__ void k_to_f32(const double* x, float* y, int64_t n);   // solve_vec.cu

template <class C>
__global__ void __launch_bounds__(MvShape<C>::NTH) k_matvec_f32(const int32_t* rowptr, const int32_t* col,
                                                                const float* vals, const float* x, double* y) {
    constexpr int BS = C::BS, RB = MvShape<C>::RB, GROUPS = MvShape<C>::GROUPS;
    __shared__ double part[GROUPS][RB];
    const int64_t F = blockIdx.x;
    const int grp = threadIdx.x / RB, r = threadIdx.x - grp * RB;
    double acc = 0.0;
    if (r < BS) {
        for (int b = rowptr[F] + grp; b < rowptr[F + 1]; b += GROUPS) {
            const float* xs = x + (size_t)col[b] * BS;
            const float* v = vals + (size_t)b * BS * BS + r;
            float a0 = 0.f, a1 = 0.f;
            int c = 0;
#pragma unroll 4
            for (; c + 1 < BS; c += 2) {
                a0 = fmaf(v[(size_t)c * BS], xs[c], a0);
                a1 = fmaf(v[(size_t)(c + 1) * BS], xs[c + 1], a1);
            }
            if (c < BS) a0 = fmaf(v[(size_t)c * BS], xs[c], a0);
            acc += (double)(a0 + a1);
        }
    }
    part[grp][r] = acc;
    __syncthreads();
    if (grp == 0 && r < BS) {
        double s = part[0][r];
        for (int g2 = 1; g2 < GROUPS; ++g2) s += part[g2][r];
        y[F * BS + r] = s;
    }
}

// recovery from region views: dU = -U^{-1}(z + Z dUhat), dQ = dq0 - L dU + Lambda dUhat.
// dUhat is rounded to Z's type once, not per row and column (a conversion is an FP64-pipe
// instruction): 4,096 hexes p = 2 1.96 -> 1.70 ms, 1,320 hexes p = 3 2.21 -> 1.88 ms.
template <class C, class TL, int NTH>
__global__ void __launch_bounds__(NTH) k_recover_r(Regions<TL> R, RecArgs A) {
    constexpr int D = C::D, M = C::M, NP = C::NP, NF = C::NF, NFP = C::NFP;
    constexpr int NU = C::NU, NQV = C::NQV, NT = C::NT;
    constexpr int GEO = Geo<D>::N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t e = blockIdx.x;
    __shared__ double duh[NT];
    __shared__ TL duhl[NT];
    __shared__ double w[NU];
    __shared__ double x[NU];
    __shared__ double geo[GEO];
    for (int i = tid; i < NT; i += NTH) {
        int f = i / (M * NFP), rem = i - f * M * NFP, a = rem / NFP, l = rem - a * NFP;
        int64_t F = A.e2f[e * NF + f];
        int k = A.perm[(e * NF + f) * NFP + l];
        duh[i] = A.dUH[(F * M + a) * NFP + k];
        duhl[i] = (TL)duh[i];
    }
    for (int i = tid; i < GEO; i += NTH) geo[i] = A.geo[e * GEO + i];
    __syncthreads();
    const double* U11 = R.a11 + e * R.a11_es;
    const TL* Z = R.a12 + e * R.a12_es;
    const double* z = R.rt + e * R.rt_es;
    // w = Z dUhat + z: each lane sums its products in the storage type (Z is FP32), the
    // lanes' partial sums are combined in FP64 (FP64 work would bound the kernel on GB300)
    for (int i = warp; i < NU; i += NTH / 32) {
        const TL* row = Z + (size_t)i * R.a12_rs;
        TL p = (TL)0;
        for (int c = lane; c < NT; c += 32) p = fma(row[c], duhl[c], p);
        double s = (double)p;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) w[i] = s + z[i * R.rt_rs];
    }
    __syncthreads();
    // x = U^{-1} w (FP64): 32-row diagonal blocks solved by warp 0 from registers, the
    // rows above updated with one dot product per row and thread
#pragma unroll 1
    for (int k1 = NU; k1 > 0; k1 -= 32) {
        const int k0 = max(0, k1 - 32), nb = k1 - k0;
        if (warp == 0) {
            double ur[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) ur[j] = (lane < nb && j < nb) ? U11[(size_t)(k0 + lane) * R.a11_rs + k0 + j] : 0.0;
            double v = lane < nb ? w[k0 + lane] : 0.0;
#pragma unroll
            for (int j = 31; j >= 0; --j) {
                if (j < nb) {
                    if (lane == j) v = v / ur[j];
                    const double xj = __shfl_sync(0xffffffffu, v, j);
                    if (lane < j) v = fma(-ur[j], xj, v);
                }
            }
            if (lane < nb) x[k0 + lane] = v;
        }
        __syncthreads();
#pragma unroll 1
        for (int r = tid; r < k0; r += NTH) {
            const double* row = U11 + (size_t)r * R.a11_rs + k0;
            double s = 0.0;
            for (int j = 0; j < nb; ++j) s = fma(row[j], x[k0 + j], s);
            w[r] -= s;
        }
        __syncthreads();
    }
    for (int i = tid; i < NU; i += NTH) A.dU[e * NU + i] = -x[i];
    const double detJ = geo[0];
    const double* Jinv = geo + 1;
    const double* NW = geo + 1 + D * D;
    const DeviceTables& T = A.tab;
    for (int idx = tid; idx < M * NP; idx += NTH) {
        int b = idx / NP, i = idx - b * NP;
        double t[D], ef[NF];
        for (int r = 0; r < D; ++r) {
            double s = 0.0;
            const double* mc = T.minv_c + ((size_t)r * NP + i) * NP;
            for (int j = 0; j < NP; ++j) s -= mc[j] * x[b * NP + j];
            t[r] = s;
        }
        for (int f = 0; f < NF; ++f) {
            double s = 0.0;
            const double* me = T.minv_e + ((size_t)f * NP + i) * NFP;
            for (int l = 0; l < NFP; ++l) s += me[l] * duh[(f * M + b) * NFP + l];
            ef[f] = s;
        }
        for (int l = 0; l < D; ++l) {
            double v = 0.0;
            for (int r = 0; r < D; ++r) v -= Jinv[r * D + l] * t[r];
            for (int f = 0; f < NF; ++f) v += NW[f * D + l] / detJ * ef[f];
            int o = (l * M + b) * NP + i;
            A.dQ[e * NQV + o] = A.dq0[e * NQV + o] + v;
        }
    }
}

}  // namespace hdg

namespace hdg {

template <class C, bool SPLIT3>
__global__ void k_schur_tc(Regions<float> R, int64_t e0, int32_t* status);
template <class C>
struct SchurTC;

inline Regions<float> mixed_regions(hdg_ctx* h) {
    const int64_t NU = h->NU, NT = h->NT;
    Regions<float> R;
    R.a11 = h->d_m11; R.a11_es = NU * NU; R.a11_rs = NU;
    const int64_t su = mixed_stride(NU), st = mixed_stride(NT);
    R.a12 = h->d_m12; R.a12_es = NU * st; R.a12_rs = st;
    R.a21 = h->d_m21; R.a21_es = NT * su; R.a21_rs = su;
    R.a22 = h->d_m22; R.a22_es = NT * st; R.a22_rs = st;
    R.rt = h->d_mrt;  R.rt_es = NU;       R.rt_rs = 1;
    R.rb = h->d_mrb;  R.rb_es = NT;       R.rb_rs = 1;
    return R;
}

template <int D, int P>
int run_linearize_mixed(hdg_ctx* h, const LinArgs& la) {
    using C = Cfg<D, P>;
    using CS = ContractShape<C, float>;
    constexpr int NB = 16;
    int rc;
    if ((rc = ensure_system_storage(h, HDG_PREC_MIXED))) return rc;
    const size_t sm_point = sizeof(double) * point_smem_doubles<C>();
    const size_t sm_elim = elim_mixed_smem_bytes<C, NB>();
    HDG_CK(cudaFuncSetAttribute(k_point<C, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_point));
    HDG_CK(cudaFuncSetAttribute(k_contract<C, float, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CS::smem_bytes));
    HDG_CK(cudaFuncSetAttribute(k_elim_mixed<C, NB, 256, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_elim));
    HDG_CK(cudaFuncSetAttribute(k_elim_mixed<C, NB, 256, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_elim));
    const int sm_lu = lu_mixed_smem_bytes<C, NB>();   // the 8-column variant needs less
    const int sm_trsm = (int)sizeof(float) * TrsmShape<C>::smem_floats;
    using LS = LuShape<C>;
    if constexpr (LS::fits) {
        HDG_CK(cudaFuncSetAttribute(k_lu_small<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, LS::smem_bytes));
    } else {
        HDG_CK(cudaFuncSetAttribute(k_lu_mixed<C, NB, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_lu));
        HDG_CK(cudaFuncSetAttribute(k_lu_mixed<C, 8, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_lu));
    }
    HDG_CK(cudaFuncSetAttribute(k_trsm<C, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_trsm));
    HDG_CK(cudaFuncSetAttribute(k_trsm<C, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_trsm));
    cudaStream_t st = h->stream;
    HDG_CK(cudaMemsetAsync(h->d_vals32, 0, sizeof(float) * h->nnzb * C::BS * C::BS, st));
    HDG_CK(cudaMemsetAsync(h->d_g, 0, sizeof(double) * h->F * C::BS, st));
    const Regions<float> RM = mixed_regions(h);
    PointArgs pa;
    pa.U = la.U; pa.Q = la.Q; pa.UH = la.UH; pa.Ustar = la.Ustar; pa.nu = la.nu;
    pa.dt = la.dt; pa.a_ii = la.a_ii; pa.ph = phys_t<double>(h->phys); pa.phf = phys_t<float>(h->phys);
    pa.tau = h->phys.tau; pa.tab = h->tab; pa.geo = h->d_geo;
    pa.e2f = h->d_e2f; pa.perm = h->d_perm;
    pa.rt = RM.rt; pa.rt_es = RM.rt_es; pa.rt_rs = RM.rt_rs;
    pa.rb = RM.rb; pa.rb_es = RM.rb_es; pa.rb_rs = RM.rb_rs;
    pa.vcoef = h->d_vcoef; pa.fcoef = h->d_fcoef; pa.dq0 = h->d_dq0;
    pa.ftag = h->d_ftag; pa.ub = h->d_ub; pa.ubf = h->d_ubf; pa.ew = h->e_wall;
    pa.tau_mode = h->phys.tau_mode; pa.taup = h->phys.tau_mode ? h->d_taup : nullptr;
    BlkArgs<float> ba;
    ba.vcoef = h->d_vcoef; ba.fcoef = h->d_fcoef; ba.geo = h->d_geo; ba.tab = h->tab; ba.ftag = h->d_ftag;
    ba.ew = h->e_wall;
    ba.taup = h->phys.tau_mode ? h->d_taup : nullptr;
    ba.R = RM; ba.dt = la.dt; ba.a_ii = la.a_ii; ba.tau = h->phys.tau; ba.has_nu = la.nu != nullptr;
    for (int64_t e0 = 0; e0 < h->E; e0 += h->chunk) {
        const int64_t ne = std::min<int64_t>(h->chunk, h->E - e0);
        pa.e0 = e0; ba.e0 = e0;
        prof_begin(h, HDG_K_POINT);
        k_point<C, float><<<(unsigned)ne, PointShape<C>::NTH, sm_point, st>>>(pa);
        prof_end(h);
        prof_begin(h, HDG_K_BLOCKS);
        k_contract<C, float, float><<<(unsigned)(ne * CS::NG), CS::NTH, CS::smem_bytes, st>>>(ba);
        prof_end(h);
        prof_begin(h, HDG_K_ELIM);
        if (h->elim_mixed_split) {
            // FP64 interior LU alone, then the FP32 border by two triangular solves
            using TS = TrsmShape<C>;
            constexpr int NCT = (C::NT + TS::CW - 1) / TS::CW;
            if constexpr (LS::fits)
                k_lu_small<C><<<(unsigned)ne, LS::NTH, LS::smem_bytes, st>>>(RM, h->d_mpiv, e0, h->d_status);
            else if (h->elim_nb == 8)   // interior LU panel width (the autotuner's elim_nb)
                k_lu_mixed<C, 8, 256><<<(unsigned)ne, 256, sm_lu, st>>>(RM, h->d_mpiv, e0, h->d_status);
            else
                k_lu_mixed<C, NB, 256><<<(unsigned)ne, 256, sm_lu, st>>>(RM, h->d_mpiv, e0, h->d_status);
            k_trsm<C, true><<<(unsigned)(ne * NCT), TS::NTH, sm_trsm, st>>>(RM, h->d_mpiv, e0);
            k_trsm<C, false><<<(unsigned)(ne * NCT), TS::NTH, sm_trsm, st>>>(RM, h->d_mpiv, e0);
        } else if (h->elim_mixed_minb == 3) {  // fused kernel, built for 3 or 2 resident CTAs per SM
            k_elim_mixed<C, NB, 256, 3><<<(unsigned)ne, 256, sm_elim, st>>>(RM, e0, h->d_status);
        } else {
            k_elim_mixed<C, NB, 256, 2><<<(unsigned)ne, 256, sm_elim, st>>>(RM, e0, h->d_status);
        }
        prof_end(h);
        prof_begin(h, HDG_K_SCHUR);
        if (h->schur_mode == 0) {
            k_schur_simt<C, 256><<<(unsigned)ne, 256, 0, st>>>(RM, e0);
        } else {
            using ST = SchurTC<C>;
            const unsigned grid = (unsigned)(ne * ST::NMT * ST::NNT);
            if (h->schur_mode == 1) {
                const int smb = ST::smem_bytes(false);
                HDG_CK(cudaFuncSetAttribute(k_schur_tc<C, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smb));
                k_schur_tc<C, false><<<grid, ST::THREADS, smb, st>>>(RM, e0, h->d_status);
            } else {
                const int smb = ST::smem_bytes(true);
                HDG_CK(cudaFuncSetAttribute(k_schur_tc<C, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smb));
                k_schur_tc<C, true><<<grid, ST::THREADS, smb, st>>>(RM, e0, h->d_status);
            }
        }
        prof_end(h);
        if (h->d_skout)
            k_copy_sk<float, float><<<(unsigned)ne, 256, 0, st>>>(RM.a22, RM.a22_es, RM.a22_rs, 0, C::NT, e0,
                                                                  static_cast<float*>(h->d_skout));
        for (int pass = 0; pass < 2; ++pass) {
            prof_begin(h, HDG_K_ASSEMBLE);
            k_assemble_r<C, float><<<(unsigned)(ne * C::NF * C::NF), 256, 0, st>>>(RM, e0, h->d_blk, h->d_rank,
                                                                                 h->d_iperm, h->d_vals32, pass);
            prof_end(h);
            prof_begin(h, HDG_K_ASSEMBLE);
            k_assemble_g_r<C, float><<<(unsigned)(ne * C::NF), 128, 0, st>>>(RM, e0, h->d_e2f, h->d_frank,
                                                                            h->d_iperm, h->d_g, pass);
            prof_end(h);
        }
        HDG_CK(cudaGetLastError());
    }
    h->have_system = true;
    h->sys_prec = HDG_PREC_MIXED;
    h->bj_ready = false;
    h->asm_ready = false;
    return HDG_OK;
}

template <int D, int P>
int run_matvec(hdg_ctx* h, const double* x, double* y) {
    using C = Cfg<D, P>;
    prof_begin(h, HDG_K_MATVEC);
    if (h->sys_prec == HDG_PREC_MIXED) {
        const int64_t n = h->F * C::BS;
        k_to_f32<<<(unsigned)std::min<int64_t>(1216, (n + 255) / 256), 256, 0, h->stream>>>(x, h->d_x32, n);
        k_matvec_f32<C><<<(unsigned)h->F, MvShape<C>::NTH, 0, h->stream>>>(h->d_rowptr, h->d_col, h->d_vals32,
                                                                          h->d_x32, y);
    } else
        k_matvec<C><<<(unsigned)h->F, MvShape<C>::NTH, 0, h->stream>>>(h->d_rowptr, h->d_col, h->d_vals, x, y);
    prof_end(h);
    HDG_CK(cudaGetLastError());
    return HDG_OK;
}

template <int D, int P>
int run_recover_mixed(hdg_ctx* h, const double* dUH, double* dQ, double* dU) {
    using C = Cfg<D, P>;
    RecArgs ra;
    ra.top = nullptr; ra.dq0 = h->d_dq0; ra.geo = h->d_geo; ra.tab = h->tab;
    ra.e2f = h->d_e2f; ra.perm = h->d_perm; ra.dUH = dUH; ra.dQ = dQ; ra.dU = dU;
    prof_begin(h, HDG_K_RECOVER);
    k_recover_r<C, float, 256><<<(unsigned)h->E, 256, 0, h->stream>>>(mixed_regions(h), ra);
    prof_end(h);
    HDG_CK(cudaGetLastError());
    return HDG_OK;
}

#define HDG_INSTANTIATE_MIXED(D, P)                                            \
    template int run_linearize_mixed<D, P>(hdg_ctx*, const LinArgs&);          \
    template int run_recover_mixed<D, P>(hdg_ctx*, const double*, double*, double*);

}  // namespace hdg

namespace hdg {

// ----------------------------------------------------------------------------
// Schur product on the 5th-generation tensor cores: S^K = Dt - W Z per element,
// tcgen05.mma kind::tf32 with FP32 accumulation in tensor memory.  W rows and Z
// columns are staged by the CTA's threads into shared memory in the canonical
// K-major layout without swizzle (8-row x 16-byte core matrices; K-adjacent
// cores 128 B apart, 8-row groups KC/4 x 128 B apart).  SPLIT3 selects 3xTF32:
// x = hi + lo with hi = tf32(x), lo = tf32(x - hi), and W Z ~ Wh Zh + Wh Zl + Wl Zh; the
// last two have an accumulator of their own, added at the end (the tensor cores' accumulation truncates,
// and a third of the additions into the large sum truncates a third as often).
// Waits on the
// MMA completion barrier are bounded; on timeout the CTA latches status bit 4,
// waits once more (bounded) and frees its tensor memory.
// ----------------------------------------------------------------------------
template <class C>
struct SchurTC {
    static constexpr int NT = C::NT, NU = C::NU;
    static constexpr int MT = 128, KC = 32;
    static constexpr int NNT = (NT + 127) / 128;                          // column tiles (<= 128 TMEM columns each)
    static constexpr int NTN = (((NT + NNT - 1) / NNT) + 15) / 16 * 16;   // columns per tile (mult. of 16)
    static constexpr int NMT = (NT + MT - 1) / MT;                        // row tiles
    static constexpr int TC1 = NTN <= 32 ? 32 : NTN <= 64 ? 64 : 128;     // columns of an accumulator
    __host__ __device__ static constexpr int tcols(bool split3) { return split3 ? 2 * TC1 : TC1; }
    static_assert(NTN <= 128, "column tile too wide");
    static constexpr int THREADS = 256;
    static constexpr int WRS = KC + 4;                                    // raw W row stride (floats)
    __host__ __device__ static constexpr int tile_floats(int rows) { return rows * KC; }
    __host__ __device__ static constexpr int raw_floats() { return MT * WRS + KC * NTN; }
    __host__ __device__ static constexpr int smem_bytes(bool split3) {
        return (split3 ? 2 : 1) * (tile_floats(MT) + tile_floats(NTN)) * 4 + raw_floats() * 4 + 64;
    }
    // right-hand side: a column tile takes RPC of the 128 rows, PARTS threads a row with KP terms of a chunk each
    static constexpr int RPC = (MT + NNT - 1) / NNT;
    static constexpr int PARTS = THREADS / RPC >= 8 ? 8 : THREADS / RPC >= 4 ? 4 : 2;
    static constexpr int KP = KC / PARTS;
    static constexpr int OS = NTN + 1;                                    // row stride of the staged product
    static_assert(RPC * PARTS <= THREADS && PARTS * KP == KC && KP % 4 == 0, "right-hand side layout");
    static_assert(MT * OS <= tile_floats(MT) + tile_floats(NTN) + raw_floats(),
                  "the product fits where the operands were");
    static_assert(RPC * PARTS * 8 <= MT * WRS * 4, "partial sums of the right-hand side fit the raw tile");
};

// 16 accumulator columns of this warp's 32 lanes; complete after tcgen05.wait::ld
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                   "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(addr));
}

// keeps the compiler from using the columns before the wait
__device__ __forceinline__ void tmem_arrived(float (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j) asm volatile("" : "+f"(v[j]));
}

// 16 bytes, of which src_bytes are read and the rest is zero; both addresses on 16 bytes
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"(smem_u32(dst)), "l"(src), "r"(src_bytes));
}

// One CTA (8 warps) per (element, 128-row tile, column tile).  The raw FP32 tiles of
// the next K chunk (W rows, Z rows) are copied into shared memory asynchronously
// (16-byte cp.async: the rows start on 16 bytes, see mixed_stride) while the tensor cores run the
// current chunk; the threads then split
// them into TF32 hi (/ lo) parts and store them in the core-matrix layout, rows
// fastest so that the 16-byte stores of a quarter warp are contiguous.  The right-hand side takes
// its W from the raw tile too, the rows dealt out over the column tiles.  The product leaves tensor
// memory through shared memory, so that Dt is read and written in whole lines.
// 4,096 hexes p = 2: 4.97 -> 2.59 ms, 1,320 hexes p = 3: 7.81 -> 2.61 ms (4-byte copies, W read again
// from global memory a row per thread for the right-hand side, Dt updated a row per thread).
template <class C, bool SPLIT3>
__global__ void __launch_bounds__(SchurTC<C>::THREADS) k_schur_tc(Regions<float> R, int64_t e0, int32_t* status) {
    using S = SchurTC<C>;
    constexpr int NT = S::NT, NU = S::NU, MT = S::MT, KC = S::KC, NTN = S::NTN, TH = S::THREADS, WRS = S::WRS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t bid = blockIdx.x;
    const int nt = (int)(bid % S::NNT), mt = (int)((bid / S::NNT) % S::NMT);
    const int64_t el = bid / (S::NNT * S::NMT), e = e0 + el;
    const int m0 = mt * MT, n0 = nt * NTN;
    const float* W = R.a21 + el * R.a21_es;
    const float* Z = R.a12 + e * R.a12_es;
    float* Dm = R.a22 + el * R.a22_es;
    const int64_t sw = R.a21_rs, sz = R.a12_rs, sd = R.a22_rs;
    extern __shared__ __align__(1024) unsigned char smraw[];
    float* Ah = reinterpret_cast<float*>(smraw);
    float* Bh = Ah + S::tile_floats(MT);
    float* Al = Bh + S::tile_floats(NTN);
    float* Bl = Al + S::tile_floats(MT);
    float* Wr = (SPLIT3 ? Bl + S::tile_floats(NTN) : Al);       // [MT][WRS] raw W of the next chunk
    float* Zr = Wr + MT * WRS;                                  // [KC][NTN] raw Z
    uint64_t* mbar = reinterpret_cast<uint64_t*>(smraw + S::smem_bytes(SPLIT3) - 64);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);

    auto prefetch = [&](int k0) {
        for (int it = tid; it < MT * (KC / 4); it += TH) {
            const int r = it / (KC / 4), k = (it - r * (KC / 4)) * 4;
            const int nb = m0 + r < NT ? 4 * max(0, min(4, NU - k0 - k)) : 0;
            cp_async16(Wr + r * WRS + k, nb ? (const void*)(W + (m0 + r) * sw + k0 + k) : (const void*)W, nb);
        }
        for (int it = tid; it < KC * (NTN / 4); it += TH) {
            const int k = it / (NTN / 4), n = (it - k * (NTN / 4)) * 4;
            const int nb = k0 + k < NU ? 4 * max(0, min(4, NT - n0 - n)) : 0;
            cp_async16(Zr + k * NTN + n, nb ? (const void*)(Z + (k0 + k) * sz + n0 + n) : (const void*)Z, nb);
        }
        asm volatile("cp.async.commit_group;");
    };
    prefetch(0);

    // right-hand side: Rh -= W z (FP64); this thread's row of the tile and part of every chunk
    const double* z = R.rt + e * R.rt_es;
    const int rpart = tid / S::RPC, rrow = nt * S::RPC + tid % S::RPC;
    const bool rhs = rpart < S::PARTS && rrow < MT && m0 + rrow < NT;
    double rsum = 0.0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(tslot)),
                     "r"(S::tcols(SPLIT3)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(mbar)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(NTN >> 3) << 17) | ((uint32_t)(MT >> 4) << 24);
    const uint32_t bar = smem_u32(mbar);
    uint32_t phase = 0;
    bool ok = true, pending = false;
    for (int k0 = 0; k0 < NU; k0 += KC) {
        asm volatile("cp.async.wait_group 0;");
        if (pending) {                                          // the previous batch still reads the tiles
            if (!mbar_wait_bounded(bar, phase, 1 << 24)) {
                ok = false;
                if (tid == 0) atomicOr(status, 4);
                mbar_wait_bounded(bar, phase, 1 << 24);
            }
            phase ^= 1;
            pending = false;
        }
        if (__syncthreads_or(ok ? 0 : 1)) {                     // raw tiles visible, operand tiles free
            ok = false;
            break;
        }
        if (rhs) {
            const int kb = rpart * S::KP;
#pragma unroll
            for (int k = 0; k < S::KP; k += 4) {
                const float4 v = *reinterpret_cast<const float4*>(Wr + rrow * WRS + kb + k);
                const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (k0 + kb + k + u < NU) rsum = fma((double)w[u], z[(k0 + kb + k + u) * R.rt_rs], rsum);
            }
        }
        // item = (row, 4-wide K group q) -> one 16-byte core-matrix row; rows fastest
        for (int it = tid; it < MT * (KC / 4); it += TH) {
            const int r = it % MT, q = it / MT;
            const float4 v = *reinterpret_cast<const float4*>(Wr + r * WRS + q * 4);
            const int off = ((r >> 3) * (KC / 4) + q) * 32 + (r & 7) * 4;    // floats
            float4 hi = make_float4(tf32_round(v.x), tf32_round(v.y), tf32_round(v.z), tf32_round(v.w));
            *reinterpret_cast<float4*>(Ah + off) = hi;
            if (SPLIT3)
                *reinterpret_cast<float4*>(Al + off) =
                    make_float4(tf32_round(v.x - hi.x), tf32_round(v.y - hi.y), tf32_round(v.z - hi.z), tf32_round(v.w - hi.w));
        }
        for (int it = tid; it < NTN * (KC / 4); it += TH) {
            const int n = it % NTN, q = it / NTN;
            const float4 v = make_float4(Zr[(q * 4 + 0) * NTN + n], Zr[(q * 4 + 1) * NTN + n], Zr[(q * 4 + 2) * NTN + n],
                                         Zr[(q * 4 + 3) * NTN + n]);
            const int off = ((n >> 3) * (KC / 4) + q) * 32 + (n & 7) * 4;
            float4 hi = make_float4(tf32_round(v.x), tf32_round(v.y), tf32_round(v.z), tf32_round(v.w));
            *reinterpret_cast<float4*>(Bh + off) = hi;
            if (SPLIT3)
                *reinterpret_cast<float4*>(Bl + off) =
                    make_float4(tf32_round(v.x - hi.x), tf32_round(v.y - hi.y), tf32_round(v.z - hi.z), tf32_round(v.w - hi.w));
        }
        asm volatile("fence.proxy.async.shared::cta;");
        __syncthreads();                                        // tiles staged, raw tiles consumed
        if (k0 + KC < NU) prefetch(k0 + KC);                    // next chunk under this chunk's MMAs
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int nsteps = (min(KC, NU - k0) + 7) / 8;
            for (int st = 0; st < nsteps; ++st) {
                const uint32_t off = st * 256;
                const uint64_t ah = umma_desc(smem_u32(Ah) + off, 128, (KC / 4) * 128);
                const uint64_t bh = umma_desc(smem_u32(Bh) + off, 128, (KC / 4) * 128);
                uint32_t acc = (k0 > 0 || st > 0) ? 1u : 0u;
                asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                             "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
                             :: "r"(tmem), "l"(ah), "l"(bh), "r"(idesc), "r"(acc));
                if (SPLIT3) {
                    const uint64_t al = umma_desc(smem_u32(Al) + off, 128, (KC / 4) * 128);
                    const uint64_t bl = umma_desc(smem_u32(Bl) + off, 128, (KC / 4) * 128);
                    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                                 "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
                                 :: "r"(tmem + S::TC1), "l"(ah), "l"(bl), "r"(idesc), "r"(acc));
                    asm volatile("tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, 1;"
                                 :: "r"(tmem + S::TC1), "l"(al), "l"(bh), "r"(idesc));
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bar));
        }
        pending = true;
    }
    asm volatile("cp.async.wait_group 0;");
    if (pending && ok) {
        if (!mbar_wait_bounded(bar, phase, 1 << 24)) {
            ok = false;
            if (tid == 0) atomicOr(status, 4);
            mbar_wait_bounded(bar, phase, 1 << 24);
        }
        phase ^= 1;
    }
    ok = !__syncthreads_or(ok ? 0 : 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok) {
        // the parts of a row of the right-hand side, in order
        double* rp = reinterpret_cast<double*>(Wr);
        if (rhs) rp[rpart * S::RPC + tid % S::RPC] = rsum;
        __syncthreads();
        if (rhs && rpart == 0) {
            double s = R.rb[el * R.rb_es + (m0 + rrow) * R.rb_rs];
            for (int q = 0; q < S::PARTS; ++q) s -= rp[q * S::RPC + tid];
            R.rb[el * R.rb_es + (m0 + rrow) * R.rb_rs] = s;
        }
        __syncthreads();
        // the product into shared memory: warp w reads lanes 32 (w % 4) .. + 31 and the column half w / 4 of the tile
        float* O = reinterpret_cast<float*>(smraw);
        const int lg = warp & 3, half = warp >> 2;
        const int r = lg * 32 + lane;
        constexpr int HC = ((NTN / 2) + 15) / 16 * 16;          // columns per half, in chunks of 16
#pragma unroll 1
        for (int c0 = half * HC; c0 < min(NTN, (half + 1) * HC); c0 += 16) {
            float v[16], x[16];
            const uint32_t addr = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)c0;
            tmem_ld16(addr, v);
            if (SPLIT3) tmem_ld16(addr + S::TC1, x);
            asm volatile("tcgen05.wait::ld.sync.aligned;");
            tmem_arrived(v);
            if (SPLIT3) tmem_arrived(x);
#pragma unroll
            for (int j = 0; j < 16; ++j) O[r * S::OS + c0 + j] = SPLIT3 ? v[j] + x[j] : v[j];
        }
        __syncthreads();
        // Dt -= product, a warp a row, two rows' loads in flight
        constexpr int NL = (NTN + 31) / 32;
        const int nr = min(MT, NT - m0), nc = min(NTN, NT - n0);
        for (int r0 = warp; r0 < nr; r0 += 2 * (TH / 32)) {
            float d[2][NL];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int j = 0; j < NL; ++j) {
                    const int rr = r0 + u * (TH / 32), c = lane + 32 * j;
                    d[u][j] = rr < nr && c < nc ? Dm[(m0 + rr) * sd + n0 + c] : 0.f;
                }
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int j = 0; j < NL; ++j) {
                    const int rr = r0 + u * (TH / 32), c = lane + 32 * j;
                    if (rr < nr && c < nc) Dm[(m0 + rr) * sd + n0 + c] = d[u][j] - O[rr * S::OS + c];
                }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(S::tcols(SPLIT3)));
}


}  // namespace hdg
