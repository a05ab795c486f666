// A2 on quads and hexes: contraction of the point coefficients with the basis
// tables into the element blocks.
//
// For a component pair (a, b) the element rows are
//   C[i][c] = sum_g A_0[g][i] phi_c(g) - sum_r sum_g A_r[g][i] psi_r,c(g) (+ theta_f,c(g) on trace columns),
//   A_k[g][i] = sum_r' dphi_r'[g][i] o_r',k[g],
// with psi_r = phi (M^{-1} C_r) and theta_f = phi (M^{-1} E_f) the q variations of unit U and Uhat columns
// along reference direction r (affine elements: N_f / |J| = +-grad xi_r(f), so the faces need no
// coefficients of their own).  phi_c, psi_r,c and theta_f,c are all products of 1-D functions that differ
// from the basis on axis r only, so each sum runs one axis at a time with p + 3 functions on axis r
// (the p + 1 columns of 1-D M^{-1} C times the basis, and the lifts of the two end points).  A thread
// streams the points of one (pair, i): (p+2)^d terms of A_k, then per axis the partial sums in
// registers.  The face rows are the same with the trace basis as rows over the face's points; of the
// element's columns only those that meet the face couple (on the other axes everything is a product).
// Pairs without a viscous part (a = 0 without artificial viscosity, and dF_momentum / dE) stop at A_0.
//
// Multiply-adds per hex p = 2 element: 2.3e6, where applying one side of the sum factorisation to every
// column and the dense face products took 5.9e6.  One warp (two for p = 3) per CTA and 1..8 pairs; the
// rows are collected in shared memory and leave in whole lines.  512 hexes p = 2, FP64: 7.27 -> 3.17 ms
// (1.9 at the FP64 pipe's rate, which is 74 % active); 693 hexes p = 1 1.81 -> 0.63 ms; mixed form, 4,096
// hexes p = 2: 10.1 -> 5.3 ms (3xTF32 tensor-core tiles before, bound by forming their operands), 1,320 hexes
// p = 3: 10.9 -> 8.1 ms, of which the interior block's sums in FP64 take 0.1 to 0.2.  The row factors come
// from the 3-D tables: with products of 1-D ones the FP32 form is 10 % faster but its blocks at p = 3 lose a
// fifth of their accuracy.
#pragma once

namespace hdg {

template <class TL>
struct BlkArgs {
    const void* vcoef; const void* fcoef;   // Jacobian coefficients in the accumulation type
    const int32_t* ftag;                    // [E][nf] or NULL
    const double* geo;
    DeviceTables tab;
    Regions<TL> R;
    double dt, a_ii, tau;
    double ew;                              // wall internal energy of tag-3 faces
    const double* taup;                     // [chunk][nf][Nfq] per-point tau (state-dependent), or NULL
    int has_nu;                             // artificial viscosity: (0, 0) has a viscous part too
    int64_t e0;
};

template <class C, class TA>
struct ContractShape {
    static constexpr int NP = C::NP, N1 = C::P + 1, Q1 = C::P + 2, D = C::D, M = C::M;
    static constexpr int NCB = C::NP + C::NF * C::NFP;            // columns of one component
    static constexpr int PPC = NP >= 27 ? 1 : 32 / NP;            // pairs per CTA
    static constexpr int NTH = (PPC * NP + 31) / 32 * 32;
    static constexpr int NG = (M * M + PPC - 1) / PPC;            // CTAs per element
    static constexpr int NVIS = D * (D + 1) + M;                  // pairs with a viscous part
    static constexpr int NK = 1 + D;
    static constexpr int CV = D * NK * C::NQ, CF = C::NF * NK * C::NFQ;   // coefficients of a pair
    static constexpr int FPR = (NP / C::NFP) < C::NF ? (NP / C::NFP) : C::NF;   // faces of a round of face rows
    static constexpr int BS = NP | 1;                             // stride of the collected rows, [column][row]
    static constexpr int smem_words = PPC * (CV + CF + NCB * BS) + Q1 * N1 + Q1 * (N1 + 2) + N1 * N1 + 2 * N1;
    static constexpr size_t smem_bytes = smem_words * sizeof(TA) + (C::NFP * C::NFP) * sizeof(TA);
};

// component pair of position q: the viscous ones first
template <int D>
__device__ __forceinline__ void pair_at(int q, int& a, int& b) {
    constexpr int M = D + 2, NM = D * (D + 1), NVIS = NM + M;
    if (q < NM) { a = 1 + q / (D + 1); b = q % (D + 1); }
    else if (q < NVIS) { a = M - 1; b = q - NM; }
    else if (q < NVIS + M) { a = 0; b = q - NVIS; }
    else { a = q - NVIS - M + 1; b = M - 1; }
}

// sums of x(g) over the tensor points (axis 0 fastest) against the 1-D functions of every axis, NA axes;
// axis AX (or none, AX < 0) takes the N1 + 2 functions of tx, the others the N1 basis functions of tb.
// put(i0, i1, i2, v): function indices per axis (0 on absent axes).
template <int NA, int N1, int Q1, int AX, class T, class X, class Put>
__device__ __forceinline__ void tensor_sums(const T* tb, const T* tx, X x, Put put) {
    constexpr int E0 = N1 + (AX == 0 ? 2 : 0), E1 = NA > 1 ? N1 + (AX == 1 ? 2 : 0) : 1, E2 = NA > 2 ? N1 + (AX == 2 ? 2 : 0) : 1;
    const T* t0 = AX == 0 ? tx : tb;
    const T* t1 = AX == 1 ? tx : tb;
    const T* t2 = AX == 2 ? tx : tb;
    constexpr int G1 = NA > 1 ? Q1 : 1, G2 = NA > 2 ? Q1 : 1;
#pragma unroll 1
    for (int g2 = 0; g2 < G2; ++g2) {
        T u[E1][E0];
#pragma unroll
        for (int e1 = 0; e1 < E1; ++e1)
#pragma unroll
            for (int e0 = 0; e0 < E0; ++e0) u[e1][e0] = T(0);
#pragma unroll 1
        for (int g1 = 0; g1 < G1; ++g1) {
            T t[E0];
#pragma unroll
            for (int e0 = 0; e0 < E0; ++e0) t[e0] = T(0);
#pragma unroll
            for (int g0 = 0; g0 < Q1; ++g0) {
                const T v = x(g0, g1, g2);
#pragma unroll
                for (int e0 = 0; e0 < E0; ++e0) t[e0] = fma(t0[g0 * E0 + e0], v, t[e0]);
            }
#pragma unroll
            for (int e1 = 0; e1 < E1; ++e1) {
                const T w = NA > 1 ? t1[g1 * E1 + e1] : T(1);
#pragma unroll
                for (int e0 = 0; e0 < E0; ++e0) u[e1][e0] = fma(w, t[e0], u[e1][e0]);
            }
        }
#pragma unroll
        for (int e2 = 0; e2 < E2; ++e2) {
            const T w = NA > 2 ? t2[g2 * E2 + e2] : T(1);
#pragma unroll
            for (int e1 = 0; e1 < E1; ++e1)
#pragma unroll
                for (int e0 = 0; e0 < E0; ++e0) put(e0, e1, e2, w * u[e1][e0]);
        }
    }
}

template <class C, class TA, class TL>
__global__ void __launch_bounds__(ContractShape<C, TA>::NTH) k_contract(BlkArgs<TL> A) {
    using S = ContractShape<C, TA>;
    constexpr int D = C::D, M = C::M, NP = C::NP, NQ = C::NQ, NF = C::NF, NFP = C::NFP, NFQ = C::NFQ;
    constexpr int N1 = S::N1, Q1 = S::Q1, NK = S::NK, PPC = S::PPC, NTH = S::NTH, BS = S::BS, NCB = S::NCB;
    constexpr int GEO = Geo<D>::N;
    const int tid = threadIdx.x;
    const int64_t el = blockIdx.x / S::NG, e = A.e0 + el;
    const int q0 = (int)(blockIdx.x % S::NG) * PPC, npair = min(PPC, M * M - q0);
    const DeviceTables& T = A.tab;
    constexpr bool F32 = sizeof(TA) == 4;
    const TA* tdphi = F32 ? (const TA*)T.fdphi : (const TA*)T.dphi;   // row tables: one rounding per entry
    const TA* tmu = F32 ? (const TA*)T.fmu : (const TA*)T.mu;
    extern __shared__ __align__(16) unsigned char craw[];
    TA* buf = reinterpret_cast<TA*>(craw);          // [PPC][NCB][BS] rows of the blocks, [column][row]
    TA* cv = buf + PPC * NCB * BS;                  // [PPC][D][NK][NQ]
    TA* cf = cv + PPC * S::CV;                      // [PPC][NF][NK][NFQ]
    TA* tb = cf + PPC * S::CF;                      // [Q1][N1] basis
    TA* tx = tb + Q1 * N1;                          // [Q1][N1 + 2] minus basis times M^{-1} C; lifts of the two ends, signed
    TA* dc = tx + Q1 * (N1 + 2);                    // [N1][N1] M^{-1} C
    TA* le = dc + N1 * N1;                          // [2][N1] lifts of the two ends, signed
    TA* mf = le + 2 * N1;                           // [NFP][NFP] face mass
    for (int i = tid; i < Q1 * N1; i += NTH) tb[i] = (TA)T.b1[i];
    for (int i = tid; i < Q1 * (N1 + 2); i += NTH) {
        const int g = i / (N1 + 2), j = i - g * (N1 + 2);
        double v = 0.0;
        for (int k = 0; k < N1; ++k)
            v += T.b1[g * N1 + k] * (j < N1 ? -T.minv_c[(size_t)k * NP + j]
                                            : (j == N1 ? -1.0 : 1.0) * T.minv_e[((size_t)(j - N1) * NP + k) * NFP]);
        tx[i] = (TA)v;
    }
    for (int i = tid; i < N1 * N1; i += NTH) dc[i] = (TA)T.minv_c[(size_t)(i / N1) * NP + i % N1];
    for (int i = tid; i < 2 * N1; i += NTH)
        le[i] = (TA)((i < N1 ? -1.0 : 1.0) * T.minv_e[((size_t)(i / N1) * NP + i % N1) * NFP]);
    for (int i = tid; i < NFP * NFP; i += NTH) mf[i] = (TA)T.mf[i];
    for (int p = 0; p < npair; ++p) {
        int a, b;
        pair_at<D>(q0 + p, a, b);
        const TA* sv = reinterpret_cast<const TA*>(A.vcoef) + (((size_t)el * M + a) * M + b) * (size_t)S::CV;
        for (int i = tid; i < S::CV; i += NTH) cv[p * S::CV + i] = sv[i];
        for (int i = tid; i < S::CF; i += NTH) {
            const int f = i / (NK * NFQ), r = i - f * NK * NFQ;
            cf[p * S::CF + i] = reinterpret_cast<const TA*>(A.fcoef)[((((size_t)el * NF + f) * M + a) * M + b) * (size_t)(NK * NFQ) + r];
        }
    }
    const double* G = A.geo + e * GEO;
    const double detJ = G[0];
    const double* NW = G + 1 + D * D;
    double* A11 = A.R.a11 + e * A.R.a11_es;
    TL* A12 = A.R.a12 + e * A.R.a12_es;
    TL* A21 = A.R.a21 + el * A.R.a21_es;
    TL* A22 = A.R.a22 + el * A.R.a22_es;
    __syncthreads();

    // ---- trace rows: the flux rows of S::FPR faces at a time ----
    for (int fr = 0; fr < NF; fr += S::FPR) {
        constexpr int RW = S::FPR * NFP;                    // rows of a round
        const int p = tid / RW, rr = tid - p * RW, f = fr + rr / NFP, lam = rr % NFP;
        const bool act = p < npair && f < NF;
        if (act) {
            int a, b;
            pair_at<D>(q0 + p, a, b);
            const bool vis = q0 + p < S::NVIS || (A.has_nu && a == b);
            TA* out = buf + (size_t)p * NCB * BS + rr;      // column c at out[c * BS]
            for (int c = 0; c < NCB; ++c) out[c * BS] = TA(0);
            const TA* o = cf + p * S::CF + f * NK * NFQ;
            const int n = f >> 1, side = f & 1, jn = side ? N1 - 1 : 0;
            int st[D];                                       // node stride of every axis
            st[0] = 1;
            for (int r = 1; r < D; ++r) st[r] = st[r - 1] * N1;
            const int t1 = n == 0 ? 1 : 0, t2 = n == 2 ? 1 : 2;   // tangential axes (t2 in 3-D only)
            // column of the node with tangential indices l1, l2 and normal index k
            auto ucol = [&](int l1, int l2, int k) { return l1 * st[t1] + (D == 3 ? l2 * st[D == 3 ? t2 : 0] : 0) + k * st[n]; };
            // column of node (index i on axis x, j on axis y) of face f2 (x, y its tangential axes, either order)
            auto tcol = [&](int f2, int x, int i, int j) {
                const int r2 = f2 >> 1;
                if (D == 2) return NP + f2 * NFP + i;
                const int lo = r2 == 0 ? 1 : 0;              // the lower tangential axis of f2
                return NP + f2 * NFP + (x == lo ? i + N1 * j : j + N1 * i);
            };
            auto row = [&](int s1, int s2) { return tmu[(s1 + Q1 * s2) * NFP + lam]; };
            const double* nw = NW + f * D;
            double nrm = 0.0;
            for (int k = 0; k < D; ++k) nrm += nw[k] * nw[k];
            nrm = sqrt(nrm);
            // kind 0: uhat of this face
            tensor_sums<D - 1, N1, Q1, -1, TA>(tb, tx, [&](int s1, int s2, int) { return row(s1, s2) * o[s1 + Q1 * s2]; },
                [&](int l1, int l2, int, TA v) { out[(NP + f * NFP + l1 + N1 * l2) * BS] += v; });
            if (vis) {
                // q along the normal: every node of a line through the face, and the faces f and opposite
                TA kn[NFP];
#pragma unroll
                for (int l = 0; l < NFP; ++l) kn[l] = TA(0);
                const TA* on = o + (1 + n) * NFQ;
                tensor_sums<D - 1, N1, Q1, -1, TA>(tb, tx, [&](int s1, int s2, int) { return row(s1, s2) * on[s1 + Q1 * s2]; },
                    [&](int l1, int l2, int, TA v) { kn[l1 + N1 * l2] += v; });
#pragma unroll
                for (int l = 0; l < NFP; ++l) {
                    const int l1 = l % N1, l2 = l / N1;
                    for (int k = 0; k < N1; ++k) out[ucol(l1, l2, k) * BS] -= kn[l] * dc[jn * N1 + k];
                    for (int s2 = 0; s2 < 2; ++s2) out[(NP + (2 * n + s2) * NFP + l) * BS] += kn[l] * le[s2 * N1 + jn];
                }
                // q along the tangential axes: the face's own nodes, and the edges of the faces across
                const TA* o1 = o + (1 + t1) * NFQ;
                tensor_sums<D - 1, N1, Q1, 0, TA>(tb, tx, [&](int s1, int s2, int) { return row(s1, s2) * o1[s1 + Q1 * s2]; },
                    [&](int l1, int l2, int, TA v) {
                        if (l1 < N1) out[ucol(l1, l2, jn) * BS] += v;
                        else out[tcol(2 * t1 + l1 - N1, n, jn, l2) * BS] += v;
                    });
                if constexpr (D == 3) {
                    const TA* o2 = o + (1 + t2) * NFQ;
                    tensor_sums<D - 1, N1, Q1, 1, TA>(tb, tx, [&](int s1, int s2, int) { return row(s1, s2) * o2[s1 + Q1 * s2]; },
                        [&](int l1, int l2, int, TA v) {
                            if (l2 < N1) out[ucol(l1, l2, jn) * BS] += v;
                            else out[tcol(2 * t2 + l2 - N1, n, jn, l1) * BS] += v;
                        });
                }
            }
            if (a == b) {                                    // tau u: the face mass, weighted by tau at the points if it varies
                if (A.taup) {                                // in FP64 in both forms: rounded once, as the constant tau's is
                    const double* tp = A.taup + (el * NF + f) * NFQ;
                    tensor_sums<D - 1, N1, Q1, -1, double>(T.b1, nullptr,
                        [&](int s1, int s2, int) { const int s = s1 + Q1 * s2; return T.mu[s * NFP + lam] * (nrm * T.wf[s] * tp[s]); },
                        [&](int l1, int l2, int, double v) { out[ucol(l1, l2, jn) * BS] += (TA)v; });
                } else {
                    const TA taun = (TA)(A.tau * nrm);
                    for (int l = 0; l < NFP; ++l) out[ucol(l % N1, l / N1, jn) * BS] += taun * mf[lam * NFP + l];
                }
            }
        }
        __syncthreads();
        for (int p2 = 0; p2 < npair; ++p2) {
            int a, b;
            pair_at<D>(q0 + p2, a, b);
            const int nr = min(S::FPR, NF - fr) * NFP;
            for (int idx = tid; idx < nr * NCB; idx += NTH) {
                const int rw = idx / NCB, c = idx - rw * NCB, ff = fr + rw / NFP;
                const TA v = buf[((size_t)p2 * NCB + c) * BS + rw];
                const int64_t trow = (ff * M + a) * NFP + rw % NFP;
                if (c < NP) A21[trow * A.R.a21_rs + b * NP + c] = (TL)v;
                else {
                    const int f2 = (c - NP) / NFP, l2 = (c - NP) % NFP;
                    A22[trow * A.R.a22_rs + (f2 * M + b) * NFP + l2] = (TL)v;
                }
            }
        }
        __syncthreads();
    }

    // ---- element rows: volume terms collected, then dt times the flux rows of the faces a node lies on ----
    {
        const int p = tid / NP, i = tid - p * NP;
        if (p < npair) {
            int a, b;
            pair_at<D>(q0 + p, a, b);
            const bool vis = q0 + p < S::NVIS || (A.has_nu && a == b);
            TA* out = buf + (size_t)p * NCB * BS + i;
            for (int c = 0; c < NCB; ++c) out[c * BS] = TA(0);
            const TA* o = cv + p * S::CV;
            // A_k at a point: the test function's gradient against the coefficients of kind k
            auto point = [&](int k) {
                return [&, k](int g0, int g1, int g2) {
                    const int g = g0 + Q1 * (g1 + Q1 * g2);
                    const TA* og = o + k * NQ + g;
                    TA v = tdphi[(size_t)g * NP + i] * og[0];
#pragma unroll
                    for (int r = 1; r < D; ++r) v = fma(tdphi[((size_t)r * NQ + g) * NP + i], og[r * NK * NQ], v);
                    return v;
                };
            };
            auto put_u = [&](int j0, int j1, int j2, TA v) { out[(j0 + N1 * (j1 + N1 * j2)) * BS] += v; };
            tensor_sums<D, N1, Q1, -1, TA>(tb, tx, point(0), put_u);
            if (vis) {
                tensor_sums<D, N1, Q1, 0, TA>(tb, tx, point(1), [&](int j0, int j1, int j2, TA v) {
                    if (j0 < N1) put_u(j0, j1, j2, v);
                    else out[(NP + (j0 - N1) * NFP + j1 + N1 * j2) * BS] += v;
                });
                tensor_sums<D, N1, Q1, 1, TA>(tb, tx, point(2), [&](int j0, int j1, int j2, TA v) {
                    if (j1 < N1) put_u(j0, j1, j2, v);
                    else out[(NP + (2 + j1 - N1) * NFP + j0 + N1 * j2) * BS] += v;
                });
                if constexpr (D == 3)
                    tensor_sums<D, N1, Q1, 2, TA>(tb, tx, point(3), [&](int j0, int j1, int j2, TA v) {
                        if (j2 < N1) put_u(j0, j1, j2, v);
                        else out[(NP + (4 + j2 - N1) * NFP + j0 + N1 * j1) * BS] += v;
                    });
            }
        }
        __syncthreads();
        for (int p2 = 0; p2 < npair; ++p2) {
            int a, b;
            pair_at<D>(q0 + p2, a, b);
            for (int idx = tid; idx < NP * NCB; idx += NTH) {
                const int ii = idx / NCB, c = idx - ii * NCB;
                const TA v = buf[((size_t)p2 * NCB + c) * BS + ii];
                const int64_t col = c < NP ? b * NP + c : (((c - NP) / NFP) * M + b) * NFP + (c - NP) % NFP;
                TA fs = TA(0);
                for (int k = 0; k < D; ++k) {
                    const int nfc = T.node_face[ii * D + k];
                    if (nfc < 0) continue;
                    const int64_t trow = ((nfc / NFP) * M + a) * NFP + nfc % NFP;
                    fs += (TA)(c < NP ? A21[trow * A.R.a21_rs + col] : A22[trow * A.R.a22_rs + col]);
                }
                const int64_t row = a * NP + ii;
                if (c < NP) {                                // the interior block is FP64 in both forms: so are its sums
                    double w = fma(A.dt, (double)fs, (double)v);
                    if (a == b) w += detJ / A.a_ii * T.mhat[ii * NP + c];
                    A11[row * A.R.a11_rs + col] = w;
                } else {
                    A12[row * A.R.a12_rs + col] = (TL)fma((TA)A.dt, fs, v);
                }
            }
        }
    }
    // ---- trace rows of boundary faces that are not flux rows: algebraic in (uhat, u) ----
    if (A.ftag) {
        __syncthreads();
        for (int p2 = 0; p2 < npair; ++p2) {
            int a, b;
            pair_at<D>(q0 + p2, a, b);
            for (int f = 0; f < NF; ++f) {
                const int tag = A.ftag[e * NF + f];
                if (boundary_row_is_flux<M>(tag, a)) continue;
                double nrm = 0.0;
                for (int k = 0; k < D; ++k) nrm += NW[f * D + k] * NW[f * D + k];
                // d bhat_a / d uhat_b = cb, d bhat_a / d u_b = cu, both times the face mass
                TA cb = (TA)(a == b ? 1.0 : 0.0), cu = TA(0);
                if (tag == 3 && a == M - 1 && b == 0) cb = (TA)(-A.ew);
                if (tag == 2 && a == b) cu = (TA)(-1);
                const TA nr = (TA)sqrt(nrm);
                for (int idx = tid; idx < NFP * NCB; idx += NTH) {
                    const int lam = idx / NCB, c = idx - lam * NCB;
                    const int64_t trow = (f * M + a) * NFP + lam;
                    if (c < NP) {
                        TA vu = TA(0);
                        for (int k = 0; k < D; ++k) {
                            const int nfc = T.node_face[c * D + k];
                            if (nfc >= 0 && nfc / NFP == f) vu = mf[lam * NFP + nfc % NFP];
                        }
                        A21[trow * A.R.a21_rs + b * NP + c] = (TL)(cu * nr * vu);
                    } else {
                        const int f2 = (c - NP) / NFP, l2 = (c - NP) % NFP;
                        A22[trow * A.R.a22_rs + (f2 * M + b) * NFP + l2] = (TL)(f2 == f ? cb * nr * mf[lam * NFP + l2] : TA(0));
                    }
                }
            }
        }
    }
}

}  // namespace hdg
