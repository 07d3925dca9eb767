// Eigendecomposition of the L x L Gram matrix S = Z^T Z for the nuclear-norm
// prox (Eq. "prox-L*") of FP32 plans, in one CTA.
//
// The prox needs V diag(f) V^T with f_j = min(1, c_j / sigma_j) (dual form,
// Algorithm 2 step 5) or max(0, 1 - c_j / sigma_j) (prox form), sigma_j =
// sqrt(lambda_j). Only eigenpairs with sigma_j > c_j make f_j differ from its
// limit (1 for the dual, 0 for the prox), so only those "active" pairs must be
// accurate; on GB300 FP64 is ~1/64 of the FP32 rate, so the work is split:
//
//  1. FP32 cyclic Jacobi (round-robin parallel ordering) on S, warm-started
//     from the previous call's eigenvectors V0 (A = V0^T S V0), gives every
//     eigenpair to FP32 accuracy; warm calls skip it while V0 still
//     diagonalises S to 2e-5 (late in a solve, when S changes slowly).
//  2. The active eigenvectors are refined in FP64 against the rest of the
//     basis with first-order correction steps (one from a warm basis, two
//     cold) of an approximate eigendecomposition (Ogita & Aishima 2018): with
//     b_j the basis (the active vectors themselves, then the inactive FP32
//     eigenvectors), T = B^T S X, R = I - B^T X, lambda_c = T_cc / (1 - R_cc),
//     the correction of x_c along b_j (j != c) is
//     (T_jc + lambda_c R_jc) / (lambda_c - lambda_j), and R_jc / 2
//     (orthogonalisation only) along x_c itself or for near-equal eigenvalues
//     (their mixing leaves f, continuous in sigma, unchanged to first order).
//     The eigenvalues are the last step's Rayleigh quotients lambda_c.
//  3. Cholesky QR keeps the active vectors orthonormal in FP64.
//  4. The factor is returned in low-rank form: M = I - sum_active (1 - f) x x^T
//     (dual) or sum_active f x x^T (prox), as r, g and the active x.
#include <algorithm>
#include <cmath>

#include "hs_device.cuh"
#include "hs_internal.h"

namespace hs {

constexpr int EIG_T = 1024;
constexpr int LD32 = MAX_L_NUC + 1;

// Block-wide sum of doubles, returned to every thread (red: 33 doubles).
__device__ __forceinline__ double eig_bsum(double v, double* red) { return block_sum_all(v, red); }

// Round-robin (circle method) schedule for n indices, n even: in round r the
// index n-1 meets r and (r + i) meets (r - i) (mod n-1) for i = 1 .. n/2-1.
// pairs[r * n/2 + k] = p | q << 8 (p < q) is the k-th pair of round r (thread r
// lists its round).
__device__ void rr_schedule(int n, unsigned short* pairs) {
    for (int r = threadIdx.x; r < n - 1; r += blockDim.x) {
        int k = 0;
        for (int i = 0; i < n; ++i) {
            int pi;
            if (i == n - 1) pi = r;
            else if (i == r) pi = n - 1;
            else pi = ((2 * r - i) % (n - 1) + (n - 1)) % (n - 1);
            if (i < pi) pairs[r * (n / 2) + k++] = (unsigned short)(i | (pi << 8));
        }
    }
}

// Rotation (c, s) that zeroes a_pq of the 2 x 2 block [[a_pp, a_pq], [a_pq, a_qq]]
// (Golub & Van Loan Alg. 8.4.1). FP32: fast reciprocal and reciprocal square
// root (the FP32 sweeps only need FP32-orthogonal rotations).
__device__ __forceinline__ void jac_rot(float app, float aqq, float apq, float& c, float& s) {
    const float tau = __fdividef(aqq - app, 2.f * apq);
    const float t = copysignf(1.f, tau) * __frcp_rn(fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f)));
    c = rsqrtf(fmaf(t, t, 1.f));
    s = t * c;
}
// FP64: the division and the roots of the library cost ~20 dependent FP64 instructions
// each at 1/64 of the FP32 rate, and a round waits for them. The tangent is taken from the
// approximate FP64 reciprocal (about 20 bits) and FP32: a rotation then leaves ~1e-6 of a_pq, which
// later rounds remove. What has to be FP64 is c^2 + s^2 = 1: one Newton step of (1 + t^2)^-1/2,
// then c and s both by the first order of what 1 - c^2 - s^2 (exact to 2^-106 by fused
// multiply-adds) still is. With a second Newton step in its place the rounding of c alone, always the same
// way, stretched the 64 columns of V by 8e-15 in nine sweeps (now 2e-16; the prox of a
// 60-channel cube with 3 active pairs was 1.2e-14 off for it).
__device__ __forceinline__ void jac_rot(double app, double aqq, double apq, double& c, double& s) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(2.0 * apq));
    float tau = (float)((aqq - app) * r);
    if (isnan(tau)) tau = 0.f;   // equal diagonal over a subnormal a_pq
    const double t = (double)copysignf(__frcp_rn(fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau);
    const double u = fma(t, t, 1.0);
    double y = (double)rsqrtf((float)u);
    y = fma(0.5 * y, fma(-(u * y), y, 1.0), y);
    c = y;
    s = t * y;
    const double e = 0.5 * fma(-s, s, fma(-c, c, 1.0));
    c = fma(e, c, c);
    s = fma(e, s, s);
}

// Cyclic Jacobi, round-robin parallel ordering, on the symmetric N x N matrix
// in A (leading dimension LDJ), accumulating V <- V J. Each round, thread k < N/2
// computes the rotation (c_k, s_k) of pair k = (p, q) from a_pp, a_qq, a_pq
// (J_pp = J_qq = c, J_pq = s, J_qp = -s); then thread (i, j) of the (N/2)^2
// grid applies A <- J^T A J to the 2 x 2 block (rows of pair i, columns of
// pair j):
//   rows   (p, q) <- (c_i row_p - s_i row_q, s_i row_p + c_i row_q)
//   cols   (p, q) <- (c_j col_p - s_j col_q, s_j col_p + c_j col_q),
// and rotates columns (p_j, q_j) of V in rows i and i + N/2. Every entry belongs
// to one thread per round, so A and V are updated in place. A rotation is
// applied only when |a_pq| exceeds skip sqrt(|a_pp a_qq|) and floor_rel ||A||_F;
// sweeps stop when the off-diagonal Frobenius norm is at most off_rel ||A||_F,
// when a sweep applies no rotation, or after max_sweeps.
template <typename T, int N>
__device__ void jacobi_blocks(T* A, T* V, unsigned short* pairs, double skip, double floor_rel,
                              double off_rel, int max_sweeps, Cx<T>* cs, double* red, int* flag) {
    constexpr int LDJ = MAX_L_NUC + 1;
    constexpr int NP = N / 2;
    constexpr int LG = (N >= 64) ? 6 : (N >= 32) ? 5 : (N >= 16) ? 4 : (N >= 8) ? 3 : (N >= 4) ? 2 : 1;
    const int tid = threadIdx.x, nt = blockDim.x;
    const T skip2 = (T)(skip * skip);
    const int bi = tid / NP, bj = tid - (tid / NP) * NP;   // block of this thread (tid < NP^2)
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        T nrmT = 0, offT = 0;   // per-thread partial sums in the working precision
        for (int k = tid; k < N * N; k += nt) {
            const int i = k >> LG, j = k & (N - 1);
            const T x = A[i * LDJ + j];
            nrmT = fma(x, x, nrmT);
            if (i != j) offT = fma(x, x, offT);
        }
        const double nrm = eig_bsum((double)nrmT, red);
        const double off = eig_bsum((double)offT, red);
        if (!(off > off_rel * off_rel * nrm)) break;
        if (sweep == 0) {   // the round-robin schedule, built only when a sweep runs
            rr_schedule(N, pairs);
            __syncthreads();
        }
        const T flo = (T)(floor_rel * sqrt(nrm));
        if (tid == 0) *flag = 0;
        __syncthreads();
        for (int r = 0; r < N - 1; ++r) {
            const unsigned short* pr = pairs + r * NP;
            if (tid < NP) {
                const int pq = pr[tid], p = pq & 0xff, q = pq >> 8;
                const T apq = A[p * LDJ + q], app = A[p * LDJ + p], aqq = A[q * LDJ + q];
                T c = 1, s = 0;
                const T ab = fabs(apq);
                if (ab > flo && ab * ab > skip2 * fabs(app * aqq)) {
                    jac_rot(app, aqq, apq, c, s);
                    *flag = 1;
                }
                Cx<T> v;
                v.x = c;
                v.y = s;
                cs[tid] = v;
            }
            __syncthreads();
            if (tid < NP * NP) {
                const int pqi = pr[bi], pqj = pr[bj];
                const int pi = pqi & 0xff, qi = pqi >> 8, pj = pqj & 0xff, qj = pqj >> 8;
                const Cx<T> csi = cs[bi], csj = cs[bj];
                const T ci = csi.x, si = csi.y, cj = csj.x, sj = csj.y;
                const T a00 = A[pi * LDJ + pj], a01 = A[pi * LDJ + qj];
                const T a10 = A[qi * LDJ + pj], a11 = A[qi * LDJ + qj];
                const T v00 = V[bi * LDJ + pj], v01 = V[bi * LDJ + qj];
                const T v10 = V[(bi + NP) * LDJ + pj], v11 = V[(bi + NP) * LDJ + qj];
                const T r0x = ci * a00 - si * a10, r0y = ci * a01 - si * a11;
                const T r1x = si * a00 + ci * a10, r1y = si * a01 + ci * a11;
                T b00 = cj * r0x - sj * r0y, b01 = sj * r0x + cj * r0y;
                T b10 = cj * r1x - sj * r1y, b11 = sj * r1x + cj * r1y;
                if (sizeof(T) == 4 && bi == bj && si != T(0)) {   // FP32: the rotated pair is decoupled
                    b01 = T(0);
                    b10 = T(0);
                }
                A[pi * LDJ + pj] = b00;
                A[pi * LDJ + qj] = b01;
                A[qi * LDJ + pj] = b10;
                A[qi * LDJ + qj] = b11;
                V[bi * LDJ + pj] = cj * v00 - sj * v01;
                V[bi * LDJ + qj] = sj * v00 + cj * v01;
                V[(bi + NP) * LDJ + pj] = cj * v10 - sj * v11;
                V[(bi + NP) * LDJ + qj] = sj * v10 + cj * v11;
            }
            __syncthreads();
        }
        const int any = *flag;
        __syncthreads();
        if (!any) break;
    }
}

// Dispatch on the padded size n (power of two, 2..64). B and W are unused
// scratch kept for the callers' layouts.
template <typename T>
__device__ void jacobi_n(int n, T* A, T* B, T* V, T* W, unsigned short* pairs, double skip,
                         double floor_rel, double off_rel, int max_sweeps, Cx<T>* cs, double* red, int* flag) {
    (void)B;
    (void)W;
#define HS_JAC(NN) jacobi_blocks<T, NN>(A, V, pairs, skip, floor_rel, off_rel, max_sweeps, cs, red, flag)
    switch (n) {
        case 2: HS_JAC(2); break;
        case 4: HS_JAC(4); break;
        case 8: HS_JAC(8); break;
        case 16: HS_JAC(16); break;
        case 32: HS_JAC(32); break;
        default: HS_JAC(64); break;
    }
#undef HS_JAC
}

// One CTA of EIG_T threads; dynamic shared memory layout below.
__global__ void __launch_bounds__(EIG_T) k_eig_mixed(const double* __restrict__ Sg, int L,
                                                    const double* __restrict__ w_sv, double thr,
                                                    int dual, double* __restrict__ Mf,
                                                    double* __restrict__ sv_out,
                                                    float* __restrict__ warm, int* __restrict__ r_out) {
    extern __shared__ __align__(16) unsigned char eig_smem[];
    constexpr int SL = MAX_L_NUC * LD32;                 // one 64 x 65 slot
    float* V32 = (float*)eig_smem;                       // slot 0
    float* W32 = V32 + SL;                               // slot 1 (Jacobi scratch)
    float* A32 = W32 + SL;                               // slot 2
    float* B32 = A32 + SL;                               // slot 3 (Jacobi scratch, warm-start temp)
    float* T32 = B32;
    double* Sd = (double*)(B32 + SL);                    // 64 x 65 doubles each from here
    double* X = Sd + SL;                                 // active vectors (columns)
    double* Y = X + SL;
    double* Rb = Y + SL;
    // FP64 view over float slots 2-3 once the FP32 Jacobi matrix is dead
    double* Tb = (double*)A32;
    __shared__ double red[33];
    __shared__ float2 cs32[MAX_L_NUC / 2];
    __shared__ unsigned short partner[(MAX_L_NUC - 1) * MAX_L_NUC / 2];
    __shared__ int flag;
    __shared__ double lam32[MAX_L_NUC], lamr[MAX_L_NUC], fv[MAX_L_NUC];
    __shared__ float lamf[MAX_L_NUC];
    __shared__ int order[MAX_L_NUC];
    __shared__ int r_act;
    const int tid = threadIdx.x, nt = blockDim.x;
    int n = 2;
    while (n < L) n <<= 1;
    // ---- load S (FP64) and its FP32 copy
    for (int k = tid; k < n * n; k += nt) {
        const int i = k / n, j = k - i * n;
        const double v = (i < L && j < L) ? Sg[i * L + j] : 0.0;
        Sd[i * MAX_L_NUC + j] = v;
        A32[i * LD32 + j] = (float)v;
        V32[i * LD32 + j] = (warm && i < L && j < L) ? warm[i * L + j] : (i == j ? 1.f : 0.f);
    }
    __syncthreads();
    if (warm) {   // A = V0^T S V0 (FP32), then symmetrise; 2 x 2 output blocks per thread
        const int nh = n >> 1;
        for (int k = tid; k < nh * nh; k += nt) {   // T = S V0
            const int i = 2 * (k / nh), j = 2 * (k % nh);
            float a00 = 0.f, a01 = 0.f, a10 = 0.f, a11 = 0.f;
            for (int m = 0; m < n; ++m) {
                const float s0 = A32[i * LD32 + m], s1 = A32[(i + 1) * LD32 + m];
                const float v0 = V32[m * LD32 + j], v1 = V32[m * LD32 + j + 1];
                a00 = fmaf(s0, v0, a00);
                a01 = fmaf(s0, v1, a01);
                a10 = fmaf(s1, v0, a10);
                a11 = fmaf(s1, v1, a11);
            }
            T32[i * LD32 + j] = a00;
            T32[i * LD32 + j + 1] = a01;
            T32[(i + 1) * LD32 + j] = a10;
            T32[(i + 1) * LD32 + j + 1] = a11;
        }
        __syncthreads();
        for (int k = tid; k < nh * nh; k += nt) {   // A = V0^T T
            const int i = 2 * (k / nh), j = 2 * (k % nh);
            float a00 = 0.f, a01 = 0.f, a10 = 0.f, a11 = 0.f;
            for (int m = 0; m < n; ++m) {
                const float u0 = V32[m * LD32 + i], u1 = V32[m * LD32 + i + 1];
                const float t0 = T32[m * LD32 + j], t1 = T32[m * LD32 + j + 1];
                a00 = fmaf(u0, t0, a00);
                a01 = fmaf(u0, t1, a01);
                a10 = fmaf(u1, t0, a10);
                a11 = fmaf(u1, t1, a11);
            }
            A32[i * LD32 + j] = a00;
            A32[i * LD32 + j + 1] = a01;
            A32[(i + 1) * LD32 + j] = a10;
            A32[(i + 1) * LD32 + j + 1] = a11;
        }
        __syncthreads();
        for (int k = tid; k < n * n; k += nt) {
            const int i = k / n, j = k - i * n;
            if (i < j) {
                const float a = 0.5f * (A32[i * LD32 + j] + A32[j * LD32 + i]);
                A32[i * LD32 + j] = a;
                A32[j * LD32 + i] = a;
            }
        }
        __syncthreads();
    }
    // ---- 1. FP32 Jacobi on every eigenpair
    // warm-started calls run at most one FP32 sweep, and none while the previous
    // basis still diagonalises S to 2e-5 (relative off-diagonal Frobenius norm,
    // about twice the FP32 rounding of V0^T S V0): the active pairs are made exact in
    // FP64 below from a basis that accurate, and the basis is swept again as
    // soon as S has drifted further
    jacobi_n<float>(n, A32, B32, V32, W32, partner, 1e-7, 2e-7, warm ? 2e-5 : 2e-6, warm ? 1 : 15, cs32, red,
                    &flag);
    // ---- eigenvalues, descending order (rank by counting), warm start for the next call
    if (tid < L) {
        lamf[tid] = A32[tid * LD32 + tid];
        lam32[tid] = (double)lamf[tid];
    }
    if (tid == 0) r_act = 0;
    __syncthreads();
    if (tid < L) {   // rank of eigenvalue tid; active when sigma > c_rank (1 - 1e-3)
        // a NaN (from a non-finite input) ranks below every number, so the ranks stay a
        // permutation and every index taken from `order` stays in range
        int rk = 0;
        const float li = isnan(lamf[tid]) ? -INFINITY : lamf[tid];
        for (int j = 0; j < L; ++j) {
            const float lj = isnan(lamf[j]) ? -INFINITY : lamf[j];
            rk += (lj > li) || (lj == li && j < tid);
        }
        order[rk] = tid;
        const double c = thr * (w_sv ? w_sv[rk] : 1.0) * (1.0 - 1e-3);
        if ((double)fmaxf(li, 0.f) > c * c) atomicMax(&r_act, rk + 1);
    }
    if (warm)
        for (int k = tid; k < L * L; k += nt) warm[k] = V32[(k / L) * LD32 + (k % L)];
    __syncthreads();
    if (tid == 0 && r_out) *r_out = r_act;
    const int r = r_act;
    if (r > 0) {
        // active vectors in FP64
        for (int k = tid; k < L * r; k += nt) {
            const int i = k / r, c = k - i * r;
            X[i * MAX_L_NUC + c] = (double)V32[i * LD32 + order[c]];
        }
        __syncthreads();
        // ---- 2. FP64 correction steps of the active vectors against the whole basis
        // (the first-order step squares the FP32 error: one suffices from a warm basis)
        const int nsteps = warm ? 1 : 2;
        for (int step = 0; step < nsteps; ++step) {
            // Y = S X
            for (int k = tid; k < L * r; k += nt) {
                const int i = k / r, c = k - i * r;
                double acc = 0.0;
                for (int m = 0; m < L; ++m) acc = fma(Sd[i * MAX_L_NUC + m], X[m * MAX_L_NUC + c], acc);
                Y[i * MAX_L_NUC + c] = acc;
            }
            __syncthreads();
            // T_jc = b_j . Y_c, R_jc = delta_jc - b_j . X_c   (b_j = X_j for j < r, else V32 column)
            for (int k = tid; k < L * r; k += nt) {
                const int j = k / r, c = k - j * r;
                double t = 0.0, q = 0.0;
                if (j < r) {
                    for (int m = 0; m < L; ++m) {
                        const double b = X[m * MAX_L_NUC + j];
                        t = fma(b, Y[m * MAX_L_NUC + c], t);
                        q = fma(b, X[m * MAX_L_NUC + c], q);
                    }
                } else {
                    const int col = order[j];
                    for (int m = 0; m < L; ++m) {
                        const double b = (double)V32[m * LD32 + col];
                        t = fma(b, Y[m * MAX_L_NUC + c], t);
                        q = fma(b, X[m * MAX_L_NUC + c], q);
                    }
                }
                Tb[j * MAX_L_NUC + c] = t;
                Rb[j * MAX_L_NUC + c] = (j == c ? 1.0 : 0.0) - q;
            }
            __syncthreads();
            if (tid < r) lamr[tid] = Tb[tid * MAX_L_NUC + tid] / (1.0 - Rb[tid * MAX_L_NUC + tid]);
            __syncthreads();
            const double delta = 1e-5 * fmax(fabs(lamr[0]), 1e-300);
            // E_jc into Tb (overwrites T in place: each entry read once by its own thread)
            for (int k = tid; k < L * r; k += nt) {
                const int j = k / r, c = k - j * r;
                const double t = Tb[j * MAX_L_NUC + c], q = Rb[j * MAX_L_NUC + c];
                double e;
                const double gap = lamr[c] - (j < r ? lamr[j] : lam32[order[j]]);
                e = (j != c && fabs(gap) > delta) ? (t + lamr[c] * q) / gap : 0.5 * q;
                Tb[j * MAX_L_NUC + c] = e;
            }
            __syncthreads();
            // X_new = X + B E  (into Y)
            for (int k = tid; k < L * r; k += nt) {
                const int i = k / r, c = k - i * r;
                double acc = X[i * MAX_L_NUC + c];
                for (int j = 0; j < r; ++j) acc = fma(X[i * MAX_L_NUC + j], Tb[j * MAX_L_NUC + c], acc);
                for (int j = r; j < L; ++j)
                    acc = fma((double)V32[i * LD32 + order[j]], Tb[j * MAX_L_NUC + c], acc);
                Y[i * MAX_L_NUC + c] = acc;
            }
            __syncthreads();
            for (int k = tid; k < L * r; k += nt) {
                const int i = k / r, c = k - i * r;
                X[i * MAX_L_NUC + c] = Y[i * MAX_L_NUC + c];
            }
            __syncthreads();
        }
        // ---- 3. orthonormalise the active vectors (Cholesky QR: G = X^T X = R^T R,
        //      X <- X R^{-1}; X is orthonormal to first order already, so G ~ I)
        for (int k = tid; k < r * r; k += nt) {
            const int a = k / r, b = k - a * r;
            if (a <= b) {
                double acc = 0.0;
                for (int m = 0; m < L; ++m) acc = fma(X[m * MAX_L_NUC + a], X[m * MAX_L_NUC + b], acc);
                Tb[a * LD32 + b] = acc;
            }
        }
        __syncthreads();
        if (tid < 32) {   // upper-triangular R in place of G, one warp, lanes over columns
            for (int j = 0; j < r; ++j) {
                if (tid == 0) {
                    double d = Tb[j * LD32 + j];
                    for (int k = 0; k < j; ++k) d -= Tb[k * LD32 + j] * Tb[k * LD32 + j];
                    Tb[j * LD32 + j] = sqrt(fmax(d, 1e-300));
                }
                __syncwarp();
                const double rjj = Tb[j * LD32 + j];
                for (int i = j + 1 + tid; i < r; i += 32) {
                    double v = Tb[j * LD32 + i];
                    for (int k = 0; k < j; ++k) v -= Tb[k * LD32 + j] * Tb[k * LD32 + i];
                    Tb[j * LD32 + i] = v / rjj;
                }
                __syncwarp();
            }
        }
        __syncthreads();
        for (int m = tid; m < L; m += nt) {   // row m of X times R^{-1} (forward substitution)
            for (int j = 0; j < r; ++j) {
                double v = X[m * MAX_L_NUC + j];
                for (int k = 0; k < j; ++k) v -= X[m * MAX_L_NUC + k] * Tb[k * LD32 + j];
                X[m * MAX_L_NUC + j] = v / Tb[j * LD32 + j];
            }
        }
        __syncthreads();
        // eigenvalues: the last step's Rayleigh quotients (second-order accurate)
        if (tid < r) {
            const double sig = sqrt(fmax(lamr[tid], 0.0));
            const double c = thr * (w_sv ? w_sv[tid] : 1.0);
            double f;
            if (dual) f = (sig > c) ? c / sig : 1.0;
            else f = (sig > c) ? 1.0 - c / sig : 0.0;
            if (sv_out) sv_out[tid] = sig;
            fv[tid] = f;   // factor of active vector tid
        }
        __syncthreads();
    }
    if (sv_out)
        for (int j = r + tid; j < L; j += nt) sv_out[j] = sqrt(fmax(lam32[order[j]], 0.0));
    // ---- 4. low-rank factor: M = I + sum_c (f_c - 1) y_c y_c^T (dual) or sum_c f_c y_c y_c^T
    if (tid == 0) {
        Mf[LR_R] = (double)r;
        Mf[LR_BASE] = dual ? 1.0 : 0.0;
    }
    float* Ff = reinterpret_cast<float*>(Mf + LR_DOUBLES);   // FP32 copies for the apply kernel
    if (tid < r) {
        const double g = dual ? fv[tid] - 1.0 : fv[tid];
        Mf[LR_G + tid] = g;
        Ff[LRF_G + tid] = (float)g;
    }
    for (int k = tid; k < L * r; k += nt) {
        const int i = k / r, c = k - i * r;
        const double x = X[i * MAX_L_NUC + c];
        const float xh = (float)x;
        Mf[LR_X + c * MAX_L_NUC + i] = x;
        Ff[LRF_XH + c * MAX_L_NUC + i] = xh;
        Ff[LRF_XL + c * MAX_L_NUC + i] = (float)(x - (double)xh);
    }
}

// ---------------------------------------------------------------- cold calls (FP32 plans)
// Eigendecomposition without a basis to start from (nuclear prox and singular values
// outside the iteration): same steps and result as k_eig_mixed, laid out for the ~6
// full Jacobi sweeps such a call needs.
//  * k_eig_mixed keeps A and V in shared memory: 16 accesses of 1024 threads, two barriers
//    and ~2800 cycles for every 32 rotations. Here the indices come in blocks of two, 4
//    indices (two blocks) to a position; thread (I, J) keeps the 4 x 4 blocks of A and V of
//    positions I and J in registers. A round rotates the 4 pairs across the two blocks of
//    every position (two stages of two disjoint pairs; in the first round of a sweep also
//    the pairs inside the blocks), so a sweep is N / 2 - 1 rounds instead of N - 1 and moves
//    half the data per rotation. The blocks then advance as in a round-robin tournament:
//    columns by warp shuffles, rows of A through shared memory, rows of V not at all.
//  * Rotations are corrected to c^2 + s^2 = 1 (a reciprocal root alone let the
//    eigenvalues drift up by 2-4e-6 of the largest; singular values of the 256 x 256,
//    L = 60 cube are now 1.1e-6 from FP64, 4.1e-6 before).
//  * The FP64 dot products of the correction steps are split over 8 lanes each when there are
//    few: one thread per dot product left 60 dependent FP64 multiply-adds to wait for.
//  * The last orthonormalisation is a product with the inverse Cholesky factor to first
//    order (G = I + E: X (I - U), U = strict upper part of E plus half its diagonal) while no entry
//    of E^2 (r active vectors: at most r times the largest entry squared) passes FP64 rounding; else
//    the factorisation.
// us per prox at 64 x 64, before -> after: L = 60 with 2 active pairs 499 -> 349, all 60 active
// 1357 -> 1246; L = 20 146 -> 99; L = 6 74 -> 49. A round takes ~2300 cycles, of
// which the rotations' serial chain and the barriers are the larger part.
// put(k, sums) for k < count, where f(k, m0, dm, s) adds the terms m0, m0 + dm, ... of entry
// k's two sums to s: by 8 lanes per entry while that leaves at most 4 entries to a
// group (few active vectors: the length of one sum is what a step waits for), else by
// one thread per entry (many: FP64 throughput).
template <typename F, typename P> __device__ __forceinline__ void each_dot(int count, F f, P put) {
    const int nt = blockDim.x, tid = threadIdx.x;
    if (2 * count <= nt) {
        const int sub = tid & 7;
        const unsigned mask = 0xffu << (tid & 24);
        for (int k = tid >> 3; k < count; k += nt >> 3) {
            double2 v = make_double2(0.0, 0.0);
            f(k, sub, 8, v);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                v.x += __shfl_xor_sync(mask, v.x, o);
                v.y += __shfl_xor_sync(mask, v.y, o);
            }
            if (sub == 0) put(k, v);
        }
    } else {
        for (int k = tid; k < count; k += nt) {
            double2 v = make_double2(0.0, 0.0);
            f(k, 0, 1, v);
            put(k, v);
        }
    }
    __syncthreads();
}

constexpr int LDD = MAX_L_NUC + 1;   // row stride of the FP64 matrices (8 lanes down a column: distinct banks)
constexpr size_t EIG_COLD_SMEM = (size_t)5 * MAX_L_NUC * LDD * sizeof(double) + MAX_L_NUC * LD32 * sizeof(float);

constexpr int EIG_COLD_T = 512;   // 256 for A, 256 for V while the sweeps run

template <int N>
__global__ void __launch_bounds__(EIG_COLD_T, 1) k_eig_cold(const double* __restrict__ Sg, int L,
                                                         const double* __restrict__ w_sv, double thr, int dual,
                                                         double* __restrict__ Mf, double* __restrict__ sv_out,
                                                         int* __restrict__ r_out) {
    extern __shared__ __align__(16) unsigned char eig_smem[];
    constexpr int NS = N / 4;   // positions
    double* Sd = (double*)eig_smem;
    double* X = Sd + MAX_L_NUC * LDD;    // active vectors (columns)
    double* Y = X + MAX_L_NUC * LDD;
    double* Rb = Y + MAX_L_NUC * LDD;
    double* Tb = Rb + MAX_L_NUC * LDD;
    float* V32 = (float*)(Tb + MAX_L_NUC * LDD);
    float4* rows = (float4*)X;           // rows of A on the move, while the sweeps run: [NS][4][NS]
    __shared__ float2 red[EIG_COLD_T / 32];
    __shared__ float2 cs[2][NS][6];      // rotations of a round: pairs (0,2) (1,3) | (0,3) (1,2) | (0,1) (2,3)
    __shared__ double dinv[MAX_L_NUC];
    __shared__ float lamf[MAX_L_NUC];
    __shared__ double lam32[MAX_L_NUC], lamr[MAX_L_NUC], fv[MAX_L_NUC];
    __shared__ int order[MAX_L_NUC];
    __shared__ int r_act, emax;
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int k = tid; k < L * L; k += nt) Sd[(k / L) * LDD + k % L] = Sg[k];
    if (tid == 0) {
        r_act = 0;
        emax = 0;
    }
    __syncthreads();
    // The sweeps run on S times a power of two that brings its largest diagonal entry to [1, 2):
    // the sum of all its squares, which decides whether to sweep, left the FP32 range from singular
    // values of 1e9 on (and the sweeps were left out). In range no bit depends on it.
    // (The largest exponent from the high words; scaled in FP32 while that cannot overflow: FP64 multiply-adds
    // and the library's scalbn took 4 us here.)
    int mh = 0;
    for (int k = tid & 31; k < L; k += 32) mh = max(mh, __double2hiint(Sd[k * LDD + k]));
    mh = __reduce_max_sync(0xffffffffu, mh) >> 20;
    const int ex = mh > 0 && mh < 2047 ? mh - 1023 : 0;
    const bool near = abs(ex) <= 64;
    const double down = __hiloint2double((1023 - ex) << 20, 0), up = __hiloint2double((1023 + ex) << 20, 0);
    const float downf = (float)down;
    // ---- 1. FP32 Jacobi, position k = indices 4k .. 4k + 3 at the start of every sweep.
    // Threads of the lower half hold blocks of A, those of the upper half blocks of V and apply a
    // round's rotations while the next round's are computed.
    const int half = tid >> 8, t0 = tid & 255;
    const bool in = t0 < NS * NS, inA = in && half == 0;
    const int I = in ? t0 / NS : 0, J = t0 % NS;
    float a[4][4];   // A[rows of position I][columns of J], or V[4I .. 4I + 3][columns of J]
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = 4 * I + p, j = 4 * J + q;
            if (half) a[p][q] = (in && i == j) ? 1.f : 0.f;
            else if (!in || i >= L || j >= L) a[p][q] = 0.f;
            else a[p][q] = near ? (float)Sd[i * LDD + j] * downf : (float)(Sd[i * LDD + j] * down);
        }
    constexpr int PA[6] = {0, 1, 0, 1, 0, 2}, PB[6] = {2, 3, 3, 2, 1, 3};
    // blocks advance: first block of position 0 stays, position 1 gets position 0's second,
    // position k position k - 1's first; second blocks come from position k + 1, the last
    // position's from its own first
    auto shift = [&]() {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float t = a[x][q], b = a[x][2 + q];
                const float up = __shfl_up_sync(0xffffffffu, J == 0 ? b : t, 1, NS);
                const float dn = __shfl_down_sync(0xffffffffu, b, 1, NS);
                a[x][q] = J == 0 ? t : up;
                a[x][2 + q] = J == NS - 1 ? t : dn;
            }
    };
    auto cols = [&](const float2* c, int k) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float y = a[x][PA[k]], z = a[x][PB[k]];
            a[x][PA[k]] = c[k].x * y - c[k].y * z;
            a[x][PB[k]] = c[k].y * y + c[k].x * z;
        }
    };
    for (int sweep = 0; sweep < 15; ++sweep) {
        float o2 = 0.f, d2 = 0.f;
        if (inA)
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (I == J && p == q) d2 = fmaf(a[p][q], a[p][q], d2);
                    else o2 = fmaf(a[p][q], a[p][q], o2);
                }
        o2 = warp_sumf(o2);
        d2 = warp_sumf(d2);
        if ((tid & 31) == 0) red[tid >> 5] = make_float2(o2, d2);
        __syncthreads();
        float off = 0.f, nrm = 0.f;
#pragma unroll
        for (int k = 0; k < EIG_COLD_T / 64; ++k) {   // the warps that hold A
            off += red[k].x;
            nrm += red[k].x + red[k].y;
        }
        if (!(off > 4e-12f * nrm)) break;
        const float flo = 2e-7f * sqrtf(nrm);
        int any = 0;
        for (int r = 0; r < N / 2 - 1; ++r) {
            const int nk = r == 0 ? 6 : 4;
            float2(*rc)[6] = cs[r & 1];
            int rot = 0;
            if (inA && I == J) {
                float m[4][4];
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) m[p][q] = a[p][q];
#pragma unroll
                for (int st = 0; st < 3; ++st) {   // two disjoint pairs at a time, without branches
                    if (2 * st >= nk) break;
                    float c[2], s[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int p = PA[2 * st + e], q = PB[2 * st + e];
                        const float ab = fabsf(m[p][q]);
                        const bool on = ab > flo && ab * ab > 1e-14f * fabsf(m[p][p] * m[q][q]);
                        const float tau = __fdividef(m[q][q] - m[p][p], 2.f * m[p][q]);
                        const float u = fmaf(tau, tau, 1.f);
                        const float t = copysignf(__fdividef(1.f, fabsf(tau) + u * rsqrtf(u)), tau);
                        const float w = fmaf(t, t, 1.f), d = rsqrtf(w);
                        const float f = fmaf(0.5f * d, fmaf(-w * d, d, 1.f), d);
                        c[e] = on ? f : 1.f;
                        s[e] = on ? t * f : 0.f;
                        rot |= on;
                        rc[I][2 * st + e] = make_float2(c[e], s[e]);
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int p = PA[2 * st + e], q = PB[2 * st + e];
                            const float y = m[p][x], z = m[q][x];
                            m[p][x] = c[e] * y - s[e] * z;
                            m[q][x] = s[e] * y + c[e] * z;
                        }
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int p = PA[2 * st + e], q = PB[2 * st + e];
                            const float y = m[x][p], z = m[x][q];
                            m[x][p] = c[e] * y - s[e] * z;
                            m[x][q] = s[e] * y + c[e] * z;
                        }
                }
            }
            const int go = __syncthreads_or(rot);
            any |= go;
            if (half == 0) {
                if (go) {
                    float2 ri[6], rj[6];
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        if (k < nk) {
                            ri[k] = rc[I][k];
                            rj[k] = rc[J][k];
                        }
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        if (k < nk)
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                const float y = a[PA[k]][x], z = a[PB[k]][x];
                                a[PA[k]][x] = ri[k].x * y - ri[k].y * z;
                                a[PB[k]][x] = ri[k].y * y + ri[k].x * z;
                            }
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        if (k < nk) cols(rj, k);
                }
                shift();
                if (in)
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        rows[(I * 4 + x) * NS + J] = make_float4(a[x][0], a[x][1], a[x][2], a[x][3]);
            }
            __syncthreads();
            if (half == 0) {
                if (in)
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const int ft = I == 0 ? x : (I == 1 ? 2 + x : (I - 1) * 4 + x);
                        const int fb = I == NS - 1 ? I * 4 + x : (I + 1) * 4 + 2 + x;
                        const float4 t = rows[ft * NS + J], b = rows[fb * NS + J];
                        a[x][0] = t.x; a[x][1] = t.y; a[x][2] = t.z; a[x][3] = t.w;
                        a[2 + x][0] = b.x; a[2 + x][1] = b.y; a[2 + x][2] = b.z; a[2 + x][3] = b.w;
                    }
            } else {
                if (go) {
                    float2 rj[6];
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        if (k < nk) rj[k] = rc[J][k];
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        if (k < nk) cols(rj, k);
                }
                shift();
            }
        }
        if (!any) break;   // uniform: the rounds' barriers agreed on it
    }
    if (in) {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (half) V32[(4 * I + p) * LD32 + 4 * J + q] = a[p][q];
                else if (I == J && p == q) lamf[4 * I + p] = a[p][q];
            }
    }
    __syncthreads();
    if (tid < L) {   // descending rank (NaN last, so the ranks stay a permutation); active when sigma > c (1 - 1e-3)
        int rk = 0;
        const float li = isnan(lamf[tid]) ? -INFINITY : lamf[tid];
        for (int j = 0; j < L; ++j) {
            const float lj = isnan(lamf[j]) ? -INFINITY : lamf[j];
            rk += (lj > li) || (lj == li && j < tid);
        }
        lam32[tid] = (double)lamf[tid] * up;
        order[rk] = tid;
        const double c = thr * (w_sv ? w_sv[rk] : 1.0) * (1.0 - 1e-3);
        if ((double)fmaxf(li, 0.f) * up > c * c) atomicMax(&r_act, rk + 1);
    }
    __syncthreads();
    const int r = r_act;
    if (tid == 0 && r_out) *r_out = r;
    if (r > 0) {
        for (int k = tid; k < L * r; k += nt) {
            const int i = k / r, c = k - i * r;
            X[i * LDD + c] = (double)V32[i * LD32 + order[c]];
        }
        __syncthreads();
        // ---- 2. FP64 correction steps of the active vectors against the whole basis
        for (int step = 0; step < 2; ++step) {
            each_dot(L * r,   // Y = S X
                     [&](int k, int m, int dm, double2& v) {
                         const int i = k / r, c = k - i * r;
                         for (; m < L; m += dm) v.x = fma(Sd[i * LDD + m], X[m * LDD + c], v.x);
                     },
                     [&](int k, double2 v) { Y[(k / r) * LDD + k % r] = v.x; });
            each_dot(L * r,   // T_jc = b_j . Y_c, R_jc = delta_jc - b_j . X_c
                     [&](int k, int m, int dm, double2& v) {
                         const int j = k / r, c = k - j * r, col = order[j];
                         if (j > c && j < r) return;   // active against active: symmetric
                         for (; m < L; m += dm) {
                             const double b = j < r ? X[m * LDD + j] : (double)V32[m * LD32 + col];
                             v.x = fma(b, Y[m * LDD + c], v.x);
                             v.y = fma(b, X[m * LDD + c], v.y);
                         }
                     },
                     [&](int k, double2 v) {
                         const int j = k / r, c = k - j * r;
                         if (j > c && j < r) return;
                         const double q = (j == c ? 1.0 : 0.0) - v.y;
                         Tb[j * LDD + c] = v.x;
                         Rb[j * LDD + c] = q;
                         if (j < c) {
                             Tb[c * LDD + j] = v.x;
                             Rb[c * LDD + j] = q;
                         }
                     });
            if (tid < r) lamr[tid] = Tb[tid * LDD + tid] / (1.0 - Rb[tid * LDD + tid]);
            __syncthreads();
            const double delta = 1e-5 * fmax(fabs(lamr[0]), 1e-300);
            for (int k = tid; k < L * r; k += nt) {   // E_jc in place of T
                const int j = k / r, c = k - j * r;
                const double t = Tb[j * LDD + c], q = Rb[j * LDD + c];
                const double gap = lamr[c] - (j < r ? lamr[j] : lam32[order[j]]);
                Tb[j * LDD + c] = (j != c && fabs(gap) > delta) ? (t + lamr[c] * q) / gap : 0.5 * q;
            }
            __syncthreads();
            each_dot(L * r,   // X + B E into Y
                     [&](int k, int j, int dj, double2& v) {
                         const int i = k / r, c = k - i * r;
                         for (; j < L; j += dj) {
                             const double b = j < r ? X[i * LDD + j] : (double)V32[i * LD32 + order[j]];
                             v.x = fma(b, Tb[j * LDD + c], v.x);
                         }
                     },
                     [&](int k, double2 v) {
                         const int i = k / r, c = k - i * r;
                         Y[i * LDD + c] = X[i * LDD + c] + v.x;
                     });
            for (int k = tid; k < L * r; k += nt) {
                const int i = k / r, c = k - i * r;
                X[i * LDD + c] = Y[i * LDD + c];
            }
            __syncthreads();
        }
        // ---- 3. orthonormalise the active vectors, G = X^T X
        each_dot(r * r,
                 [&](int k, int m, int dm, double2& v) {
                     const int i = k / r, c = k - i * r;
                     if (i <= c)
                         for (; m < L; m += dm) v.x = fma(X[m * LDD + i], X[m * LDD + c], v.x);
                 },
                 [&](int k, double2 v) {
                     const int i = k / r, c = k - i * r;
                     if (i > c) return;
                     Tb[i * LDD + c] = v.x;
                     const double e = v.x - (i == c ? 1.0 : 0.0);
                     if (!(r * e * e <= 1e-16)) atomicMax(&emax, 1);
                 });
        if (emax == 0) {   // X (I - U)
            each_dot(L * r,
                     [&](int k, int j, int dj, double2& v) {
                         const int i = k / r, c = k - i * r;
                         for (; j <= c; j += dj) {
                             const double u = j < c ? Tb[j * LDD + c] : 0.5 * (Tb[c * LDD + c] - 1.0);
                             v.x = fma(X[i * LDD + j], u, v.x);
                         }
                     },
                     [&](int k, double2 v) {
                         const int i = k / r, c = k - i * r;
                         Y[i * LDD + c] = X[i * LDD + c] - v.x;
                     });
            for (int k = tid; k < L * r; k += nt) {
                const int i = k / r, c = k - i * r;
                X[i * LDD + c] = Y[i * LDD + c];
            }
        } else {   // Cholesky QR, right-looking: column j of R eliminates from G and X together
            for (int j = 0; j < r; ++j) {
                if (tid == 0) {
                    const double d = fmax(Tb[j * LDD + j], 1e-30);
                    double y = (double)rsqrtf((float)d);
                    y = fma(0.5 * y, fma(-(d * y), y, 1.0), y);
                    dinv[j] = fma(0.5 * y, fma(-(d * y), y, 1.0), y);
                }
                __syncthreads();
                const double d2 = dinv[j] * dinv[j];
                const int nc = r - 1 - j;
                for (int k = tid; k < (nc + L) * nc; k += nt) {   // rows of G above the diagonal, then rows of X
                    const int i = k / nc, c = j + 1 + k - i * nc;
                    const double f = d2 * Tb[j * LDD + c];
                    if (i < nc) {
                        if (j + 1 + i <= c)
                            Tb[(j + 1 + i) * LDD + c] = fma(-Tb[j * LDD + j + 1 + i], f, Tb[(j + 1 + i) * LDD + c]);
                    } else {
                        X[(i - nc) * LDD + c] = fma(-X[(i - nc) * LDD + j], f, X[(i - nc) * LDD + c]);
                    }
                }
                __syncthreads();
            }
            for (int k = tid; k < L * r; k += nt) {
                const int i = k / r, c = k - i * r;
                X[i * LDD + c] *= dinv[c];
            }
        }
        if (tid < r) {
            const double sig = sqrt(fmax(lamr[tid], 0.0));
            const double c = thr * (w_sv ? w_sv[tid] : 1.0);
            if (sv_out) sv_out[tid] = sig;
            fv[tid] = dual ? ((sig > c) ? c / sig : 1.0) : ((sig > c) ? 1.0 - c / sig : 0.0);
        }
        __syncthreads();
    }
    if (sv_out)
        for (int j = r + tid; j < L; j += nt) sv_out[j] = sqrt(fmax(lam32[order[j]], 0.0));
    // ---- 4. low-rank factor, as in k_eig_mixed
    if (tid == 0) {
        Mf[LR_R] = (double)r;
        Mf[LR_BASE] = dual ? 1.0 : 0.0;
    }
    float* Ff = reinterpret_cast<float*>(Mf + LR_DOUBLES);
    if (tid < r) {
        const double g = dual ? fv[tid] - 1.0 : fv[tid];
        Mf[LR_G + tid] = g;
        Ff[LRF_G + tid] = (float)g;
    }
    for (int k = tid; k < L * r; k += nt) {
        const int i = k / r, c = k - i * r;
        const double x = X[i * LDD + c];
        const float xh = (float)x;
        Mf[LR_X + c * MAX_L_NUC + i] = x;
        Ff[LRF_XH + c * MAX_L_NUC + i] = xh;
        Ff[LRF_XL + c * MAX_L_NUC + i] = (float)(x - (double)xh);
    }
}

size_t eig_mixed_smem() {
    return (size_t)4 * MAX_L_NUC * LD32 * sizeof(float) + (size_t)4 * MAX_L_NUC * LD32 * sizeof(double);
}

// FP64 plans: the whole Gram matrix is diagonalised by the FP64 Jacobi method;
// f and the low-rank factor as in k_eig_mixed (all eigenpairs are FP64-accurate).
__global__ void __launch_bounds__(EIG_T) k_eig_f64(const double* __restrict__ Sg, int L,
                                                  const double* __restrict__ w_sv, double thr, int dual,
                                                  double* __restrict__ Mf, double* __restrict__ sv_out,
                                                  int* __restrict__ r_out) {
    extern __shared__ __align__(16) unsigned char eig_smem[];
    constexpr int SL = MAX_L_NUC * LD32;
    double* A = (double*)eig_smem;
    double* B = A + SL;
    double* V = B + SL;
    double* W = V + SL;
    __shared__ double red[33];
    __shared__ double lam[MAX_L_NUC], fv[MAX_L_NUC];
    __shared__ double2 cs[MAX_L_NUC / 2];
    __shared__ int order[MAX_L_NUC];
    __shared__ unsigned short partner[(MAX_L_NUC - 1) * MAX_L_NUC / 2];
    __shared__ int flag;
    const int tid = threadIdx.x, nt = blockDim.x;
    int n = 2;
    while (n < L) n <<= 1;
    for (int k = tid; k < n * n; k += nt) {
        const int i = k / n, j = k - i * n;
        A[i * LD32 + j] = (i < L && j < L) ? Sg[i * L + j] : 0.0;
        V[i * LD32 + j] = (i == j) ? 1.0 : 0.0;
    }
    __syncthreads();
    jacobi_n<double>(n, A, B, V, W, partner, 1e-17, 1e-18, 1e-16, 40, cs, red, &flag);
    if (tid < L) lam[tid] = A[tid * LD32 + tid];
    __syncthreads();
    if (tid < L) {   // NaN ranks last (the ranks stay a permutation)
        int rk = 0;
        const double li = isnan(lam[tid]) ? -INFINITY : lam[tid];
        for (int j = 0; j < L; ++j) {
            const double lj = isnan(lam[j]) ? -INFINITY : lam[j];
            rk += (lj > li) || (lj == li && j < tid);
        }
        order[rk] = tid;
    }
    __syncthreads();
    if (tid == 0) {
        int r = 0;
        for (int j = 0; j < L; ++j) {
            const double sig = sqrt(fmax(lam[order[j]], 0.0));
            const double c = thr * (w_sv ? w_sv[j] : 1.0);
            double f;
            if (dual) f = (sig > c) ? c / sig : 1.0;
            else f = (sig > c) ? 1.0 - c / sig : 0.0;
            fv[j] = f;
            if (sv_out) sv_out[j] = sig;
            if (sig > c) r = j + 1;
        }
        if (r_out) *r_out = r;
    }
    __syncthreads();
    // low-rank factor over the pairs with sigma > c (f differs from its limit only there)
    __shared__ int r_act;
    if (tid == 0) {
        int r = 0;
        for (int j = 0; j < L; ++j)
            if (sqrt(fmax(lam[order[j]], 0.0)) > thr * (w_sv ? w_sv[j] : 1.0)) r = j + 1;
        r_act = r;
        Mf[LR_R] = (double)r;
        Mf[LR_BASE] = dual ? 1.0 : 0.0;
    }
    __syncthreads();
    const int r = r_act;
    if (tid < r) Mf[LR_G + tid] = dual ? fv[tid] - 1.0 : fv[tid];
    for (int k = tid; k < L * r; k += nt) {
        const int i = k / r, c = k - i * r;
        Mf[LR_X + c * MAX_L_NUC + i] = V[i * LD32 + order[c]];
    }
}

hs_status eig_f64_launch(const double* S, int L, const double* w_sv, double thr, int dual, double* Mf,
                         double* sv_out, int* r_out, cudaStream_t s) {
    const size_t sm = (size_t)4 * MAX_L_NUC * LD32 * sizeof(double);
    // as many threads as a round has 2 x 2 blocks (n^2 / 4, n the padded size): small matrices
    // are bound by the barriers and block sums of a round (L = 6: one warp instead of 32)
    int n = 2;
    while (n < L) n <<= 1;
    const int threads = std::max(n * n / 4, 64) > EIG_T ? EIG_T : std::max(n * n / 4, 64);
    k_eig_f64<<<1, threads, sm, s>>>(S, L, w_sv, thr, dual, Mf, sv_out, r_out);
    HS_CHECK_LAUNCH();
    return HS_OK;
}

hs_status eig_init() {
    static bool done = false;
    if (done) return HS_OK;
    HS_CHECK_CUDA(cudaFuncSetAttribute(k_eig_mixed, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)eig_mixed_smem()));
    HS_CHECK_CUDA(cudaFuncSetAttribute(k_eig_cold<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EIG_COLD_SMEM));
    HS_CHECK_CUDA(cudaFuncSetAttribute(k_eig_cold<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EIG_COLD_SMEM));
    HS_CHECK_CUDA(cudaFuncSetAttribute(k_eig_cold<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EIG_COLD_SMEM));
    HS_CHECK_CUDA(cudaFuncSetAttribute(k_eig_cold<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EIG_COLD_SMEM));
    HS_CHECK_CUDA(cudaFuncSetAttribute(k_eig_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(4 * MAX_L_NUC * LD32 * sizeof(double))));
    done = true;
    return HS_OK;
}

hs_status eig_mixed_launch(const double* S, int L, const double* w_sv, double thr, int dual,
                           double* Mf, double* sv_out, float* warm, int* r_out, cudaStream_t s) {
#define HS_COLD(N) k_eig_cold<N><<<1, EIG_COLD_T, EIG_COLD_SMEM, s>>>(S, L, w_sv, thr, dual, Mf, sv_out, r_out)
    if (warm) k_eig_mixed<<<1, EIG_T, eig_mixed_smem(), s>>>(S, L, w_sv, thr, dual, Mf, sv_out, warm, r_out);
    else if (L <= 4)   // a round or two: 44.2 us against 45.2 at L = 2
        k_eig_mixed<<<1, EIG_T, eig_mixed_smem(), s>>>(S, L, w_sv, thr, dual, Mf, sv_out, nullptr, r_out);
    else if (L <= 8) HS_COLD(8);
    else if (L <= 16) HS_COLD(16);
    else if (L <= 32) HS_COLD(32);
    else HS_COLD(64);
#undef HS_COLD
    HS_CHECK_LAUNCH();
    return HS_OK;
}

}  // namespace hs
