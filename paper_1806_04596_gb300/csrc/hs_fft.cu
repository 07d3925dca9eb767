// Batched 2-D FFT of the oversampled grid with the zero-padding / scaling Z
// fused into the first pass and the crop / scale / real part of Z^T fused
// into the last pass (Sec. 2.1: Phi_l = Theta_l G_l F Z).
//
// The image is real, so its spectrum is Hermitian, F(-k) = conj F(k), and only
// the half plane 0 <= kx <= Kx/2 is ever formed. The plan mirrors every
// visibility with u < 0 to (-u, -v) (its value is conjugated: G_l row for row
// the same weights on the mirrored cells), so windows reach only columns
// kx = -3 .. Kx/2 + 4: Kc = Kx/2 + 8 stored columns, column c holding kx = c - 3,
// on a grid of pitch Kw (Kc rounded up to whole gridding strips).
//   Forward Phi:  X (real) --rows, r2c--> tmp (ny x Kc) --cols--> grid (Ky x Kw)
//   Adjoint:      grid --cols, inverse, keep ny rows--> tmp --rows, c2r, crop--> X
// Row passes are complex transforms of N = Kx/2 = nx points over pixel pairs
// (z_m = x_2m + i x_2m+1); the split into the spectrum of the real row, with
// the 7 mirrored columns around it, follows the last pass, and the adjoint's
// first pass folds those columns back (Re of the sum over the half plane is the
// sum over the Hermitian whole). Only the ny image rows are ever transformed
// along x: the other Ky - ny rows of Z x are zero in the forward direction and
// discarded by Z^T in the adjoint. Against the whole plane this halves the
// grid, the intermediate and the transforms.
//
// Each CTA transforms G lines held in shared memory with a self-sorting Stockham
// schedule: radix-8 passes, one radix-4 or radix-2 pass when log2 is not a
// multiple of 3, then one radix-3 or radix-5 pass for lines of 3 2^a or 5 2^a.
// Every thread keeps its E operands of a pass in registers (8, 24 or 40), so
// one copy of the lines suffices. The first pass loads straight from global
// memory (padding, scaling: of its 8 operands only 4 are nonzero), the last
// stores straight to global memory (crop). Line element k sits at
// k + k/8 in shared memory: the radix-8 stores of a pass, 8 elements apart, then
// fall in distinct banks (unpadded they met 8 ways in the row passes).
#include <algorithm>

#include "hs_device.cuh"
#include "hs_internal.h"

namespace hs {

enum FftMode { ROW_FWD = 0, COL_FWD = 1, COL_INV = 2, ROW_INV = 3 };

template <typename R> struct FftArgs {
    const void* in;
    void* out;
    const Cx<R>* tw;   // exp(-2 pi i m / K): K = N (columns), K = 2 N (rows)
    const R* cxs;      // Z scale along x (nx)
    const R* cys;      // Z scale along y (ny)
    int N;             // points of a line: Ky (columns), nx (rows)
    int lg2;           // log2 of N's power-of-two part
    int lgG;           // log2 of the lines per CTA
    int nx, ny, Ky, Kc, Kw;
    int vec;           // the image is aligned for pixel-pair accesses
    const int4* rng;   // cells reached, per channel
};

template <typename R> __device__ __forceinline__ Cx<R> twiddle(const Cx<R>* tw, int m, int dir) {
    Cx<R> t = tw[m];
    if (dir > 0) t.y = -t.y;
    return t;
}

__device__ __forceinline__ constexpr int lpad(int k) { return k + (k >> 3); }

// 3- and 5-point DFTs with kernel exp(DIR 2 pi i q r / n), in place.
template <typename R, int DIR> __device__ __forceinline__ void dft3(Cx<R>* a) {
    typedef Cx<R> CT;
    const R s = (R)(DIR * 0.86602540378443864676);
    const CT t1 = cadd(a[1], a[2]), t2 = csub(a[1], a[2]);
    const CT m = cx<R>(fma((R)-0.5, t1.x, a[0].x), fma((R)-0.5, t1.y, a[0].y));
    a[0] = cadd(a[0], t1);
    a[1] = cx<R>(fma(-s, t2.y, m.x), fma(s, t2.x, m.y));
    a[2] = cx<R>(fma(s, t2.y, m.x), fma(-s, t2.x, m.y));
}
template <typename R, int DIR> __device__ __forceinline__ void dft5(Cx<R>* a) {
    typedef Cx<R> CT;
    const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;
    const R s1 = (R)(DIR * 0.95105651629515357212), s2 = (R)(DIR * 0.58778525229247312917);
    const CT t1 = cadd(a[1], a[4]), t2 = cadd(a[2], a[3]), t3 = csub(a[1], a[4]), t4 = csub(a[2], a[3]);
    const CT m1 = cx<R>(fma(c2, t2.x, fma(c1, t1.x, a[0].x)), fma(c2, t2.y, fma(c1, t1.y, a[0].y)));
    const CT m2 = cx<R>(fma(c1, t2.x, fma(c2, t1.x, a[0].x)), fma(c1, t2.y, fma(c2, t1.y, a[0].y)));
    const CT n1 = cx<R>(fma(s2, t4.x, s1 * t3.x), fma(s2, t4.y, s1 * t3.y));
    const CT n2 = cx<R>(fma(-s1, t4.x, s2 * t3.x), fma(-s1, t4.y, s2 * t3.y));
    a[0] = cadd(a[0], cadd(t1, t2));
    a[1] = cx<R>(m1.x - n1.y, m1.y + n1.x);
    a[4] = cx<R>(m1.x + n1.y, m1.y - n1.x);
    a[2] = cx<R>(m2.x - n2.y, m2.y + n2.x);
    a[3] = cx<R>(m2.x + n2.y, m2.y - n2.x);
}

// First-pass loads: operand r (of 8) of butterfly j of a line, element k = j + r N/8.
// The image occupies k < N/4 and k >= 3 N/4 (of a line or of its pixel pairs),
// so operands 2 .. 5 are zero in the forward modes.
template <typename R, int MODE>
__device__ __forceinline__ Cx<R> fft_load(const FftArgs<R>& a, const int4& rg, int la, int lb, int N, int k, int r) {
    typedef Cx<R> CT;
    if (MODE == ROW_FWD) {   // Z: pad and scale; pixels 2 m + N/2 (mod 2 N) of row lb
        if (r >= 2 && r < 6) return cx<R>(0, 0);
        const int ix = r < 2 ? 2 * k + (N >> 1) : 2 * k - 3 * (N >> 1);
        const R* x = (const R*)a.in + ((int64_t)la * a.ny + lb) * a.nx + ix;
        const R cy = a.cys[lb];
        const CT s = *reinterpret_cast<const CT*>(a.cxs + ix);
        CT v;
        if (a.vec) v = *reinterpret_cast<const CT*>(x);
        else v = cx<R>(x[0], x[1]);
        return cx<R>(cy * s.x * v.x, cy * s.y * v.y);
    } else if (MODE == COL_FWD) {   // only the ny image rows are nonzero
        if (r >= 2 && r < 6) return cx<R>(0, 0);
        const int iy = r < 2 ? k + (N >> 2) : k - 3 * (N >> 2);
        return ((const CT*)a.in)[((int64_t)la * a.ny + iy) * a.Kc + lb];
    } else if (MODE == COL_INV) {
        if (!row_reached(rg, k)) return cx<R>(0, 0);
        return ((const CT*)a.in)[((int64_t)la * a.Ky + k) * a.Kw + lb];
    } else {
        // ROW_INV: fold the mirrored columns (C(k), 0 <= k <= N), then the complex input
        // of the real inverse, ((A + B) + i w (A - B)) / 2 with A = C(k), B = conj C(N - k),
        // w = exp(2 pi i k / 2N) (both ends real and counted twice at k = 0)
        const CT* T = (const CT*)a.in + ((int64_t)la * a.ny + lb) * a.Kc + 3;
        auto at = [&](int q) { return q + 3 < rg.x ? T[q] : cx<R>(0, 0); };   // rg.y is the pitch here
        auto folded = [&](int q) {
            CT v = at(q);
            if (q <= 3) {
                const CT m = at(-q);
                v.x += m.x;
                v.y -= m.y;
            }
            if (q >= N - 4) {
                const CT m = at(2 * N - q);
                v.x += m.x;
                v.y -= m.y;
            }
            return v;
        };
        if (k == 0) {
            const R p = at(0).x, q = at(N).x;
            return cx<R>(p + q, p - q);
        }
        const CT A = folded(k);
        const CT C = folded(N - k);
        const CT d = cx<R>(A.x - C.x, A.y + C.y);
        const CT w = twiddle<R>(a.tw, k, 1);
        const CT e = cmul(w, d);   // i e = (-e.y, e.x)
        return cx<R>((R)0.5 * ((A.x + C.x) - e.y), (R)0.5 * ((A.y - C.y) + e.x));
    }
}

// Last-pass stores of element k (known to lie inside the crop in the inverse modes).
template <typename R, int MODE>
__device__ __forceinline__ void fft_store(const FftArgs<R>& a, const int4& rg, int la, int lb, int N, int k, bool upper,
                                          Cx<R> v) {
    typedef Cx<R> CT;
    if (MODE == COL_FWD) {
        if (row_reached(rg, k)) ((CT*)a.out)[((int64_t)la * a.Ky + k) * a.Kw + lb] = v;
    } else if (MODE == COL_INV) {   // keep the ny image rows
        const int iy = upper ? k - 3 * (N >> 2) : k + (N >> 2);
        ((CT*)a.out)[((int64_t)la * a.ny + iy) * a.Kc + lb] = v;
    } else if (MODE == ROW_INV) {   // crop, scale: pixels 2 k + N/2 (mod 2 N)
        const int ix = upper ? 2 * k - 3 * (N >> 1) : 2 * k + (N >> 1);
        R* x = (R*)a.out + ((int64_t)la * a.ny + lb) * a.nx + ix;
        const R cy = a.cys[lb];
        const CT s = *reinterpret_cast<const CT*>(a.cxs + ix);
        v = cx<R>(cy * s.x * v.x, cy * s.y * v.y);
        if (a.vec) {
            *reinterpret_cast<CT*>(x) = v;
        } else {
            x[0] = v.x;
            x[1] = v.y;
        }
    }
}

// Operands per thread: several butterflies per pass, so that long lines come G
// to a CTA within 512 threads (NREP) and the odd radix divides them.
template <int ODD, int NREP> __host__ __device__ constexpr int fft_elems() {
    return ODD == 1 ? 8 * NREP : (ODD == 3 ? 24 : 40);
}

// One Stockham pass of radix RAD with sub-transform length 2^lgNs over the
// CTA's G lines; LG > 0 fixes N = ODD 2^LG at compile time.
template <typename R, int DIR, int MODE, int RAD, int LG, int ODD, int NREP, int LGG>
__device__ __forceinline__ void fft_pass(const FftArgs<R>& a, const int4& rg, Cx<R>* sm, int lgNs, bool first,
                                         bool last, int la, int line0) {
    typedef Cx<R> CT;
    constexpr bool COLS = (MODE == COL_FWD || MODE == COL_INV);
    constexpr int E = fft_elems<ODD, NREP>();
    constexpr int PER = E / RAD;
    const int N = LG > 0 ? (ODD << LG) : a.N;
    const int nb = N / RAD;
    const int nthr = blockDim.x, tid = threadIdx.x;
    const int LD = N + (N >> 3);
    const bool to_global = last && MODE != ROW_FWD;
    CT v[E];
    int gs[PER], js[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int w = tid + i * nthr;
        const int g = COLS ? (w & ((1 << LGG) - 1)) : w / nb;
        const int j = COLS ? (w >> LGG) : w - g * nb;
        gs[i] = g;
        js[i] = j;
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
            const int k = j + r * nb;
            v[i * RAD + r] = first ? fft_load<R, MODE>(a, rg, la, line0 + g, N, k, r)
                                   : sm[COLS ? ((lpad(k) << LGG) + g) : (g * LD + lpad(k))];
        }
    }
    if (!first) __syncthreads();   // every read of this pass precedes any write
    constexpr int TS = COLS ? 1 : 2;   // table points per N-point root
    const int tstep = TS * (N >> lgNs) / RAD;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int j = js[i], g = gs[i];
        const int kk = j & ((1 << lgNs) - 1);
        CT* u = v + i * RAD;
        if (lgNs > 0) {   // the first pass has unit twiddles
            if (RAD == 8) {
                // w^1, w^2, w^4 from the table, the others as products (one rounding each)
                CT t[8];
                t[1] = a.tw[kk * tstep];
                t[2] = a.tw[2 * kk * tstep];
                t[4] = a.tw[4 * kk * tstep];
                t[3] = cmul(t[1], t[2]);
                t[5] = cmul(t[1], t[4]);
                t[6] = cmul(t[2], t[4]);
                t[7] = cmul(t[3], t[4]);
#pragma unroll
                for (int r = 1; r < 8; ++r) {
                    if (DIR > 0) t[r].y = -t[r].y;
                    u[r] = cmul(u[r], t[r]);
                }
            } else {
#pragma unroll
                for (int r = 1; r < RAD; ++r) u[r] = cmul(u[r], twiddle<R>(a.tw, r * kk * tstep, DIR));
            }
        }
        if (RAD == 8) {
            dft8<R, DIR>(u);
        } else if (RAD == 4) {
            dft4<DIR>(u[0], u[1], u[2], u[3]);
        } else if (RAD == 2) {
            const CT t0 = cadd(u[0], u[1]);
            u[1] = csub(u[0], u[1]);
            u[0] = t0;
        } else if (RAD == 3) {
            dft3<R, DIR>(u);
        } else {
            dft5<R, DIR>(u);
        }
        const int base = (j >> lgNs) * (RAD << lgNs) + kk;
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
            const int k = base + (r << lgNs);
            if (!to_global) {
                sm[COLS ? ((lpad(k) << LGG) + g) : (g * LD + lpad(k))] = u[r];
            } else if (MODE == COL_FWD) {
                fft_store<R, MODE>(a, rg, la, line0 + g, N, k, false, u[r]);
            } else if (RAD == 8 || RAD == 4) {   // k = j + r N / RAD: the kept quarters are whole operands
                if (r < RAD / 4) fft_store<R, MODE>(a, rg, la, line0 + g, N, k, false, u[r]);
                else if (r >= RAD - RAD / 4) fft_store<R, MODE>(a, rg, la, line0 + g, N, k, true, u[r]);
            } else {
                if (k < (N >> 2)) fft_store<R, MODE>(a, rg, la, line0 + g, N, k, false, u[r]);
                else if (k >= 3 * (N >> 2)) fft_store<R, MODE>(a, rg, la, line0 + g, N, k, true, u[r]);
            }
        }
    }
    if (!to_global) __syncthreads();
}

// Spectrum of the real rows from the N-point transforms Z of their pixel pairs:
// X(k) = (Z(k) + conj Z(N - k)) / 2 + exp(-2 pi i k / 2N) (Z(k) - conj Z(N - k)) / 2i for
// k = 0 .. N, and X(-k) = conj X(k) in the mirrored columns at both ends.
template <typename R, int ODD, int NREP>
__device__ __forceinline__ void row_split(const FftArgs<R>& a, const int4& rg, const Cx<R>* sm, int N, int la, int line0) {
    typedef Cx<R> CT;
    const int tpr = N / fft_elems<ODD, NREP>();   // threads per row
    const int g = threadIdx.x / tpr, t = threadIdx.x - g * tpr;
    const CT* z = sm + g * (N + (N >> 3));
    CT* out = (CT*)a.out + ((int64_t)la * a.ny + line0 + g) * a.Kc;
    for (int c = t; c < N + 8; c += tpr) {
        if (c >= rg.x) break;
        const int kx = c - 3;
        const bool mir = kx < 0 || kx > N;
        const int k = kx < 0 ? -kx : (kx > N ? 2 * N - kx : kx);
        const CT p = z[k == N ? 0 : lpad(k)], q = z[k == 0 ? 0 : lpad(N - k)];
        const CT e = cx<R>((R)0.5 * (p.x + q.x), (R)0.5 * (p.y - q.y));
        const CT o = cx<R>((R)0.5 * (p.y + q.y), (R)-0.5 * (p.x - q.x));
        const CT w = a.tw[k];
        CT x = cx<R>(e.x + (w.x * o.x - w.y * o.y), e.y + (w.x * o.y + w.y * o.x));
        if (mir) x.y = -x.y;
        out[c] = x;
    }
}

// Registers: column lines of 512 (FP32) come 512 threads to a CTA, three CTAs to an SM.
template <typename R, int ODD, int NREP> __host__ __device__ constexpr int fft_max_threads() {
    return (ODD == 5 || (ODD == 3 && sizeof(R) == 8)) ? 256 : 512;
}
template <typename R, int ODD, int NREP> __host__ __device__ constexpr int fft_min_ctas() {
    return ODD == 1 ? (NREP > 2 ? 1 : (sizeof(R) == 4 ? (NREP == 2 ? 2 : 3) : (NREP == 2 ? 1 : 2))) : 1;
}

// DIR = -1: forward transform (exp(-2 pi i kn / K)); DIR = +1: unnormalised inverse.
// LG > 0: lines of ODD 2^LG points fixed at compile time (the pass schedule and
// every index computation fold to constants); 0: from the arguments. Column
// modes take 2^LGG columns per CTA, row modes the number of rows in a.lgG.
template <typename R, int DIR, int MODE, int LG, int ODD, int NREP, int LGG>
__global__ void __launch_bounds__(fft_max_threads<R, ODD, NREP>(), fft_min_ctas<R, ODD, NREP>())
    k_fft(const FftArgs<R> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<R>* sm = reinterpret_cast<Cx<R>*>(smem_raw);
    constexpr bool COLS = (MODE == COL_FWD || MODE == COL_INV);
    const int la = blockIdx.y;
    const int line0 = COLS ? (blockIdx.x << LGG) : (blockIdx.x << a.lgG);
    const int4 rg = a.rng[la];
    if (COLS && !col_reached(rg, line0)) return;   // the whole group (8 columns divide the bounds)
#define HS_PASS(RAD, NS, FIRST, LAST) \
    fft_pass<R, DIR, MODE, RAD, LG, ODD, NREP, LGG>(a, rg, sm, NS, FIRST, LAST, la, line0)
    if constexpr (LG > 0) {
        constexpr int N8 = LG / 3, REM = LG % 3;
#pragma unroll
        for (int p = 0; p < N8; ++p) HS_PASS(8, 3 * p, p == 0, ODD == 1 && REM == 0 && p == N8 - 1);
        if constexpr (REM == 2) HS_PASS(4, 3 * N8, false, ODD == 1);
        if constexpr (REM == 1) HS_PASS(2, 3 * N8, false, ODD == 1);
    } else {
        const int n8 = a.lg2 / 3, rem = a.lg2 - 3 * n8;
        HS_PASS(8, 0, true, ODD == 1 && rem == 0 && n8 == 1);
        for (int p = 1; p < n8; ++p) HS_PASS(8, 3 * p, false, ODD == 1 && rem == 0 && p == n8 - 1);
        if (rem == 2) HS_PASS(4, 3 * n8, false, ODD == 1);
        if (rem == 1) HS_PASS(2, 3 * n8, false, ODD == 1);
    }
    if constexpr (ODD == 3) HS_PASS(3, LG > 0 ? LG : a.lg2, false, true);
    if constexpr (ODD == 5) HS_PASS(5, LG > 0 ? LG : a.lg2, false, true);
#undef HS_PASS
    if constexpr (MODE == ROW_FWD) row_split<R, ODD, NREP>(a, rg, sm, LG > 0 ? (ODD << LG) : a.N, la, line0);
}

// ---------------------------------------------------------------- launches
static int64_t g_l2_bytes = 0;
constexpr int FFT_SMEM_MAX = 200 * 1024;

template <typename R, int DIR, int MODE, int LG, int ODD, int NREP, int LGG>
static hs_status run_fft(const FftArgs<R>& a, dim3 grid, int threads, size_t smem, cudaStream_t s) {
    static const cudaError_t opted = cudaFuncSetAttribute(
        k_fft<R, DIR, MODE, LG, ODD, NREP, LGG>, cudaFuncAttributeMaxDynamicSharedMemorySize, FFT_SMEM_MAX);
    HS_CHECK_CUDA(opted);
    if (grid.y == 0) return HS_OK;   // set-up only (fft_prepare)
    k_fft<R, DIR, MODE, LG, ODD, NREP, LGG><<<grid, threads, smem, s>>>(a);
    HS_CHECK_LAUNCH();
    return HS_OK;
}

// nl channels from l0, starting at in / out (a channel range of the plan's buffers).
template <typename R, int DIR, int MODE>
static hs_status launch_fft(Plan* p, const void* in, void* out, int l0, int nl, cudaStream_t s) {
    constexpr bool cols = (MODE == COL_FWD || MODE == COL_INV);
    FftArgs<R> a{};
    a.in = in;
    a.out = out;
    a.nx = p->g.nx;
    a.ny = p->g.ny;
    a.Ky = p->g.Ky;
    a.Kc = p->g.Kc;
    a.Kw = p->g.Kw;
    a.cxs = (const R*)p->cxs;
    a.cys = (const R*)p->cys;
    a.tw = (const Cx<R>*)(cols ? p->twy : p->twx);
    a.N = cols ? p->g.Ky : p->g.nx;
    const void* img = MODE == ROW_FWD ? in : out;
    a.rng = p->rng + l0;
    a.vec = ((uintptr_t)img % sizeof(Cx<R>)) == 0;
    int odd = 1;
    for (int r : {3, 5})
        if (a.N % r == 0) odd = r;
    a.lg2 = 0;
    while ((odd << a.lg2) < a.N) ++a.lg2;
    if ((odd << a.lg2) != a.N || a.lg2 < 3)
        return fail(HS_ERR_ARG, "FFT: line length %d is not r 2^m with r in {1, 3, 5}", a.N);
    const int tpl = a.N / (odd == 1 ? 8 : (odd == 3 ? 24 : 40));   // threads per line (one butterfly set each)
    const size_t line = (size_t)(a.N + a.N / 8) * sizeof(Cx<R>);
    if constexpr (cols) {
        // 64-byte segments of a row (8 columns FP32, 4 FP64) where the lines take at most
        // 80 KB (two CTAs per SM), else 32-byte segments (whole sectors)
        const int lgg = (line << (sizeof(R) == 4 ? 3 : 2)) <= (size_t)80 * 1024 ? (sizeof(R) == 4 ? 3 : 2)
                                                                               : (sizeof(R) == 4 ? 2 : 1);
        a.lgG = lgg;
        const size_t smem = line << lgg;
        if (smem > (size_t)FFT_SMEM_MAX) return fail(HS_ERR_ARG, "FFT: line length %d too long", a.N);
        const int nrep = odd == 1 ? std::max(1, (tpl << lgg) / 512) : 1;
        const int threads = (tpl << lgg) / nrep;
        const dim3 grid(a.Kc >> lgg, nl);
#define HS_FFT(LG_, ODD_, NREP_, LGG_) \
    if (odd == ODD_ && lgg == LGG_ && nrep == NREP_ && (LG_ == 0 || a.lg2 == LG_)) \
        return run_fft<R, DIR, MODE, LG_, ODD_, NREP_, LGG_>(a, grid, threads, smem, s);
        if constexpr (sizeof(R) == 4) {
            HS_FFT(7, 1, 1, 3)
            HS_FFT(8, 1, 1, 3)
            HS_FFT(9, 1, 1, 3)
            HS_FFT(10, 1, 2, 3)
            HS_FFT(11, 1, 2, 2)
            HS_FFT(12, 1, 4, 2)
            HS_FFT(7, 3, 1, 3)
            HS_FFT(8, 3, 1, 3)
            HS_FFT(7, 5, 1, 3)
            HS_FFT(8, 5, 1, 2)
            HS_FFT(0, 1, 1, 3)
            HS_FFT(0, 3, 1, 3)
            HS_FFT(0, 5, 1, 3)
            HS_FFT(0, 3, 1, 2)
            HS_FFT(0, 5, 1, 2)
        } else {
            HS_FFT(8, 1, 1, 2)
            HS_FFT(9, 1, 1, 2)
            HS_FFT(12, 1, 2, 1)
            HS_FFT(0, 1, 1, 2)
            HS_FFT(0, 1, 1, 1)
            HS_FFT(0, 3, 1, 2)
            HS_FFT(0, 5, 1, 2)
            HS_FFT(0, 3, 1, 1)
            HS_FFT(0, 5, 1, 1)
        }
    } else {
        // 256 threads per CTA, fewer while the rows would not give every SM two CTAs
        int lgG = 0;
        while ((tpl << (lgG + 1)) <= 256 && (p->g.ny % (2 << lgG)) == 0) ++lgG;
        while (lgG > 0 && (tpl << lgG) > 32 && (int64_t)p->g.L * (p->g.ny >> lgG) < 2 * 152) --lgG;
        a.lgG = lgG;
        const size_t smem = line << lgG;
        const int threads = tpl << lgG;
        const dim3 grid(p->g.ny >> lgG, nl);
        constexpr int lgg = 0, nrep = 1;
        if constexpr (sizeof(R) == 4) {
            HS_FFT(6, 1, 1, 0)
            HS_FFT(7, 1, 1, 0)
            HS_FFT(8, 1, 1, 0)
            HS_FFT(9, 1, 1, 0)
            HS_FFT(10, 1, 1, 0)
            HS_FFT(11, 1, 1, 0)
            HS_FFT(7, 3, 1, 0)
            HS_FFT(8, 3, 1, 0)
            HS_FFT(7, 5, 1, 0)
            HS_FFT(8, 5, 1, 0)
        } else {
            HS_FFT(7, 1, 1, 0)
            HS_FFT(8, 1, 1, 0)
        }
        HS_FFT(0, 1, 1, 0)
        HS_FFT(0, 3, 1, 0)
        HS_FFT(0, 5, 1, 0)
    }
#undef HS_FFT
    return fail(HS_ERR_ARG, "FFT: no kernel for lines of %d points", a.N);
}

// Size of the L2, for the chunk rule below (at plan creation).
hs_status fft_init() {
    static bool done = false;
    if (done) return HS_OK;
    int dev = 0, l2 = 0;
    HS_CHECK_CUDA(cudaGetDevice(&dev));
    HS_CHECK_CUDA(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev));
    g_l2_bytes = l2;
    done = true;
    return HS_OK;
}

// Opts the kernels of this plan's line lengths into their shared memory, so that
// no first launch inside a stream capture has to.
template <typename R> static hs_status fft_prepare_t(Plan* p) {
    HS_TRY((launch_fft<R, -1, ROW_FWD>(p, nullptr, nullptr, 0, 0, nullptr)));
    HS_TRY((launch_fft<R, -1, COL_FWD>(p, nullptr, nullptr, 0, 0, nullptr)));
    HS_TRY((launch_fft<R, 1, COL_INV>(p, nullptr, nullptr, 0, 0, nullptr)));
    return launch_fft<R, 1, ROW_INV>(p, nullptr, nullptr, 0, 0, nullptr);
}
hs_status fft_prepare(Plan* p) {
    if (!p->half) return plane_fft_init();
    return p->prec == HS_F32 ? fft_prepare_t<float>(p) : fft_prepare_t<double>(p);
}

hs_status fft_forward(Plan* p, const void* X, cudaStream_t s) {
    if (!p->half) return plane_fft_forward(p, X, s);
    const int L = p->g.L;
    if (p->prec == HS_F32) {
        HS_TRY((launch_fft<float, -1, ROW_FWD>(p, X, p->tmp, 0, L, s)));
        HS_TRY((launch_fft<float, -1, COL_FWD>(p, p->tmp, p->grid, 0, L, s)));
    } else {
        HS_TRY((launch_fft<double, -1, ROW_FWD>(p, X, p->tmp, 0, L, s)));
        HS_TRY((launch_fft<double, -1, COL_FWD>(p, p->tmp, p->grid, 0, L, s)));
    }
    return HS_OK;
}

// Channels per adjoint chunk that keep a chunk's traffic within a quarter of the
// L2: the column pass of a chunk streams its half-plane grid (Ky Kw cells per
// channel) and writes the ny x Kc intermediate, which the row pass reads right after, so the intermediate can stay on chip. The row pass of chunk c runs on
// the plan's side stream, overlapping the column pass of chunk c + 1; the plan's
// autotuner keeps the chunked form only where it measures faster
// (p->fft_adj_chunk, default all channels).
int fft_adjoint_chunk(const Plan* p) {
    const int64_t per = ((int64_t)p->g.Ky * p->g.Kw + (int64_t)p->g.ny * p->g.Kc) * (int64_t)p->csize();
    const int64_t budget = g_l2_bytes > 0 ? g_l2_bytes / 4 : ((int64_t)16 << 20);
    return (int)std::max<int64_t>(1, std::min<int64_t>(p->g.L, budget / std::max<int64_t>(per, 1)));
}

template <typename R> static hs_status fft_adjoint_t(Plan* p, R* X, cudaStream_t s) {
    const int L = p->g.L, C = std::max(1, std::min(L, p->fft_adj_chunk > 0 ? p->fft_adj_chunk : L));
    const int64_t gch = (int64_t)p->g.Ky * p->g.Kw, tch = (int64_t)p->g.ny * p->g.Kc, xch = p->N();
    const bool side = C < L && p->fft_side != nullptr;
    cudaStream_t s2 = side ? p->fft_side : s;
    for (int l0 = 0; l0 < L; l0 += C) {
        const int n = std::min(C, L - l0);
        const Cx<R>* g = (const Cx<R>*)p->grid + l0 * gch;
        Cx<R>* t = (Cx<R>*)p->tmp + l0 * tch;
        if (p->half) HS_TRY((launch_fft<R, 1, COL_INV>(p, g, t, l0, n, s)));
        else HS_TRY(plane_fft_cols_inv(p, g, t, l0, n, s));
        if (side) {
            HS_CHECK_CUDA(cudaEventRecord(p->fft_ev_col, s));
            HS_CHECK_CUDA(cudaStreamWaitEvent(s2, p->fft_ev_col, 0));
        }
        if (p->half) HS_TRY((launch_fft<R, 1, ROW_INV>(p, t, X + l0 * xch, l0, n, s2)));
        else HS_TRY(plane_fft_rows_inv(p, t, X + l0 * xch, l0, n, s2));
    }
    if (side) {
        HS_CHECK_CUDA(cudaEventRecord(p->fft_ev_join, s2));
        HS_CHECK_CUDA(cudaStreamWaitEvent(s, p->fft_ev_join, 0));
    }
    return HS_OK;
}

hs_status fft_adjoint(Plan* p, void* X, cudaStream_t s) {
    if (p->prec == HS_F32) return fft_adjoint_t<float>(p, (float*)X, s);
    return fft_adjoint_t<double>(p, (double*)X, s);
}

}  // namespace hs
