// k_radial.cu -- the muffin-tin side of the mixed product basis and of the
// Coulomb matrix, from the LAPW radial functions of an atom (Sec. III.B-C).
//
// For every L, in FP64:
//   - the products u_lp u_l'p' (lp <= l'p', |l - l'| <= L <= l + l'), each
//     normalised, and for L = 0 the constant function, projected out of them;
//   - the overlap matrix of the products and its largest eigenpairs;
//     eigenfunctions with eigenvalue above the threshold are linearly
//     independent, and the P largest of them (L = 0: P - 1 after the constant)
//     become the functions M_aLP, orthonormal, each with its largest eigenvector
//     component positive;
//   - the multipole moments mu_aLP = int M r^(L+2) dr (Sec. III.C), the radial
//     integrals R = int M u_lp u_l'p' r^2 dr, and the on-site Coulomb integrals
//     C_PP' = 4 pi/(2L+1) int int M_P(r) M_P'(r') r<^L/r>^(L+1) r^2 r'^2 dr dr'.
// A multipole-free combination of the M_aLP makes no potential outside its
// sphere, so every Coulomb matrix element with a mu = 0 function of the
// transform of Sec. III.C is one of these on-site integrals, the same for every
// q: launch_onsite_fill writes them into v_t (Fig. 1's channel blocks).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "hfx_internal.cuh"

namespace hfx {

namespace {

constexpr double kPi = 3.14159265358979323846;

// GB300's FP64 pipe does about two FMAs per cycle and SM, so what bounds this
// file is FP64 issue and the latency of serial chains, not memory.  The products
// and the integrals are spread over the chip; only the eigenproblem stays in one
// block per L, and there only the P wanted eigenpairs are computed (Householder
// tridiagonal form, bisection, inverse iteration) instead of all of them by
// Jacobi rotations, whose n^2/2 rotations per sweep are a serial chain.
// One atom, lmax = Lmax = 4, P = 3, 600 points: 189 ms with one block per L for
// everything (170 ms of it pow() in the on-site double integral), 0.52 ms now (copies included).

constexpr int RP_THREADS = 128;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// sum over the block (a multiple of 32 threads, at most 1024); red: 33 doubles
__device__ double block_sum(double v, double *red) {
    v = warp_sum(v);
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < (blockDim.x + 31) / 32 ? red[threadIdx.x] : 0.0;
        t = warp_sum(t);
        if (threadIdx.x == 0) red[32] = t;
    }
    __syncthreads();
    v = red[32];
    __syncthreads();
    return v;
}

// The products u_lp u_l'p' of every L, normalised (one block each), and for L = 0
// with the constant function projected out.  A product that vanishes identically
// becomes a zero row: its eigenvalue is 0, below every threshold.
__global__ void __launch_bounds__(RP_THREADS) radial_products_kernel(int n_r, const double *__restrict__ r,
                                                                     const double *__restrict__ w,
                                                                     const double *__restrict__ u,
                                                                     const int2 *__restrict__ prod,
                                                                     const int *__restrict__ ncL, int maxc,
                                                                     double *__restrict__ f) {
    const int c = blockIdx.x, L = blockIdx.y, tid = threadIdx.x;
    if (c >= ncL[L]) return;
    __shared__ double red[33];
    const int2 ab = prod[L * maxc + c];
    const double *ua = u + (size_t)ab.x * n_r, *ub = u + (size_t)ab.y * n_r;
    double *fc = f + ((size_t)L * maxc + c) * n_r;
    double s = 0.0, s1 = 0.0, s0 = 0.0;
    for (int i = tid; i < n_r; i += RP_THREADS) {
        const double v = ua[i] * ub[i], wr = w[i] * r[i] * r[i];
        s += wr * v * v;
        if (L == 0) {
            s1 += wr * v;
            s0 += wr;
        }
    }
    s = block_sum(s, red);
    const double inv = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
    double sub = 0.0;
    if (L == 0) {   // <const|f> const, const = 1/sqrt(int r^2 dr)
        s1 = block_sum(s1, red);
        s0 = block_sum(s0, red);
        sub = inv * s1 / s0;
    }
    for (int i = tid; i < n_r; i += RP_THREADS) fc[i] = s > 0.0 ? inv * (ua[i] * ub[i]) - sub : 0.0;
}

// Partial overlaps O_z[L][a][b] (a >= b) of the products over one of OV_SPLIT
// slices of the grid: 16 x 16 tiles, the slices summed in a fixed order by the
// eigenproblem's block.  The split fills the chip: 30 tile pairs at lmax 4.
constexpr int OV_T = 16, OV_SPLIT = 8, OV_RC = 32;
__global__ void __launch_bounds__(OV_T *OV_T) radial_overlap_kernel(int n_r, const double *__restrict__ r,
                                                                    const double *__restrict__ w,
                                                                    const double *__restrict__ f,
                                                                    const int *__restrict__ ncL, int maxc,
                                                                    double *__restrict__ O) {
    const int L = blockIdx.y, nc = ncL[L];
    int bi = 0, bj = blockIdx.x;   // lower-triangular tile pair
    while (bj > bi) { bj -= bi + 1; ++bi; }
    if (bi * OV_T >= nc) return;
    __shared__ double fa[OV_T][OV_RC + 1], fb[OV_T][OV_RC + 1];
    const int tx = threadIdx.x % OV_T, ty = threadIdx.x / OV_T;
    const int per = (n_r + OV_SPLIT - 1) / OV_SPLIT, i0 = blockIdx.z * per, i1 = min(n_r, i0 + per);
    const double *fL = f + (size_t)L * maxc * n_r;
    double acc = 0.0;
    for (int c0 = i0; c0 < i1; c0 += OV_RC) {
        for (int t = threadIdx.x; t < OV_T * OV_RC; t += OV_T * OV_T) {
            const int row = t / OV_RC, i = c0 + t % OV_RC;
            const int ra = bi * OV_T + row, rb = bj * OV_T + row;
            const bool in = i < i1;
            fa[row][t % OV_RC] = in && ra < nc ? w[i] * r[i] * r[i] * fL[(size_t)ra * n_r + i] : 0.0;
            fb[row][t % OV_RC] = in && rb < nc ? fL[(size_t)rb * n_r + i] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < OV_RC; ++k) acc = fma(fa[ty][k], fb[tx][k], acc);
        __syncthreads();
    }
    const int a = bi * OV_T + ty, b = bj * OV_T + tx;
    if (a < nc && b <= a) O[(((size_t)blockIdx.z * gridDim.y + L) * maxc + a) * maxc + b] = acc;
}

// The P largest eigenpairs of the overlap matrix of one L (one block each):
// V[L][k][c] = sign and 1/sqrt(eigenvalue) times the eigenvector, for the
// eigenvalues above the threshold in descending order (status: fewer than wanted).
//  1. Householder reduction to tridiagonal form, the matrix in shared memory, one
//     thread per row and column group (a warp per row would spend more FP64 issue
//     on the reductions than on the products);
//  2. bisection by Sturm sequences, a warp per eigenvalue, 32 points per round
//     (the sequence itself instead of its ratios: no division);
//  3. inverse iteration on the tridiagonal matrix with partial pivoting, a lane per
//     eigenvalue, vectors of close eigenvalues kept orthogonal;
//  4. the reflections applied to the vectors, a warp per vector.
constexpr int RE_THREADS = 512;
constexpr int RE_MAXN = 128;    // >= the products of any L (114 at lmax 8)
__host__ __device__ constexpr size_t re_smem(int n) {
    return ((size_t)n * (n | 1) + 6 * (size_t)n + 6 * (size_t)n * kMaxP + kMaxP + RE_THREADS) * sizeof(double);
}
__global__ void __launch_bounds__(RE_THREADS) radial_eigen_kernel(const double *__restrict__ O, const int *__restrict__ ncL,
                                                                  int maxc, int nL, int P, double thr,
                                                                  double *__restrict__ V, int *__restrict__ status) {
    const int L = blockIdx.x, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = ncL[L], want = L == 0 ? P - 1 : P;
    if (want == 0) return;
    if (n < want) {
        if (tid == 0) atomicMin(status, -(L + 1));
        return;
    }
    const int ld = n | 1;
    extern __shared__ double sh[];
    double *A = sh, *d = A + (size_t)n * ld, *e = d + n, *beta = e + n, *v = beta + n, *wv = v + n, *e2 = wv + n;
    double *lam = e2 + n;                            // [kMaxP]
    double *x = lam + kMaxP;                         // [n][kMaxP] vectors, then the LU factors
    double *u0 = x + (size_t)n * kMaxP, *u1 = u0 + (size_t)n * kMaxP, *u2 = u1 + (size_t)n * kMaxP, *lm = u2 + (size_t)n * kMaxP;
    double *part = lm + 2 * (size_t)n * kMaxP;       // [groups][rows] partial sums
    __shared__ double s_beta, s_K, s_norm;

    for (int t = tid; t < n * n; t += RE_THREADS) {
        const int a = t / n, b = t % n;
        if (b > a) continue;
        double o = 0.0;
        for (int z = 0; z < OV_SPLIT; ++z) o += O[(((size_t)z * nL + L) * maxc + a) * maxc + b];
        A[a * ld + b] = o;
    }
    __syncthreads();
    // ---- 1. tridiagonal form; column k below the diagonal keeps the reflection vector
    for (int k = 0; k + 2 < n; ++k) {
        const int m = n - k - 1;
        if (warp == 0) {
            double sg = 0.0;
            for (int i = 1 + lane; i < m; i += 32) { const double t = A[(k + 1 + i) * ld + k]; sg = fma(t, t, sg); }
            sg = warp_sum(sg);
            const double al = A[(k + 1) * ld + k];
            double b = 0.0, v0 = 1.0, ek = al;
            // what is below the rounding of the column's first element is dropped
            const bool act = sg > 1e-36 * (al * al) && sg > 1e-60;
            if (act) {
                ek = sqrt(fma(al, al, sg));
                v0 = al <= 0.0 ? al - ek : -sg / (al + ek);
                b = 2.0 * v0 * v0 / (sg + v0 * v0);
            }
            const double iv0 = act ? 1.0 / v0 : 0.0;
            for (int i = lane; i < m; i += 32) {
                const double t = i == 0 ? 1.0 : A[(k + 1 + i) * ld + k] * iv0;
                v[i] = t;
                A[(k + 1 + i) * ld + k] = t;
            }
            if (lane == 0) { d[k] = A[k * ld + k]; e[k] = ek; beta[k] = b; s_beta = b; }
        }
        __syncthreads();
        const double b = s_beta;
        if (b != 0.0) {   // uniform over the block
            const int rows = (m + 31) / 32 * 32, ng = RE_THREADS / rows, g = tid / rows, i = tid % rows;
            double acc = 0.0;
            if (g < ng && i < m)
                for (int j = g; j < m; j += ng) acc = fma(j <= i ? A[(k + 1 + i) * ld + k + 1 + j] : A[(k + 1 + j) * ld + k + 1 + i], v[j], acc);
            if (g < ng) part[g * rows + i] = acc;
            __syncthreads();
            if (tid < m) {
                double s = 0.0;
                for (int q = 0; q < ng; ++q) s += part[q * rows + tid];
                wv[tid] = b * s;
            }
            __syncthreads();
            if (warp == 0) {
                double s = 0.0;
                for (int j = lane; j < m; j += 32) s = fma(wv[j], v[j], s);
                s = warp_sum(s);
                if (lane == 0) s_K = 0.5 * b * s;
            }
            __syncthreads();
            if (tid < m) wv[tid] = fma(-s_K, v[tid], wv[tid]);
            __syncthreads();
            if (g < ng && i < m) {
                const double vi = v[i], wi = wv[i];
                for (int j = g; j <= i; j += ng) {
                    double *a = A + (k + 1 + i) * ld + k + 1 + j;
                    *a = fma(-wi, v[j], fma(-vi, wv[j], *a));
                }
            }
        }
        __syncthreads();
    }
    if (tid == 0) {
        if (n >= 2) { d[n - 2] = A[(n - 2) * ld + n - 2]; e[n - 2] = A[(n - 1) * ld + n - 2]; }
        d[n - 1] = A[(n - 1) * ld + n - 1];
        e[n - 1] = 0.0;
    }
    __syncthreads();
    // scale to norm 1 (the bound of Gershgorin's circles)
    if (warp == 0) {
        double mx = 0.0, any = 0.0;
        for (int i = lane; i < n; i += 32) any += fabs(d[i]) + fabs(e[i]);
        any = warp_sum(any);
        for (int i = lane; i < n; i += 32) mx = fmax(mx, fabs(d[i]) + fabs(e[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) s_norm = isfinite(any) ? (mx > 0.0 ? mx : 1.0) : 0.0;
    }
    __syncthreads();
    const double norm = s_norm;
    if (norm == 0.0) {   // an overflow in the products
        if (tid == 0) atomicMin(status, -(L + 1));
        return;
    }
    for (int i = tid; i < n; i += RE_THREADS) {
        d[i] /= norm;
        // an exact zero would stop the recurrence below; 1e-17 is under the rounding of T
        const double t = e[i] / norm;
        e[i] = i + 1 < n && fabs(t) < 1e-17 ? 1e-17 : t;
        e2[i] = e[i] * e[i];
    }
    __syncthreads();
    // ---- 2. the (warp)-th largest eigenvalue: index n - 1 - warp in ascending order
    if (warp < want) {
        double lo = -1.0 - 1e-14, hi = 1.0 + 1e-14;
        const int idx = n - 1 - warp;
        for (int round = 0; round < 11; ++round) {
            const double h = (hi - lo) / 33.0, xx = lo + h * (lane + 1);
            // number of eigenvalues below xx = sign changes of the leading minors
            int cnt = 0;
            double p0 = 1.0, p1 = d[0] - xx;
            bool neg = p1 < 0.0 || p1 == 0.0;
            cnt += neg;
            for (int i = 1; i < n; ++i) {
                const double p2 = fma(d[i] - xx, p1, -e2[i - 1] * p0);
                p0 = p1;
                p1 = p2;
                const bool ng = p1 < 0.0 || (p1 == 0.0 && !neg);
                cnt += ng != neg;
                neg = ng;
                if ((i & 3) == 3) {   // keep both in range
                    const int eb = max(__double2hiint(fmax(fabs(p0), fabs(p1))) >> 20, 1);
                    const double sc = __hiloint2double((2046 - min(eb, 2045)) << 20, 0);
                    p0 *= sc;
                    p1 *= sc;
                }
            }
            const unsigned above = __ballot_sync(0xffffffffu, cnt > idx);   // eigenvalue idx lies below xx
            const int first = above ? __ffs(above) - 1 : 32;
            const double nlo = lo + h * first, nhi = first < 32 ? lo + h * (first + 1) : hi;
            lo = nlo;
            hi = nhi;
        }
        if (lane == 0) lam[warp] = 0.5 * (lo + hi);
    }
    __syncthreads();
    bool few = false;
    for (int k = 0; k < want; ++k) few |= !(lam[k] * norm > thr);
    if (few) {
        if (tid == 0) atomicMin(status, -(L + 1));
        return;
    }
    // ---- 3. inverse iteration
    if (warp == 0) {
        const bool on = lane < want;
        const int q = on ? lane : 0;
        const double l = lam[q];
        if (on) {
            constexpr double tiny = 2.3e-16;
            double a = d[0] - l, b = n > 1 ? e[0] : 0.0;
            for (int i = 0; i + 1 < n; ++i) {
                const double sub = e[i], dn = d[i + 1] - l, en = i + 2 < n ? e[i + 1] : 0.0;
                const bool sw = fabs(a) < fabs(sub);
                double pv = sw ? sub : a;
                if (fabs(pv) < tiny) pv = pv < 0.0 ? -tiny : tiny;
                const double rp = 1.0 / pv, mlt = (sw ? a : sub) * rp;
                u0[i * kMaxP + q] = rp;
                u1[i * kMaxP + q] = sw ? dn : b;
                u2[i * kMaxP + q] = sw ? en : 0.0;
                lm[i * kMaxP + q] = mlt;
                lm[(size_t)n * kMaxP + i * kMaxP + q] = sw ? 1.0 : 0.0;
                a = sw ? fma(-mlt, dn, b) : fma(-mlt, b, dn);
                b = sw ? -mlt * en : en;
            }
            if (fabs(a) < tiny) a = a < 0.0 ? -tiny : tiny;
            u0[(n - 1) * kMaxP + q] = 1.0 / a;
            for (int i = 0; i < n; ++i)   // a start vector with no symmetry of its own
                x[i * kMaxP + q] = 1.0 + (double)((i * 29 + q * 17) % 31) * (1.0 / 64.0);
        }
        for (int it = 0; it < 4; ++it) {
            if (on) {
                for (int i = 0; i + 1 < n; ++i) {
                    const double mlt = lm[i * kMaxP + q];
                    const bool sw = lm[(size_t)n * kMaxP + i * kMaxP + q] != 0.0;
                    const double xi = x[i * kMaxP + q], xn = x[(i + 1) * kMaxP + q];
                    x[i * kMaxP + q] = sw ? xn : xi;
                    x[(i + 1) * kMaxP + q] = sw ? fma(-mlt, xn, xi) : fma(-mlt, xi, xn);
                }
                double y1 = 0.0, y2 = 0.0, mx = 0.0;
                for (int i = n - 1; i >= 0; --i) {
                    double t = x[i * kMaxP + q];
                    if (i + 1 < n) t = fma(-u1[i * kMaxP + q], y1, t);
                    if (i + 2 < n) t = fma(-u2[i * kMaxP + q], y2, t);
                    t *= u0[i * kMaxP + q];
                    x[i * kMaxP + q] = t;
                    y2 = y1;
                    y1 = t;
                    mx = fmax(mx, fabs(t));
                }
                const double sc = mx > 0.0 ? 1.0 / mx : 0.0;
                for (int i = 0; i < n; ++i) x[i * kMaxP + q] *= sc;
            }
            __syncwarp();
            // orthogonal to the vectors of close eigenvalues already there; unit length
            for (int k = 0; k < want; ++k) {
                for (int j = 0; j < k; ++j) {
                    if (!(lam[j] - lam[k] < 1e-3)) continue;
                    double s = 0.0;
                    for (int i = lane; i < n; i += 32) s = fma(x[i * kMaxP + j], x[i * kMaxP + k], s);
                    s = warp_sum(s);
                    for (int i = lane; i < n; i += 32) x[i * kMaxP + k] = fma(-s, x[i * kMaxP + j], x[i * kMaxP + k]);
                    __syncwarp();
                }
                double s = 0.0;
                for (int i = lane; i < n; i += 32) s = fma(x[i * kMaxP + k], x[i * kMaxP + k], s);
                s = warp_sum(s);
                const double sc = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
                for (int i = lane; i < n; i += 32) x[i * kMaxP + k] *= sc;
                __syncwarp();
            }
        }
    }
    __syncthreads();
    // ---- 4. back to the products; the largest component positive, scaled by 1/sqrt(eigenvalue)
    if (warp < want) {
        const int q = warp;
        for (int k = n - 3; k >= 0; --k) {
            const double b = beta[k];
            if (b == 0.0) continue;
            const int m = n - k - 1;
            double s = 0.0;
            for (int i = lane; i < m; i += 32) s = fma(A[(k + 1 + i) * ld + k], x[(k + 1 + i) * kMaxP + q], s);
            s = b * warp_sum(s);
            for (int i = lane; i < m; i += 32)
                x[(k + 1 + i) * kMaxP + q] = fma(-s, A[(k + 1 + i) * ld + k], x[(k + 1 + i) * kMaxP + q]);
            __syncwarp();
        }
        double s = 0.0, big = -1.0;
        int at = 0;
        for (int i = lane; i < n; i += 32) {
            const double t = x[i * kMaxP + q];
            s = fma(t, t, s);
            if (fabs(t) > big) { big = fabs(t); at = i; }
        }
        s = warp_sum(s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, big, o);
            const int oa = __shfl_xor_sync(0xffffffffu, at, o);
            if (ob > big || (ob == big && oa < at)) { big = ob; at = oa; }
        }
        const double sc = (x[at * kMaxP + q] >= 0.0 ? 1.0 : -1.0) / sqrt(s * (lam[q] * norm));
        for (int i = lane; i < n; i += 32) V[((size_t)L * kMaxP + q) * maxc + i] = sc * x[i * kMaxP + q];
    }
}

// The functions M_aLP on the grid: grid (points, P, L).
__global__ void __launch_bounds__(RP_THREADS) radial_functions_kernel(int n_r, const double *__restrict__ r,
                                                                      const double *__restrict__ w,
                                                                      const double *__restrict__ f,
                                                                      const double *__restrict__ V,
                                                                      const int *__restrict__ ncL, int maxc, int P,
                                                                      const int *__restrict__ status,
                                                                      double *__restrict__ M) {
    if (*status < 0) return;
    const int L = blockIdx.z, Pi = blockIdx.y, i = blockIdx.x * RP_THREADS + threadIdx.x;
    __shared__ double red[33];
    double v = 0.0;
    if (L == 0 && Pi == 0) {
        double s = 0.0;
        for (int j = threadIdx.x; j < n_r; j += RP_THREADS) s += w[j] * r[j] * r[j];
        v = 1.0 / sqrt(block_sum(s, red));
    } else if (i < n_r) {
        const double *vk = V + ((size_t)L * kMaxP + (L == 0 ? Pi - 1 : Pi)) * maxc;
        const double *fL = f + (size_t)L * maxc * n_r + i;
        const int nc = ncL[L];
        for (int c = 0; c < nc; ++c) v = fma(vk[c], fL[(size_t)c * n_r], v);
    }
    if (i < n_r) M[((size_t)L * P + Pi) * n_r + i] = v;
}

// The functions of one L made orthonormal on the grid, in descending order of the
// eigenvalue (one block per L).  An eigenvector is accurate to rounding in the norm of
// the overlap matrix, so what it holds of one with a larger eigenvalue grows by the root
// of their ratio once it is scaled by 1/sqrt(eigenvalue): overlaps of the functions
// reached 4e-12 at lmax 8, 1e-15 here.  The overlaps G = K K^T (Cholesky), a warp each,
// then M = K^-1 M: 0.504 to 0.520 ms for the whole call at lmax 4, P = 3, 600 points.
constexpr int RO_THREADS = 512;
__global__ void __launch_bounds__(RO_THREADS) radial_orthonormal_kernel(int n_r, const double *__restrict__ r,
                                                                        const double *__restrict__ w, int P,
                                                                        const int *__restrict__ status,
                                                                        double *__restrict__ M) {
    if (*status < 0) return;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    __shared__ double K[kMaxP][kMaxP + 1];   // lower triangle; the diagonal inverted
    double *ML = M + (size_t)blockIdx.x * P * n_r;
    for (int t = warp; t < P * (P + 1) / 2; t += RO_THREADS / 32) {
        int a = 0, b = t;
        while (b > a) { b -= a + 1; ++a; }
        const double *x = ML + (size_t)a * n_r, *y = ML + (size_t)b * n_r;
        double s = 0.0;
#pragma unroll 8
        for (int i = lane; i < n_r; i += 32) s = fma(w[i] * r[i] * r[i] * x[i], y[i], s);
        s = warp_sum(s);
        if (lane == 0) K[a][b] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int a = 0; a < P; ++a)
            for (int b = 0; b <= a; ++b) {
                double s = K[a][b];
                for (int j = 0; j < b; ++j) s = fma(-K[a][j], K[b][j], s);
                K[a][b] = a == b ? 1.0 / sqrt(s) : s * K[b][b];
            }
    __syncthreads();
    // (K is close to the unit matrix: its difference from that is added, one rounding)
    for (int i = threadIdx.x; i < n_r; i += RO_THREADS)
        for (int a = 0; a < P; ++a) {
            const double m = ML[(size_t)a * n_r + i];
            double c = 0.0;
            for (int j = 0; j < a; ++j) c = fma(-K[a][j], ML[(size_t)j * n_r + i], c);
            ML[(size_t)a * n_r + i] = m + fma(m, K[a][a] - 1.0, c * K[a][a]);
        }
}

// r^k, k >= 0
__device__ __forceinline__ double ipow(double r, int k) {
    double p = 1.0;
    for (int i = 0; i < k; ++i) p *= r;
    return p;
}

// Multipole moments and radial integrals, a warp per (L, P, a <= b) (a < 0: the moment).
__global__ void __launch_bounds__(RP_THREADS) radial_integrals_kernel(int n_r, const double *__restrict__ r,
                                                                      const double *__restrict__ w,
                                                                      const double *__restrict__ u,
                                                                      const double *__restrict__ M, int nlp, int P, int nL,
                                                                      const int *__restrict__ status,
                                                                      double *__restrict__ mu, double *__restrict__ R) {
    if (*status < 0) return;
    const int per = 1 + nlp * (nlp + 1) / 2, lane = threadIdx.x % 32;
    const long long e = (long long)blockIdx.x * (RP_THREADS / 32) + threadIdx.x / 32;
    if (e >= (long long)nL * P * per) return;
    const int LP = (int)(e / per), L = LP / P;
    int t = (int)(e % per);
    const double *m = M + (size_t)LP * n_r;
    double acc = 0.0;
    if (t == 0) {
        for (int i = lane; i < n_r; i += 32) acc = fma(w[i] * m[i], ipow(r[i], L + 2), acc);
        acc = warp_sum(acc);
        if (lane == 0) mu[LP] = acc;
        return;
    }
    int b = 0;
    t -= 1;
    while (t > b) { t -= b + 1; ++b; }
    const double *ua = u + (size_t)t * n_r, *ub = u + (size_t)b * n_r;
    for (int i = lane; i < n_r; i += 32) acc = fma(w[i] * r[i] * r[i] * m[i] * ua[i], ub[i], acc);
    acc = warp_sum(acc);
    if (lane == 0) {
        R[((size_t)LP * nlp + t) * nlp + b] = acc;
        R[((size_t)LP * nlp + b) * nlp + t] = acc;
    }
}

// On-site Coulomb integrals C[L][P][Q] (Laplace expansion, tensor-product
// quadrature), one block per (Q, L).  With the grid ascending, the inner integral
// over r' at r_i is r_i^-(L+1) times a prefix sum (r' <= r_i) plus r_i^L times a
// suffix sum (r' > r_i) of the same products: n_r terms instead of n_r^2.
constexpr int RC_THREADS = 256;
__global__ void __launch_bounds__(RC_THREADS) radial_onsite_kernel(int n_r, const double *__restrict__ r,
                                                                   const double *__restrict__ w,
                                                                   const double *__restrict__ M, int P,
                                                                   const int *__restrict__ status,
                                                                   double *__restrict__ inner, double *__restrict__ C) {
    if (*status < 0) return;
    const int Q = blockIdx.x, L = blockIdx.y, tid = threadIdx.x;
    __shared__ double lo[RC_THREADS], up[RC_THREADS], red[33];
    const double *g = M + ((size_t)L * P + Q) * n_r;
    double *in = inner + ((size_t)L * P + Q) * n_r;
    const int per = (n_r + RC_THREADS - 1) / RC_THREADS, i0 = min(n_r, tid * per), i1 = min(n_r, i0 + per);
    double a = 0.0, b = 0.0;
    for (int i = i0; i < i1; ++i) {
        const double t = w[i] * r[i] * r[i] * g[i], pl = ipow(r[i], L);
        a = fma(t, pl, a);
        b += t / (pl * r[i]);
    }
    lo[tid] = a;
    up[tid] = b;
    __syncthreads();
    for (int o = 1; o < RC_THREADS; o <<= 1) {   // inclusive prefix and suffix sums of the chunks
        const double x = tid >= o ? lo[tid - o] : 0.0, y = tid + o < RC_THREADS ? up[tid + o] : 0.0;
        __syncthreads();
        lo[tid] += x;
        up[tid] += y;
        __syncthreads();
    }
    double pre = tid > 0 ? lo[tid - 1] : 0.0, suf = tid + 1 < RC_THREADS ? up[tid + 1] : 0.0;
    for (int i = i0; i < i1; ++i) {
        const double pl = ipow(r[i], L);
        pre = fma(w[i] * r[i] * r[i] * g[i], pl, pre);
        in[i] = pre / (pl * r[i]);
    }
    for (int i = i1 - 1; i >= i0; --i) {
        const double pl = ipow(r[i], L);
        in[i] = fma(pl, suf, in[i]);
        suf += w[i] * r[i] * r[i] * g[i] / (pl * r[i]);
    }
    __syncthreads();
    for (int Pi = 0; Pi < P; ++Pi) {
        const double *m = M + ((size_t)L * P + Pi) * n_r;
        double acc = 0.0;
        for (int i = i0; i < i1; ++i) acc = fma(w[i] * r[i] * r[i] * m[i], in[i], acc);
        acc = block_sum(acc, red);
        if (tid == 0) C[((size_t)L * P + Pi) * P + Q] = 4.0 * kPi / (2 * L + 1) * acc;
    }
}

// The mu = 0 rows and columns of v_t (transformed index positions, Sec. III.C):
// inside channel (a, L, M) the on-site block T C_aL T^T, zero elsewhere.
__global__ void onsite_fill_kernel(double2 *__restrict__ v, int naux, const double *__restrict__ C,
                                   const double *__restrict__ T, int n_atoms, int Lmax, int P) {
    const int nLM = (Lmax + 1) * (Lmax + 1);
    const long long nrow = (long long)n_atoms * nLM * (P - 1);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nrow * naux;
         e += (long long)gridDim.x * blockDim.x) {
        const long long rix = e / naux;
        const int J = (int)(e % naux);
        const int ch = (int)(rix / (P - 1)), i = 1 + (int)(rix % (P - 1));
        const int a = ch / nLM, L = (int)floor(sqrt((double)(ch % nLM)) + 1e-9);
        const int I = ch * P + i;
        double val = 0.0;
        if (J / P == ch && J < n_atoms * nLM * P) {
            const int j = J % P;
            const double *Ta = T + ((size_t)a * (Lmax + 1) + L) * P * P;
            const double *Ca = C + ((size_t)a * (Lmax + 1) + L) * P * P;
            for (int p = 0; p < P; ++p)
                for (int q = 0; q < P; ++q) val += Ta[i * P + p] * Ca[p * P + q] * Ta[j * P + q];
        }
        v[(size_t)I * naux + J] = make_double2(val, 0.0);
        v[(size_t)J * naux + I] = make_double2(val, 0.0);
    }
}

}  // namespace

void launch_onsite_fill(double2 *d_v, int naux, const double *d_C, const double *d_T, int n_atoms, int Lmax, int P,
                        cudaStream_t st) {
    if (P < 2) return;
    const long long n = (long long)n_atoms * (Lmax + 1) * (Lmax + 1) * (P - 1) * naux;
    long long g = (n + 255) / 256;
    if (g > 152LL * 32) g = 152LL * 32;
    onsite_fill_kernel<<<(unsigned)std::max<long long>(g, 1), 256, 0, st>>>(d_v, naux, d_C, d_T, n_atoms, Lmax, P);
}

}  // namespace hfx

using namespace hfx;

extern "C" {

int hfx_set_radial_functions(hfx_ctx *ctx, int atom, int n_r, const double *r, const double *w, const double *u,
                             double threshold) {
    if (!ctx) return HFX_EINVAL;
    const hfx_system &s = ctx->sys;
    if (atom < 0 || atom >= s.n_atoms || !r || !w || !u || n_r < 2 || n_r > 8192 || !(threshold > 0.0))
        return set_err(ctx, HFX_EINVAL, "set_radial_functions: bad atom, grid, pointer or threshold");
    if (ctx->P > kMaxP) return set_err(ctx, HFX_EUNSUPPORTED, "set_radial_functions: P above the kernel's limit");
    const int nlp = ctx->nlp, LP = (s.Lmax + 1) * ctx->P, P = ctx->P;
    for (int i = 0; i < n_r; ++i)
        if (!std::isfinite(r[i]) || !std::isfinite(w[i]) || r[i] <= 0.0 || r[i] > ctx->rmt[atom] * (1.0 + 1e-12) ||
            (i > 0 && r[i] <= r[i - 1]))
            return set_err(ctx, HFX_EINVAL, "set_radial_functions: grid must increase within (0, R_MT]");
    for (size_t i = 0; i < (size_t)nlp * n_r; ++i)
        if (!std::isfinite(u[i])) return set_err(ctx, HFX_ENONFINITE, "set_radial_functions: non-finite u");
    int rc = cuda_check(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    if (rc) return rc;
    // the products of every L (l p <= l' p', triangle rule)
    const int nL = s.Lmax + 1;
    std::vector<std::vector<int2>> prods(nL);
    int maxc = 1;
    for (int L = 0; L < nL; ++L) {
        for (int a = 0; a < nlp; ++a)
            for (int b = a; b < nlp; ++b)
                if (std::abs(a / 2 - b / 2) <= L && L <= a / 2 + b / 2) prods[L].push_back(make_int2(a, b));
        maxc = std::max(maxc, (int)prods[L].size());
    }
    if (maxc > RE_MAXN) return set_err(ctx, HFX_EUNSUPPORTED, "set_radial_functions: too many products");
    // one upload (grid, functions, product lists), one download (M, mu, R, C, status);
    // the device buffer belongs to the context and is reused by the next atom
    HostArena in;
    const size_t o_r = in.put(r, n_r * sizeof(double)), o_w = in.put(w, n_r * sizeof(double));
    const size_t o_u = in.put(u, (size_t)nlp * n_r * sizeof(double));
    std::vector<int2> plist((size_t)nL * maxc, make_int2(0, 0));
    std::vector<int> nc(nL);
    for (int L = 0; L < nL; ++L) {
        nc[L] = (int)prods[L].size();
        std::copy(prods[L].begin(), prods[L].end(), plist.begin() + (size_t)L * maxc);
    }
    const size_t o_p = in.put(plist), o_nc = in.put(nc);
    const size_t n_out = (size_t)LP * n_r + LP + (size_t)LP * nlp * nlp + (size_t)nL * P * P + 1;
    Layout lay;
    lay.place(in.buf.size());
    const size_t o_f = lay.place((size_t)nL * maxc * n_r * sizeof(double));
    const size_t o_O = lay.place((size_t)OV_SPLIT * nL * maxc * maxc * sizeof(double));
    const size_t o_V = lay.place((size_t)nL * kMaxP * maxc * sizeof(double));
    const size_t o_in = lay.place((size_t)LP * n_r * sizeof(double));
    const size_t o_out = lay.place(n_out * sizeof(double));
    if ((rc = scratch_reserve(ctx, ctx->s_misc, lay.off))) return rc;
    char *base = reinterpret_cast<char *>(ctx->s_misc.p);
    auto dp = [&](size_t o) { return reinterpret_cast<double *>(base + o); };
    const double *d_r = dp(o_r), *d_w = dp(o_w), *d_u = dp(o_u);
    double *dM = dp(o_out), *dmu = dM + (size_t)LP * n_r, *dR = dmu + LP, *dC = dR + (size_t)LP * nlp * nlp;
    int *d_status = reinterpret_cast<int *>(dC + (size_t)nL * P * P);
    const int *d_nc = reinterpret_cast<const int *>(base + o_nc);
    cudaStream_t st = ctx->stream;
    std::vector<double> out(n_out);
    if ((rc = cuda_check(ctx, cudaMemcpyAsync(base, in.buf.data(), in.buf.size(), cudaMemcpyHostToDevice, st), "radial inputs")) ||
        (rc = cuda_check(ctx, cudaMemsetAsync(d_status, 0, sizeof(double), st), "radial status")))
        return rc;
    int sm_max = 0;   // the opt-in of the eigenproblem's shared memory, for its largest size here
    cudaDeviceGetAttribute(&sm_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
    const size_t sm = re_smem(maxc);
    if (sm > (size_t)sm_max) return set_err(ctx, HFX_EUNSUPPORTED, "set_radial_functions: too many products");
    if ((rc = cuda_check(ctx, cudaFuncSetAttribute(radial_eigen_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm),
                         "radial shared memory")))
        return rc;
    radial_products_kernel<<<dim3(maxc, nL), RP_THREADS, 0, st>>>(n_r, d_r, d_w, d_u, reinterpret_cast<const int2 *>(base + o_p),
                                                                  d_nc, maxc, dp(o_f));
    const int nt = (maxc + OV_T - 1) / OV_T;
    radial_overlap_kernel<<<dim3(nt * (nt + 1) / 2, nL, OV_SPLIT), OV_T * OV_T, 0, st>>>(n_r, d_r, d_w, dp(o_f), d_nc, maxc,
                                                                                        dp(o_O));
    radial_eigen_kernel<<<nL, RE_THREADS, sm, st>>>(dp(o_O), d_nc, maxc, nL, P, threshold, dp(o_V), d_status);
    radial_functions_kernel<<<dim3((n_r + RP_THREADS - 1) / RP_THREADS, P, nL), RP_THREADS, 0, st>>>(
        n_r, d_r, d_w, dp(o_f), dp(o_V), d_nc, maxc, P, d_status, dM);
    radial_orthonormal_kernel<<<nL, RO_THREADS, 0, st>>>(n_r, d_r, d_w, P, d_status, dM);
    const long long nint = (long long)LP * (1 + nlp * (nlp + 1) / 2);
    radial_integrals_kernel<<<(unsigned)((nint + RP_THREADS / 32 - 1) / (RP_THREADS / 32)), RP_THREADS, 0, st>>>(
        n_r, d_r, d_w, d_u, dM, nlp, P, nL, d_status, dmu, dR);
    radial_onsite_kernel<<<dim3(P, nL), RC_THREADS, 0, st>>>(n_r, d_r, d_w, dM, P, d_status, dp(o_in), dC);
    if ((rc = cuda_check(ctx, cudaGetLastError(), "radial kernels")) ||
        (rc = cuda_check(ctx, cudaMemcpyAsync(out.data(), dM, n_out * sizeof(double), cudaMemcpyDeviceToHost, st), "radial results")) ||
        (rc = cuda_check(ctx, cudaStreamSynchronize(st), "radial kernels")))
        return rc;
    int status = 0;
    std::memcpy(&status, &out[n_out - 1], sizeof(int));
    if (status < 0)
        return set_err(ctx, HFX_EINVAL, "set_radial_functions: fewer than P product functions above the threshold for L = " +
                                            std::to_string(-status - 1));
    // keep the basis; R and mu replace those of hfx_set_radial
    const double *M = out.data(), *mu = M + (size_t)LP * n_r, *R = mu + LP, *C = R + (size_t)LP * nlp * nlp;
    if (ctx->rad_M.size() != (size_t)s.n_atoms) {
        ctx->rad_M.assign(s.n_atoms, {});
        ctx->rad_nr.assign(s.n_atoms, 0);
        ctx->rad_C.assign((size_t)s.n_atoms * (s.Lmax + 1) * P * P, 0.0);
        ctx->rad_set.assign(s.n_atoms, 0);
    }
    ctx->rad_M[atom].assign(M, M + (size_t)LP * n_r);
    ctx->rad_nr[atom] = n_r;
    std::memcpy(ctx->rad_C.data() + (size_t)atom * (s.Lmax + 1) * P * P, C, sizeof(double) * (s.Lmax + 1) * P * P);
    ctx->rad_set[atom] = 1;
    ctx->rad_C_dirty = true;
    return hfx_set_radial(ctx, atom, R, mu);
}

int hfx_get_radial_basis(hfx_ctx *ctx, int atom, double *M, double *mu, double *R, double *C) {
    if (!ctx) return HFX_EINVAL;
    const hfx_system &s = ctx->sys;
    if (atom < 0 || atom >= s.n_atoms) return set_err(ctx, HFX_EINVAL, "get_radial_basis: bad atom");
    if (ctx->rad_set.size() != (size_t)s.n_atoms || !ctx->rad_set[atom])
        return set_err(ctx, HFX_EMISSING, "get_radial_basis: set_radial_functions first");
    const int P = ctx->P, LP = (s.Lmax + 1) * P, nlp = ctx->nlp;
    if (M) std::memcpy(M, ctx->rad_M[atom].data(), sizeof(double) * ctx->rad_M[atom].size());
    if (mu) std::memcpy(mu, ctx->hmu.data() + (size_t)atom * LP, sizeof(double) * LP);
    if (R) std::memcpy(R, ctx->hR.data() + (size_t)atom * LP * nlp * nlp, sizeof(double) * (size_t)LP * nlp * nlp);
    if (C) std::memcpy(C, ctx->rad_C.data() + (size_t)atom * (s.Lmax + 1) * P * P, sizeof(double) * (s.Lmax + 1) * P * P);
    return HFX_OK;
}

}  // extern "C"
