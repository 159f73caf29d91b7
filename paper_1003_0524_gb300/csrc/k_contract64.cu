// k_contract64.cu -- the FP64 contraction (the "plain FP64 GPU" build):
// Y' = U Z (dense block and mu=0 blocks of Fig. 1; U the upper triangle of v_t
// with half its diagonal, v_t = U + U^H) and the per-pair P' = sum_m Z_m^H Y'_m,
// whose P' + P'^H is the pair's term of Eq. vec-mat-vec, with DFMA on the CUDA cores.
// Where v is Hermitian only within a tolerance, all of v_t is applied and Z^H Y is the term.
#include <algorithm>
#include <cmath>

#include "hfx_internal.cuh"

namespace hfx {

namespace {

// Batched complex GEMM, C = op(A) B, K = K1 * K2 split into two strides.
//
// Bound by FP64 issue: about two FMAs per cycle and SM, so one warp's FMA occupies
// its scheduler for ~64 cycles and the shared-memory and address work hides behind
// it.  What counts is how few products are padding and how evenly they spread over
// the SMs, hence small tiles: 64 threads in 8 x 8, R x R outputs each, tile edge 8 R
// for R = 2..5 (zgemm64_tile).  Z^H Y of 64 pairs of 40 bands, K = 5256: 22.8 ms with
// 64 x 64 tiles and one block per pair, 4.5 ms with 40 x 40 tiles and the K sum
// split over blocks.
// upper: A is square in (row, k2) and only its upper triangle with half the diagonal
// is applied: K starts at the tile's first row.
// herm: C is Hermitian; only the tiles on and above the diagonal are computed, the
// others are their conjugates.
constexpr int TK = 8, T8 = 8;

template <int R>
__global__ void __launch_bounds__(64) zgemm64_kernel(const ZGemmBatch *__restrict__ batches) {
    constexpr int T = T8 * R;
    const ZGemmBatch b = batches[blockIdx.z];
    const int i0 = blockIdx.y * T, j0 = blockIdx.x * T;
    if (i0 >= b.M || j0 >= b.N || (b.herm && j0 < i0)) return;
    __shared__ double2 As[TK][T + 1];
    __shared__ double2 Bs[TK][T + 1];
    const int tx = threadIdx.x % T8, ty = threadIdx.x / T8;
    double2 acc[R][R];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = make_double2(0.0, 0.0);
    const long long K = (long long)b.K1 * b.K2;
    const bool akf = b.sAk2 == 1, bkf = b.sBk2 == 1;   // K is the contiguous index: read along it
    for (long long k0 = b.upper ? i0 : 0; k0 < K; k0 += TK) {
        for (int t = threadIdx.x; t < TK * T; t += 64) {
            const int kk = akf ? t % TK : t / T, r = akf ? t / TK : t % T;
            const long long k = k0 + kk;
            double2 v = make_double2(0.0, 0.0);
            if (k < K && i0 + r < b.M) {
                const long long k1 = b.K1 == 1 ? 0 : k / b.K2, k2 = k - k1 * b.K2;
                v = b.A[(i0 + r) * b.sAi + k1 * b.sAk1 + k2 * b.sAk2];
                if (b.conjA) v.y = -v.y;
                if (b.upper && k <= i0 + r) {
                    const double w = k == i0 + r ? 0.5 : 0.0;
                    v = make_double2(w * v.x, w * v.y);
                }
            }
            As[kk][r] = v;
        }
        for (int t = threadIdx.x; t < TK * T; t += 64) {
            const int kk = bkf ? t % TK : t / T, c = bkf ? t / TK : t % T;
            const long long k = k0 + kk;
            double2 v = make_double2(0.0, 0.0);
            if (k < K && j0 + c < b.N) {
                const long long k1 = b.K1 == 1 ? 0 : k / b.K2, k2 = k - k1 * b.K2;
                v = b.B[k1 * b.sBk1 + k2 * b.sBk2 + (j0 + c) * b.sBj];
            }
            Bs[kk][c] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            double2 a[R], bb[R];
#pragma unroll
            for (int i = 0; i < R; ++i) a[i] = As[kk][ty + T8 * i];
#pragma unroll
            for (int j = 0; j < R; ++j) bb[j] = Bs[kk][tx + T8 * j];
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) acc[i][j] = cfma(a[i], bb[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int r = i0 + ty + T8 * i, c = j0 + tx + T8 * j;
            if (r >= b.M || c >= b.N) continue;
            b.C[r * b.sCi + c * b.sCj] = acc[i][j];
            if (b.herm && j0 > i0) b.C[c * b.sCi + r * b.sCj] = make_double2(acc[i][j].x, -acc[i][j].y);
        }
}

// Tile factor R: least padded work, the larger tile at equal padding; with few blocks
// per SM their uneven number counts too (the LAPW transform of 8 k points, 314 x 314
// outputs: 160 tiles of 64 on 152 SMs took two block times, 7.14 ms with the copies;
// 3.92 ms with 16 x 16 tiles and the Hermitian half).
int zgemm64_r(int M, int N, long long nbatch) {
    int best = 2;
    double cost = 1e300;
    for (int r = 2; r <= 5; ++r) {
        const long long T = T8 * r, tm = (M + T - 1) / T, tn = (N + T - 1) / T;
        const double waves = (double)(nbatch * tm * tn) / 152.0;
        const double c = (double)(tm * T) * (double)(tn * T) * (waves < 16.0 ? std::ceil(waves) / waves : 1.0);
        if (c <= cost) { cost = c; best = r; }
    }
    return best;
}

// Y' rows of the mu=0 functions: per channel, the (P-1) x P block of U times the
// channel's [mu!=0, mu=0...] rows of Z (Fig. 1 on-site blocks): the coupling to the
// mu!=0 function lies above the diagonal, of the mu=0 functions those from i on count,
// i itself half (full: those of v_t, all of them).
__global__ void block64_kernel(const QDesc *__restrict__ qd, const double2 *const *__restrict__ VB,
                               const double2 *__restrict__ Z, double2 *__restrict__ Y, long long RSc, int nch, int P,
                               int N0, int full) {
    const QDesc q = qd[blockIdx.y];
    const double2 *vb = VB[blockIdx.y];
    long long total = q.ncols * N0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        int u = (int)(e % N0);
        long long col = q.colbase + e / N0;
        int ch = u / (P - 1), i = u % (P - 1);
        const double2 *z = Z + col * RSc;
        const double2 *row = vb + ((size_t)ch * (P - 1) + i) * P;
        double2 acc = cmul(row[0], z[N0 + ch]);
        for (int s = full ? 1 : i + 1; s < P; ++s) {
            const double w = !full && s == i + 1 ? 0.5 : 1.0;
            acc = cfma(make_double2(w * row[s].x, w * row[s].y), z[ch * (P - 1) + s - 1], acc);
        }
        Y[col * RSc + u] = acc;
    }
}

}  // namespace

int zgemm64_tile(int M, int N, long long nbatch) { return T8 * zgemm64_r(M, N, nbatch); }

void launch_zgemm64(const ZGemmBatch *d_b, int nbatch, int maxM, int maxN, cudaStream_t st) {
    if (nbatch == 0) return;
    const int r = zgemm64_r(maxM, maxN, nbatch), T = T8 * r;
    const dim3 grid((unsigned)((maxN + T - 1) / T), (unsigned)((maxM + T - 1) / T), (unsigned)nbatch);
    switch (r) {
    case 2: zgemm64_kernel<2><<<grid, 64, 0, st>>>(d_b); break;
    case 3: zgemm64_kernel<3><<<grid, 64, 0, st>>>(d_b); break;
    case 4: zgemm64_kernel<4><<<grid, 64, 0, st>>>(d_b); break;
    default: zgemm64_kernel<5><<<grid, 64, 0, st>>>(d_b); break;
    }
}

void launch_block64(const QDesc *d_q, int nq, const double2 *const *d_VB, const double2 *d_Z, double2 *d_Y,
                    long long RSc, int nch, int P, int N0, int full, long long maxcols, cudaStream_t st) {
    if (N0 == 0 || nq == 0) return;
    long long per = maxcols * N0;
    long long g = (per + 255) / 256;
    if (g > 4096) g = 4096;
    dim3 grid((unsigned)g, (unsigned)nq);
    block64_kernel<<<grid, 256, 0, st>>>(d_q, d_VB, d_Z, d_Y, RSc, nch, P, N0, full);
}

}  // namespace hfx
