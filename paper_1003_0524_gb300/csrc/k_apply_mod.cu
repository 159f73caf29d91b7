// k_apply_mod.cu -- the Coulomb apply Y' = U Z of large dense blocks as exact integer
// products modulo nine small numbers (tcgen05.mma kind::f16 with BF16 operands).
//
// Every row of U (the dense-block rows of the upper triangle of v_t with half its
// diagonal) and every column of Z is scaled by a power of two and rounded to complex
// integers a, b of Euclidean norm below 2^39.39.  Then |Re|, |Im| of sum_k a_k b_k stay
// below M / 2 for M = m_1 ... m_9 = 2^79.79, and the sum is known exactly from its
// residues modulo the m_i (Chinese remainder theorem).  Modulo m, a product of primes
// = 1 mod 4, there is a j with j^2 = -1, and x + i y -> (x + j y, x - j y) turns one
// complex product into two real ones.  So a complex product costs 18 real products of
// residues |r| <= 255, instead of the 40 of the digit scheme (ten digit products for
// each of the four real products of the embedding [[Re, -Im], [Im, Re]]).
//
// A residue is an integer of at most 8 bits, exact in BF16; a product sum over 256 K
// values stays below 2^24 and is exact in the FP32 accumulators, after which the
// accumulator is reduced modulo m on the CUDA cores and added up as a small integer.
// The only error is the rounding of the operands, whose units are at most 2^-38.39 of
// the line's norm.  The norm is at most sqrt(2 D) times the largest component, so up to
// 6144 functions a unit is at most 2^-31.6 of that component, however the line is
// distributed, where the digits have 2^-32 to 2^-31 of it and drop products besides.
// Error of Y' over its largest element, D = 1280, 2660, 6144, by a model of both
// roundings: elements of equal size 4e-11, 5e-11, 9e-11 (digits 1e-10 at each), Gaussian
// 5e-11, 5e-11, 9e-11 (1.4e-9, 1.8e-9, 1.9e-9), decaying 4e-12 (5e-9 to 1e-8).  Eight
// moduli (norms below 2^35.04) were 11 % fewer products, but at equal size 7e-10, 1.9e-9,
// 1.4e-9, above the digits.
//
// The residues of Z and of Y' take 36 bytes per complex element each (the digits of Z
// and Y' in FP64 16 each), so the scheme pays where the products outweigh the extra
// traffic; apply_mod_usable holds the rule and its figures.
#include <algorithm>
#include <cmath>
#include <string>

#include "tc_ptx.cuh"

namespace hfx {

using namespace tc;

namespace {

// ------------------------------------------------------------- moduli
constexpr int NM = 9, NRP = 2 * NM;                       // moduli; residue planes (x + j y, x - j y per modulus)
constexpr int kMod[NM] = {509, 505, 493, 481, 461, 457, 449, 433, 421};
constexpr float kHalfBits = 39.399f;                      // (log2 M - 1) / 2 = 39.39907, rounded down

constexpr int mod_root(int m) {
    for (int j = 1; j < m; ++j)
        if ((j * j + 1) % m == 0) return j;
    return 0;
}
constexpr int mod_inv(int a, int m) {
    for (int x = 1; x < m; ++x)
        if ((long long)a * x % m == 1) return x;
    return 0;
}
constexpr int balanced(long long a, int m) {
    const int r = (int)(((a % m) + m) % m);
    return r > m / 2 ? r - m : r;
}
constexpr int others(int i) {                             // M / m_i mod m_i
    long long p = 1;
    for (int k = 0; k < NM; ++k)
        if (k != i) p = p * kMod[k] % kMod[i];
    return (int)p;
}
constexpr double mod_product() {
    double p = 1.0;
    for (int k = 0; k < NM; ++k) p *= kMod[k];
    return p;
}
// round(2^64 c / m)
constexpr unsigned long long frac64(int c, int m) {
    unsigned long long q = 0, r = (unsigned long long)c;
    for (int b = 0; b < 64; ++b) {
        r *= 2;
        q = 2 * q + (r >= (unsigned long long)m ? 1 : 0);
        if (r >= (unsigned long long)m) r -= m;
    }
    return 2 * r >= (unsigned long long)m ? q + 1 : q;
}
struct ModTab {
    float m[NM] = {}, inv[NM] = {};                       // modulus and its reciprocal
    float c13[NM] = {}, c26[NM] = {};                     // 2^13, 2^26 mod m
    float d0[NM] = {}, d13[NM] = {}, d26[NM] = {};        // j, j 2^13, j 2^26 mod m
    // x mod M = M frac(sum_i (p_i + q_i) re_i), y = M frac(sum_i (p_i - q_i) im_i): 64-bit
    // fractions, the low word as a signed number
    int re_lo[NM] = {}, im_lo[NM] = {};
    unsigned re_hi[NM] = {}, im_hi[NM] = {};
};
constexpr ModTab make_tab() {
    ModTab t;
    for (int i = 0; i < NM; ++i) {
        const int m = kMod[i], j = mod_root(m), oi = mod_inv(others(i), m);
        t.m[i] = (float)m;
        t.inv[i] = 1.0f / (float)m;
        t.c13[i] = (float)balanced(1LL << 13, m);
        t.c26[i] = (float)balanced(1LL << 26, m);
        t.d0[i] = (float)balanced(j, m);
        t.d13[i] = (float)balanced((long long)j << 13, m);
        t.d26[i] = (float)balanced((long long)j << 26, m);
        const unsigned long long wr = frac64((int)((long long)mod_inv(2, m) * oi % m), m);
        const unsigned long long wi = frac64((int)((long long)mod_inv(2 * j % m, m) * oi % m), m);
        t.re_lo[i] = (int)(unsigned)wr;
        t.re_hi[i] = (unsigned)(wr >> 32) + ((unsigned)wr >> 31);
        t.im_lo[i] = (int)(unsigned)wi;
        t.im_hi[i] = (unsigned)(wi >> 32) + ((unsigned)wi >> 31);
    }
    return t;
}
__constant__ ModTab kTab = make_tab();
// U is scaled by kKappa = M / 2^79 besides its power of two, so that a result is its
// 64-bit fraction times a power of two, 2^kFracExp for operands of scale 1
constexpr double kKappa = mod_product() / 604462909807314587353088.0;
constexpr int kFracExp = 79 - 64;
static_assert(kKappa > 1.7387, "2^(2 kHalfBits + 1) exceeds M");

// ------------------------------------------------------------- residues
__device__ __forceinline__ uint64_t f2_both(float x) { return f2_pack(__float_as_uint(x), __float_as_uint(x)); }

// |N| < 2^39.4 as three pieces N = p2 2^26 + p1 2^13 + p0, |p0|, |p1| <= 4096,
// |p2| < 10810
__device__ __forceinline__ void pieces_of(long long N, float (&p)[3]) {
    const unsigned long long v = (unsigned long long)N + 0x2001000ULL;   // 2^25 + 2^12
    const uint32_t vl = (uint32_t)v, vh = (uint32_t)(v >> 32);
    p[0] = __uint_as_float(0x4B000000u | (vl & 0x1fffu)) - 8392704.0f;
    p[1] = __uint_as_float(0x4B000000u | ((vl >> 13) & 0x1fffu)) - 8392704.0f;
    p[2] = __int_as_float(0x4B400000 + (int)__funnelshift_r(vl, vh, 26)) - 12582912.0f;
}
// The pieces of round(|x| 2^s) with the sign of x (0 for zeros and subnormals)
__device__ __forceinline__ void int_pieces(double x, int s, float (&p)[3]) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int E = (int)((hi >> 20) & 0x7ffu);
    const int sh = E ? max(1074 - E - s, 0) : 64;         // one bit below the unit; >= 12 by |x| 2^s < 2^40
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const unsigned long long q = ((sh < 64 ? m >> sh : 0ULL) + 1) >> 1;
    const unsigned long long neg = (unsigned long long)((long long)(int)hi >> 63);
    pieces_of((long long)((q ^ neg) - neg), p);
}

// p - m round(p / m) for packed integers |p| < 2^24: at most 255 (the rounding of p / m may
// miss the nearest integer by 0.002)
__device__ __forceinline__ uint64_t f2_reduce(uint64_t p, int i) {
    const uint64_t magic = f2_both(12582912.0f);
    const uint64_t k = f2_sub(f2_fma(p, f2_both(kTab.inv[i]), magic), magic);
    return f2_fma(k, f2_both(-kTab.m[i]), p);
}
__device__ __forceinline__ uint32_t f2_bf16(uint64_t v) { return __byte_perm((uint32_t)v, (uint32_t)(v >> 32), 0x7632); }

// The residues of two complex integers (packed pieces) modulo m_i as BF16 pairs:
// x + j y and x - j y, from sums below 254 (10810 + 4096 + 1) + 254 (10810 + 2 4096) < 2^23.1.
__device__ __forceinline__ void residues(const uint64_t (&X)[3], const uint64_t (&Y)[3], int i, uint32_t &plus, uint32_t &minus) {
    const uint64_t a = f2_fma(X[2], f2_both(kTab.c26[i]), f2_fma(X[1], f2_both(kTab.c13[i]), X[0]));
    const uint64_t b = f2_fma(Y[2], f2_both(kTab.d26[i]), f2_fma(Y[1], f2_both(kTab.d13[i]), f2_mul(Y[0], f2_both(kTab.d0[i]))));
    plus = f2_bf16(f2_reduce(f2_add(a, b), i));
    minus = f2_bf16(f2_reduce(f2_sub(a, b), i));
}
__device__ __forceinline__ uint64_t f2_pieces(float a, float b) { return f2_pack(__float_as_uint(a), __float_as_uint(b)); }

// Sum of squares as s 2^(2 (ref - 1023)), ref the largest biased exponent so far: a
// running scale, so that any magnitude of the data is covered.
struct SquareSum {
    int ref = 0;
    float s = 0.0f;
    __device__ __forceinline__ void rescale(int to) {     // to >= ref
        s = to - ref > 60 ? 0.0f : s * __int_as_float((127 - 2 * min(to - ref, 60)) << 23);
        ref = to;
    }
    __device__ __forceinline__ float part(double x) const {   // x 2^-(ref - 1023), truncated to 20 bits
        const uint32_t hi = (uint32_t)__double2hiint(x);
        const int E = (int)((hi >> 20) & 0x7ffu), e = E - ref + 127;
        return E && e > 0 ? __uint_as_float(((uint32_t)e << 23) | ((hi & 0xfffffu) << 3)) : 0.0f;
    }
    __device__ __forceinline__ void add(const double2 &v) {
        const int e = (int)max(((uint32_t)__double2hiint(v.x) >> 20) & 0x7ffu, ((uint32_t)__double2hiint(v.y) >> 20) & 0x7ffu);
        if (e > ref) rescale(e);
        const float a = part(v.x), b = part(v.y);
        s = fmaf(a, a, fmaf(b, b, s));
    }
    __device__ __forceinline__ void join(int r2, float s2) {
        if (r2 > ref) rescale(r2);
        SquareSum o;
        o.ref = r2;
        o.s = s2;
        if (ref > r2) o.rescale(ref);
        s += o.s;
    }
    // power of two that takes the norm just below 2^bits (margins: the truncation of
    // part(), the FP32 sum, the rounding of up to 2 x 6144 components to integers)
    __device__ __forceinline__ int scale(float bits) const {
        if (!(s > 0.0f)) return 0;
        return (int)floorf(bits - 0.002f - 0.5f * log2f(s)) - (ref - 1023);
    }
};

// ------------------------------------------------------------- U
// Residues of the dense-block rows of U: one block per row r of one q; planes
// UR[t][row][Kp], zero below the diagonal and in the padding.
__global__ void __launch_bounds__(256) mod_u_kernel(const double2 *__restrict__ VD, __nv_bfloat16 *__restrict__ UR,
                                                    int *__restrict__ uexp, int D, int naux, int N0, int Dp, int Kp) {
    const int r = blockIdx.x, tid = threadIdx.x;
    __shared__ int s_ref[8], s_e;
    __shared__ float s_s[8];
    const double2 *row = VD + (size_t)r * naux + N0;
    auto get = [&](int k) {
        double2 v = make_double2(0.0, 0.0);
        if (r < D && k >= r && k < D) {
            v = row[k];
            const double w = k == r ? 0.5 * kKappa : kKappa;
            v.x *= w;
            v.y *= w;
        }
        return v;
    };
    SquareSum n;
    for (int k = r + tid; k < D; k += 256) n.add(get(k));
    for (int o = 16; o > 0; o >>= 1) n.join(__shfl_xor_sync(0xffffffffu, n.ref, o), __shfl_xor_sync(0xffffffffu, n.s, o));
    if (tid % 32 == 0) { s_ref[tid / 32] = n.ref; s_s[tid / 32] = n.s; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 8; ++w) n.join(s_ref[w], s_s[w]);
        s_e = n.scale(kHalfBits);
        uexp[r] = s_e;
    }
    __syncthreads();
    const int e = s_e;
    for (int k = 4 * tid; k < Kp; k += 1024) {
        float x[4][3], y[4][3];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const double2 v = get(k + t);
            int_pieces(v.x, e, x[t]);
            int_pieces(v.y, e, y[t]);
        }
#pragma unroll
        for (int i = 0; i < NM; ++i) {
            uint32_t p[2], q[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint64_t X[3], Y[3];
#pragma unroll
                for (int u = 0; u < 3; ++u) { X[u] = f2_pieces(x[2 * h][u], x[2 * h + 1][u]); Y[u] = f2_pieces(y[2 * h][u], y[2 * h + 1][u]); }
                residues(X, Y, i, p[h], q[h]);
            }
            __nv_bfloat16 *d = UR + ((size_t)(2 * i) * Dp + r) * Kp + k;
            *reinterpret_cast<uint2 *>(d) = make_uint2(p[0], p[1]);
            *reinterpret_cast<uint2 *>(d + (size_t)Dp * Kp) = make_uint2(q[0], q[1]);
        }
    }
}

// ------------------------------------------------------------- Z
// The digits of Z (all rows, for Z^H Y) and the residues of its dense rows (for the
// apply), from the interstitial rows (F32: the interstitial kernel's plane ZI [g][col] of
// FP32 pairs in units of 2^cexp[col]; else Z itself, where a caller's projections are in
// it) and the muffin-tin rows of Z; the layout and the passes of slice_z_kernel, with the
// sum of squares of the dense rows beside the maximum.  Bound by memory: 32 bytes read, 52 written per element.
constexpr int MZ_COLS = 8, MZ_THREADS = 256, MZ_NJ = MZ_THREADS / MZ_COLS, MZ_CH = 4 * MZ_NJ, MZ_CS = MZ_CH + 8;
constexpr size_t kMzSmem = (size_t)(2 * NPL + NRP) * MZ_COLS * MZ_CS * sizeof(__nv_bfloat16);
template <bool F32>
__global__ void __launch_bounds__(MZ_THREADS, 3) mod_z_kernel(const float4 *__restrict__ ZI, long long NCi,
                                                           const int *__restrict__ cexp,
                                                           const double2 *__restrict__ Z, long long RSc,
                                                           const QDesc *__restrict__ qd, int nmt, int N0, int N0pad, int HS,
                                                           int RS, int Kp, long long NC, __nv_bfloat16 *__restrict__ XS,
                                                           __nv_bfloat16 *__restrict__ ZR, int *__restrict__ xexp,
                                                           int *__restrict__ zexp) {
    constexpr int NJ = MZ_NJ, CH = MZ_CH, CS = MZ_CS;
    extern __shared__ __align__(16) unsigned char mz_smem[];
    __nv_bfloat16 *stage = reinterpret_cast<__nv_bfloat16 *>(mz_smem);   // [2 planes x part | residue plane][column][CS]
    __shared__ unsigned long long red[MZ_THREADS / 32][MZ_COLS];
    __shared__ int rref[MZ_THREADS / 32][MZ_COLS];
    __shared__ float rsum[MZ_THREADS / 32][MZ_COLS];
    const QDesc q = qd[blockIdx.y];
    const long long c0 = (long long)blockIdx.x * MZ_COLS;
    if (c0 >= q.ncols) return;
    const int tid = threadIdx.x, c = tid % MZ_COLS, j = tid / MZ_COLS;
    const bool live = c0 + c < q.ncols;
    const long long col = q.colbase + (live ? c0 + c : c0);
    const double2 *z = Z + col * RSc;
    const float4 *zi = ZI + col;
    const int ce = F32 ? cexp[col] : 0;
    unsigned long long mx = 0;
    SquareSum n;
    for (int i = j; i < (F32 ? nmt : nmt + q.nipw); i += NJ) {
        const double2 v = z[i];
        mx = max(mx, max(abs_bits(v.x), abs_bits(v.y)));
        if (i >= N0) n.add(v);
    }
    if (F32) {
        // sums of integers below 2^30 in units of the column's exponent: no scale needed
        uint32_t mf = 0;
        float s = 0.0f;
#pragma unroll 8
        for (int g = j; g < q.nipw; g += NJ) {
            const float4 v = zi[(size_t)g * NCi];
            mf = max(mf, max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.z) & 0x7fffffffu));
            s = fmaf(v.x, v.x, fmaf(v.z, v.z, s));
        }
        const unsigned long long mp = abs_bits(f32pair_to_f64_int(__uint_as_float(mf), 0.0f, ce));   // 0 below the normal range
        mx = max(mx, mp);
        if (mp) n.join(1023 + ce + 16, s * 0x1p-32f);
    }
#pragma unroll
    for (int o = 8; o <= 16; o <<= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int r2 = __shfl_xor_sync(0xffffffffu, n.ref, o);
        const float s2 = __shfl_xor_sync(0xffffffffu, n.s, o);
        n.join(r2, s2);
    }
    if (tid % 32 < MZ_COLS) { red[tid / 32][c] = mx; rref[tid / 32][c] = n.ref; rsum[tid / 32][c] = n.s; }
    __syncthreads();
    n = SquareSum();
#pragma unroll
    for (int w = 0; w < MZ_THREADS / 32; ++w) { mx = max(mx, red[w][c]); n.join(rref[w][c], rsum[w][c]); }
    const int e = line_exp_bits(mx), sb = n.scale(kHalfBits);
    if (j == 0 && live) { xexp[col] = e; zexp[col] = sb; }
    const int nd = nmt - N0;                       // muffin-tin rows among the dense ones
    const long long plane = NC * RS, rplane = NC * Kp;
    uint4 v[4];                                    // this thread's four rows of a chunk, as they are
    auto fetch = [&](int u) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int dr = u + t - N0pad;          // dense row
            v[t] = make_uint4(0, 0, 0, 0);
            if (F32 && dr >= nd) {
                if (dr < q.D) v[t] = *reinterpret_cast<const uint4 *>(zi + (size_t)(dr - nd) * NCi);
            } else if (dr >= 0) {
                if (dr < q.D) v[t] = *reinterpret_cast<const uint4 *>(z + N0 + dr);
            } else if (u + t < N0) {
                v[t] = *reinterpret_cast<const uint4 *>(z + u + t);
            }
        }
    };
    fetch(4 * j);
    const int uend = max(HS, N0pad + Kp);
    for (int u0 = 0; u0 < uend; u0 += CH) {
        __syncthreads();                           // the chunk before has been stored
        {
            Digits sr[4], si[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) slice_row(v[t], F32 && u0 + 4 * j + t - N0pad >= nd, e, ce, sr[t], si[t]);
#pragma unroll
            for (int p = 0; p < NPL; ++p) {
                __nv_bfloat16 *s = stage + (size_t)((2 * p) * MZ_COLS + c) * CS + 4 * j;
                *reinterpret_cast<uint2 *>(s) = make_uint2(pack_digits(sr[0].s[p], sr[1].s[p]), pack_digits(sr[2].s[p], sr[3].s[p]));
                *reinterpret_cast<uint2 *>(s + MZ_COLS * CS) =
                    make_uint2(pack_digits(si[0].s[p], si[1].s[p]), pack_digits(si[2].s[p], si[3].s[p]));
            }
        }
        if (u0 + CH > N0pad) {
            float x[4][3], y[4][3];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (F32 && u0 + 4 * j + t - N0pad >= nd) {
                    pieces_of(pair_round<20>(__uint_as_float(v[t].x), __uint_as_float(v[t].y), sb + ce), x[t]);
                    pieces_of(pair_round<20>(__uint_as_float(v[t].z), __uint_as_float(v[t].w), sb + ce), y[t]);
                } else {
                    int_pieces(__hiloint2double((int)v[t].y, (int)v[t].x), sb, x[t]);
                    int_pieces(__hiloint2double((int)v[t].w, (int)v[t].z), sb, y[t]);
                }
            }
            uint64_t X[2][3], Y[2][3];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    X[h][u] = f2_pieces(x[2 * h][u], x[2 * h + 1][u]);
                    Y[h][u] = f2_pieces(y[2 * h][u], y[2 * h + 1][u]);
                }
#pragma unroll
            for (int i = 0; i < NM; ++i) {
                uint32_t p[2], m[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) residues(X[h], Y[h], i, p[h], m[h]);
                __nv_bfloat16 *s = stage + (size_t)((2 * NPL + 2 * i) * MZ_COLS + c) * CS + 4 * j;
                *reinterpret_cast<uint2 *>(s) = make_uint2(p[0], p[1]);
                *reinterpret_cast<uint2 *>(s + MZ_COLS * CS) = make_uint2(m[0], m[1]);
            }
        }
        if (u0 + CH < uend) fetch(u0 + CH + 4 * j);   // the next chunk, while this one is stored
        __syncthreads();
        const int nplane = u0 + CH > N0pad ? 2 * NPL + NRP : 2 * NPL;
        for (int t = tid; t < nplane * MZ_COLS * (CH / 8); t += MZ_THREADS) {
            const int x = t % (CH / 8), line = t / (CH / 8), cc = line % MZ_COLS, pp = line / MZ_COLS, u = u0 + 8 * x;
            if (c0 + cc >= q.ncols) continue;
            const uint4 w = *reinterpret_cast<const uint4 *>(stage + (size_t)line * CS + 8 * x);
            const long long cl = q.colbase + c0 + cc;
            if (pp < 2 * NPL) {                    // pp = 2 plane + part
                if (u < HS) __stcs(reinterpret_cast<uint4 *>(XS + (pp >> 1) * plane + cl * RS + (pp & 1) * HS + u), w);
            } else if (u >= N0pad && u < N0pad + Kp) {
                __stcs(reinterpret_cast<uint4 *>(ZR + (pp - 2 * NPL) * rplane + cl * Kp + (u - N0pad)), w);
            }
        }
    }
}

// ------------------------------------------------------------- products
// Tile: 256 columns of Z (M) x 256 rows of U (N) of one residue plane, shared by the two
// CTAs of a cluster (cta_group::2): each loads 128 columns and 128 rows, 64 bytes per
// cycle and SM at the full MMA rate, where a CTA by itself with 128 x 256 would need 96
// (10.4 ms against 7.9 on 96000 columns of 2660 functions with eight moduli; 9.2 with nine; the digit products: 16.7).  K from the tile's first row on (U is upper
// triangular); three stages of 128 K values (64 KB; with twice the stages of half the size the
// issuing thread's waits and commits left the tensor cores idle a third of the time); two
// accumulators of 256 TMEM columns, so that the drain of one K group of 256 overlaps the
// products of the next.  CTA r holds rows [64 r, 64 r + 64) and [128 + 64 r, 192 + 64 r)
// of the tile: in the diagonal block (the first K group) the first chunk meets only rows
// [0, 128), the first 64 of either CTA, as one MMA of N = 128, and the second takes two; in the later groups one MMA of N = 256 takes all, so a row's TMEM column depends on
// the group.  warpgroup 0: warp 0 TMA, warp 1 MMA (CTA 0 only); warpgroups 1, 2: epilogue
// (TMEM lane quarter = column of Z, half = the rows of CTA 0 or 1).
// A finished tile leaves through shared memory (a warp's 32 columns x 64 rows as two
// swizzled boxes) by TMA stores: storing 32 bytes per lane and column straight to memory
// took 4200 cycles of the 11300 a tile's products take.
//
// Tiles of one residue plane: {q, first row | K chunks << 16, first column, end of the q's
// columns}, by q, groups of M_COLGROUP column tiles, row tiles, columns of the group (the
// tiles running at once share a few rows of U and columns of Z in L2); the planes one
// after the other.
struct MParams {
    const int4 *tiles;
    int ntiles, nplane;      // all planes; of one
    int Dp;
    long long NC;
    short *YR;               // [t][col][Kp] residues of Y'
    int Kp;
    int *err;
};

constexpr int M_BM = 256, M_BN = 256, M_KC = 128, M_STAGES = 3, M_COLGROUP = 4;
// per CTA and stage: two blocks of 64 K values of the columns, then two of the rows
constexpr int M_KB = 64, M_AB = M_BM / 2 * M_KB * 2, M_BB = M_BN / 2 * M_KB * 2, M_STAGE = 2 * (M_AB + M_BB);
constexpr int M_GROUP = 256 / M_KC;                        // chunks per exact K group
constexpr int M_OUT = 8 * 4096;                            // staging of the results: 4 KB per epilogue warp
constexpr int M_THREADS = 384;
constexpr int M_REG_LAUNCH = 168, M_REG_CTRL = 64, M_REG_EPI = 216;
static_assert(4 * M_REG_CTRL + 8 * M_REG_EPI <= 12 * M_REG_LAUNCH, "register split exceeds the launch allocation");

// Walks a CTA pair's tiles; the next descriptor is loaded one tile ahead.
struct MWalk {
    const MParams &p;
    int e, t, step, left;    // entry, plane; tiles still to do
    int4 nx;
    __device__ MWalk(const MParams &p_, int first, int step_) : p(p_), e(first), t(0), step(step_) {
        left = first < p.ntiles ? (p.ntiles - first + step - 1) / step : 0;
        wrap();
        if (left > 0) nx = p.tiles[e];
    }
    __device__ __forceinline__ void wrap() {
        while (e >= p.nplane) { e -= p.nplane; ++t; }
    }
    // the next tile and its plane; false at the end
    __device__ __forceinline__ bool next(int4 &d, int &plane) {
        if (left == 0) return false;
        d = nx;
        plane = t;
        if (--left > 0) {
            e += step;
            wrap();
            nx = p.tiles[e];
        }
        return true;
    }
};
__device__ __forceinline__ int mt_row0(const int4 &d) { return d.y & 0xffff; }
__device__ __forceinline__ int mt_chunks(const int4 &d) { return d.y >> 16; }

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(M_THREADS, 1)
    mod_gemm_kernel(const __grid_constant__ CUtensorMap tmZ, const __grid_constant__ CUtensorMap tmU,
                    const __grid_constant__ CUtensorMap tmY, const MParams p) {
    extern __shared__ __align__(1024) unsigned char mg_smem[];
    uintptr_t base = (reinterpret_cast<uintptr_t>(mg_smem) + 1023) & ~(uintptr_t)1023;
    unsigned char *stages = reinterpret_cast<unsigned char *>(base);
    // full, tempty: those of CTA 0 count for the pair; empty, tfull: each CTA its own
    __shared__ uint64_t full_bar[M_STAGES], empty_bar[M_STAGES], tfull_bar[2], tempty_bar[2], mma_done;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int rank = (int)cluster_rank(), first = blockIdx.x / 2, step = gridDim.x / 2;
    if (threadIdx.x == 0) {
        for (int s = 0; s < M_STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&tfull_bar[s], 1);
            mbar_init(&tempty_bar[s], 16);
        }
        mbar_init(&mma_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc_pair(&tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(M_REG_CTRL));
        if (warp == 0 && lane == 0) {
            int s = 0, issued = 0, plane;
            uint32_t ph = 0;
            MWalk walk(p, first, step);
            int4 tl;
            while (!abort_flag && walk.next(tl, plane)) {
                const int yz = (int)(plane * p.NC) + tl.z + rank * (M_BM / 2);
                const int yu = (tl.x * NRP + plane) * p.Dp + mt_row0(tl) + rank * 64;
                const int nchunk = mt_chunks(tl);
                bool stop = false;
                for (int kc = 0; kc < nchunk; ++kc) {
                    if (!mbar_wait(&empty_bar[s], ph ^ 1, &abort_flag, p.err, kDevTimeoutTma)) { stop = true; break; }
                    const uint32_t st = saddr(stages + (size_t)s * M_STAGE), full = in_cta0(&full_bar[s]);
                    if (rank == 0) mbar_expect_tx(&full_bar[s], 2 * M_STAGE);
                    const int x = mt_row0(tl) + kc * M_KC;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {   // (K past the padded end is filled with zeros)
                        tma_load_2d_pair(st + h * M_AB, &tmZ, full, x + h * M_KB, yz);
                        tma_load_2d_pair(st + 2 * M_AB + h * M_BB, &tmU, full, x + h * M_KB, yu);
                        tma_load_2d_pair(st + 2 * M_AB + h * M_BB + M_BB / 2, &tmU, full, x + h * M_KB, yu + 128);
                    }
                    ++issued;
                    if (++s == M_STAGES) { s = 0; ph ^= 1; }
                }
                if (stop) break;
            }
            if (abort_flag && rank == 0) {   // the loads of both CTAs report here; CTA 1 waits at the end
                for (int i = 0; i < M_STAGES && i < issued; ++i) mbar_drain(&full_bar[i], 0), mbar_drain(&full_bar[i], 1);
            }
        } else if (warp == 1 && lane == 0 && rank == 0) {
            int s = 0, b = 0, plane;
            uint32_t ph = 0, eph = 0;
            bool ok = true;
            MWalk walk(p, first, step);
            int4 tl;
            constexpr uint32_t id_half = idesc_bf16(M_BM, M_BN / 2), id_full = idesc_bf16(M_BM, M_BN);
            while (ok && walk.next(tl, plane)) {
                const int nchunk = mt_chunks(tl);
                for (int g0 = 0; g0 < nchunk && ok; g0 += M_GROUP) {
                    if (!mbar_wait(&tempty_bar[b], eph ^ 1, &abort_flag, p.err, kDevTimeoutMma)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t acc = tmem + b * M_BN;
                    for (int kc = g0; kc < min(nchunk, g0 + M_GROUP); ++kc) {
                        if (!mbar_wait(&full_bar[s], ph, &abort_flag, p.err, kDevTimeoutMma)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t a0 = saddr(stages + (size_t)s * M_STAGE), b0 = a0 + 2 * M_AB;
                        const uint64_t da = desc_sw128(a0), db = desc_sw128(b0);
                        // K step ks: 32 bytes further in its block of 64 K values
                        auto at = [](int ks, int block) { return (uint64_t)(2 * (ks % 4) + ks / 4 * (block >> 4)); };
                        if (g0 == 0) {
#pragma unroll
                            for (int ks = 0; ks < M_KC / 16; ++ks) {
                                umma_bf16_pair(acc, da + at(ks, M_AB), db + at(ks, M_BB), id_half, kc || ks ? 1u : 0u);
                                if (kc)
                                    umma_bf16_pair(acc + M_BN / 2, da + at(ks, M_AB), db + at(ks, M_BB) + (M_BB / 2 >> 4), id_half,
                                                   ks ? 1u : 0u);
                            }
                        } else {
#pragma unroll
                            for (int ks = 0; ks < M_KC / 16; ++ks)
                                umma_bf16_pair(acc, da + at(ks, M_AB), db + at(ks, M_BB), id_full, kc > g0 || ks ? 1u : 0u);
                        }
                        umma_commit_pair(&empty_bar[s]);
                        if (++s == M_STAGES) { s = 0; ph ^= 1; }
                    }
                    if (!ok) break;
                    umma_commit_pair(&tfull_bar[b]);
                    b ^= 1;
                    if (!b) eph ^= 1;
                }
            }
            umma_drain_pair(&mma_done);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(M_REG_EPI));
        const int quarter = warp % 4, half = (warp - 4) / 4;
        int b = 0, plane;
        uint32_t eph = 0;
        bool ok = true;
        unsigned char *out = stages + (size_t)M_STAGES * M_STAGE + (warp - 4) * 4096;
        MWalk walk(p, first, step);
        int4 tl;
        const uint64_t magic = f2_both(12582912.0f);
        while (ok && walk.next(tl, plane)) {
            const uint64_t inv = f2_both(kTab.inv[plane >> 1]), neg = f2_both(-kTab.m[plane >> 1]);   // this plane's modulus
            const int ngroups = (mt_chunks(tl) + M_GROUP - 1) / M_GROUP;
            // rows of the tile that exist in the padded planes (columns that the last, short
            // diagonal block never wrote lie beyond)
            const int rows = min(M_BN, p.Kp - mt_row0(tl));
            uint64_t acc[M_BN / 4];   // packed pairs: this half's rows, 64 of each half of the tile
#pragma unroll
            for (int i = 0; i < M_BN / 4; ++i) acc[i] = 0;
            for (int g = 0; g < ngroups; ++g) {
                if (!mbar_wait(&tfull_bar[b], eph, &abort_flag, p.err, kDevTimeoutEpi)) { ok = false; break; }
                tc_fence_after();
                // the TMEM columns of this half's two runs of 64 rows
                const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + b * M_BN + half * (g == 0 ? 64 : 128);
                const uint32_t tb1 = tb + (g == 0 ? 128 : 64);
                auto take = [&](const uint32_t (&x)[32], int c) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        // exact integers below 2^24: reduced modulo m and added
                        const uint64_t v = f2_pack(x[i], x[i + 1]);
                        const uint64_t k = f2_sub(f2_fma(v, inv, magic), magic);
                        acc[(c + i) / 2] = f2_add(acc[(c + i) / 2], f2_fma(k, neg, v));
                    }
                };
                // 32 columns are reduced while the next 32 are on their way
                uint32_t xa[32], xb[32];
                tmem_ld32(tb, xa);
                tmem_wait_ld();
                tmem_ld32(tb + 32, xb);
                take(xa, 0);
                tmem_wait_ld();
                tmem_ld32(tb1, xa);
                take(xb, 32);
                tmem_wait_ld();
                tmem_ld32(tb1 + 32, xb);
                take(xa, 64);
                tmem_wait_ld();
                tc_fence_before();   // everything read: hand the accumulator back
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(in_cta0(&tempty_bar[b]));
                take(xb, 96);
                b ^= 1;
                if (!b) eph ^= 1;
            }
            if (!ok) break;
            // residues as 16-bit integers: rows half * 64 + [0, 64), then 128 more
            const int col = tl.z + rank * (M_BM / 2) + quarter * 32;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (lane == 0) bulk_wait_read();   // the staging is free again
                __syncwarp();
#pragma unroll
                for (int c = 0; c < 64; c += 8) {
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint64_t v = acc[(h * 64 + c) / 2 + i];
                        const uint64_t k = f2_sub(f2_fma(v, inv, magic), magic);
                        // 1.5 2^23 + r: the low half of its bits is r in two's complement
                        const uint64_t r = f2_add(f2_fma(k, neg, v), magic);
                        w[i] = __byte_perm((uint32_t)r, (uint32_t)(r >> 32), 0x5410);
                    }
                    // 128-byte swizzle of the box: 16-byte piece c / 8 of column `lane`
                    *reinterpret_cast<uint4 *>(out + lane * 128 + (((c / 8) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
                const int row = h * 128 + half * 64;
                if (col + 32 <= tl.w) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0 && row < rows) {
                        tma_store_2d(&tmY, saddr(out), mt_row0(tl) + row, (int)(plane * p.NC) + col);
                        bulk_commit();
                    }
                } else {
                    // the last columns of a q: the box would reach into the next one's
                    __syncwarp();
                    for (int i = lane; i < 32 * 8; i += 32) {
                        const int cc = i / 8, piece = i % 8;
                        if (col + cc < tl.w && row < rows)
                            *reinterpret_cast<uint4 *>(p.YR + (plane * p.NC + col + cc) * p.Kp + mt_row0(tl) + row + piece * 8) =
                                *reinterpret_cast<const uint4 *>(out + cc * 128 + ((piece ^ (cc & 7)) << 4));
                    }
                    __syncwarp();
                }
            }
        }
        if (lane == 0) bulk_wait();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // no CTA leaves while the other's MMAs, copies or arrivals can still reach it
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 512);
    }
}

// ------------------------------------------------------------- Y
// From the residues of Y' (dense rows) and the FP64 mu = 0 rows Y0 [col][N0] to the digits
// of Y' for Z^H Y.  One block per column: the values F 2^e of the dense rows (F: the 64-bit
// fraction of the residues, see ModTab) stay in shared memory between the pass that finds
// the column's exponent and the one that cuts the digits.  Bound by memory: 36 bytes
// read and 16 written per element, and the ~110 integer operations of an element.
constexpr int MY_THREADS = 256;
__device__ __forceinline__ int bit_length(long long f) { return 64 - __clzll(f < 0 ? -f : f); }

// digits of F 2^(x - 32) relative to 2^0, i.e. of N = round(F 2^x), |N| <= 2^32 (ties to even)
__device__ __forceinline__ Digits slice_i64(long long F, int x) {
    const unsigned long long a = F < 0 ? (unsigned long long)(-F) : (unsigned long long)F;
    unsigned long long q;
    if (x >= 0) {
        q = a << min(x, 63);   // |N| < 2^32: no bit is lost
    } else {
        const int s = min(-x, 63);
        q = (a + ((1ULL << (s - 1)) - 1) + ((a >> s) & 1ULL)) >> s;
        if (-x > 63) q = 0;
    }
    const unsigned long long neg = (unsigned long long)(F >> 63);
    return digits_of((long long)((q ^ neg) - neg));
}

__global__ void __launch_bounds__(MY_THREADS) mod_y_kernel(const short *__restrict__ YR, const double2 *__restrict__ Y0,
                                                           const QDesc *__restrict__ qd, const int *__restrict__ uexp, int Dp,
                                                           const int *__restrict__ zexp, int N0, int N0pad, int HS, int RS,
                                                           int Kp, long long NC, __nv_bfloat16 *__restrict__ YS,
                                                           int *__restrict__ yexp) {
    extern __shared__ __align__(16) unsigned char my_smem[];
    longlong2 *val = reinterpret_cast<longlong2 *>(my_smem);   // [4][Kp / 4]: row 4 g + t at [t][g]
    __shared__ int red[MY_THREADS / 32];
    const QDesc q = qd[blockIdx.y];
    const int *ue = uexp + (size_t)q.iq * Dp;
    const int tid = threadIdx.x, ng = Kp / 4;
    const long long plane = NC * RS, rplane = NC * Kp;
    for (long long cc = blockIdx.x; cc < q.ncols; cc += gridDim.x) {
        const long long col = q.colbase + cc;
        const int sb = zexp[col];
        int emax = -100000;
        for (int u = tid; u < N0; u += MY_THREADS) {
            const double2 v = Y0[col * N0 + u];
            const unsigned long long b = max(abs_bits(v.x), abs_bits(v.y));
            if (b) emax = max(emax, line_exp_bits(b));
        }
        for (int g = tid; 4 * g < q.D; g += MY_THREADS) {
            long long lr[4] = {0, 0, 0, 0}, li[4] = {0, 0, 0, 0};
            unsigned hr[4] = {0, 0, 0, 0}, hi[4] = {0, 0, 0, 0};
#pragma unroll
            for (int i = 0; i < NM; ++i) {
                const short *src = YR + (long long)(2 * i) * rplane + col * Kp + 4 * g;
                const uint2 p = __ldcs(reinterpret_cast<const uint2 *>(src));
                const uint2 m = __ldcs(reinterpret_cast<const uint2 *>(src + rplane));
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const uint32_t pw = t < 2 ? p.x : p.y, mw = t < 2 ? m.x : m.y;
                    const int a = t & 1 ? (int)pw >> 16 : (int)(short)pw, b = t & 1 ? (int)mw >> 16 : (int)(short)mw;
                    lr[t] += (long long)(a + b) * kTab.re_lo[i];
                    hr[t] += (unsigned)(a + b) * kTab.re_hi[i];
                    li[t] += (long long)(a - b) * kTab.im_lo[i];
                    hi[t] += (unsigned)(a - b) * kTab.im_hi[i];
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                longlong2 f;
                f.x = (long long)((unsigned long long)lr[t] + ((unsigned long long)hr[t] << 32));
                f.y = (long long)((unsigned long long)li[t] + ((unsigned long long)hi[t] << 32));
                val[t * ng + g] = f;
                if (4 * g + t < q.D && (f.x | f.y))
                    emax = max(emax, max(bit_length(f.x), bit_length(f.y)) + kFracExp - ue[4 * g + t] - sb);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
        if (tid % 32 == 0) red[tid / 32] = emax;
        __syncthreads();
        int e = red[0];
#pragma unroll
        for (int w = 1; w < MY_THREADS / 32; ++w) e = max(e, red[w]);
        if (e <= -100000) e = 0;
        if (tid == 0) yexp[col] = e;
        for (int u = 4 * tid; u < HS; u += 4 * MY_THREADS) {
            Digits sr[4], si[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int dr = u + t - N0pad;
                if (dr >= 0) {
                    // (dr and t: N0pad is a multiple of 4, so row dr sits at [t][(u - N0pad) / 4])
                    const bool in = dr < q.D;
                    const longlong2 f = in ? val[t * ng + (u - N0pad) / 4] : make_longlong2(0, 0);
                    const int x = in ? kFracExp - ue[dr] - sb + 32 - e : 0;
                    sr[t] = slice_i64(f.x, x);
                    si[t] = slice_i64(f.y, x);
                } else {
                    const double2 v = u + t < N0 ? Y0[col * N0 + u + t] : make_double2(0.0, 0.0);
                    sr[t] = slice4f(v.x, e);
                    si[t] = slice4f(v.y, e);
                }
            }
#pragma unroll
            for (int p = 0; p < NPL; ++p) {
                const uint2 wr = make_uint2(pack_digits(sr[0].s[p], sr[1].s[p]), pack_digits(sr[2].s[p], sr[3].s[p]));
                const uint2 wi = make_uint2(pack_digits(si[0].s[p], si[1].s[p]), pack_digits(si[2].s[p], si[3].s[p]));
                *reinterpret_cast<uint2 *>(YS + p * plane + col * RS + u) = wr;
                *reinterpret_cast<uint2 *>(YS + p * plane + col * RS + HS + u) = wi;
            }
        }
        __syncthreads();   // val and red are free for the next column
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// From 1664 dense functions on.  Builds with residues and with digits, ms:
//   functions        1285         1425         1625         1825         2025
//   8 k, 120 bands   20.4 / 18.7  21.9 / 20.7  24.6 / 24.4  28.2 / 28.5  30.2 / 32.2
//   8 k, 40 bands    3.62 / 3.47                            4.82 / 4.96
// (20 and 8 bands occupied: 154000 and 20500 columns; the products take 0.65 to 0.75 of
// those of the digits from 1425 on, the extra residues grow with the size alone), and
//   functions               1285         1625         1925         2425         6125
//   one k, 4800 columns     3.05 / 3.04  3.57 / 3.57  4.17 / 4.15  5.14 / 5.33  13.1 / 14.4
//   one k, 320 columns      0.80 / 0.81  0.92 / 0.92  1.01 / 1.03  1.17 / 1.21  2.56 / 2.69
// Few columns do not change the line much: below it they lose up to 0.03 ms (48 columns:
// 0.48 / 0.50 at 1285).  Up to 6144, where the unit of the residues still is no larger
// than the largest one of the digits (2^-31 of a line's largest element, see above).
bool apply_mod_usable(int maxD) { return maxD >= 1664 && maxD <= 6144; }

int apply_mod_products() { return NRP; }

ModSizes apply_mod_sizes(int maxD) {
    ModSizes z;
    z.Kp = (maxD + M_KB - 1) / M_KB * M_KB;
    z.Dp = (maxD + M_BN - 1) / M_BN * M_BN;
    z.u_elems = (size_t)NRP * z.Dp * z.Kp;
    z.col_bytes = (size_t)NRP * z.Kp * 2;
    return z;
}

int apply_mod_prepare_u(hfx_ctx *ctx, const double2 *d_VD, __nv_bfloat16 *d_UR, int *d_uexp, int D, int naux, int N0,
                        const ModSizes &z) {
    mod_u_kernel<<<z.Dp, 256, 0, ctx->stream>>>(d_VD, d_UR, d_uexp, D, naux, N0, z.Dp, z.Kp);
    return cuda_check(ctx, cudaGetLastError(), "residues of U");
}

int apply_mod_tiles(const QDesc *h_q, int nq, std::vector<unsigned char> &out) {
    std::vector<int4> tiles;
    for (int i = 0; i < nq; ++i) {
        const QDesc &q = h_q[i];
        const int kend = (q.D + M_KC - 1) / M_KC * M_KC;
        const long long cend = q.colbase + q.ncols;
        for (long long g0 = q.colbase; g0 < cend; g0 += (long long)M_BM * M_COLGROUP)
            for (int r = 0; r < q.D; r += M_BN)
                for (int j = 0; j < M_COLGROUP; ++j) {
                    const long long c = g0 + (long long)j * M_BM;
                    if (c < cend) tiles.push_back(make_int4(q.iq, r | ((kend - r) / M_KC) << 16, (int)c, (int)cend));
                }
    }
    if (tiles.size() > (size_t)0x7fffffff / NRP) return -1;
    out.assign(reinterpret_cast<const unsigned char *>(tiles.data()),
               reinterpret_cast<const unsigned char *>(tiles.data()) + tiles.size() * sizeof(int4));
    return (int)tiles.size();
}

int apply_mod_slice_z(hfx_ctx *ctx, const float4 *d_ZI, const int *d_cexp, const double2 *d_Z, long long RSc,
                      const QDesc *d_q, int nq, long long NC, long long maxcols, int nmt, int N0, int N0pad, int HS, int RS,
                      const ModSizes &z, __nv_bfloat16 *d_ZS, __nv_bfloat16 *d_ZR, int *d_xexp, int *d_zexp) {
    if (nq == 0 || maxcols == 0) return HFX_OK;
    const dim3 grid((unsigned)((maxcols + MZ_COLS - 1) / MZ_COLS), (unsigned)nq);
    auto go = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMzSmem);
        kern<<<grid, MZ_THREADS, kMzSmem, ctx->stream>>>(d_ZI, NC, d_cexp, d_Z, RSc, d_q, nmt, N0, N0pad, HS, RS, z.Kp, NC, d_ZS,
                                                         d_ZR, d_xexp, d_zexp);
    };
    if (d_ZI) go(mod_z_kernel<true>);
    else go(mod_z_kernel<false>);
    return cuda_check(ctx, cudaGetLastError(), "residues of Z");
}

int apply_mod_run(hfx_ctx *ctx, const __nv_bfloat16 *d_UR_all, int nk, const __nv_bfloat16 *d_ZR, short *d_YR, long long NC,
                  const ModSizes &z, const void *d_tiles, int nplane) {
    if (nplane == 0) return HFX_OK;
    if (NC > 0x7fffffffLL / NRP || (long long)nk * NRP * z.Dp > 0x7fffffffLL)
        return set_err(ctx, HFX_EUNSUPPORTED, "batch has too many columns for 32-bit TMA coordinates");
    int rc;
    CUtensorMap mZ, mU, mY;
    if ((rc = make_map_2d_sw(ctx, &mZ, d_ZR, (long long)NRP * NC, z.Kp, M_BM / 2, M_KB, 128)) ||
        (rc = make_map_2d_sw(ctx, &mU, d_UR_all, (long long)nk * NRP * z.Dp, z.Kp, 64, M_KB, 128)) ||
        (rc = make_map_2d_sw(ctx, &mY, d_YR, (long long)NRP * NC, z.Kp, 32, 64, 128)))
        return rc;
    MParams p;
    p.tiles = reinterpret_cast<const int4 *>(d_tiles);
    p.nplane = nplane;
    p.ntiles = nplane * NRP;
    p.Dp = z.Dp;
    p.Kp = z.Kp;
    p.NC = NC;
    p.YR = d_YR;
    p.err = ctx->d_err;
    const size_t smem = (size_t)M_STAGES * M_STAGE + M_OUT + 1024;
    cudaFuncSetAttribute(mod_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    {
        // the register split of the kernel assumes this launch allocation
        cudaFuncAttributes fa;
        if ((rc = cuda_check(ctx, cudaFuncGetAttributes(&fa, mod_gemm_kernel), "apply attributes"))) return rc;
        if (fa.numRegs < M_REG_LAUNCH)
            return set_err(ctx, HFX_EUNSUPPORTED, "apply compiled with fewer registers than its warpgroup split needs");
    }
    const int pairs = std::max(1, std::min(num_sms() / 2, p.ntiles));
    mod_gemm_kernel<<<2 * pairs, M_THREADS, smem, ctx->stream>>>(mZ, mU, mY, p);
    return cuda_check(ctx, cudaGetLastError(), "modular apply");
}

int apply_mod_slice_y(hfx_ctx *ctx, const short *d_YR, const double2 *d_Y0, const QDesc *d_q, int nq, const int *d_uexp,
                      const int *d_zexp, long long NC, long long maxcols, int N0, int N0pad, int HS, int RS, const ModSizes &z,
                      __nv_bfloat16 *d_YS, int *d_yexp) {
    if (nq == 0 || maxcols == 0) return HFX_OK;
    const size_t smem = (size_t)z.Kp * sizeof(longlong2);
    cudaFuncSetAttribute(mod_y_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const dim3 grid((unsigned)std::min<long long>(maxcols, 152 * 64), (unsigned)nq);
    mod_y_kernel<<<grid, MY_THREADS, smem, ctx->stream>>>(d_YR, d_Y0, d_q, d_uexp, z.Dp, d_zexp, N0, N0pad, HS, RS, z.Kp, NC,
                                                          d_YS, d_yexp);
    return cuda_check(ctx, cudaGetLastError(), "slices of Y");
}

}  // namespace hfx
