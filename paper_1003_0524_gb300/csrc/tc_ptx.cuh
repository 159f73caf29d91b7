// tc_ptx.cuh -- inline-PTX helpers for the tensor-core kernels (sm_103a):
// mbarriers with bounded waits, TMA tile loads, tcgen05 MMA / commit / TMEM
// allocation and loads, shared-memory matrix descriptors, and the
// fixed-point slice helpers shared by every slice GEMM.
#pragma once

#include "hfx_internal.cuh"

namespace hfx {
namespace tc {

constexpr unsigned long long kWaitNs = 2000000000ULL;  // 2 s

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P1;\n\tmbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\tselp.b32 %0, 1, 0, P1;\n\t}"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    return ok;
}
// Bounded wait.  Returns false (and raises the CTA abort flag and the global
// error word) if the phase did not complete in time or the CTA is aborting.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int *err,
                                          int code) {
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            unsigned long long now = gtimer();
            if (t0 == 0) t0 = now;
            else if (now - t0 > kWaitNs) {
                *abort_flag = 1;
                atomicCAS(err, 0, code);
                return false;
            }
        }
    }
}
// Bounded wait on a barrier that nothing completes, for the fault-injection
// hook of the tests: gives up after ns nanoseconds like mbar_wait does.
__device__ __forceinline__ bool mbar_wait_ns(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int *err,
                                             int code, unsigned long long ns) {
    unsigned long long t0 = gtimer();
    for (;;) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (gtimer() - t0 > ns) {
            *abort_flag = 1;
            atomicCAS(err, 0, code);
            return false;
        }
    }
}
// Best-effort bounded wait used only while draining after an abort.
__device__ __forceinline__ void mbar_drain(uint64_t *bar, uint32_t parity) {
    unsigned long long t0 = gtimer();
    while (!mbar_try(bar, parity)) {
        if (gtimer() - t0 > kWaitNs) return;
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::
            "r"(dst),
        "l"((uint64_t)map), "r"(saddr(bar)), "r"(x), "r"(y)
        : "memory");
}

// 1-D bulk copy global -> shared (both 16-byte aligned, bytes a multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"((uint64_t)src), "r"(bytes), "r"(saddr(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
                 : "memory");
}

// The MMA thread's last step: wait (bounded) until every tcgen05.mma it issued
// has completed, so that TMEM is never freed under an MMA still in flight
// (after an abort nothing else waits for them).  bar: an mbarrier of count 1
// used for nothing else.
__device__ __forceinline__ void umma_drain(uint64_t *bar) {
    umma_commit(bar);
    mbar_drain(bar, 0);
}

// ---- a pair of CTAs (cluster of two) working on one tile: cta_group::2
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// address of the same shared-memory object in CTA 0 of the cluster
__device__ __forceinline__ uint32_t in_cta0(const void *p) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(saddr(p)));
    return a;
}
// Relaxed: a release at cluster scope would wait for this thread's global stores (it held
// the drains of the modular apply at twice their time).  What it has to order, the
// tcgen05.ld of an accumulator before the MMAs that overwrite it, is complete by
// tcgen05.wait::ld and fenced by tcgen05.fence::before_thread_sync.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// a tile from shared memory to global memory (bulk group of the issuing thread)
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"((uint64_t)map), "r"(src),
                 "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// a tile into this CTA's shared memory that reports to a barrier of either CTA
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
        "[%2];" ::"r"(dst),
        "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t *slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// M = 256 over the pair (CTA 0 rows 0..127); N: the first half of B's rows in CTA 0
__device__ __forceinline__ void umma_bf16_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// arrive at the barrier at this address in both CTAs when the MMAs so far are done
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(saddr(bar)),
        "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void umma_drain_pair(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar)) : "memory");
    mbar_drain(bar, 0);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,"
        "%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, K-major operand, 128-byte swizzle:
// 8-row atoms of 1024 bytes (stride-byte-offset), leading offset unused.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes (rows
// 16 bytes apart); lbo = byte distance of the two core matrices adjacent in
// K, sbo = byte distance of core matrices adjacent in M/N.
__device__ __forceinline__ uint64_t desc_ns(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// K-major operand, 64-byte swizzle (rows of 32 BF16): 8-row atoms of 512 bytes.
__device__ __forceinline__ uint64_t desc_sw64(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

// The ten kept slice products s_a t_b (a + b <= 3) fall in four weight classes
// w = a + b, one TMEM accumulator of N columns each, class w at columns w N.
// The slice planes of B sit back to back in shared memory, so the products of
// one A slice a with B slices b, b + 1, ... form one MMA of width (count) N
// whose output starts at column (a + b) N.

// Instruction descriptor: BF16 x BF16 -> FP32, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}


// ------------------------------------------------------------- slices
constexpr int NPL = 4;      // slices per operand

// The slicing below runs on the integer units: GB300's FP64 pipe is far too
// narrow for a pass over every element of the projections.

// |x| as an integer that orders like |x| (non-negative doubles order like
// their bit patterns)
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
}

// exponent e with max < 2^e, from abs_bits(max) (0 for an all-zero line)
__device__ __forceinline__ int line_exp_bits(unsigned long long b) {
    if (b == 0) return 0;
    int E = (int)(b >> 52);
    return E == 0 ? -1021 : E - 1022;
}

// x (|x| < 2^e) as four balanced base-256 digits s_0..s_3 of
// N = round(x 2^(32-e)) (nearest, ties to even): x ~ sum_i s_i 2^(e-8(i+1)),
// |s_0| <= 256, |s_1..3| <= 128.  Each digit comes as the FP32 number whose upper
// half is its BF16 pattern (a digit has at most 8 significant bits).
//
// Ties are not rare: outputs of the slice products (T_n, Z, Y) carry few bits below
// the last digit, so the rounding of ties decides about 1e-10 of V^x.
// About 35 instructions: with 128 (1 + 256 + 65536) added to N, the three low digits
// are bytes, and a byte put under the exponent of 2^23 less 2^23 + 128 is the digit as
// a float.  Taking the digits one by one in 64 bits took twice as many and held the
// slicing of Y at 0.7 of the copy bandwidth (6.6 ms for 30 GB, 4.8 ms now).
struct Digits { uint32_t s[4]; };
// the digits of N, |N| <= 2^32
__device__ __forceinline__ Digits digits_of(long long N) {
    const unsigned long long v = (unsigned long long)N + 0x808080ULL;
    const uint32_t vl = (uint32_t)v, vh = (uint32_t)(v >> 32);
    Digits d;
    d.s[0] = __float_as_uint(__int_as_float(0x4B400000 + (int)__funnelshift_r(vl, vh, 24)) - 12582912.0f);
    d.s[1] = __float_as_uint(__uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7442)) - 8388736.0f);
    d.s[2] = __float_as_uint(__uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7441)) - 8388736.0f);
    d.s[3] = __float_as_uint(__uint_as_float(__byte_perm(vl, 0x4B000000u, 0x7440)) - 8388736.0f);
    return d;
}
__device__ __forceinline__ Digits slice4f(double x, int e) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int E = (int)((hi >> 20) & 0x7ffu);
    // N = m 2^-sh; sh >= 21 because |x| < 2^e; zeros and subnormals give 0
    const int sh = E ? 1043 + e - E : 64;
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const int s1 = min(sh, 63);
    const unsigned long long r = m + ((1ULL << (s1 - 1)) - 1) + ((m >> s1) & 1ULL);
    const unsigned long long q = sh < 64 ? r >> s1 : 0ULL;
    const unsigned long long neg = (unsigned long long)((long long)(int)hi >> 63);
    return digits_of((long long)((q ^ neg) - neg));
}
// x 2^p as an integer with F fraction bits, truncated (|x| 2^(p + F) < 2^62)
__device__ __forceinline__ long long f32_fixed(float x, int k) {   // k = p + F
    const uint32_t b = __float_as_uint(x);
    const int E = (int)((b >> 23) & 0xffu), sh = E - 150 + k;
    const unsigned long long m = E ? (unsigned long long)((b & 0x7fffffu) | 0x800000u) : 0ULL;
    const unsigned long long a = sh >= 0 ? m << min(sh, 39) : (sh > -24 ? m >> -sh : 0ULL);
    return (int)b < 0 ? -(long long)a : (long long)a;
}
// round((s + e) 2^p), to nearest even as far as 2^-F of a unit
template <int F> __device__ __forceinline__ long long pair_round(float s, float e, int p) {
    const long long V = f32_fixed(s, p + F) + f32_fixed(e, p + F);
    return (V + ((1LL << (F - 1)) - 1) + ((V >> F) & 1)) >> F;
}
// the BF16 patterns of two digits (their FP32 bits) in one word
__device__ __forceinline__ uint32_t pack_digits(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x7632); }

// The same digits as BF16 numbers.
__device__ __forceinline__ void slice4(double x, int e, __nv_bfloat16 *o /* 4 */) {
    const Digits d = slice4f(x, e);
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = __ushort_as_bfloat16((unsigned short)(d.s[i] >> 16));
}

// Combine the four exact class sums of one K group (units 2^(eA+eB-16)) and
// add them, scaled by sc, into the compensated pair (hi, lo).
__device__ __forceinline__ void class_accumulate(float a0, float a1, float a2, float a3, float sc, float &hi,
                                                 float &lo) {
    float c = fmaf(a3, 0x1p-8f, a2);
    c = fmaf(c, 0x1p-8f, a1);
    float x = a0 * sc;
    float s = hi + x;
    float bb = s - hi;
    float er = (hi - (s - bb)) + (x - bb);
    hi = s;
    lo += er + c * (0x1p-8f * sc);
}

// Packed FP32 pairs (two columns per instruction; each lane rounds to nearest
// exactly as the scalar operation does).
__device__ __forceinline__ uint64_t f2_pack(uint32_t x, uint32_t y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(x), "r"(y));
    return r;
}
__device__ __forceinline__ float2 f2_unpack(uint64_t v) {
    uint32_t x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(x), "=r"(y) : "l"(v));
    return make_float2(__uint_as_float(x), __uint_as_float(y));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// s + e = h + l exactly, s = fl(h + l), for two columns at once
__device__ __forceinline__ void f2_two_sum(uint64_t h, uint64_t l, float2 &s, float2 &e) {
    const uint64_t t = f2_add(h, l), bb = f2_sub(t, h);
    s = f2_unpack(t);
    e = f2_unpack(f2_add(f2_sub(h, f2_sub(t, bb)), f2_sub(l, bb)));
}
// 32 bytes to global memory (32-byte aligned) in one store, not kept in L2
__device__ __forceinline__ void st_global_32(void *p, const float4 &a, const float4 &b) {
    asm volatile("st.global.cs.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(__float_as_uint(a.x)),
                 "r"(__float_as_uint(a.y)), "r"(__float_as_uint(a.z)), "r"(__float_as_uint(a.w)), "r"(__float_as_uint(b.x)),
                 "r"(__float_as_uint(b.y)), "r"(__float_as_uint(b.z)), "r"(__float_as_uint(b.w))
                 : "memory");
}

// class_accumulate (sc = 1) for two columns at once; a_w hold the class sums
// of the two columns as packed pairs.
__device__ __forceinline__ void class_accumulate2(uint64_t a0, uint64_t a1, uint64_t a2, uint64_t a3, uint64_t &hi,
                                                  uint64_t &lo) {
    const uint64_t s8 = f2_pack(0x3b800000u, 0x3b800000u);   // 2^-8, 2^-8
    uint64_t c = f2_fma(a3, s8, a2);
    c = f2_fma(c, s8, a1);
    const uint64_t s = f2_add(hi, a0);
    const uint64_t bb = f2_sub(s, hi);
    const uint64_t er = f2_add(f2_sub(hi, f2_sub(s, bb)), f2_sub(a0, bb));
    hi = s;
    lo = f2_add(lo, f2_fma(c, s8, er));
}

// the bits of ldexpf(1, k), also where it is subnormal, zero or infinite
__device__ __forceinline__ uint32_t pow2_bits(int k) {
    return k >= -126 ? (uint32_t)(min(k, 128) + 127) << 23 : (k >= -149 ? 1u << (k + 149) : 0u);
}

// class_accumulate for two columns with per-column scales sc (packed pair)
__device__ __forceinline__ void class_accumulate2_sc(uint64_t a0, uint64_t a1, uint64_t a2, uint64_t a3, uint64_t sc,
                                                     uint64_t &hi, uint64_t &lo) {
    const uint64_t s8 = f2_pack(0x3b800000u, 0x3b800000u);   // 2^-8, 2^-8
    uint64_t c = f2_fma(a3, s8, a2);
    c = f2_fma(c, s8, a1);
    const uint64_t x = f2_mul(a0, sc);
    const uint64_t s = f2_add(hi, x);
    const uint64_t bb = f2_sub(s, hi);
    const uint64_t er = f2_add(f2_sub(hi, f2_sub(s, bb)), f2_sub(x, bb));
    hi = s;
    lo = f2_add(lo, f2_fma(c, f2_mul(s8, sc), er));
}

// x * 2^k as a double for a normal FP32 x (or zero), built from the bits of x
// with 32-bit integer operations: no FP64 conversion.  FP32 subnormals give 0.
// The scaled exponent must stay in the normal FP64 range.
__device__ __forceinline__ double f32_to_f64_scaled(float x, int k) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t e = (b >> 23) & 0xffu;
    const uint32_t hi = e ? (b & 0x80000000u) | ((e + 896u + (uint32_t)k) << 20) | ((b & 0x7fffffu) >> 3) : 0u;
    const uint32_t lo = e ? b << 29 : 0u;
    return __hiloint2double((int)hi, (int)lo);
}

// (h + l) * 2^k for FP32 h, l: the two exact scaled conversions and one FP64
// add, the correctly rounded sum (exact when the exponents of h and l are
// within 29).  One FP64 operation per output: GB300's FP64 pipe is narrow, and
// the epilogues convert one value per output element.
__device__ __forceinline__ double f32pair_to_f64(float h, float l, int k) {
    return f32_to_f64_scaled(h, k) + f32_to_f64_scaled(l, k);
}

// The same value by integer operations only (no FP64 operation): both terms
// on a common 62-bit fixed point 38 bits below the larger exponent, added, and
// rounded to 53 bits, to nearest even.  Correctly rounded when the exponents
// of h and l are within 38; a smaller term further below is truncated there
// (at most one unit in the last place).  Results below the normal range give 0.
__device__ __forceinline__ double f32pair_to_f64_int(float h, float l, int k) {
    const uint32_t bh = __float_as_uint(h), bl = __float_as_uint(l);
    const int beh = (bh >> 23) & 0xff, bel = (bl >> 23) & 0xff;
    long long mh = (long long)((bh & 0x7fffffu) | (beh ? 0x800000u : 0u));
    long long ml = (long long)((bl & 0x7fffffu) | (bel ? 0x800000u : 0u));
    if (bh >> 31) mh = -mh;
    if (bl >> 31) ml = -ml;
    const int eh = (beh ? beh : 1) - 150, el = (bel ? bel : 1) - 150;   // value = m * 2^e
    const int emax = mh ? (ml ? max(eh, el) : eh) : el;
    const int e0 = emax - 38;
    const int dh = eh - e0, dl = el - e0;                                // the larger term: shift 38
    // (a signed term times 2^d as a product: left shifts of negative values are not defined)
    const long long S = (dh >= 0 ? mh * (1LL << dh) : (dh > -63 ? mh >> -dh : (mh < 0 ? -1 : 0))) +
                        (dl >= 0 ? ml * (1LL << dl) : (dl > -63 ? ml >> -dl : (ml < 0 ? -1 : 0)));
    if (S == 0) return 0.0;
    const unsigned long long sgn = S < 0 ? (1ULL << 63) : 0ULL;
    unsigned long long a = S < 0 ? (unsigned long long)(-S) : (unsigned long long)S;
    const int lz = __clzll(a);
    a <<= lz;                                                           // bit 63 set
    unsigned long long m = a >> 11;                                     // 53 bits
    const unsigned long long rem = a & 0x7ffULL;
    if (rem > 0x400ULL || (rem == 0x400ULL && (m & 1ULL))) ++m;         // may carry to 2^53: exponent + 1 below
    const long long bexp = (long long)(e0 + k - lz) + 63 + 1023;        // biased exponent of the leading bit
    if (bexp < 1) return 0.0;
    return __longlong_as_double((long long)(sgn | (((unsigned long long)(bexp - 1) << 52) + m)));
}

// The digits of one complex row of a column with exponent e: an FP64 pair, or an FP32
// pair (s_r, e_r, s_i, e_i) in units of 2^ce.
__device__ __forceinline__ void slice_row(const uint4 &v, bool f32, int e, int ce, Digits &re, Digits &im) {
    if (f32) {
        re = digits_of(pair_round<24>(__uint_as_float(v.x), __uint_as_float(v.y), 32 - e + ce));
        im = digits_of(pair_round<24>(__uint_as_float(v.z), __uint_as_float(v.w), 32 - e + ce));
    } else {
        re = slice4f(__hiloint2double((int)v.y, (int)v.x), e);
        im = slice4f(__hiloint2double((int)v.w, (int)v.z), e);
    }
}

// S + E += a * b for double-FP32 a = (ah, al), b = (bh, bl): the product's
// rounding error from an FMA, the cross terms to first order, S updated by an
// exact two-sum whose error joins E.  Relative error about 2^-46.
__device__ __forceinline__ void df_mac(float ah, float al, float bh, float bl, float &S, float &E) {
    const float p = ah * bh;
    const float pe = fmaf(ah, bh, -p);
    const float cross = fmaf(ah, bl, al * bh);
    const float s = S + p;
    const float bb = s - S;
    const float err = (S - (s - bb)) + (p - bb);
    S = s;
    E += err + (pe + cross);
}

// (h, l) -> (s, e) with s = fl(h + l) and s + e = h + l exactly (two-sum)
__device__ __forceinline__ void two_sum(float h, float l, float &s, float &e) {
    s = h + l;
    const float bb = s - h;
    e = (h - (s - bb)) + (l - bb);
}

// 2^d as a float for d <= 0 (0 below the normal range)
__device__ __forceinline__ float pow2f_neg(int d) { return d >= -126 ? __int_as_float((127 + d) << 23) : 0.0f; }

int make_map_2d(hfx_ctx *ctx, CUtensorMap *m, const void *ptr, long long rows, long long cols, int box_rows);
int make_map_2d_sw(hfx_ctx *ctx, CUtensorMap *m, const void *ptr, long long rows, long long cols, int box_rows,
                   int box_cols, int swizzle_bytes);
int num_sms();

}  // namespace tc
}  // namespace hfx
