// Tile-level device functions of the contraction kernels.  One call computes one work tile of
// one step; the per-step kernels map blocks to tiles, the persistent kernel claims tiles from a
// global work list.  Inside one persistent launch an arena address is rewritten by later steps, so an SM
// must never see a stale L1 line: operand loads bypass L1 (ld.global.cg), or, where only 8-byte
// asynchronous copies fit (which pass through L1), come after the block's wait for the operand's producer,
// an acquire at GPU scope, or read leaves and program results, complete before the launch.
#pragma once

#include <cstdint>

#include "kernels.cuh"

namespace tn {

template <typename T> struct Cx;
template <> struct Cx<float> { using t = float2; };
template <> struct Cx<double> { using t = double2; };
template <typename T> using cx_t = typename Cx<T>::t;

__device__ __forceinline__ float2 cmake(float r, float i) { return make_float2(r, i); }
__device__ __forceinline__ double2 cmake(double r, double i) { return make_double2(r, i); }

template <typename C>
__device__ __forceinline__ void cfma(C &acc, const C &a, const C &b) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}

template <typename C> __device__ __forceinline__ C ldc(const C *p) { return __ldcg(p); }

template <typename C> __device__ __forceinline__ C cscale(C v, decltype(C::x) s) {
    return cmake(v.x * s, v.y * s);
}

// Error-free transformations (Knuth's TwoSum; the FMA form of Dekker's TwoProduct, as used by
// Ogita, Rump and Oishi for accurate dot products), written with round-to-nearest intrinsics so
// that the compiler neither contracts nor reorders them: a + b = s + err and a * b = p + err
// exactly.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &err) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// A sum kept as an unevaluated pair hi + lo (about 44 significant bits); adds x = xh + xl.
__device__ __forceinline__ void df_add(float &hi, float &lo, float xh, float xl) {
    float s, t;
    two_sum(hi, xh, s, t);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(xl, t));
}

// The sum of one output of a small step.  In complex64 Re and Im are kept as hi + lo pairs of exact
// products and exact pairwise sums, rounded once when the output is stored: these steps are most of a
// circuit's steps, and with plain FP32 multiply-adds their several roundings per output (rather than
// the one of storing it) tripled the error of small amplitudes.
template <typename T> struct SmallSum;
template <> struct SmallSum<float> {
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    __device__ __forceinline__ void mac(float2 a, float2 b) {
        const float p1 = __fmul_rn(a.x, b.x), e1 = __fmaf_rn(a.x, b.x, -p1);
        const float p2 = __fmul_rn(a.y, b.y), e2 = __fmaf_rn(a.y, b.y, -p2);
        const float p3 = __fmul_rn(a.x, b.y), e3 = __fmaf_rn(a.x, b.y, -p3);
        const float p4 = __fmul_rn(a.y, b.x), e4 = __fmaf_rn(a.y, b.x, -p4);
        float s1, t1, s2, t2;
        two_sum(p1, -p2, s1, t1);
        two_sum(p3, p4, s2, t2);
        df_add(rh, rl, s1, __fadd_rn(__fsub_rn(e1, e2), t1));
        df_add(ih, il, s2, __fadd_rn(__fadd_rn(e3, e4), t2));
    }
    __device__ __forceinline__ void join(int32_t off) {
        const float orh = __shfl_xor_sync(0xffffffffu, rh, off), orl = __shfl_xor_sync(0xffffffffu, rl, off);
        const float oih = __shfl_xor_sync(0xffffffffu, ih, off), oil = __shfl_xor_sync(0xffffffffu, il, off);
        df_add(rh, rl, orh, orl);
        df_add(ih, il, oih, oil);
    }
    __device__ __forceinline__ float2 value() const { return cmake(__fadd_rn(rh, rl), __fadd_rn(ih, il)); }
};
template <> struct SmallSum<double> {
    double2 acc = {0.0, 0.0};
    __device__ __forceinline__ void mac(double2 a, double2 b) { cfma(acc, a, b); }
    __device__ __forceinline__ void join(int32_t off) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
    }
    __device__ __forceinline__ double2 value() const { return acc; }
};

// frexp-style exponent of the float with bit pattern `bits` (0 for zero): x = f * 2^e with f in
// [0.5, 1).  Subnormal maxima are treated as 2^-126.
__device__ __forceinline__ int32_t scale_exponent(uint32_t bits) {
    if (bits == 0u) return 0;
    int32_t e = (int32_t)((bits >> 23) & 0xffu);
    // a max-abs of 2^126 or more keeps e = 126, so that the scale 2^-e stays a normal float (the
    // scaled values then stay below 4); the exponent bookkeeping uses the same e
    return e == 0 ? -126 : (e - 126 > 126 ? 126 : e - 126);
}

// Exact 2^e built from the IEEE-754 exponent field (e within the normal range of T; the scale
// exponents used here stay in [-128, 128]).
template <typename T> __device__ __forceinline__ T pow2(int32_t e);
template <> __device__ __forceinline__ float pow2<float>(int32_t e) {
    e = e < -126 ? -126 : (e > 127 ? 127 : e);
    return __int_as_float((e + 127) << 23);
}
template <> __device__ __forceinline__ double pow2<double>(int32_t e) {
    e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// The same without the limits, for scales: scale_exponent is in [-126, 126], and sums of two are taken only where
// each is below 60 in magnitude.
template <typename T> __device__ __forceinline__ T pow2_scale(int32_t e);
template <> __device__ __forceinline__ float pow2_scale<float>(int32_t e) { return __int_as_float((e + 127) << 23); }
template <> __device__ __forceinline__ double pow2_scale<double>(int32_t e) {
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// Staged and small steps spend no multiplication on A's scale where none is needed: both scales go on B (fold),
// whose entries only grow by that when A's exponent is negative -- the products are those of scaled operands -- and
// a positive exponent of A is left out (set to 0: products, sums and stored values are larger by 2^eA, which their
// max-abs and exponents then say).  Neither costs range: scaling B down by A's exponent would, entries far
// below B's largest would become subnormal.  Exponents of 60 or more scale each operand on its own (false).
__device__ __forceinline__ bool scales_fold(int32_t eA, int32_t eB) {
    return (uint32_t)(eA + 59) < 119u && (uint32_t)(eB + 59) < 119u;
}
__device__ __forceinline__ bool leave_out_scale(int32_t &eA, int32_t eB) {
    const bool fold = scales_fold(eA, eB);
    if (fold) eA = min(eA, 0);
    return fold;
}

__device__ __forceinline__ float absmax2(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }
__device__ __forceinline__ float absmax2(double2 v) { return (float)fmax(fabs(v.x), fabs(v.y)); }

// Digits by division (dims that are not powers of two), kept out of line: inlined at each of its
// uses in every tile shape, the 64-bit divisions were most of the kernels' code (k_persist 1.2 MB),
// which does not stay in the instruction caches.
static __device__ __noinline__ int64_t group_off_div(const Groups *g, int64_t idx) {
    int64_t off = 0;
#pragma unroll 1
    for (int32_t i = 0; i < g->n; ++i) {
        const int64_t q = idx / g->dim[i];
        off += (idx - q * g->dim[i]) * g->sa[i];
        idx = q;
    }
    return off;
}
static __device__ __noinline__ longlong2 group_off2_div(const Groups *g, int64_t idx) {
    longlong2 off = make_longlong2(0, 0);
#pragma unroll 1
    for (int32_t i = 0; i < g->n; ++i) {
        const int64_t q = idx / g->dim[i], d = idx - q * g->dim[i];
        off.x += d * g->sa[i];
        off.y += d * g->sb[i];
        idx = q;
    }
    return off;
}

// Offset contributed by the digits of `idx` over a group list (stride `sa`).
__device__ __forceinline__ int64_t group_off(const Groups &g, int64_t idx) {
    if (!g.pow2) return group_off_div(&g, idx);
    int64_t off = 0;
#pragma unroll 4
    for (int32_t i = 0; i < g.n; ++i) off += ((idx >> g.lsb[i]) & g.mask[i]) * g.sa[i];
    return off;
}

// Offsets in A and B of a shared-leg multi-index.
__device__ __forceinline__ void group_off2(const Groups &g, int64_t idx, int64_t &oa, int64_t &ob) {
    if (!g.pow2) {
        const longlong2 o = group_off2_div(&g, idx);
        oa = o.x;
        ob = o.y;
        return;
    }
    oa = 0;
    ob = 0;
#pragma unroll 4
    for (int32_t i = 0; i < g.n; ++i) {
        const int64_t d = (idx >> g.lsb[i]) & g.mask[i];
        oa += d * g.sa[i];
        ob += d * g.sb[i];
    }
}

// The same, out of line (for uses that are unrolled or rare).
static __device__ __noinline__ int64_t group_off_call(const Groups *g, int64_t idx) { return group_off(*g, idx); }
static __device__ __noinline__ longlong2 group_off2_call(const Groups *g, int64_t idx) {
    int64_t a, b;
    group_off2(*g, idx, a, b);
    return make_longlong2(a, b);
}

// Copy a descriptor into shared memory (all threads), followed by a barrier.
__device__ __forceinline__ void load_desc(StepDesc &dst, const StepDesc *src) {
    const int4 *s = reinterpret_cast<const int4 *>(src);
    int4 *d = reinterpret_cast<int4 *>(&dst);
    for (int i = threadIdx.x; i < (int)(sizeof(StepDesc) / sizeof(int4)); i += blockDim.x)
        d[i] = __ldcg(s + i);
    __syncthreads();
}
static_assert(sizeof(StepDesc) % sizeof(int4) == 0 && alignof(StepDesc) % sizeof(int4) == 0 &&
                  alignof(StepHead) % sizeof(int4) == 0,
              "descriptors are copied in 16-byte pieces");

// The same copy in two halves, so that the loads can be in flight while thread 0 waits on the
// step's dependencies: desc_fetch issues them (one 16-byte piece per thread and round), desc_store
// writes the pieces to shared memory (the caller then synchronises).
constexpr int kDescPieces = (int)(sizeof(StepDesc) / sizeof(int4));
constexpr int kDescRounds = (kDescPieces + kThreads - 1) / kThreads;
__device__ __forceinline__ void desc_fetch(int4 (&r)[kDescRounds], const StepDesc *src) {
    const int4 *s = reinterpret_cast<const int4 *>(src);
#pragma unroll
    for (int q = 0; q < kDescRounds; ++q) {
        const int i = threadIdx.x + q * kThreads;
        if (i < kDescPieces) r[q] = __ldcg(s + i);
    }
}
__device__ __forceinline__ void desc_store(const int4 (&r)[kDescRounds], StepDesc &dst) {
    int4 *d = reinterpret_cast<int4 *>(&dst);
#pragma unroll
    for (int q = 0; q < kDescRounds; ++q) {
        const int i = threadIdx.x + q * kThreads;
        if (i < kDescPieces) d[i] = r[q];
    }
}

__device__ __forceinline__ float warp_max(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Block-wide max of non-negative values, then one atomicMax on the bit pattern (non-negative
// floats order like their bit patterns).  Ends with a barrier.
__device__ __forceinline__ void publish_max(float v, uint32_t *slot, float *red) {
    v = warp_max(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f;
        v = warp_max(v);
        if (lane == 0 && v > 0.f) atomicMax(slot, __float_as_uint(v));
    }
    __syncthreads();
}

template <typename C>
__device__ __forceinline__ const C *operand(const StepHead &d, const JobPtrs &j, bool is_a) {
    const bool leaf = is_a ? (d.flags & FLAG_A_LEAF) : (d.flags & FLAG_B_LEAF);
    const int64_t off = is_a ? d.a_off : d.b_off;
    return leaf ? static_cast<const C *>(j.leaf) + off : reinterpret_cast<const C *>(j.arena) + off;
}

__device__ __forceinline__ void step_scales(const StepHead &d, const JobPtrs &j, int32_t &eA, int32_t &eB) {
    eA = scale_exponent(__ldcg(j.maxbits + d.node_a));
    eB = scale_exponent(__ldcg(j.maxbits + d.node_b));
}

__device__ __forceinline__ void write_exponent(const StepHead &d, const JobPtrs &j, int32_t eA, int32_t eB) {
    j.exp2[d.node_c] = __ldcg(j.exp2 + d.node_a) + eA + __ldcg(j.exp2 + d.node_b) + eB;
}

// Shared-memory scratch needed by any tile function, per element type.
template <typename T> struct Scratch {
    using C = cx_t<T>;
    static constexpr int TK_MM = sizeof(T) == 4 ? 8 : 4;   // shared-index chunk of local_mm
    static constexpr int rows = kRowsMaxKN * sizeof(C) + kRowsMaxK * sizeof(int64_t);
    // GEMM: two stages of operand tiles, the largest 8 shared indices of 128 + 32 rows (complex64), of 32 + 32
    // (complex128), and the index arrays
    static constexpr int tile_rows = sizeof(T) == 4 ? 160 : 64;
    static constexpr int tile = 2 * 8 * (tile_rows + 2) * (int)sizeof(C) + (tile_rows + 48) * (int)sizeof(int64_t);
    static constexpr int dot = (kThreads / 32) * kDotMaxOut * sizeof(double2) + 2 * kDotMaxOut * sizeof(int64_t);
    // subtree programs: the register-tiled GEMM's operand tiles and offsets, or the REDUCE mode's
    // offset table and FP64 partials
    static constexpr int mm = (TK_MM * (257 + 65) * (int)sizeof(C) + (256 + 64) * 4 + TK_MM * 8 + 15) / 16 * 16;
    static constexpr int local = mm > 1024 * 8 + (kThreads / 32) * 16 ? mm : 1024 * 8 + (kThreads / 32) * 16;
    static constexpr int m1 = rows > tile ? rows : tile;
    static constexpr int m2 = dot > local ? dot : local;
    static constexpr int bytes = m1 > m2 ? m1 : m2;
};

// ------------------------------------------------------------------------------ ROWS
// Tiny-bond contraction (N <= NT <= 16, K <= 64): B (K x N) is staged in shared memory, each
// thread owns output rows m, reads their K entries of A through the index map and writes N
// consecutive outputs.  The K entries of a row are loaded in bursts of KC independent loads, so
// a row pays one memory latency per burst instead of one per entry.  HBM traffic: one read of A,
// one write of C.
template <typename T, int NT>
__device__ void tile_rows(const StepDesc &d, int64_t tile, const JobPtrs &j, char *smem, float *red) {
    using C = cx_t<T>;
    constexpr int KC = 8;
    C *Bs = reinterpret_cast<C *>(smem);
    int64_t *kA = reinterpret_cast<int64_t *>(smem + kRowsMaxKN * sizeof(C));
    const int32_t N = (int32_t)d.N, K = (int32_t)d.K;
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    const T sA = pow2<T>(-eA), sB = pow2<T>(-eB);
    const C *__restrict__ A = operand<C>(d, j, true);
    const C *__restrict__ B = operand<C>(d, j, false);
    C *__restrict__ Cp = reinterpret_cast<C *>(j.arena) + d.c_off;
    for (int32_t i = threadIdx.x; i < K * N; i += blockDim.x) {
        int32_t k = i / N, n = i - k * N;
        int64_t oa, ob;
        group_off2(d.k, k, oa, ob);
        ob += group_off(d.n, n);
        Bs[i] = cscale(ldc(B + ob), sB);
        if (n == 0) kA[k] = oa;
    }
    __syncthreads();
    const int64_t m_begin = tile * (int64_t)d.tile_rows;
    const int64_t m_end = min(d.M, m_begin + (int64_t)d.tile_rows);
    float mx = 0.f;
    for (int64_t m = m_begin + threadIdx.x; m < m_end; m += blockDim.x) {
        const C *Arow = A + group_off(d.m, m);
        C acc[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) acc[n] = cmake((T)0, (T)0);
        for (int32_t k0 = 0; k0 < K; k0 += KC) {
            C a[KC];
#pragma unroll
            for (int kk = 0; kk < KC; ++kk)
                a[kk] = (k0 + kk < K) ? ldc(Arow + kA[k0 + kk]) : cmake((T)0, (T)0);
#pragma unroll
            for (int kk = 0; kk < KC; ++kk) {
                if (k0 + kk >= K) break;
                const C av = cscale(a[kk], sA);
                const C *Bk = Bs + (k0 + kk) * N;
#pragma unroll
                for (int n = 0; n < NT; ++n)
                    if (n < N) cfma(acc[n], av, Bk[n]);
            }
        }
        C *out = Cp + m * N;
#pragma unroll
        for (int n = 0; n < NT; ++n)
            if (n < N) {
                out[n] = acc[n];
                mx = fmaxf(mx, absmax2(acc[n]));
            }
    }
    publish_max(mx, j.maxbits + d.node_c, red);
    if (tile == 0 && threadIdx.x == 0) write_exponent(d, j, eA, eB);
}

// A small step (the criterion of the subtree programs) that runs as a work tile of its own, complex64:
// an output per thread, summed as the programs do (SmallSum), so that its value does not depend on
// where it runs.
__device__ __forceinline__ void tile_small(const StepDesc &d, const JobPtrs &j, char *smem, float *red) {
    int2 *kt = reinterpret_cast<int2 *>(smem);   // [K <= 256] offsets in A and B
    const int32_t N = (int32_t)d.N, K = (int32_t)d.K, O = (int32_t)d.M * N;
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    const bool fold = leave_out_scale(eA, eB);
    const float sA = fold ? 1.f : pow2<float>(-eA), sB = pow2<float>(fold ? -eA - eB : -eB);
    const float2 *__restrict__ A = operand<float2>(d, j, true);
    const float2 *__restrict__ B = operand<float2>(d, j, false);
    float2 *__restrict__ Cp = reinterpret_cast<float2 *>(j.arena) + d.c_off;
    for (int32_t k = threadIdx.x; k < K; k += blockDim.x) {
        const longlong2 o = group_off2_call(&d.k, k);
        kt[k] = make_int2((int32_t)o.x, (int32_t)o.y);
    }
    __syncthreads();
    float mx = 0.f;
    for (int32_t o = threadIdx.x; o < O; o += blockDim.x) {
        const float2 *a = A + group_off_call(&d.m, o / N), *b = B + group_off_call(&d.n, o % N);
        SmallSum<float> sum;
#pragma unroll 4
        for (int32_t k = 0; k < K; ++k) sum.mac(cscale(ldc(a + kt[k].x), sA), cscale(ldc(b + kt[k].y), sB));
        const float2 v = sum.value();
        Cp[o] = v;
        mx = fmaxf(mx, absmax2(v));
    }
    publish_max(mx, j.maxbits + d.node_c, red);
    if (threadIdx.x == 0) write_exponent(d, j, eA, eB);
}

// Shared-memory layout of the large operand and of C of a staged step: element i of the dense row-major
// tensor sits at swz(i) -- inside each run of 16 elements (128 bytes) its 16-byte pairs are exchanged
// by an exclusive or with the higher index bits, so that threads that read or write elements 16 or more
// apart spread over the banks.  Pairs stay pairs (16-byte copies work), and swz is linear over index
// bits: swz(i | j) = swz(i) ^ swz(j) for disjoint bits.
__host__ __device__ __forceinline__ uint32_t swz(uint32_t i) {
    const uint32_t x = i >> 4;
    return i ^ (((x ^ (x >> 3) ^ (x >> 6) ^ (x >> 9)) & 7u) << 1);
}

// Block-wide max of non-negative values, returned to every thread.  Ends with a barrier.
__device__ __forceinline__ float block_max(float v, float *red) {
    v = warp_max(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f;
    v = warp_max(v);
    __syncthreads();
    return v;
}

// Phase cycle accounting of the profiling variant of the dataflow kernel (PROF), compiled out of
// the other one.
template <bool PROF>
__device__ __forceinline__ void prof_phase(long long *prof, int slot, long long &t) {
    if (PROF && threadIdx.x == 0) {
        const long long t1 = clock64();
        atomicAdd((unsigned long long *)(prof + slot), (unsigned long long)(t1 - t));
        atomicAdd((unsigned long long *)(prof + kProfSlots + slot), 1ull);
        t = t1;
    }
}

// cp.async of a staged step's A into its shared-memory layout (committed; the caller waits): swizzled for
// power-of-two dims -- the index bits of rows and shared indices are then disjoint, and the address of an
// entry is the exclusive or of its two parts -- else linear, where the parts add up.
__device__ __forceinline__ void stage_a(const StepHead &d, const JobPtrs &j, float2 *As, int32_t MK, bool p2) {
    const float2 *__restrict__ A = operand<float2>(d, j, true);
#pragma unroll 2
    for (int32_t i = threadIdx.x; 2 * i + 1 < MK; i += kThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(As + (p2 ? swz(2 * i) : 2 * i))),
                     "l"(A + 2 * i)
                     : "memory");
    if ((MK & 1) && threadIdx.x == 0)   // one entry, or no power of two
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(As + MK - 1)),
                     "l"(A + MK - 1)
                     : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Step staged whole through shared memory (complex64, FLAG_A_SMEM; one tile covers the step): A is
// copied with 16-byte cp.async into the swizzled layout -- or, for a continuation of a chain (a_res), is
// there already, left by the previous step -- and B, scaled and dense, goes next to it.  Each thread owns
// R rows x NC columns: the CG = rows_groups(N, NC) column groups lie on neighbouring lanes, the threads
// of a group rstep rows apart.  C then stays in shared memory (c_in_smem: the next step of the chain
// consumes it; the block's max-abs of C is returned) or leaves it in coalesced 16-byte stores.  Memory
// traffic: one read of A and B, one write of C (B alone inside a chain).  Ends with a barrier.
// Bound by shared-memory loads and the FMA pipe alike: a load instruction returns 128 bytes a cycle to the
// registers of the SM whether or not its lanes share addresses, so a shared index costs a warp 2 R + 2 NC
// cycles there against R NC of the pipe; 4 x 8 (24 against 32) keeps both short, where 2 x 16 took 36.
// With the column groups on lanes, a load of A has 32 / CG different rows, which the swizzle spreads over
// the banks, and one of B CG neighbouring pairs of columns.  Packed multiply-adds (fma.rn.f32x2) with B's
// parts duplicated were slower: 16 bytes an entry.
// Measured on 2432 24-qubit amplitudes (18 such steps in two chains each, 128 x 64 x 32, 256 x 32 x 32 and
// 512 x 16 x 16 the largest): the dataflow kernel 2.05 ms; 2.99 ms with 2 x 16 thread tiles, N <= 16
// only and the wider steps as separate GEMM tiles.
// next: the step that continues the chain (null: none); its B is fetched while this step multiplies.
// ahead: this step's B was fetched that way.
constexpr int kAheadPer = kRowsAhead / kThreads;
__device__ __forceinline__ int32_t b_entries(const StepHead &d) {
    const int nc = rows_nc(d.tile_shape);
    return (int32_t)d.K * rows_groups(d.N, nc) * nc;
}
__device__ __forceinline__ void b_ahead_offsets(const StepHead &d, const JobPtrs &j, int32_t (&o)[kAheadPer]) {
    if (d.tile_shape == kRowsShapeSmall) return;
    const int32_t *tab = reinterpret_cast<const int32_t *>(j.ktab + d.ktab_off) + d.M + d.K;
    const int32_t n = b_entries(d);
#pragma unroll
    for (int q = 0; q < kAheadPer; ++q) {
        const int32_t i = threadIdx.x + q * kThreads;
        o[q] = i < n ? __ldg(tab + i) : -2;
    }
}
__device__ __forceinline__ void b_ahead_copy(const StepHead &d, const JobPtrs &j, float2 *raw,
                                             const int32_t (&o)[kAheadPer]) {
    if (d.tile_shape == kRowsShapeSmall) return;
    const float2 *B = operand<float2>(d, j, false);
#pragma unroll
    for (int q = 0; q < kAheadPer; ++q) {
        const int32_t i = threadIdx.x + q * kThreads;
        if (o[q] >= 0)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(raw + i)),
                         "l"(B + o[q])
                         : "memory");
        else if (o[q] == -1) raw[i] = make_float2(0.f, 0.f);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int NC, int R, bool PROF>
__device__ float rows_smem_core(const StepHead &d, const JobPtrs &j, char *smem, char *dyn, float *red, int32_t eA,
                                int32_t eB, bool a_res, bool ahead, const StepHead *next, long long *prof) {
    long long tp = 0;
    if (PROF && threadIdx.x == 0) tp = clock64();
    using C = float2;
    const int32_t M = (int32_t)d.M, N = (int32_t)d.N, K = (int32_t)d.K, MK = M * K;
    const int32_t CG = rows_groups(N, NC), NB = CG * NC, rstep = kThreads / CG;
    const int tid = threadIdx.x, cg = tid & (CG - 1);
    // the step's table: byte offsets in A of its rows and of its shared indices, element offsets in B of
    // its (k, column) entries (-1: no such column)
    const int32_t *__restrict__ tab = reinterpret_cast<const int32_t *>(j.ktab + d.ktab_off);
    int32_t *kat = reinterpret_cast<int32_t *>(smem);
    C *As = reinterpret_cast<C *>(dyn);
    char *Bp = smem + kRowsTabBytes;
    if (K * NB * 8 > Scratch<float>::bytes - kRowsTabBytes) Bp = dyn + (MK * 8 + 15) / 16 * 16;
    C *Bs = reinterpret_cast<C *>(Bp);
    const C *__restrict__ B = operand<C>(d, j, false);
    const bool p2 = (d.flags & FLAG_A_POW2) != 0, c_in_smem = next != nullptr;
    if (!a_res) stage_a(d, j, As, MK, p2);
    const int32_t m0 = tid / CG;
    uint32_t row[R];   // absent rows read row 0
#pragma unroll
    for (int r = 0; r < R; ++r) row[r] = m0 + r * rstep < M ? (uint32_t)__ldg(tab + m0 + r * rstep) : 0u;
    if (tid < K) kat[tid] = __ldg(tab + M + tid);
    int32_t onext[kAheadPer];   // where the next step's B entries are
    if (c_in_smem) b_ahead_offsets(*next, j, onext);
    const bool fold = scales_fold(eA, eB);
    const float sB = pow2<float>(fold ? -eA - eB : -eB);
    C *raw = As + kRowsSmemElems;
    if (!a_res) asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (ahead) {   // each thread reads what it copied itself
#pragma unroll
        for (int q = 0; q < kAheadPer; ++q) {
            const int32_t i = tid + q * kThreads;
            if (i < K * NB) Bs[i] = cscale(raw[i], sB);
        }
    }
#pragma unroll 4
    for (int32_t i = tid + (ahead ? kRowsAhead : 0); i < K * NB; i += kThreads) {
        const int32_t o = __ldg(tab + M + K + i);
        Bs[i] = o >= 0 ? cscale(ldc(B + o), sB) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (c_in_smem) b_ahead_copy(*next, j, raw, onext);
    if (!fold) {
        const float sA = pow2<float>(-eA);
#pragma unroll 1
        for (int32_t i = tid; i < MK; i += kThreads) As[i] = cscale(As[i], sA);   // swizzled or not: B may follow
        __syncthreads();
    }
    prof_phase<PROF>(prof, 7, tp);
    C acc[R][NC];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NC; ++n) acc[r][n] = make_float2(0.f, 0.f);
    const C *Bk = Bs + 2 * cg;   // column n of the thread: (n / 2) 2 CG + 2 cg + n mod 2
    const uint32_t carry = p2 ? 0u : ~0u;   // x + y = (x ^ y) + 2 (x & y)
#pragma unroll 2
    for (int32_t k = 0; k < K; ++k, Bk += NB) {
        const uint32_t ko = (uint32_t)kat[k];
        C a[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            a[r] = *reinterpret_cast<const C *>(reinterpret_cast<const char *>(As) + (row[r] ^ ko) +
                                                (2 * (row[r] & ko) & carry));
#pragma unroll
        for (int n = 0; n < NC; n += 2) {
            const float4 bb = *reinterpret_cast<const float4 *>(Bk + n * CG);
            const C b0 = make_float2(bb.x, bb.y), b1 = make_float2(bb.z, bb.w);
#pragma unroll
            for (int r = 0; r < R; ++r) cfma(acc[r][n], a[r], b0);
#pragma unroll
            for (int r = 0; r < R; ++r) cfma(acc[r][n + 1], a[r], b1);
        }
    }
    __syncthreads();   // every thread is done reading A and B
    prof_phase<PROF>(prof, 11, tp);
    float mx = 0.f;
    // columns past N are sums of zeros
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < NC; ++n) mx = fmaxf(mx, absmax2(acc[r][n]));
    if (NB == N) {   // a power of two: row and column bits are disjoint, and a pair is one 16-byte piece
        uint32_t cs[NC / 2];
#pragma unroll
        for (int n = 0; n < NC / 2; ++n) cs[n] = swz((uint32_t)(2 * n * CG + 2 * cg));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int32_t m = m0 + r * rstep;
            const uint32_t mrow = swz((uint32_t)(m * N));
            if (m < M) {
#pragma unroll
                for (int n = 0; n < NC / 2; ++n)
                    *reinterpret_cast<float4 *>(As + (mrow ^ cs[n])) =
                        make_float4(acc[r][2 * n].x, acc[r][2 * n].y, acc[r][2 * n + 1].x, acc[r][2 * n + 1].y);
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int32_t m = m0 + r * rstep;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int32_t c = (n / 2) * 2 * CG + 2 * cg + (n & 1);
                if (m < M && c < N) As[swz((uint32_t)(m * N + c))] = acc[r][n];
            }
        }
    }
    if (c_in_smem) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // the next step's B and the head after it
        const float cmax = block_max(mx, red);
        prof_phase<PROF>(prof, 15, tp);
        return cmax;
    }
    __syncthreads();
    C *__restrict__ Cp = reinterpret_cast<C *>(j.arena) + d.c_off;   // 256-byte aligned
    const int32_t MN = M * N;
    for (int32_t i = 2 * tid; i + 1 < MN; i += 2 * kThreads)
        *reinterpret_cast<float4 *>(Cp + i) = *reinterpret_cast<const float4 *>(As + swz((uint32_t)i));
    if ((MN & 1) && tid == 0) Cp[MN - 1] = As[swz((uint32_t)(MN - 1))];
    publish_max(mx, j.maxbits + d.node_c, red);
    prof_phase<PROF>(prof, 15, tp);
    return 0.f;
}

// A small step (the criterion of the subtree programs: at most 256 outputs) staged the same way, an
// output per thread, summed as the programs do.  Its table: A offsets of rows and shared indices as
// above, then element offsets in B of the shared indices and of the columns.
template <bool PROF>
__device__ float rows_smem_small(const StepHead &d, const JobPtrs &j, char *dyn, float *red, int32_t eA, int32_t eB,
                                 bool a_res, const StepHead *next, long long *prof) {
    long long tp = 0;
    if (PROF && threadIdx.x == 0) tp = clock64();
    using C = float2;
    const int32_t M = (int32_t)d.M, N = (int32_t)d.N, K = (int32_t)d.K, o = threadIdx.x;
    const int32_t *__restrict__ tab = reinterpret_cast<const int32_t *>(j.ktab + d.ktab_off);
    C *As = reinterpret_cast<C *>(dyn);
    const bool p2 = (d.flags & FLAG_A_POW2) != 0, c_in_smem = next != nullptr, act = o < M * N;
    if (!a_res) {
        stage_a(d, j, As, M * K, p2);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    }
    if (c_in_smem) {
        int32_t onext[kAheadPer];
        b_ahead_offsets(*next, j, onext);
        b_ahead_copy(*next, j, As + kRowsSmemElems, onext);
    }
    const bool fold = scales_fold(eA, eB);
    const float sA = fold ? 1.f : pow2<float>(-eA), sB = pow2<float>(fold ? -eA - eB : -eB);
    const uint32_t row = act ? (uint32_t)__ldg(tab + o / N) : 0u, carry = p2 ? 0u : ~0u;
    const C *B = operand<C>(d, j, false) + (act ? __ldg(tab + M + 2 * K + o % N) : 0);
    SmallSum<float> sum;
#pragma unroll 4
    for (int32_t k = 0; k < K; ++k) {
        const uint32_t ko = (uint32_t)__ldg(tab + M + k);
        const C a = *reinterpret_cast<const C *>(reinterpret_cast<const char *>(As) + (row ^ ko) +
                                                 (2 * (row & ko) & carry));
        sum.mac(cscale(a, sA), cscale(ldc(B + __ldg(tab + M + K + k)), sB));
    }
    __syncthreads();   // every thread is done reading A
    prof_phase<PROF>(prof, 11, tp);
    const C v = sum.value();
    if (c_in_smem) {
        if (act) As[swz((uint32_t)o)] = v;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        return block_max(act ? absmax2(v) : 0.f, red);
    }
    if (act) (reinterpret_cast<C *>(j.arena) + d.c_off)[o] = v;
    publish_max(act ? absmax2(v) : 0.f, j.maxbits + d.node_c, red);
    return 0.f;
}

// The thread tile of a staged step: the smallest that covers it (see rows_shape).
template <bool PROF>
__device__ __forceinline__ float rows_smem_any(const StepHead &d, const JobPtrs &j, char *smem, char *dyn, float *red,
                                               int32_t eA, int32_t eB, bool a_res, bool ahead, const StepHead *next,
                                               long long *prof) {
    switch (d.tile_shape) {
        case 0: return rows_smem_core<rows_nc(0), rows_r(0), PROF>(d, j, smem, dyn, red, eA, eB, a_res, ahead, next, prof);
        case 1: return rows_smem_core<rows_nc(1), rows_r(1), PROF>(d, j, smem, dyn, red, eA, eB, a_res, ahead, next, prof);
        case 2: return rows_smem_core<rows_nc(2), rows_r(2), PROF>(d, j, smem, dyn, red, eA, eB, a_res, ahead, next, prof);
        case 3: return rows_smem_core<rows_nc(3), rows_r(3), PROF>(d, j, smem, dyn, red, eA, eB, a_res, ahead, next, prof);
        default: return rows_smem_small<PROF>(d, j, dyn, red, eA, eB, a_res, next, prof);
    }
}

// A ROWS step staged through shared memory on its own.
__device__ __forceinline__ void tile_rows_smem(const StepDesc &d, const JobPtrs &j, char *smem, char *dyn,
                                               float *red) {
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    leave_out_scale(eA, eB);
    rows_smem_any<false>(d, j, smem, dyn, red, eA, eB, false, false, nullptr, nullptr);
    if (threadIdx.x == 0) write_exponent(d, j, eA, eB);
}

// A chain of staged steps linked by chain_next, run by one block of the persistent kernel: the first
// step reads A from the arena, each later one takes the previous step's C, kept in shared memory,
// as its A, and the last writes its C to the arena.  The per-step power-of-two scaling is that of the
// separate steps: a continuation's A exponent comes from the block max of the previous C, which is the
// value the separate steps would publish, so results are bit-identical to running the steps one
// by one; the exponents of the inner nodes stay in registers and only the last node's max-abs and
// exponent are written.  The heads of the steps are fetched two steps ahead into a ring of three, and
// the next step's B and its scale one step ahead, so that inside a chain no step waits for them.
// Thread 0 writes the indices of the continuation steps to chain[].  Returns their count.
constexpr int kHeadPieces = (int)(sizeof(StepHead) / 16);
__device__ __forceinline__ void head_copy(StepHead &dst, const StepDesc *src) {   // asynchronous, not committed
    if (threadIdx.x < kHeadPieces)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(reinterpret_cast<char *>(&dst) + 16 * threadIdx.x)),
                     "l"(reinterpret_cast<const char *>(static_cast<const StepHead *>(src)) + 16 * threadIdx.x)
                     : "memory");
}

template <bool PROF>
__device__ __forceinline__ int32_t rows_chain(const StepDesc &d, const JobPtrs &j, char *smem, char *dyn, float *red,
                                              StepHead *ring, int32_t *chain, long long *prof) {
    head_copy(ring[1], j.steps + d.chain_next);
    asm volatile("cp.async.commit_group;" ::: "memory");
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    int32_t xa = __ldcg(j.exp2 + d.node_a), xb = __ldcg(j.exp2 + d.node_b);
    if (threadIdx.x < kHeadPieces)
        reinterpret_cast<int4 *>(ring)[threadIdx.x] = reinterpret_cast<const int4 *>(&d)[threadIdx.x];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    int32_t n = 0, at = 0;   // step of the chain, its place in the ring
    while (true) {
        const StepHead &cur = ring[at];
        const int32_t after = at == 2 ? 0 : at + 1;
        // read here: past the step's last barrier the head's place belongs to the copy of the step after
        // the next one, which other lanes may have started
        const int32_t cont = cur.chain_next;
        const StepHead *next = cont >= 0 ? ring + after : nullptr;
        uint32_t next_max = 0;
        int32_t next_exp = 0;
        if (next) {
            if (next->chain_next >= 0) head_copy(ring[after == 2 ? 0 : after + 1], j.steps + next->chain_next);
            asm volatile("cp.async.commit_group;" ::: "memory");
            next_max = __ldcg(j.maxbits + next->node_b);
            next_exp = __ldcg(j.exp2 + next->node_b);
        }
        leave_out_scale(eA, eB);
        const float cmax = rows_smem_any<PROF>(cur, j, smem, dyn, red, eA, eB, n > 0, n > 0, next, prof);
        const int32_t xc = xa + eA + xb + eB;
        if (!next) {
            if (threadIdx.x == 0) j.exp2[cur.node_c] = xc;
            return n;
        }
        if (threadIdx.x == 0) chain[n] = cont;
        ++n;
        at = after;
        xa = xc;
        eA = scale_exponent(__float_as_uint(cmax));
        eB = scale_exponent(next_max);
        xb = next_exp;
    }
}

template <typename T>
__device__ __forceinline__ void tile_rows_dispatch(const StepDesc &d, int64_t tile, const JobPtrs &j,
                                                   char *smem, float *red, char *dyn) {
    if constexpr (sizeof(T) == 4) {
        if (d.flags & FLAG_SMALL) {
            tile_small(d, j, smem, red);
            return;
        }
        if (d.flags & FLAG_A_SMEM) {
            tile_rows_smem(d, j, smem, dyn, red);
            return;
        }
    }
    if (d.N <= 1) tile_rows<T, 1>(d, tile, j, smem, red);
    else if (d.N <= 2) tile_rows<T, 2>(d, tile, j, smem, red);
    else if (d.N <= 4) tile_rows<T, 4>(d, tile, j, smem, red);
    else if (d.N <= 8) tile_rows<T, 8>(d, tile, j, smem, red);
    else tile_rows<T, 16>(d, tile, j, smem, red);
}

// ------------------------------------------------------------------------------ TILE (GEMM)
// General contraction on CUDA cores: a TM x TN output tile, RM x RN outputs per thread, the shared index
// in chunks of KS TK: the block's KS thread groups take TK shared indices of a chunk each (their sums are
// added in a fixed order at the end).  Operand chunks are gathered through the index maps into shared
// memory with cp.async, chunk c + 1 while chunk c is multiplied, running along whichever index is
// contiguous in the operand, so that a warp reads whole sectors.  The scales are applied where no product
// loses range: to the sums while the unscaled products are the larger ones, else together to B's entries (the
// products are then those of scaled operands) or, for exponents so large that unscaled entries could leave
// FP32's range, to the entries of both.  Each thread scales the entries that it copied itself, before the
// barrier that publishes them.
// Bound by the FMA pipe (56 % of it at two blocks per SM) and by the last wave of tiles, which run alone
// on their SMs: 128 x 64 tiles with 8 x 4 outputs a thread spent as much per multiply-add and had the
// longer tail.  Measured, a 64 x 64 x 512 complex64 tile: 236 k cycles, 308 k with register-staged gathers
// along the rows.  Few outputs with a long shared index take KS = 4: 8 x 8 x 512 took 250 k cycles in a
// 64 x 64 tile and takes 45 k in 16 x 16.  From eight such tiles on their threads, two rows and two columns each, wait
// for shared memory too long in a full batch: 64 x 64 x 512 takes 32 x 32 tiles of 4 x 4 outputs a thread, one contraction
// 51 us (37 us in 16 x 16, 96 us in 64 x 64), 1024 of them 0.64 ms (1.05 and 0.50 ms).
template <typename T, int TM, int TN, int RM, int RN, int TK, int KS>
__device__ void tile_gemm(const StepDesc &d, int64_t tile, const JobPtrs &j, char *smem, float *red) {
    using C = cx_t<T>;
    constexpr int TX = TN / RN, TY = TM / RM, KC = TK * KS, PA = TM + 1, PB = TN + 1;
    static_assert(TX * TY * KS == kThreads, "one register tile per thread");
    constexpr int RA = TM * KC / kThreads, RB = TN * KC / kThreads;
    static_assert(RA * kThreads == TM * KC && RB * kThreads == TN * KC, "operand tile split");
    static_assert((KS & (KS - 1)) == 0 && KC <= kThreads, "thread groups");
    constexpr int stage = KC * (PA + PB), tile_bytes = (2 * stage * (int)sizeof(C) + 7) / 8 * 8;
    static_assert(tile_bytes + (TM + TN + 6 * KC) * 8 <= Scratch<T>::bytes, "scratch");
    static_assert(KS / 2 * TM * TN * (int)sizeof(C) <= Scratch<T>::bytes, "partial sums");
    C *As = reinterpret_cast<C *>(smem);   // [2 stages][KC][PA], then [KC][PB] of the same stage
    int64_t *rowA = reinterpret_cast<int64_t *>(smem + tile_bytes);
    int64_t *colB = rowA + TM;
    int64_t *kAo = colB + TN, *kBo = kAo + 3 * KC;   // [3][KC], written two chunks ahead
    const int64_t M = d.M, N = d.N, K = d.K;
    const int64_t tiles_n = (N + TN - 1) / TN;
    const int64_t m0 = (tile / tiles_n) * TM, n0 = (tile % tiles_n) * TN;
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    constexpr int kLate = sizeof(T) == 4 ? 40 : 120;   // |exponents| up to which the sums are scaled
    const bool late = eA > -kLate && eA < kLate && eB > -kLate && eB < kLate;
    const int32_t es = eA + eB;
    const T sA = pow2<T>(-eA), sB = pow2<T>(late ? -es : -eB);   // A: !late; B: !late or es < 0
    const C *__restrict__ A = operand<C>(d, j, true);
    const C *__restrict__ B = operand<C>(d, j, false);
    C *__restrict__ Cp = reinterpret_cast<C *>(j.arena) + d.c_off;
    const int tid = threadIdx.x;
    const bool a_k = d.k.n > 0 && d.k.sa[0] == 1, b_k = d.k.n > 0 && d.k.sb[0] == 1;   // contiguous along k
    for (int i = tid; i < TM + TN; i += kThreads) {
        if (i < TM) rowA[i] = (m0 + i < M) ? group_off(d.m, m0 + i) : -1;
        else colB[i - TM] = (n0 + i - TM < N) ? group_off(d.n, n0 + i - TM) : -1;
    }
    const int32_t nch = (int32_t)((K + KC - 1) / KC);
    auto koffs = [&](int32_t c, int slot) {
        if (tid < KC) {
            const int64_t k = (int64_t)c * KC + tid;
            int64_t oa = -1, ob = -1;
            if (k < K) {
                if (d.k.n == 1) {
                    oa = k * d.k.sa[0];
                    ob = k * d.k.sb[0];
                } else {
                    group_off2(d.k, k, oa, ob);
                }
            }
            kAo[slot * KC + tid] = oa;
            kBo[slot * KC + tid] = ob;
        }
    };
    auto copy = [&](C *dst, const C *src, bool in) {
        if (!in) *dst = cmake((T)0, (T)0);
        else
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                         "l"(src), "n"(sizeof(C))
                         : "memory");
    };
    auto gather = [&](int st, int slot) {
        C *a = As + st * stage, *b = a + KC * PA;
        const int64_t *ka = kAo + slot * KC, *kb = kBo + slot * KC;
#pragma unroll
        for (int r = 0; r < RA; ++r) {
            const int i = tid + r * kThreads, row = a_k ? i / KC : i % TM, kk = a_k ? i % KC : i / TM;
            const int64_t o = rowA[row], ok = ka[kk];
            copy(a + kk * PA + row, A + o + ok, (o | ok) >= 0);
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const int i = tid + r * kThreads, col = b_k ? i / KC : i % TN, kk = b_k ? i % KC : i / TN;
            const int64_t o = colB[col], ok = kb[kk];
            copy(b + kk * PB + col, B + o + ok, (o | ok) >= 0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto scale_own = [&](int st) {
        C *a = As + st * stage, *b = a + KC * PA;
        if (!late) {
#pragma unroll
            for (int r = 0; r < RA; ++r) {
                const int i = tid + r * kThreads, o = a_k ? i % KC * PA + i / KC : i / TM * PA + i % TM;
                a[o] = cscale(a[o], sA);
            }
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const int i = tid + r * kThreads, o = b_k ? i % KC * PB + i / KC : i / TN * PB + i % TN;
            b[o] = cscale(b[o], sB);
        }
    };
    koffs(0, 0);
    koffs(1, 1);
    __syncthreads();
    gather(0, 0);
    const int tx = tid % TX, ty = tid / TX % TY, ks = tid / (TX * TY);
    C acc[RM][RN];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int jj = 0; jj < RN; ++jj) acc[i][jj] = cmake((T)0, (T)0);
    int slot = 1;   // of chunk c + 1
#pragma unroll 1
    for (int32_t c = 0; c < nch; ++c) {
        const int ahead = slot == 2 ? 0 : slot + 1;
        if (c + 2 < nch) koffs(c + 2, ahead);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (!late || es < 0) scale_own(c & 1);
        __syncthreads();   // chunk c is there, and chunk c - 1's stage is free
        if (c + 1 < nch) gather((c + 1) & 1, slot);
        slot = ahead;
        C *cur = As + (c & 1) * stage;
        const C *Ak = cur + ks * TK * PA + ty, *Bk = cur + KC * PA + ks * TK * PB + tx;
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            C a[RM], b[RN];
#pragma unroll
            for (int i = 0; i < RM; ++i) a[i] = Ak[kk * PA + TY * i];
#pragma unroll
            for (int jj = 0; jj < RN; ++jj) b[jj] = Bk[kk * PB + TX * jj];
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int jj = 0; jj < RN; ++jj) cfma(acc[i][jj], a[i], b[jj]);
        }
    }
    if (late && es > 0) {
        const T s = pow2<T>(-es);
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int jj = 0; jj < RN; ++jj) acc[i][jj] = cscale(acc[i][jj], s);
    }
    if constexpr (KS > 1) {   // upper half of the groups into the lower one, halving
        C *P = reinterpret_cast<C *>(smem);
#pragma unroll
        for (int h = KS / 2; h > 0; h /= 2) {
            __syncthreads();
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int jj = 0; jj < RN; ++jj)
                    if (ks >= h && ks < 2 * h) P[(((ks - h) * RM + i) * RN + jj) * (TX * TY) + tid % (TX * TY)] = acc[i][jj];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int jj = 0; jj < RN; ++jj)
                    if (ks < h) {
                        const C v = P[((ks * RM + i) * RN + jj) * (TX * TY) + tid % (TX * TY)];
                        acc[i][jj].x += v.x;
                        acc[i][jj].y += v.y;
                    }
        }
    }
    float mx = 0.f;
    if (ks == 0) {
#pragma unroll
        for (int i = 0; i < RM; ++i) {
            const int64_t m = m0 + ty + TY * i;
            if (m >= M) continue;
#pragma unroll
            for (int jj = 0; jj < RN; ++jj) {
                const int64_t n = n0 + tx + TX * jj;
                if (n < N) {
                    Cp[m * N + n] = acc[i][jj];
                    mx = fmaxf(mx, absmax2(acc[i][jj]));
                }
            }
        }
    }
    publish_max(mx, j.maxbits + d.node_c, red);
    if (tile == 0 && threadIdx.x == 0) write_exponent(d, j, eA, eB);
}

// Out of line: rare, and inlined it moved the other tile shapes about (1 % of a dense complex64 step).
static __device__ __noinline__ void tile_long32(const StepDesc &d, int64_t tile, const JobPtrs &j, char *smem,
                                                float *red) {
    tile_gemm<float, 32, 32, 4, 4, 4, 4>(d, tile, j, smem, red);
}

// ------------------------------------------------------------------------------ DOT
// Small outputs (M * N <= kDotMaxOut) with a long shared index.  DOTP: each tile reduces
// kDotChunk shared indices; products are formed in the storage precision, summed per thread in
// bursts of 8 in that precision and then in FP64.  DOTF: one tile sums the partials in a fixed order, so results are
// reproducible.  The root step of a closed network (M = N = 1) always takes this path: the final
// reduction of the amplitude is FP64.
template <typename T>
__device__ void tile_dotp(const StepDesc &d, int64_t tile, const JobPtrs &j, char *smem, char *dyn) {
    using C = cx_t<T>;
    double2(*red)[kDotMaxOut] = reinterpret_cast<double2(*)[kDotMaxOut]>(smem);
    int64_t *rowA = reinterpret_cast<int64_t *>(smem + (kThreads / 32) * kDotMaxOut * sizeof(double2));
    int64_t *colB = rowA + kDotMaxOut;
    const int32_t M = (int32_t)d.M, N = (int32_t)d.N;
    const int32_t MN = M * N;
    if (threadIdx.x < M) rowA[threadIdx.x] = group_off(d.m, threadIdx.x);
    if (threadIdx.x < N) colB[threadIdx.x] = group_off(d.n, threadIdx.x);
    __syncthreads();
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    const T sA = pow2<T>(-eA), sB = pow2<T>(-eB);
    const C *__restrict__ A = operand<C>(d, j, true);
    const C *__restrict__ B = operand<C>(d, j, false);
    // an operand whose offsets are permuted along k (complex64 only) is copied whole -- K elements,
    // 16-byte aligned in the arena -- with coalesced 16-byte copies, then gathered from shared
    // memory with plain loads (Xs)
    const bool sm_a = sizeof(T) == 4 && (d.flags & FLAG_DOT_SMEM_A) != 0;
    const bool sm_b = sizeof(T) == 4 && (d.flags & FLAG_DOT_SMEM_B) != 0;
    C *Xs = reinterpret_cast<C *>(dyn);
    if (sm_a || sm_b) {
        const C *src = sm_a ? A : B;
        const int32_t K = (int32_t)d.K;
        for (int32_t i = threadIdx.x; 2 * i + 1 < K; i += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(Xs + 2 * i)),
                         "l"(src + 2 * i)
                         : "memory");
        if ((K & 1) && threadIdx.x == 0) Xs[K - 1] = ldc(src + K - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    }
    double2 acc[kDotMaxOut];
#pragma unroll
    for (int i = 0; i < kDotMaxOut; ++i) acc[i] = make_double2(0, 0);
    const int64_t k_begin = tile * (int64_t)d.tile_rows;
    const int64_t k_end = min(d.K, k_begin + (int64_t)d.tile_rows);
    constexpr int U = 8;
    // both operands contiguous along the whole shared index (the closing trace of a matrix product):
    // 16-byte loads, two complex64 numbers each, all of a burst in flight together (8.4 M indices: 62 us;
    // 159 us when each index's loads waited for the previous index's multiply-add)
    bool stream = false;
    if constexpr (sizeof(T) == 4) {
        stream = MN == 1 && d.k.n == 1 && d.k.sa[0] == 1 && d.k.sb[0] == 1 && !sm_a && !sm_b &&
                 ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
        if (stream) {
            for (int64_t kb = k_begin + 2 * (int64_t)threadIdx.x; kb < k_end; kb += 2 * U * (int64_t)blockDim.x) {
                float4 av[U], bv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t k = kb + 2 * (int64_t)u * blockDim.x;
                    av[u] = bv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (k + 1 < k_end) {
                        av[u] = __ldcg(reinterpret_cast<const float4 *>(A + k));
                        bv[u] = __ldcg(reinterpret_cast<const float4 *>(B + k));
                    } else if (k < k_end) {
                        const C a = ldc(A + k), b = ldc(B + k);
                        av[u].x = a.x;
                        av[u].y = a.y;
                        bv[u].x = b.x;
                        bv[u].y = b.y;
                    }
                }
                C run0 = cmake(0.f, 0.f), run1 = cmake(0.f, 0.f);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    cfma(run0, cscale(cmake(av[u].x, av[u].y), sA), cscale(cmake(bv[u].x, bv[u].y), sB));
                    cfma(run1, cscale(cmake(av[u].z, av[u].w), sA), cscale(cmake(bv[u].z, bv[u].w), sB));
                }
                acc[0].x += (double)run0.x + (double)run1.x;
                acc[0].y += (double)run0.y + (double)run1.y;
            }
        }
    }
    // bursts of U shared indices per thread: offsets first, then U independent load pairs; each
    // burst is summed in the storage precision and then added in FP64
    for (int64_t kb = stream ? k_end : k_begin; kb < k_end; kb += (int64_t)U * blockDim.x) {
        int64_t oa[U], ob[U];
        if (d.ktab_off >= 0) {   // tabulated offsets: one coalesced 8-byte load per index
            const int2 *tab = j.ktab + d.ktab_off;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t k = kb + (int64_t)u * blockDim.x + threadIdx.x;
                oa[u] = -1;
                ob[u] = 0;
                if (k < k_end) {
                    const int2 t = __ldg(tab + k);
                    oa[u] = t.x;
                    ob[u] = t.y;
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t k = kb + (int64_t)u * blockDim.x + threadIdx.x;
                oa[u] = -1;
                ob[u] = 0;
                if (k < k_end) {
                    if (d.k.n == 1) {   // one fused group
                        oa[u] = k * d.k.sa[0];
                        ob[u] = k * d.k.sb[0];
                    } else {
                        group_off2(d.k, k, oa[u], ob[u]);
                    }
                }
            }
        }
        if (MN == 1) {
            // one output: all loads of the burst first, so that it pays one memory latency
            const C zero = cmake((T)0, (T)0);
            C av[U], bv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = oa[u] >= 0;
                av[u] = !in ? zero : sm_a ? Xs[oa[u] + rowA[0]] : ldc(A + oa[u] + rowA[0]);
                bv[u] = !in ? zero : sm_b ? Xs[ob[u] + colB[0]] : ldc(B + ob[u] + colB[0]);
            }
            C run = zero;
#pragma unroll
            for (int u = 0; u < U; ++u) cfma(run, cscale(av[u], sA), cscale(bv[u], sB));
            acc[0].x += (double)run.x;
            acc[0].y += (double)run.y;
            continue;
        }
        C run[kDotMaxOut];
#pragma unroll
        for (int i = 0; i < kDotMaxOut; ++i) run[i] = cmake((T)0, (T)0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (oa[u] < 0) continue;
#pragma unroll
            for (int i = 0; i < kDotMaxOut; ++i) {
                if (i < MN) {
                    const int m = i / N, n = i - m * N;
                    const C av = sm_a ? Xs[oa[u] + rowA[m]] : ldc(A + oa[u] + rowA[m]);
                    const C bv = sm_b ? Xs[ob[u] + colB[n]] : ldc(B + ob[u] + colB[n]);
                    const C a = cscale(av, sA), b = cscale(bv, sB);
                    cfma(run[i], a, b);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kDotMaxOut; ++i) {
            acc[i].x += (double)run[i].x;
            acc[i].y += (double)run[i].y;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < kDotMaxOut; ++i) {
        if (i >= MN) break;
        double x = acc[i].x, y = acc[i].y;
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            y += __shfl_down_sync(0xffffffffu, y, o);
        }
        if (lane == 0) red[warp][i] = make_double2(x, y);
    }
    __syncthreads();
    if (threadIdx.x < MN) {
        double2 s = make_double2(0, 0);
        for (int w = 0; w < kThreads / 32; ++w) { s.x += red[w][threadIdx.x].x; s.y += red[w][threadIdx.x].y; }
        j.partials[d.part_off + tile * kDotMaxOut + threadIdx.x] = s;
    }
    __syncthreads();
}

template <typename T>
__device__ void tile_dotf(const StepDesc &d, const JobPtrs &j, char *smem) {
    using C = cx_t<T>;
    double2(*red)[kDotMaxOut] = reinterpret_cast<double2(*)[kDotMaxOut]>(smem);
    const int32_t MN = (int32_t)(d.M * d.N);
    const int32_t nparts = d.tile_rows;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = 0; i < MN; ++i) {
        double x = 0, y = 0;
        for (int b = threadIdx.x; b < nparts; b += blockDim.x) {
            double2 p = __ldcg(j.partials + d.part_off + (int64_t)b * kDotMaxOut + i);
            x += p.x;
            y += p.y;
        }
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            y += __shfl_down_sync(0xffffffffu, y, o);
        }
        if (lane == 0) red[warp][i] = make_double2(x, y);
    }
    __syncthreads();
    int32_t eA, eB;
    step_scales(d, j, eA, eB);
    const int32_t e_out = __ldcg(j.exp2 + d.node_a) + eA + __ldcg(j.exp2 + d.node_b) + eB;
    if (threadIdx.x < MN) {
        double2 s = make_double2(0, 0);
        for (int w = 0; w < kThreads / 32; ++w) { s.x += red[w][threadIdx.x].x; s.y += red[w][threadIdx.x].y; }
        if (d.flags & FLAG_ROOT) {
            DeviceResult *r = static_cast<DeviceResult *>(j.result);
            r->re = s.x;
            r->im = s.y;
            r->exp2 = e_out;
        }
        if (!(d.flags & FLAG_NO_C)) {
            C v = cmake((T)s.x, (T)s.y);
            (reinterpret_cast<C *>(j.arena) + d.c_off)[threadIdx.x] = v;
            atomicMax(j.maxbits + d.node_c, __float_as_uint(absmax2(v)));
        }
    }
    if (threadIdx.x == 0) j.exp2[d.node_c] = e_out;
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ void run_tile(const StepDesc &d, int64_t tile, const JobPtrs &j, char *smem,
                                         float *red, char *dyn) {
    switch (d.kind) {
        case STEP_ROWS: tile_rows_dispatch<T>(d, tile, j, smem, red, dyn); break;
        case STEP_TILE:
            if constexpr (sizeof(T) == 4) {
                if (d.tile_rows == TILE_NARROW) tile_gemm<T, 128, 32, 4, 4, 8, 1>(d, tile, j, smem, red);
                else if (d.tile_rows == TILE_LONG_K) tile_gemm<T, 16, 16, 2, 2, 8, 4>(d, tile, j, smem, red);
                else if (d.tile_rows == TILE_LONG_K32) tile_long32(d, tile, j, smem, red);
                else tile_gemm<T, 64, 64, 4, 4, 8, 1>(d, tile, j, smem, red);
            } else {
                tile_gemm<T, 32, 32, 2, 2, 8, 1>(d, tile, j, smem, red);
            }
            break;
        case STEP_DOTP: tile_dotp<T>(d, tile, j, smem, dyn); break;
        case STEP_DOTF: tile_dotf<T>(d, j, smem); break;
        default: break;
    }
}

}  // namespace tn
