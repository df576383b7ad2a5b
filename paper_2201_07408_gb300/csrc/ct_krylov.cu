// Krylov solvers: BA-GMRES (Eq. 5), AB-GMRES (Eq. 4) and CGLS (Eqs. 2-3).
//
// Arnoldi with modified Gram-Schmidt (Sec. II): the newest Krylov vector q
// is orthogonalised against the basis one vector at a time.  A pass
// applies the previous projection (q -= h_{i-1} v_{i-1}) and forms the next
// inner product <q, v_i> in the same sweep over memory, so pass i reads q,
// v_{i-1}, v_i and writes q once.  Vectors that fit the registers of the chip
// are swept in one launch that keeps q there; longer ones take a launch a
// pass.
// Inner products: per-thread FP32 accumulation (plain FMA, or compensated
// with an FMA two-product and a two-sum), sums within a block in FP32 triples
// that keep the rounding errors, between blocks in FP64, in a fixed order
// (deterministic).  The Hessenberg column, the Givens rotations, the
// residual estimate |g_{j+1}| and the final triangular solve run in FP64 in
// one warp, so the whole solve is enqueued without host round
// trips; a device status word stops the remaining kernels on a tolerance
// stop, a lucky breakdown or a non-finite norm.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "ct_internal.cuh"

namespace ct {

constexpr int RED_BLOCK = 256;

enum : int { ST_RUN = 0, ST_TOL = 1, ST_LUCKY = 2, ST_NONFINITE = 3, ST_TIMEOUT = 4 };

// Device-resident solver state.
struct SolverState {
    int status;
    int iters;
    unsigned counter;
    int reorth_skip;
    double inv_norm;    // scale that normalises the newest basis vector
    double ref_sumsq;   // ||S v_j||^2 before orthogonalisation
    double sumsq;       // ||q||^2 after orthogonalisation
    double sumsq_pre2;  // ||q||^2 before the optional second sweep
    // CGLS scalars
    double gamma, gamma_new, delta, rr, data_rr;
};

// ---------------------------------------------------------------------------
// accumulators
// ---------------------------------------------------------------------------
// a + b as a rounded sum (returned) and its rounding error
__device__ __forceinline__ float two_sum(float a, float b, float &err)
{
    const float t = __fadd_rn(a, b);
    const float bp = __fsub_rn(t, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bp)), __fsub_rn(b, bp));
    return t;
}

// An unevaluated sum s + c + d of FP32 numbers of falling size (about 70 bits).
struct Sum3 {
    float s, c, d;
    __device__ __forceinline__ void add(const Sum3 &o)
    {
        float e1, e2, e3;
        s = two_sum(s, o.s, e1);
        c = two_sum(c, o.c, e2);
        c = two_sum(c, e1, e3);
        d = __fadd_rn(__fadd_rn(d, o.d), __fadd_rn(e2, e3));
    }
    __device__ __forceinline__ Sum3 lane_down(int o) const
    {
        return Sum3{__shfl_down_sync(0xffffffffu, s, o), __shfl_down_sync(0xffffffffu, c, o),
                    __shfl_down_sync(0xffffffffu, d, o)};
    }
    __device__ __forceinline__ double value() const { return double(s) + (double(c) + double(d)); }
};

template <int MODE>
struct Acc;

// Thread sums of products, one for each position in a group of 4 elements (four
// short chains: less rounding, and their steps overlap).
template <>
struct Acc<1> {  // FP32 FMA accumulation
    float p[4] = {};
    __device__ __forceinline__ void add(float a, float b, int e = 0) { p[e & 3] = fmaf(a, b, p[e & 3]); }
    __device__ __forceinline__ Sum3 part(int e) const { return Sum3{p[e], 0.0f, 0.0f}; }
};

template <>
struct Acc<0> {  // compensated: two-product (FMA) + two-sum in FP32
    float s[4] = {}, c[4] = {};
    __device__ __forceinline__ void add(float a, float b, int e = 0)
    {
        const float p = __fmul_rn(a, b);
        const float pe = fmaf(a, b, -p);
        float err;
        s[e & 3] = two_sum(s[e & 3], p, err);
        c[e & 3] = __fadd_rn(c[e & 3], __fadd_rn(err, pe));
    }
    __device__ __forceinline__ Sum3 part(int e) const { return Sum3{s[e], c[e], 0.0f}; }
};

template <int MODE>
__device__ __forceinline__ Sum3 thread_sum(const Acc<MODE> &a)
{
    Sum3 r = a.part(0), r2 = a.part(2);
    r.add(a.part(1));
    r2.add(a.part(3));
    r.add(r2);
    return r;
}

// Sums over a block of NT threads of two values (each only if wanted, the same
// for all threads), valid in thread 0.  FP64 additions run at 2 a clock on an
// SM: a warp-wide one occupies the unit for 16 cycles, and a tree of them in
// each of a streaming pass's warps took longer than the pass's memory traffic.
// So lanes and warps add triples of FP32 numbers that keep the rounding errors
// (Sum3), and only the block's sum goes on in FP64.  Sums near the end of
// FP32's range are added in FP64 throughout.
struct BlockPart {
    Sum3 sum;
    int big;
    double v;
};
template <int MODE>
__device__ __forceinline__ void warp_part(const Acc<MODE> &acc, BlockPart &out)
{
    Sum3 r = thread_sum(acc);
    const bool big = __any_sync(0xffffffffu, !(fabsf(r.s) <= 1e30f));
    double v = 0.0;
    if (big) {
        v = MODE == 0 || fabsf(r.s) <= 1e30f ? r.value() : double(r.s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r.add(r.lane_down(o));
    }
    if ((threadIdx.x & 31) == 0) out = BlockPart{r, big, v};
}
template <int NW>
__device__ __forceinline__ double warps_total(const BlockPart *part)
{
    const int lane = threadIdx.x & 31;
    BlockPart p = lane < NW ? part[lane] : BlockPart{{0.0f, 0.0f, 0.0f}, 0, 0.0};
    if (__any_sync(0xffffffffu, p.big)) {
        double v = p.big ? p.v : p.sum.value();
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        return v;
    }
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) p.sum.add(p.sum.lane_down(o));
    return p.sum.value();
}

template <int NT, int MODE>
__device__ __forceinline__ void block_total2(const Acc<MODE> &a, const Acc<MODE> &b, bool want_a, bool want_b,
                                             double &ta, double &tb)
{
    __shared__ BlockPart part[2][NT / 32];
    const int w = threadIdx.x >> 5;
    if (want_a) warp_part(a, part[0][w]);
    if (want_b) warp_part(b, part[1][w]);
    __syncthreads();
    ta = tb = 0.0;
    if (w == 0) {
        if (want_a) ta = warps_total<NT / 32>(part[0]);
        if (want_b) tb = warps_total<NT / 32>(part[1]);
    }
}

// The sums of n partials in a fixed order, valid in thread 0 afterwards (every
// thread of the block calls it).  load(i, a, b) reads partial i and says
// whether it is there yet; a partial that stays away for max_polls reads ends
// the wait (false, in every thread).  Four warps add: few FP64 additions in
// all, and a lane's reads go out together.
template <typename F>
__device__ __forceinline__ bool sum_partials(F load, int n, bool want_a, bool want_b, double &ta, double &tb,
                                             int max_polls = 1)
{
    __shared__ double sum[2][4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    bool ok = true;
    if (w < 4) {
        ta = tb = 0.0;
        for (int i0 = threadIdx.x; i0 < n; i0 += 4 * 128) {
            double a[4], b[4];
            int polls = 0;
            bool all;
            do {
                all = true;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    a[k] = b[k] = 0.0;
                    if (i0 + 128 * k < n) all = load(i0 + 128 * k, a[k], b[k]) && all;
                }
            } while (!all && ++polls < max_polls);
            ok = ok && all;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (want_a) ta += a[k];
                if (want_b) tb += b[k];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            if (want_a) ta += __shfl_down_sync(0xffffffffu, ta, o);
            if (want_b) tb += __shfl_down_sync(0xffffffffu, tb, o);
        }
        if (lane == 0) {
            sum[0][w] = ta;
            sum[1][w] = tb;
        }
    }
    if (w < 4) __threadfence();   // reads of the next partials stay behind these
    ok = __syncthreads_and(ok);
    if (threadIdx.x == 0) {
        ta = (sum[0][0] + sum[0][1]) + (sum[0][2] + sum[0][3]);
        tb = (sum[1][0] + sum[1][1]) + (sum[1][2] + sum[1][3]);
    }
    return ok;
}

// Stores the block's partial sums; the last block to finish sums all
// partials in a fixed order and writes the outputs (either may be null).
template <int NT, int MODE>
__device__ __forceinline__ void grid_finish(const Acc<MODE> &a, const Acc<MODE> &b, double *partials,
                                            unsigned *counter, double *out_a, double *out_b)
{
    __shared__ bool last;
    double ta, tb;
    block_total2<NT, MODE>(a, b, out_a != nullptr, out_b != nullptr, ta, tb);
    if (gridDim.x == 1) {
        if (threadIdx.x == 0) {
            if (out_a) *out_a = ta;
            if (out_b) *out_b = tb;
        }
        return;
    }
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = ta;
        partials[2 * blockIdx.x + 1] = tb;
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_partials([&](int i, double &va, double &vb) {
        if (out_a) va = __ldcg(partials + 2 * i);
        if (out_b) vb = __ldcg(partials + 2 * i + 1);
        return true;
    }, gridDim.x, out_a != nullptr, out_b != nullptr, ta, tb);
    if (threadIdx.x == 0) {
        if (out_a) *out_a = ta;
        if (out_b) *out_b = tb;
        *counter = 0u;
    }
}

// ---------------------------------------------------------------------------
// One MGS pass: q -= (*hprev) vprev (if vprev), then <q, vcur> (if vcur) and
// ||q||^2 (if out_sumsq).  Stops early on *stop, or on *skip when given.
// ---------------------------------------------------------------------------
// One group of 4 elements of the FP32 pass: q -= h v_prev (stored back),
// then the dot with v_cur and the sum of squares of the new q.
template <int MODE>
__device__ __forceinline__ void mgs_group4(float4 *q4, float4 a, float4 p, float4 c, bool has_prev, bool has_cur,
                                           bool sumsq, float h, Acc<MODE> &dot, Acc<MODE> &ss)
{
    if (has_prev) {
        a.x = fmaf(-h, p.x, a.x);
        a.y = fmaf(-h, p.y, a.y);
        a.z = fmaf(-h, p.z, a.z);
        a.w = fmaf(-h, p.w, a.w);
        *q4 = a;
    }
    if (has_cur) {
        dot.add(a.x, c.x, 0);
        dot.add(a.y, c.y, 1);
        dot.add(a.z, c.z, 2);
        dot.add(a.w, c.w, 3);
    }
    if (sumsq) {
        ss.add(a.x, a.x, 0);
        ss.add(a.y, a.y, 1);
        ss.add(a.z, a.z, 2);
        ss.add(a.w, a.w, 3);
    }
}

// The elements tid, tid + nth, ... of a pass over an FP32 basis.
template <int MODE>
__device__ __forceinline__ void pass_elements(float *__restrict__ q, const float *__restrict__ vprev, float h,
                                              const float *__restrict__ vcur, size_t len, bool vec, bool sumsq,
                                              size_t tid, size_t nth, Acc<MODE> &dot, Acc<MODE> &ss)
{
    size_t start = 0;
    if (vec) {
        const size_t n4 = len / 4;
        float4 *q4 = reinterpret_cast<float4 *>(q);
        const float4 *p4 = reinterpret_cast<const float4 *>(vprev);
        const float4 *c4 = reinterpret_cast<const float4 *>(vcur);
        const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        // two groups of 4 per step: the six 16-byte loads are in flight together
        // (basis vectors stream through L2 evict-first)
        size_t i = tid;
        for (; i + nth < n4; i += 2 * nth) {
            const size_t i1 = i + nth;
            const float4 a0 = q4[i], a1 = q4[i1];
            const float4 p0 = vprev ? __ldcs(p4 + i) : zero, p1 = vprev ? __ldcs(p4 + i1) : zero;
            const float4 c0 = vcur ? __ldcs(c4 + i) : zero, c1 = vcur ? __ldcs(c4 + i1) : zero;
            mgs_group4(q4 + i, a0, p0, c0, vprev != nullptr, vcur != nullptr, sumsq, h, dot, ss);
            mgs_group4(q4 + i1, a1, p1, c1, vprev != nullptr, vcur != nullptr, sumsq, h, dot, ss);
        }
        if (i < n4)
            mgs_group4(q4 + i, q4[i], vprev ? __ldcs(p4 + i) : zero, vcur ? __ldcs(c4 + i) : zero, vprev != nullptr,
                       vcur != nullptr, sumsq, h, dot, ss);
        start = n4 * 4;
    }
    for (size_t i = start + tid; i < len; i += nth) {
        float a = q[i];
        if (vprev) {
            a = fmaf(-h, vprev[i], a);
            q[i] = a;
        }
        if (vcur) dot.add(a, vcur[i]);
        if (sumsq) ss.add(a, a);
    }
}

// The same pass with a bf16 basis (FP32 work vector q): eight elements per
// step, the basis read as 16-byte vectors.
__device__ __forceinline__ void unpack8(const uint4 w, float (&o)[8])
{
    o[0] = bf16_lo(w.x); o[1] = bf16_hi(w.x); o[2] = bf16_lo(w.y); o[3] = bf16_hi(w.y);
    o[4] = bf16_lo(w.z); o[5] = bf16_hi(w.z); o[6] = bf16_lo(w.w); o[7] = bf16_hi(w.w);
}

// One group of 8 elements of the bf16-basis pass: q -= h v_prev (stored
// back), then the dot with v_cur and the sum of squares of the new q.
template <int MODE>
__device__ __forceinline__ void mgs_group8(float4 *q4, float4 lo, float4 hi, uint4 pw, uint4 cw, bool has_prev,
                                           bool has_cur, bool sumsq, float h, Acc<MODE> &dot, Acc<MODE> &ss)
{
    float a[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    if (has_prev) {
        float pv[8];
        unpack8(pw, pv);
#pragma unroll
        for (int e = 0; e < 8; ++e) a[e] = fmaf(-h, pv[e], a[e]);
        q4[0] = make_float4(a[0], a[1], a[2], a[3]);
        q4[1] = make_float4(a[4], a[5], a[6], a[7]);
    }
    if (has_cur) {
        float cv[8];
        unpack8(cw, cv);
#pragma unroll
        for (int e = 0; e < 8; ++e) dot.add(a[e], cv[e], e);
    }
    if (sumsq) {
#pragma unroll
        for (int e = 0; e < 8; ++e) ss.add(a[e], a[e], e);
    }
}

template <int MODE>
__device__ __forceinline__ void pass_elements(float *__restrict__ q, const __nv_bfloat16 *__restrict__ vprev, float h,
                                              const __nv_bfloat16 *__restrict__ vcur, size_t len, bool vec,
                                              bool sumsq, size_t tid, size_t nth, Acc<MODE> &dot, Acc<MODE> &ss)
{
    size_t start = 0;
    if (vec) {
        const size_t n8 = len / 8;
        float4 *q4 = reinterpret_cast<float4 *>(q);
        const uint4 *p8 = reinterpret_cast<const uint4 *>(vprev);
        const uint4 *c8 = reinterpret_cast<const uint4 *>(vcur);
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        // two groups of 8 per step: all six 16-byte loads are in flight together
        size_t i = tid;
        for (; i + nth < n8; i += 2 * nth) {
            const size_t i1 = i + nth;
            const float4 l0 = q4[2 * i], h0 = q4[2 * i + 1], l1 = q4[2 * i1], h1 = q4[2 * i1 + 1];
            const uint4 p0 = vprev ? __ldcs(p8 + i) : zero, p1 = vprev ? __ldcs(p8 + i1) : zero;
            const uint4 c0 = vcur ? __ldcs(c8 + i) : zero, c1 = vcur ? __ldcs(c8 + i1) : zero;
            mgs_group8(q4 + 2 * i, l0, h0, p0, c0, vprev != nullptr, vcur != nullptr, sumsq, h, dot, ss);
            mgs_group8(q4 + 2 * i1, l1, h1, p1, c1, vprev != nullptr, vcur != nullptr, sumsq, h, dot, ss);
        }
        if (i < n8)
            mgs_group8(q4 + 2 * i, q4[2 * i], q4[2 * i + 1], vprev ? __ldcs(p8 + i) : zero,
                       vcur ? __ldcs(c8 + i) : zero, vprev != nullptr, vcur != nullptr, sumsq, h, dot, ss);
        start = n8 * 8;
    }
    for (size_t i = start + tid; i < len; i += nth) {
        float a = q[i];
        if (vprev) {
            a = fmaf(-h, __bfloat162float(vprev[i]), a);
            q[i] = a;
        }
        if (vcur) dot.add(a, __bfloat162float(vcur[i]));
        if (sumsq) ss.add(a, a);
    }
}

template <int MODE, typename TB, int NT>
__global__ void __launch_bounds__(NT) mgs_pass_kernel(float *__restrict__ q, const TB *__restrict__ vprev,
                                                      const double *__restrict__ hprev, const TB *__restrict__ vcur,
                                                      size_t len, int vec, double *__restrict__ partials,
                                                      unsigned *__restrict__ counter, double *__restrict__ out_dot,
                                                      double *__restrict__ out_sumsq, const int *__restrict__ stop,
                                                      const int *__restrict__ skip)
{
    if ((stop && *stop) || (skip && *skip)) return;
    Acc<MODE> dot, ss;
    pass_elements<MODE>(q, vprev, vprev ? float(*hprev) : 0.0f, vcur, len, vec, out_sumsq != nullptr,
                        blockIdx.x * size_t(NT) + threadIdx.x, gridDim.x * size_t(NT), dot, ss);
    grid_finish<NT, MODE>(dot, ss, partials, counter, vcur ? out_dot : nullptr, out_sumsq);
}

// sum (a - b)^2 -> *out (recomputed data residuals)
__global__ void __launch_bounds__(RED_BLOCK) diff_sumsq_kernel(const float *__restrict__ a,
                                                               const float *__restrict__ b, size_t len,
                                                               double *__restrict__ partials,
                                                               unsigned *__restrict__ counter,
                                                               double *__restrict__ out,
                                                               const int *__restrict__ stop)
{
    if (stop && *stop) return;
    Acc<1> ss;
    for (size_t i = blockIdx.x * size_t(RED_BLOCK) + threadIdx.x; i < len;
         i += size_t(gridDim.x) * RED_BLOCK) {
        const float d = a[i] - b[i];
        ss.add(d, d);
    }
    grid_finish<RED_BLOCK, 1>(Acc<1>(), ss, partials, counter, nullptr, out);
}

static unsigned red_blocks(size_t len)
{
    size_t want = (len / 4 + RED_BLOCK - 1) / RED_BLOCK;
    size_t cap = size_t(num_sms()) * 8;
    return unsigned(std::max<size_t>(1, std::min(want, cap)));
}

static size_t partials_count() { return size_t(num_sms()) * 8 * 2; }


// Vectors of up to sweep_max() elements are orthogonalised by one kernel that
// keeps q in registers (mgs_sweep_kernel): one block of SWEEP_NT threads an SM,
// 32 elements a thread at most.
constexpr int SWEEP_NT = 512, SWEEP_ELEMS = 32;
static size_t slots_count() { return size_t(num_sms()) * 2 * 3 * 2; }
static size_t sweep_max() { return size_t(num_sms()) * SWEEP_NT * SWEEP_ELEMS; }

// Blocks of the sweep kernel, and of a single pass over as many elements (the
// same sums in the same order either way): 16 elements a thread until every SM
// has a block.
static unsigned sweep_blocks(size_t len)
{
    return unsigned(std::min((len + 16 * SWEEP_NT - 1) / (16 * SWEEP_NT), size_t(num_sms())));
}

// MGS pass over a typed basis (float or bf16 vectors; q is always float).
template <int MODE, typename TB>
static cudaError_t mgs_pass_t(float *q, const TB *vprev, const double *hprev, const TB *vcur, size_t len,
                              double *partials, unsigned *counter, double *out_dot, double *out_sumsq,
                              const int *stop, const int *skip, cudaStream_t st)
{
    constexpr size_t G = 16 / sizeof(TB);   // elements of a 16-byte group of the basis
    // in groups where the vectors are aligned (a solve's always are, whatever their length); the elements past
    // the last group, and vectors that are not aligned, one by one
    const int vec = (reinterpret_cast<uintptr_t>(q) % 16 == 0) &&
                    (!vprev || reinterpret_cast<uintptr_t>(vprev) % 16 == 0) &&
                    (!vcur || reinterpret_cast<uintptr_t>(vcur) % 16 == 0);
    ProfScope prof(PK_MGS, st);
    // past one block, single elements take all the threads that are resident at once (a sweep of 16.8 M elements, j =
    // 4: 511 us with 4 blocks an SM, 471 so; 100001 elements 61 us with 16 elements a thread, 45 so)
    if (!vec && len > 16 * SWEEP_NT) {
        int per_sm = 8;
        if (len > size_t(num_sms()) * 8 * RED_BLOCK * 4 &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mgs_pass_kernel<MODE, TB, RED_BLOCK>, RED_BLOCK, 0) !=
                cudaSuccess) {
            cudaGetLastError();
            per_sm = 4;
        }
        const size_t most = size_t(num_sms()) * std::min(std::max(per_sm, 1), 8);
        const unsigned blocks = unsigned(std::max<size_t>(1, std::min((len / 4 + RED_BLOCK - 1) / RED_BLOCK, most)));
        mgs_pass_kernel<MODE, TB, RED_BLOCK><<<blocks, RED_BLOCK, 0, st>>>(
            q, vprev, hprev, vcur, len, vec, partials, counter, out_dot, out_sumsq, stop, skip);
        return cudaGetLastError();
    }
    if (len <= sweep_max()) {
        mgs_pass_kernel<MODE, TB, SWEEP_NT><<<sweep_blocks(len), SWEEP_NT, 0, st>>>(
            q, vprev, hprev, vcur, len, vec, partials, counter, out_dot, out_sumsq, stop, skip);
        return cudaGetLastError();
    }
    // a thread's two groups a step put six 16-byte loads in flight, and 4 blocks an SM of them cover the memory's
    // latency (256^3, compensated: 34.4 us a pass; 5, 6 and 8 blocks 42.3, 39.2, 37.9); a bf16 basis moves half the
    // bytes at as many operations, and the compensated sums of 8 elements a group then take 6 (36.0, 32.7, 31.4,
    // 35.0 us with 4, 5, 6, 8; plain sums 28.7 with 4); plain sums over FP32, 5 (37.4, 35.7, 43.9, 40.1)
    constexpr int BLOCKS_PER_SM = MODE == 0 ? (G == 8 ? 6 : 4) : (G == 8 ? 4 : 5);
    const unsigned blocks = unsigned(std::min((len / G + RED_BLOCK - 1) / RED_BLOCK,
                                              size_t(num_sms()) * BLOCKS_PER_SM));
    mgs_pass_kernel<MODE, TB, RED_BLOCK><<<blocks, RED_BLOCK, 0, st>>>(q, vprev, hprev, vcur, len, vec, partials,
                                                                       counter, out_dot, out_sumsq, stop, skip);
    return cudaGetLastError();
}

static cudaError_t mgs_pass_typed(int mode, bool vbf16, float *q, const void *vprev, const double *hprev,
                                  const void *vcur, size_t len, double *partials, unsigned *counter,
                                  double *out_dot, double *out_sumsq, const int *stop, const int *skip,
                                  cudaStream_t st)
{
    auto run = [&](auto m, auto tb) {
        using TB = decltype(tb);
        return mgs_pass_t<decltype(m)::value, TB>(q, static_cast<const TB *>(vprev), hprev,
                                                  static_cast<const TB *>(vcur), len, partials, counter, out_dot,
                                                  out_sumsq, stop, skip, st);
    };
    using M0 = std::integral_constant<int, 0>;
    using M1 = std::integral_constant<int, 1>;
    if (vbf16) return mode == 0 ? run(M0(), __nv_bfloat16()) : run(M1(), __nv_bfloat16());
    return mode == 0 ? run(M0(), float()) : run(M1(), float());
}

static cudaError_t mgs_pass(int mode, float *q, const float *vprev, const double *hprev, const float *vcur, size_t len,
                            double *partials, unsigned *counter, double *out_dot, double *out_sumsq, const int *stop,
                            const int *skip, cudaStream_t st)
{
    return mgs_pass_typed(mode, false, q, vprev, hprev, vcur, len, partials, counter, out_dot, out_sumsq, stop, skip,
                          st);
}

// ---------------------------------------------------------------------------
// Small FP64 kernels of the GMRES least-squares problem.
// H, R: (k+1) x k, column-major with leading dimension k+1.
// ---------------------------------------------------------------------------
__global__ void gmres_init_kernel(SolverState *st, double *g, double *resid, int k)
{
    const double beta = sqrt(st->sumsq);
    for (int i = 0; i <= k; ++i) {
        g[i] = 0.0;
        resid[i] = -1.0;
    }
    g[0] = beta;
    resid[0] = beta;
    st->iters = 0;
    st->status = ST_RUN;
    if (!isfinite(beta)) {
        st->status = ST_NONFINITE;
    } else if (beta == 0.0) {
        st->status = ST_LUCKY;  // b (or B b) is zero: x = 0 is exact
    } else {
        st->inv_norm = 1.0 / beta;
    }
}

__global__ void sqrt_inplace_kernel(double *p) { *p = sqrt(*p); }

__global__ void reorth_decide_kernel(SolverState *st)
{
    // second sweep only when the first removed at least half of the squared
    // norm (||q_after|| <= ||q_before|| / sqrt 2)
    st->reorth_skip = !(st->sumsq <= 0.5 * st->ref_sumsq);
    st->sumsq_pre2 = st->sumsq;
}

// One warp.  The column's loads (32 rows at a time, a row a lane) are in flight
// together; only the chain of rotations is serial.
struct GivensArgs {
    int j, k;
    double *H;
    const double *H2;   // the second sweep's coefficients, or null
    double *R, *cs, *sn, *g, *resid;
    SolverState *st;
    double tol;
};
__device__ __forceinline__ void givens_step(const GivensArgs &A)
{
    const int lane = threadIdx.x & 31, j = A.j;
    const int ld = A.k + 1;
    double *h = A.H + size_t(j) * ld, *r = A.R + size_t(j) * ld;
    const double *H2 = A.H2;
    double *cs = A.cs, *sn = A.sn, *g = A.g, *resid = A.resid;
    SolverState *st = A.st;
    const double tol = A.tol;
    const double sumsq = st->sumsq, ref_sumsq = st->ref_sumsq;
    const bool second = H2 && !st->reorth_skip;
    const double g_j = g[j], resid0 = resid[0];
    bool bad = !isfinite(sumsq) || !isfinite(ref_sumsq);
    double x = 0.0;   // entry i of the column after the rotations before it
    for (int i0 = 0; i0 <= j; i0 += 32) {
        const int i = i0 + lane;
        double hv = 0.0, c = 0.0, s = 0.0, done = 0.0;
        if (i <= j) {
            hv = h[i];
            if (second) {
                hv += H2[i];
                h[i] = hv;
            }
            bad = bad || !isfinite(hv);
            if (i > 0) {   // the rotation of rows i - 1 and i
                c = cs[i - 1];
                s = sn[i - 1];
            }
        }
        const double ch = c * hv, sh = s * hv;
        for (int l = 0; l < 32 && i0 + l <= j; ++l) {
            const double cl = __shfl_sync(0xffffffffu, c, l), sl = __shfl_sync(0xffffffffu, s, l);
            const double t = fma(cl, x, __shfl_sync(0xffffffffu, sh, l));
            x = i0 + l == 0 ? __shfl_sync(0xffffffffu, hv, l) : fma(-sl, x, __shfl_sync(0xffffffffu, ch, l));
            if (lane == l) done = t;
        }
        if (i > 0 && i <= j) r[i - 1] = done;
    }
    bad = __any_sync(0xffffffffu, bad);
    // FP64 roots and quotients are long chains of slow operations: lane 0, 1, 2
    // take the roots of ||q||^2, of its value before the sweep, and of
    // x^2 + ||q||^2 at once, then the three quotients.  (Squares of sums of FP32
    // data are far inside FP64's range.)
    const double root = sqrt(lane == 0 ? sumsq : lane == 1 ? ref_sumsq : fma(x, x, sumsq));
    const double hnext = __shfl_sync(0xffffffffu, root, 0), ref = __shfl_sync(0xffffffffu, root, 1);
    const bool lucky = hnext <= 1e-14 * ref;
    const double rr = lucky ? fabs(x) : __shfl_sync(0xffffffffu, root, 2);
    const double quot = (lane == 0 ? x : lane == 1 ? (lucky ? 0.0 : hnext) : 1.0) / (lane < 2 ? rr : hnext);
    const double qc = __shfl_sync(0xffffffffu, quot, 0), qs = __shfl_sync(0xffffffffu, quot, 1);
    const double inv = __shfl_sync(0xffffffffu, quot, 2);
    if (lane > 0) return;
    h[j + 1] = hnext;
    if (bad) {
        st->status = ST_NONFINITE;
        return;
    }
    const double c = rr != 0.0 ? qc : 1.0, s = rr != 0.0 ? qs : 0.0;
    cs[j] = c;
    sn[j] = s;
    r[j] = rr;
    r[j + 1] = 0.0;
    const double g1 = -s * g_j, g0 = c * g_j;
    g[j + 1] = g1;
    g[j] = g0;
    // a column that vanishes after the rotations (a breakdown on which the
    // operator is singular) cannot reduce g[j]: the least-squares residual
    // stays, and the back substitution gives that coefficient 0
    const double res = rr != 0.0 ? fabs(g1) : hypot(g0, g1);
    resid[j + 1] = res;
    st->iters = j + 1;
    if (lucky || rr == 0.0) {
        st->status = ST_LUCKY;
    } else {
        st->inv_norm = inv;
        if (tol > 0.0 && res <= tol * resid0) st->status = ST_TOL;
    }
}
__global__ void givens_kernel(GivensArgs A)
{
    if (A.st->status != ST_RUN) return;
    givens_step(A);
}

// ---------------------------------------------------------------------------
// A whole MGS sweep of q against V_0 .. V_j in one launch, for vectors that fit
// the registers.  A pass a vector has to wait for the sum over all of q before
// it can go on, and as separate launches it spent most of its time on that
// (about 11 us a pass for 2.1 M elements, 5 us of it memory traffic; 8 us for
// 4096).  Here q stays in registers, the next basis vector is loaded while the
// sum is on its way, and the blocks exchange their partial sums through `slots`:
// each block publishes its partial and reads everyone's, adding them up in the
// order in which a single pass does, so the coefficients have the same bits.
// A slot holds SLOT_EMPTY until its block publishes; pass p uses slots p mod 3,
// and a block empties its slots of pass p - 1 once it has seen all of pass p
// (by then everyone has read them).  Two sets take turns from launch to launch:
// a launch empties the other set.  Launched cooperatively (all blocks
// resident); a wait that runs out marks the solve and ends the kernel.
// ---------------------------------------------------------------------------
constexpr unsigned long long SLOT_EMPTY = ~0ull;
// How long a block waits for another's sum, in reads (2^22: a few seconds, against microseconds that
// any wait takes between resident blocks), and a block that publishes none (-1; fault injection).
struct SweepWait {
    int max_polls = 1 << 22;
    int silent = -1;
};

__device__ __forceinline__ bool slot_get(const unsigned long long *p, double &v)
{
    unsigned long long b;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(b) : "l"(p) : "memory");
    v = __longlong_as_double((long long)b);
    return b != SLOT_EMPTY;
}
__device__ __forceinline__ void slot_put(unsigned long long *p, double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b == SLOT_EMPTY) b = 0x7ff8000000000000ull;   // (another NaN)
    asm volatile("st.release.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}

// unpacked group of 16 bytes of the basis
__device__ __forceinline__ void unpack_group(const uint4 w, float (&o)[4])
{
    o[0] = __uint_as_float(w.x); o[1] = __uint_as_float(w.y); o[2] = __uint_as_float(w.z); o[3] = __uint_as_float(w.w);
}
__device__ __forceinline__ void unpack_group(const uint4 w, float (&o)[8]) { unpack8(w, o); }

template <int MODE, typename TB, int ELEMS>
__global__ void __launch_bounds__(SWEEP_NT)
    mgs_sweep_kernel(float *q, const TB *V, size_t ldv, int j, size_t len, double *h, double *first_ss,
                     double *last_ss, unsigned long long *slots, int set, const int *stop, const int *skip,
                     SolverState *st, GivensArgs giv, SweepWait wait)
{
    constexpr int G = 16 / sizeof(TB), NG = ELEMS / G;
    const int nb = gridDim.x;
    // slots[set][pass mod 3][sum][block]
    unsigned long long *mine = slots + size_t(set) * 6 * nb + blockIdx.x;
    if (nb > 1 && threadIdx.x < 6) slots[size_t((1 - set) * 6 + threadIdx.x) * nb + blockIdx.x] = SLOT_EMPTY;
    const size_t ng = len / G, tid = blockIdx.x * size_t(SWEEP_NT) + threadIdx.x, nth = nb * size_t(SWEEP_NT);
    __shared__ double bcast;
    float a[NG][G];
    uint4 prev[NG], cur[NG];
    auto group = [&](int m) { return tid + m * nth; };
#pragma unroll
    for (int m = 0; m < NG; ++m) {
        prev[m] = cur[m] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int e = 0; e < G; ++e) a[m][e] = 0.0f;
        if (group(m) < ng) {
            const float4 *q4 = reinterpret_cast<const float4 *>(q) + group(m) * (G / 4);
#pragma unroll
            for (int e = 0; e < G; e += 4) {
                const float4 v = q4[e / 4];
                a[m][e] = v.x; a[m][e + 1] = v.y; a[m][e + 2] = v.z; a[m][e + 3] = v.w;
            }
            cur[m] = __ldcs(reinterpret_cast<const uint4 *>(V) + group(m));
        }
    }
    if ((stop && *stop) || (skip && *skip)) return;   // (read while the loads are under way)
    float hf = 0.0f;   // coefficient of V_{i-1}
    for (int i = 0; i <= j + 1; ++i) {
        Acc<MODE> dot, ss;
        const bool want_dot = i <= j, want_ss = (i == 0 && first_ss) || (i == j + 1 && last_ss);
        // (groups past the end are zero and add nothing)
#pragma unroll
        for (int m = 0; m < NG; ++m) {
            float p[G], c[G];
            unpack_group(prev[m], p);
            unpack_group(cur[m], c);
#pragma unroll
            for (int e = 0; e < G; ++e) a[m][e] = fmaf(-hf, p[e], a[m][e]);
            if (want_dot) {
#pragma unroll
                for (int e = 0; e < G; ++e) dot.add(a[m][e], c[e], e);
            }
        }
        if (want_ss) {
#pragma unroll
            for (int m = 0; m < NG; ++m) {
#pragma unroll
                for (int e = 0; e < G; ++e) ss.add(a[m][e], a[m][e], e);
            }
        }
        if (i == j + 1) {   // q is final
#pragma unroll
            for (int m = 0; m < NG; ++m) {
                if (group(m) < ng) {
                    float4 *q4 = reinterpret_cast<float4 *>(q) + group(m) * (G / 4);
#pragma unroll
                    for (int e = 0; e < G; e += 4)
                        q4[e / 4] = make_float4(a[m][e], a[m][e + 1], a[m][e + 2], a[m][e + 3]);
                }
            }
            if (!want_ss) break;
        }
        double ta, tb;
        block_total2<SWEEP_NT, MODE>(dot, ss, want_dot, want_ss, ta, tb);
        if (nb > 1) {
            unsigned long long *out = mine + (i % 3) * 2 * nb;
            if (threadIdx.x == 0 && int(blockIdx.x) != wait.silent) {
                if (want_dot) slot_put(out, ta);
                if (want_ss) slot_put(out + nb, tb);
            }
        }
        // the next vector comes in meanwhile
#pragma unroll
        for (int m = 0; m < NG; ++m) {
            prev[m] = cur[m];
            if (i < j && group(m) < ng) cur[m] = __ldcs(reinterpret_cast<const uint4 *>(V + size_t(i + 1) * ldv) + group(m));
        }
        if (nb > 1) {
            if (i == j + 1 && blockIdx.x > 0) break;   // the last sum is block 0's
            const unsigned long long *in = slots + size_t(set) * 6 * nb + (i % 3) * 2 * nb;
            const bool ok = sum_partials([&](int b, double &va, double &vb) {
                const bool ga = !want_dot || slot_get(in + b, va), gb = !want_ss || slot_get(in + nb + b, vb);
                return ga && gb;
            }, nb, want_dot, want_ss, ta, tb, wait.max_polls);
            if (!ok) {
                if (threadIdx.x == 0) st->status = ST_TIMEOUT;
                return;
            }
            if (i > 0 && threadIdx.x < 2) mine[(((i - 1) % 3) * 2 + threadIdx.x) * nb] = SLOT_EMPTY;
        }
        if (threadIdx.x == 0) {
            bcast = ta;
            if (blockIdx.x == 0) {
                if (want_dot) h[i] = ta;
                if (want_ss) *(i == 0 ? first_ss : last_ss) = tb;
            }
        }
        __syncthreads();
        hf = float(bcast);
    }
    if (blockIdx.x == 0 && threadIdx.x < 32 && giv.H) givens_step(giv);
}

// *cnt = j when iterate j exists (j <= iterations done), else 0
__global__ void iterate_count_kernel(const SolverState *st, int j, int *cnt) { *cnt = j <= st->iters ? j : 0; }

// *cnt = min(k, iterations done): the iterate x_k, or the last one when fewer exist
__global__ void iterate_upto_kernel(const SolverState *st, int k, int *cnt) { *cnt = st->iters < k ? st->iters : k; }

// y = R_j^{-1} g_j for the first *cnt columns: the least-squares coefficients
// of iterate x_j (R's first j columns and g's first j entries are final once
// iteration j is done).  One warp, a column at a time: y_i, then row l < i
// loses R[l][i] y_i; the next column's first 64 entries are loaded meanwhile.
__global__ void backsolve_kernel(const double *__restrict__ R, const double *__restrict__ g, double *__restrict__ y,
                                 const int *__restrict__ cnt, int k)
{
    extern __shared__ double rhs[];   // k
    const int it = min(*cnt, k);
    const int ld = k + 1, lane = threadIdx.x;
    for (int i = lane; i < it; i += 32) rhs[i] = g[i];
    __syncwarp();
    auto at = [&](int i, int l) { return i >= 0 && l <= i ? R[size_t(i) * ld + l] : 0.0; };
    double n0 = at(it - 1, lane), n1 = at(it - 1, lane + 32), nd = at(it - 1, it - 1);
    for (int i = it - 1; i >= 0; --i) {
        const double c0 = n0, c1 = n1, d = nd;
        n0 = at(i - 1, lane);
        n1 = at(i - 1, lane + 32);
        nd = at(i - 1, i - 1);
        const double yi = d != 0.0 ? rhs[i] / d : 0.0;
        if (lane == 0) y[i] = yi;
        if (lane < i) rhs[lane] -= c0 * yi;
        if (lane + 32 < i) rhs[lane + 32] -= c1 * yi;
        for (int l = lane + 64; l < i; l += 32) rhs[l] -= R[size_t(i) * ld + l] * yi;
        __syncwarp();
    }
}

static cudaError_t backsolve(const double *R, const double *g, double *y, const int *cnt, int k, cudaStream_t st)
{
    ProfScope prof(PK_SMALL, st);
    backsolve_kernel<<<1, 32, size_t(k) * sizeof(double), st>>>(R, g, y, cnt, k);
    return cudaGetLastError();
}

// err[j] = sqrt(err[j]) for the iterates that exist, -1 after them
__global__ void err_finish_kernel(double *err, const SolverState *st, int k)
{
    for (int j = 0; j <= k; ++j) err[j] = j <= st->iters ? sqrt(err[j]) : -1.0;
}

// x = sum_{i < count} y_i V_i ; count = *count_ptr when given, else k
template <typename TB>
__global__ void __launch_bounds__(RED_BLOCK) combine_kernel(const TB *__restrict__ V, size_t ldv, int k,
                                                            size_t len, const double *__restrict__ y,
                                                            const int *__restrict__ count_ptr,
                                                            float *__restrict__ x)
{
    extern __shared__ float ys[];
    const int count = count_ptr ? min(*count_ptr, k) : k;
    for (int i = threadIdx.x; i < count; i += RED_BLOCK) ys[i] = float(y[i]);
    __syncthreads();
    for (size_t e = blockIdx.x * size_t(RED_BLOCK) + threadIdx.x; e < len;
         e += size_t(gridDim.x) * RED_BLOCK) {
        float acc = 0.0f;
        for (int i = 0; i < count; ++i) acc = fmaf(ys[i], float(V[i * ldv + e]), acc);
        x[e] = acc;
    }
}

template <typename TB>
static cudaError_t combine_t(const TB *V, size_t ldv, int k, size_t len, const double *y, const int *count_ptr,
                             float *x, cudaStream_t st)
{
    const size_t smem = std::max<size_t>(1, size_t(k)) * sizeof(float);
    if (smem > 48 * 1024) {
        cudaError_t e = raise_dyn_smem(reinterpret_cast<const void *>(combine_kernel<TB>),
                                       std::min<size_t>(smem, 200 * 1024));
        if (e != cudaSuccess) return e;
    }
    const unsigned blocks = unsigned(std::max<size_t>(1, std::min((len + RED_BLOCK - 1) / RED_BLOCK,
                                                                  size_t(num_sms()) * 8)));
    ProfScope prof(PK_COMBINE, st);
    combine_kernel<TB><<<blocks, RED_BLOCK, smem, st>>>(V, ldv, k, len, y, count_ptr, x);
    return cudaGetLastError();
}

static cudaError_t combine(const float *V, size_t ldv, int k, size_t len, const double *y, const int *count_ptr,
                           float *x, cudaStream_t st)
{
    return combine_t<float>(V, ldv, k, len, y, count_ptr, x, st);
}

// ---------------------------------------------------------------------------
// CGLS vector kernels (coefficients from device scalars).
// ---------------------------------------------------------------------------
// y += sign * (*num / *den) * x ; optionally ||y||^2
__global__ void __launch_bounds__(RED_BLOCK) axpy_ratio_kernel(float *__restrict__ y, const float *__restrict__ x,
                                                               const double *__restrict__ num,
                                                               const double *__restrict__ den, float sign,
                                                               size_t len, double *__restrict__ partials,
                                                               unsigned *__restrict__ counter,
                                                               double *__restrict__ out_sumsq,
                                                               const int *__restrict__ stop)
{
    if (stop && *stop) return;
    const float a = sign * float(*num / *den);
    Acc<1> ss;
    for (size_t i = blockIdx.x * size_t(RED_BLOCK) + threadIdx.x; i < len;
         i += size_t(gridDim.x) * RED_BLOCK) {
        const float v = fmaf(a, x[i], y[i]);
        y[i] = v;
        ss.add(v, v);
    }
    if (out_sumsq) grid_finish<RED_BLOCK, 1>(Acc<1>(), ss, partials, counter, nullptr, out_sumsq);
}

// p = s + (*num / *den) p
__global__ void xpby_ratio_kernel(float *__restrict__ p, const float *__restrict__ s,
                                  const double *__restrict__ num, const double *__restrict__ den,
                                  size_t len, const int *__restrict__ stop)
{
    if (stop && *stop) return;
    const float b = float(*num / *den);
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < len;
         i += size_t(gridDim.x) * blockDim.x)
        p[i] = fmaf(b, p[i], s[i]);
}

__global__ void cgls_check_kernel(SolverState *st, int phase)
{
    if (st->status != ST_RUN) return;
    if (phase == 0) {  // after delta = ||A p||^2
        if (!isfinite(st->delta) || !isfinite(st->gamma)) st->status = ST_NONFINITE;
        else if (st->delta == 0.0 || st->gamma == 0.0) st->status = ST_LUCKY;
    }
}

__global__ void cgls_record_kernel(SolverState *st, double *resid, int j, int use_data, double tol)
{
    if (st->status != ST_RUN) return;
    const double v = sqrt(use_data ? st->data_rr : st->rr);
    resid[j] = v;
    st->iters = j;
    if (!isfinite(v) || !isfinite(st->gamma_new)) {
        st->status = ST_NONFINITE;
        return;
    }
    if (tol > 0.0 && v <= tol * resid[0]) st->status = ST_TOL;
}

__global__ void cgls_shift_kernel(SolverState *st)
{
    if (st->status != ST_RUN) return;
    st->gamma = st->gamma_new;
}

__global__ void cgls_init_kernel(SolverState *st, double *resid, int k)
{
    for (int i = 0; i <= k; ++i) resid[i] = -1.0;
    resid[0] = sqrt(st->rr);
    st->iters = 0;
    st->status = ST_RUN;
    if (!isfinite(st->gamma) || !isfinite(resid[0])) st->status = ST_NONFINITE;
    else if (st->gamma == 0.0) st->status = ST_LUCKY;
}

// ---------------------------------------------------------------------------
// Operator plumbing shared by the solvers.
// ---------------------------------------------------------------------------
struct OpBufs {
    float *Xc = nullptr, *Yc = nullptr;  // plane-major volume copies
    float *ypad = nullptr;               // padded sinogram
    float *t = nullptr;                  // plain sinogram
    float *acc = nullptr;                // A^T's accumulators (b_kind CT_B_AT)
};

static void take_op_bufs(Arena &ar, const GeomDev &g, OpBufs &b, bool need_t, bool need_acc)
{
    b.Xc = ar.take<float>(size_t(g.nzp) * g.nx * g.pitchX);
    b.Yc = ar.take<float>(size_t(g.nzp) * g.ny * g.pitchY);
    b.ypad = ar.take<float>(padded_sino_floats(g));
    b.t = need_t ? ar.take<float>(size_t(g.n_views) * g.nv * g.nu) : nullptr;
    b.acc = need_acc ? ar.take<float>(at_scratch_floats(g, at_scatter(g))) : nullptr;
}

// out_vol = B sino.  `sino` is a plain sinogram, scaled by (*scale) first when
// given (and normalised in place when `normalize`).
static cudaError_t apply_B(const GeomDev &g, int b_kind, float *sino, const double *scale, bool normalize,
                           OpBufs &b, float *out_vol, const int *stop, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    if (b_kind == CT_B_UN) {
        e = launch_pad_sino(g, sino, scale, normalize, b.ypad, stop, st);
        if (e == cudaSuccess) e = launch_voxel_B(g, b.ypad, out_vol, stop, st, QUAD_ROWDIFF);
        return e;
    }
    if (scale) {
        // normalise in place through the padded copy (values only), then filter / scatter
        e = launch_pad_sino(g, sino, scale, true, b.ypad, stop, st);
        if (e != cudaSuccess) return e;
    }
    if (b_kind == CT_B_FBP) {
        e = launch_ramp(g, sino, b.ypad, padded_layout(g), false, stop, st);
        if (e == cudaSuccess) e = launch_voxel_B(g, b.ypad, out_vol, stop, st, QUAD_ROWDIFF);
        return e;
    }
    return launch_project_At(g, at_scatter(g), sino, out_vol, b.acc, stop, st);   // exact transpose A^T
}

static ct_status check_common(const ct_geom *geom, const float *b, int k, const float *x,
                              const ct_solve_opts *o)
{
    if (!geom || !b || !x) return set_error(CT_EINVAL, "solver: NULL argument");
    if (k < 1) return set_error(CT_EINVAL, "solver: k must be >= 1 (got %d)", k);
    if (k > 4096) return set_error(CT_EINVAL, "solver: k must be <= 4096 (got %d)", k);
    if (o->b_kind != CT_B_UN && o->b_kind != CT_B_FBP && o->b_kind != CT_B_AT)
        return set_error(CT_EINVAL, "solver: unknown b_kind %d", o->b_kind);
    if (o->dot_mode != 0 && o->dot_mode != 1)
        return set_error(CT_EINVAL, "solver: dot_mode must be 0 or 1");
    if (!(o->tol >= 0.0)) return set_error(CT_EINVAL, "solver: tol must be >= 0");
    return o->b_kind == CT_B_FBP ? check_ramp(geom->g, "solver") : CT_OK;
}

static size_t round_ld(size_t len) { return (len + 63) & ~size_t(63); }

// Carves the GMRES workspace; with a counting arena (base == nullptr) it
// only adds up the size.
struct GmresWs {
    void *V = nullptr;      // k+1 basis vectors, float or (BA-GMRES with vol_bf16) bf16
    bool vbf16 = false;
    size_t ldv = 0;
    float *q = nullptr;     // BA-GMRES: FP32 work vector (new Krylov vector)
    OpBufs ob;
    float *tvol = nullptr;  // AB-GMRES: B v_j
    double *H = nullptr, *H2 = nullptr, *R = nullptr, *cs = nullptr, *sn = nullptr, *g = nullptr,
           *resid = nullptr, *y = nullptr, *partials = nullptr;
    double *err = nullptr;  // squared distances of the iterates to a reference image
    int *cnt = nullptr;     // iterate count for the error history
    unsigned long long *slots = nullptr;   // the blocks' partial sums of a sweep kernel
    SolverState *st = nullptr;
    const void *vec(int i) const
    {
        return static_cast<const char *>(V) + size_t(i) * ldv * (vbf16 ? 2 : 4);
    }
    void *vec(int i) { return static_cast<char *>(V) + size_t(i) * ldv * (vbf16 ? 2 : 4); }
};

static cudaError_t gmres_state_reset(GmresWs &w, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(w.slots, 0xff, slots_count() * sizeof(unsigned long long), s);
    return e == cudaSuccess ? cudaMemsetAsync(w.st, 0, sizeof(SolverState), s) : e;
}

// Bytes of the k+1 basis vectors of a BA (ab = false) or AB workspace.
static size_t basis_bytes(const GeomDev &g, int k, bool ab)
{
    const size_t len = ab ? size_t(g.n_views) * g.nv * g.nu : size_t(g.nx) * g.ny * g.nz;
    return Arena::align(round_ld(len) * size_t(k + 1) * ((!ab && g.vol_bf16) ? 2 : 4));
}

// external_basis: the basis lives elsewhere (w.V is set by the caller)
static bool carve_gmres(Arena &ar, const GeomDev &g, int k, bool ab, int b_kind, GmresWs &w,
                        bool external_basis = false)
{
    const size_t n = size_t(g.nx) * g.ny * g.nz;
    const size_t m = size_t(g.n_views) * g.nv * g.nu;
    const size_t len = ab ? m : n;
    w.ldv = round_ld(len);
    w.vbf16 = !ab && g.vol_bf16;
    if (external_basis)
        w.V = nullptr;
    else if (w.vbf16)
        w.V = ar.take<__nv_bfloat16>(w.ldv * size_t(k + 1));
    else
        w.V = ar.take<float>(w.ldv * size_t(k + 1));
    if (!ab) w.q = ar.take<float>(n);
    // BA needs a plain sinogram when B reads one (F or A^T); AB never does
    take_op_bufs(ar, g, w.ob, !ab && b_kind != CT_B_UN, b_kind == CT_B_AT);
    if (ab) w.tvol = ar.take<float>(n);
    const size_t ld = size_t(k) + 1;
    w.H = ar.take<double>(ld * k);
    w.H2 = ar.take<double>(ld);
    w.R = ar.take<double>(ld * k);
    w.cs = ar.take<double>(k);
    w.sn = ar.take<double>(k);
    w.g = ar.take<double>(ld);
    w.resid = ar.take<double>(ld);
    w.y = ar.take<double>(k);
    w.partials = ar.take<double>(partials_count());
    w.err = ar.take<double>(ld);
    w.cnt = ar.take<int>(1);
    w.slots = ar.take<unsigned long long>(slots_count());
    w.st = ar.take<SolverState>(1);
    return w.st != nullptr;
}

static size_t gmres_bytes(const GeomDev &g, int k, bool ab, int b_kind, bool external_basis = false)
{
    Arena ar;
    ar.size = ~size_t(0) >> 1;
    ar.base = nullptr;
    GmresWs w;
    carve_gmres(ar, g, k, ab, b_kind, w, external_basis);
    return ar.used;
}

// Host-resident basis streamed through the device by the copy engine.  The
// basis vectors live in page-locked host memory; the newest one is written to
// a device buffer (vnew) and copied out on a copy stream while the operators
// run; each MGS sweep brings the older vectors back into a ring of three
// device buffers, V_i into slot i mod 3, two vectors ahead of the pass that
// reads them (the copy of V_{i+2} waits for pass i, the last reader of the
// slot's previous vector).  The kernels read only device memory, so a pass
// runs at the copy's pace instead of at the kernels' own reads over the
// host link.
struct Stager {
    cudaStream_t cs = nullptr;       // copy stream
    void *ring[3] = {};              // device slots, one basis vector each
    void *vnew = nullptr;            // device copy of the newest vector
    char *host = nullptr;            // host basis, vector i at host + i * vbytes_ld
    size_t vbytes = 0;               // bytes copied per vector
    size_t vbytes_ld = 0;            // stride of the host vectors
    cudaEvent_t ev[8] = {};
    int evi = 0;
    cudaEvent_t vnew_free = nullptr; // the last copy out of vnew has finished
    cudaEvent_t ready[3] = {};       // per slot: its current vector has arrived

    cudaEvent_t next_event() { cudaEvent_t e = ev[evi]; evi = (evi + 1) % 8; return e; }
    // copies host vector i into slot i mod 3 after the work enqueued on s so far
    cudaError_t fetch(int i, cudaStream_t s)
    {
        cudaEvent_t e = next_event();
        cudaError_t r = cudaEventRecord(e, s);
        if (r == cudaSuccess) r = cudaStreamWaitEvent(cs, e, 0);
        if (r == cudaSuccess)
            r = cudaMemcpyAsync(ring[i % 3], host + size_t(i) * vbytes_ld, vbytes, cudaMemcpyHostToDevice, cs);
        if (r == cudaSuccess) r = cudaEventRecord(ready[i % 3], cs);
        return r;
    }
    // the device copy of V_i for a sweep whose newest vector is V_j (in vnew);
    // makes s wait for its arrival
    const void *vector(int i, int j, cudaStream_t s)
    {
        if (i == j) return vnew;
        cudaStreamWaitEvent(s, ready[i % 3], 0);
        return ring[i % 3];
    }
    // copies vnew out to host vector j after the work enqueued on s so far
    cudaError_t store_new(int j, cudaStream_t s)
    {
        cudaEvent_t e = next_event();
        cudaError_t r = cudaEventRecord(e, s);
        if (r == cudaSuccess) r = cudaStreamWaitEvent(cs, e, 0);
        if (r == cudaSuccess)
            r = cudaMemcpyAsync(host + size_t(j) * vbytes_ld, vnew, vbytes, cudaMemcpyDeviceToHost, cs);
        if (r == cudaSuccess) r = cudaEventRecord(vnew_free, cs);
        return r;
    }
};

// One MGS sweep (passes i = 0..j+1) over a staged basis: V_i for i < j comes
// through the ring, V_j from vnew.
// With `prefetched`, V_0 and V_1 were fetched already (at the start of the
// iteration, so that their copies overlap the operators).
static cudaError_t staged_sweep(Stager &sg, int mode, bool vbf16, float *q, int j, double *hcol, size_t len,
                                double *partials, unsigned *ctr, double *first_ss, double *last_ss,
                                const int *stop, const int *skip, cudaStream_t s, bool prefetched)
{
    cudaError_t e = cudaSuccess;
    if (!prefetched && 0 < j) e = sg.fetch(0, s);
    if (!prefetched && e == cudaSuccess && 1 < j) e = sg.fetch(1, s);
    for (int i = 0; i <= j + 1 && e == cudaSuccess; ++i) {
        const void *vprev = i > 0 ? sg.vector(i - 1, j, s) : nullptr;
        const void *vcur = i <= j ? sg.vector(i, j, s) : nullptr;
        const double *hprev = i > 0 ? hcol + (i - 1) : nullptr;
        double *odot = i <= j ? hcol + i : nullptr;
        double *oss = i == 0 ? first_ss : (i == j + 1 ? last_ss : nullptr);
        e = mgs_pass_typed(mode, vbf16, q, vprev, hprev, vcur, len, partials, ctr, odot, oss, stop, skip, s);
        // slot (i + 2) mod 3 held V_{i-1}, whose last reader was this pass
        if (e == cudaSuccess && i + 2 < j) e = sg.fetch(i + 2, s);
    }
    return e;
}

// One MGS sweep (passes i = 0..j+1) over a device basis: the sweep kernel where
// the vectors fit it, with the Givens step at its end when `giv` is given
// (givens_done), else a launch a pass.
template <int MODE, typename TB>
static cudaError_t launch_sweep(GmresWs &w, float *q, int j, double *hcol, size_t len, double *first_ss,
                                double *last_ss, int set, const int *stop, const int *skip, const GivensArgs *giv,
                                cudaStream_t s)
{
    const TB *V = static_cast<const TB *>(w.V);
    GivensArgs g{};
    if (giv) g = *giv;
    SweepWait wait;
    void *args[] = {&q,    &V,   &w.ldv, &j,    &len,  &hcol, &first_ss, &last_ss, &w.slots,
                    &set, &stop, &skip,  &w.st, &g,    &wait};
    ProfScope prof(PK_MGS, s);
    const unsigned blocks = sweep_blocks(len);
    if (blocks == 1) {   // nobody to wait for
        auto *kernel = len <= SWEEP_NT * 8 ? mgs_sweep_kernel<MODE, TB, 8> : mgs_sweep_kernel<MODE, TB, 16>;
        kernel<<<1, SWEEP_NT, 0, s>>>(q, V, w.ldv, j, len, hcol, first_ss, last_ss, w.slots, set, stop, skip, w.st, g,
                                      wait);
        return cudaGetLastError();
    }
    const FaultSpec fault = fault_spec();
    if (fault.sweep_refused) return cudaErrorCooperativeLaunchTooLarge;
    if (fault.sweep_stall == j + 1) {
        wait.max_polls = 1 << 12;
        wait.silent = int(blocks) - 1;
    }
    const void *kernel = len <= size_t(blocks) * SWEEP_NT * 16
                             ? reinterpret_cast<const void *>(mgs_sweep_kernel<MODE, TB, 16>)
                             : reinterpret_cast<const void *>(mgs_sweep_kernel<MODE, TB, SWEEP_ELEMS>);
    return cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(SWEEP_NT), args, 0, s);
}

static cudaError_t device_sweep(GmresWs &w, int mode, float *q, int j, double *hcol, size_t len, double *first_ss,
                                double *last_ss, int set, const int *stop, const int *skip, const GivensArgs *giv,
                                bool &givens_done, cudaStream_t s)
{
    // the kernel reads 16-byte groups (the basis' stride is a multiple of 64 elements, its start 256-byte aligned)
    if (len <= sweep_max() && len % (w.vbf16 ? 8 : 4) == 0 && reinterpret_cast<uintptr_t>(q) % 16 == 0) {
        cudaError_t e;
        if (w.vbf16)
            e = mode == 0 ? launch_sweep<0, __nv_bfloat16>(w, q, j, hcol, len, first_ss, last_ss, set, stop, skip, giv, s)
                          : launch_sweep<1, __nv_bfloat16>(w, q, j, hcol, len, first_ss, last_ss, set, stop, skip, giv, s);
        else
            e = mode == 0 ? launch_sweep<0, float>(w, q, j, hcol, len, first_ss, last_ss, set, stop, skip, giv, s)
                          : launch_sweep<1, float>(w, q, j, hcol, len, first_ss, last_ss, set, stop, skip, giv, s);
        if (e == cudaSuccess) {
            givens_done = giv != nullptr;
            return e;
        }
        // not all blocks can be resident (a device with part of its SMs): a launch a pass gives the same sums
        if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorLaunchOutOfResources &&
            e != cudaErrorNotSupported)
            return e;
        cudaGetLastError();
        // the launch that was to empty the other set's slots did not run: a later one must not find them full
        e = cudaMemsetAsync(w.slots, 0xff, slots_count() * sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaSuccess;
    for (int i = 0; i <= j + 1 && e == cudaSuccess; ++i)
        e = mgs_pass_typed(mode, w.vbf16, q, i > 0 ? w.vec(i - 1) : nullptr, i > 0 ? hcol + (i - 1) : nullptr,
                           i <= j ? w.vec(i) : nullptr, len, w.partials, &w.st->counter, i <= j ? hcol + i : nullptr,
                           i == 0 ? first_ss : (i == j + 1 ? last_ss : nullptr), stop, skip, s);
    return e;
}

// Enqueues the MGS sweep of iteration j (the new vector q against
// V_0..V_j) and its Givens step.
static cudaError_t arnoldi_orthogonalise(GmresWs &w, float *q, int j, int k, size_t len, const ct_solve_opts &o,
                                         cudaStream_t s, Stager *sg = nullptr)
{
    const int *stop = &w.st->status;
    unsigned *ctr = &w.st->counter;
    double *hcol = w.H + size_t(j) * (k + 1);
    cudaError_t e = fault_poison(q, j + 1, stop, s);
    if (sg) {
        if (e == cudaSuccess)
            e = staged_sweep(*sg, o.dot_mode, w.vbf16, q, j, hcol, len, w.partials, ctr, &w.st->ref_sumsq,
                             &w.st->sumsq, stop, nullptr, s, true);
        if (e != cudaSuccess) return e;
        const double *H2s = nullptr;
        if (o.reorth) {
            { ProfScope prof(PK_SMALL, s); reorth_decide_kernel<<<1, 1, 0, s>>>(w.st); }
            e = staged_sweep(*sg, o.dot_mode, w.vbf16, q, j, w.H2, len, w.partials, ctr, nullptr, &w.st->sumsq,
                             stop, &w.st->reorth_skip, s, false);
            if (e != cudaSuccess) return e;
            H2s = w.H2;
        }
        { ProfScope prof(PK_SMALL, s); givens_kernel<<<1, 32, 0, s>>>(GivensArgs{j, k, w.H, H2s, w.R, w.cs, w.sn, w.g, w.resid, w.st, o.tol}); }
        return cudaGetLastError();
    }
    GivensArgs giv{j, k, w.H, o.reorth ? w.H2 : nullptr, w.R, w.cs, w.sn, w.g, w.resid, w.st, o.tol};
    bool givens_done = false;
    if (e == cudaSuccess)
        e = device_sweep(w, o.dot_mode, q, j, hcol, len, &w.st->ref_sumsq, &w.st->sumsq, o.reorth ? 0 : j & 1, stop,
                         nullptr, o.reorth ? nullptr : &giv, givens_done, s);
    if (e == cudaSuccess && o.reorth) {
        { ProfScope prof(PK_SMALL, s); reorth_decide_kernel<<<1, 1, 0, s>>>(w.st); }
        bool unused = false;
        e = device_sweep(w, o.dot_mode, q, j, w.H2, len, nullptr, &w.st->sumsq, 1, stop, &w.st->reorth_skip, nullptr,
                         unused, s);
    }
    if (e != cudaSuccess || givens_done) return e;
    { ProfScope prof(PK_SMALL, s); givens_kernel<<<1, 32, 0, s>>>(giv); }
    return cudaGetLastError();
}

static ct_status finish_solve(SolverState *st_dev, const double *resid_dev, int k, double *resid_hist,
                              int *iters_done, cudaStream_t s, const char *who)
{
    SolverState hst;
    std::vector<double> hres(size_t(k) + 1);
    CT_CUDA(cudaMemcpyAsync(&hst, st_dev, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
    CT_CUDA(cudaMemcpyAsync(hres.data(), resid_dev, sizeof(double) * (k + 1), cudaMemcpyDeviceToHost, s));
    CT_CUDA(cudaStreamSynchronize(s));
    if (resid_hist) std::copy(hres.begin(), hres.end(), resid_hist);
    if (iters_done) *iters_done = hst.iters;
    if (hst.status == ST_NONFINITE)
        return set_error(CT_ENONFINITE, "%s: a norm became NaN/Inf after %d iterations", who, hst.iters);
    if (hst.status == ST_TIMEOUT)
        return set_error(CT_ETIMEOUT, "%s: a wait between blocks ran out after %d iterations", who, hst.iters);
    if (hst.status == ST_LUCKY) return CT_BREAKDOWN_LUCKY;
    return CT_OK;
}

static ct_status open_ws(Arena &ar, size_t bytes, const ct_solve_opts &o, cudaStream_t s)
{
    return arena_open(ar, bytes, o.workspace, o.workspace_bytes, s);
}

// ---------------------------------------------------------------------------
// BA-GMRES
// ---------------------------------------------------------------------------
// BA-GMRES in three steps, shared by the one-call solve and the persistent
// solver state (kmax: the workspace's capacity, the leading dimension of H).
//
// Start (x0 = 0): r0 = B b into q; ||r0|| starts the residual history.
static cudaError_t ba_start(const GeomDev &g, GmresWs &w, const float *b, int kmax, size_t n,
                            const ct_solve_opts &o, cudaStream_t s)
{
    cudaError_t e = gmres_state_reset(w, s);
    // zero the padded sinogram once: its border is never written afterwards
    if (e == cudaSuccess)
        e = cudaMemsetAsync(w.ob.ypad, 0, padded_sino_floats(g) * sizeof(float), s);
    if (e == cudaSuccess)
        e = apply_B(g, o.b_kind, const_cast<float *>(b), nullptr, false, w.ob, w.q, nullptr, s);
    if (e == cudaSuccess)
        e = mgs_pass(o.dot_mode, w.q, nullptr, nullptr, nullptr, n, w.partials, &w.st->counter, nullptr,
                     &w.st->sumsq, nullptr, nullptr, s);
    if (e == cudaSuccess) {
        { ProfScope prof(PK_SMALL, s); gmres_init_kernel<<<1, 1, 0, s>>>(w.st, w.g, w.resid, kmax); }
        e = cudaGetLastError();
    }
    return e;
}

// Iteration j (0-based): v_j = q / ||q|| joins the basis, q = B A v_j is
// orthogonalised against v_0..v_j, and the Givens step updates the residual.
static cudaError_t ba_iteration(const GeomDev &g, GmresWs &w, int j, int kmax, size_t n, const ct_solve_opts &o,
                                cudaStream_t s, Stager *sg = nullptr)
{
    NvtxRange iter_range("BA-GMRES iteration");
    const int *stop = &w.st->status;
    cudaError_t e = cudaSuccess;
    // a staged basis: vnew is rewritten only after its previous copy out; the
    // first two vectors of this iteration's sweep start coming in now
    if (sg) {
        e = cudaStreamWaitEvent(s, sg->vnew_free, 0);
        if (e == cudaSuccess && 0 < j) e = sg->fetch(0, s);
        if (e == cudaSuccess && 1 < j) e = sg->fetch(1, s);
    }
    // v_j = q / ||q|| stored in the basis while the projector's plane copies are built
    if (e == cudaSuccess)
        e = launch_plane_copies(g, w.q, &w.st->inv_norm, sg ? sg->vnew : w.vec(j), w.ob.Xc, w.ob.Yc, stop, s);
    if (e == cudaSuccess && sg) e = sg->store_new(j, s);
    if (e != cudaSuccess) return e;
    // q = B A v_j
    if (o.b_kind == CT_B_UN) {
        e = launch_project_A(g, w.ob.Xc, w.ob.Yc, w.ob.ypad, padded_layout(g), stop, s);
        if (e == cudaSuccess) e = launch_voxel_B(g, w.ob.ypad, w.q, stop, s, QUAD_CORNERS);
    } else {
        e = launch_project_A(g, w.ob.Xc, w.ob.Yc, w.ob.t, plain_layout(g), stop, s);
        if (e == cudaSuccess) e = apply_B(g, o.b_kind, w.ob.t, nullptr, false, w.ob, w.q, stop, s);
    }
    if (e == cudaSuccess) e = arnoldi_orthogonalise(w, w.q, j, kmax, n, o, s, sg);
    return e;
}

static ct_status bagmres(const ct_geom *geom, const float *b, int k, float *x, double *resid_hist,
                         const ct_solve_opts &o, int *iters_done, cudaStream_t s, const float *x_ref = nullptr,
                         double *err_hist = nullptr)
{
    const GeomDev &g = geom->g;
    const size_t n = geom->n;
    Arena ar;
    ct_status rc = open_ws(ar, gmres_bytes(g, k, false, o.b_kind), o, s);
    if (rc != CT_OK) return rc;
    GmresWs w;
    carve_gmres(ar, g, k, false, o.b_kind, w);
    cudaError_t e = ba_start(g, w, b, k, n, o, s);
    for (int j = 0; j < k && e == cudaSuccess; ++j) e = ba_iteration(g, w, j, k, n, o, s);
    // distance of every iterate x_j = V_j y_j to x_ref (x_out is the scratch
    // image; the final x_k is formed after)
    if (x_ref && e == cudaSuccess) {
        const unsigned vb = red_blocks(n);
        e = mgs_pass(1, const_cast<float *>(x_ref), nullptr, nullptr, nullptr, n, w.partials, &w.st->counter,
                     nullptr, &w.err[0], nullptr, nullptr, s);
        for (int j = 1; j <= k && e == cudaSuccess; ++j) {
            {
                ProfScope prof(PK_SMALL, s);
                iterate_count_kernel<<<1, 1, 0, s>>>(w.st, j, w.cnt);
            }
            e = backsolve(w.R, w.g, w.y, w.cnt, k, s);
            if (e != cudaSuccess) break;
            e = w.vbf16 ? combine_t(static_cast<const __nv_bfloat16 *>(w.V), w.ldv, k, n, w.y, w.cnt, x, s)
                        : combine(static_cast<const float *>(w.V), w.ldv, k, n, w.y, w.cnt, x, s);
            if (e == cudaSuccess) {
                ProfScope prof(PK_CGLS_VEC, s);
                diff_sumsq_kernel<<<vb, RED_BLOCK, 0, s>>>(x, x_ref, n, w.partials, &w.st->counter, &w.err[j],
                                                           nullptr);
                e = cudaGetLastError();
            }
        }
        if (e == cudaSuccess) {
            { ProfScope prof(PK_SMALL, s); err_finish_kernel<<<1, 1, 0, s>>>(w.err, w.st, k); }
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && err_hist)
            e = cudaMemcpyAsync(err_hist, w.err, sizeof(double) * (k + 1), cudaMemcpyDeviceToHost, s);
    }
    if (e == cudaSuccess) e = backsolve(w.R, w.g, w.y, &w.st->iters, k, s);
    if (e == cudaSuccess)
        e = w.vbf16 ? combine_t(static_cast<const __nv_bfloat16 *>(w.V), w.ldv, k, n, w.y, &w.st->iters, x, s)
                    : combine(static_cast<const float *>(w.V), w.ldv, k, n, w.y, &w.st->iters, x, s);
    if (e != cudaSuccess) {
        arena_close(ar);
        return cuda_error(e, "ct_bagmres_solve launch");
    }
    rc = finish_solve(w.st, w.resid, k, resid_hist, iters_done, s, "ct_bagmres_solve");
    arena_close(ar);
    return rc;
}

// ---------------------------------------------------------------------------
// Restarted BA-GMRES(m): cycles of m iterations, each on the residual
// system B A dx = B (b - A x) from dx = 0, then x += dx.
// ---------------------------------------------------------------------------
__global__ void sub_kernel(float *__restrict__ out, const float *__restrict__ a, const float *__restrict__ b,
                           size_t len)
{
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < len; i += size_t(gridDim.x) * blockDim.x)
        out[i] = a[i] - b[i];
}

__global__ void add_kernel(float *__restrict__ x, const float *__restrict__ d, size_t len)
{
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < len; i += size_t(gridDim.x) * blockDim.x)
        x[i] += d[i];
}

static ct_status bagmres_restarted(const ct_geom *geom, const float *b, int m, int cycles, float *x,
                                   double *resid_hist, const ct_solve_opts &o, int *iters_done, cudaStream_t s)
{
    const GeomDev &g = geom->g;
    const size_t n = geom->n, mm = geom->m;
    const size_t copies = size_t(g.nzp) * g.nx * g.pitchX + size_t(g.nzp) * g.ny * g.pitchY;
    float *buf = nullptr;
    cudaError_t e = scratch_alloc(reinterpret_cast<void **>(&buf), sizeof(float) * (copies + 2 * mm + n), s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(CT_ENOMEM, "ct_bagmres_restarted: %zu bytes of scratch: %s",
                         sizeof(float) * (copies + 2 * mm + n), cudaGetErrorString(e));
    }
    float *Xc = buf, *Yc = buf + size_t(g.nzp) * g.nx * g.pitchX;
    float *ax = buf + copies, *rb = ax + mm, *dx = rb + mm;
    const unsigned blocks = unsigned(std::min<size_t>((std::max(n, mm) + 255) / 256, size_t(num_sms()) * 16));
    std::vector<double> hist(size_t(m) + 1);
    int total = 0;
    ct_status rc = CT_OK;
    e = cudaMemsetAsync(x, 0, n * sizeof(float), s);
    if (resid_hist)
        for (int i = 0; i <= m * cycles; ++i) resid_hist[i] = -1.0;
    for (int c = 0; c < cycles && e == cudaSuccess; ++c) {
        const float *rhs = b;
        if (c > 0) {   // rb = b - A x
            e = launch_plane_copies(g, x, nullptr, nullptr, Xc, Yc, nullptr, s);
            if (e == cudaSuccess) e = launch_project_A(g, Xc, Yc, ax, plain_layout(g), nullptr, s);
            if (e == cudaSuccess) {
                sub_kernel<<<blocks, 256, 0, s>>>(rb, b, ax, mm);
                e = cudaGetLastError();
            }
            rhs = rb;
        }
        if (e != cudaSuccess) break;
        int it = 0;
        rc = bagmres(geom, rhs, m, dx, hist.data(), o, &it, s);
        if (rc != CT_OK && rc != CT_BREAKDOWN_LUCKY) break;
        add_kernel<<<blocks, 256, 0, s>>>(x, dx, n);
        e = cudaGetLastError();
        if (resid_hist) {
            if (c == 0) resid_hist[0] = hist[0];
            for (int j = 1; j <= it; ++j) resid_hist[total + j] = hist[j];
        }
        total += it;
        // a tolerance stop (relative to this cycle's start) or a breakdown ends the solve
        if (it < m || rc == CT_BREAKDOWN_LUCKY) break;
        if (o.tol > 0.0 && resid_hist && resid_hist[total] <= o.tol * resid_hist[0]) break;
    }
    cudaError_t e2 = cudaFreeAsync(buf, s);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (iters_done) *iters_done = total;
    if (e != cudaSuccess) return cuda_error(e, "ct_bagmres_restarted");
    return rc;
}

// ---------------------------------------------------------------------------
// AB-GMRES
// ---------------------------------------------------------------------------
static ct_status abgmres(const ct_geom *geom, const float *b, int k, float *x, double *resid_hist,
                         const ct_solve_opts &o, int *iters_done, cudaStream_t s)
{
    const GeomDev &g = geom->g;
    const size_t m = geom->m;
    Arena ar;
    ct_status rc = open_ws(ar, gmres_bytes(g, k, true, o.b_kind), o, s);
    if (rc != CT_OK) return rc;
    GmresWs w;
    carve_gmres(ar, g, k, true, o.b_kind, w);
    float *Vf = static_cast<float *>(w.V);   // data-space basis, FP32
    const int *stop = &w.st->status;
    cudaError_t e = gmres_state_reset(w, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(w.ob.ypad, 0, padded_sino_floats(g) * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(Vf, b, m * sizeof(float), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess)
        e = mgs_pass(o.dot_mode, Vf, nullptr, nullptr, nullptr, m, w.partials, &w.st->counter, nullptr,
                     &w.st->sumsq, nullptr, nullptr, s);
    if (e == cudaSuccess) {
        { ProfScope prof(PK_SMALL, s); gmres_init_kernel<<<1, 1, 0, s>>>(w.st, w.g, w.resid, k); }
        e = cudaGetLastError();
    }
    for (int j = 0; j < k && e == cudaSuccess; ++j) {
        NvtxRange iter_range("AB-GMRES iteration");
        float *vj = Vf + size_t(j) * w.ldv;
        float *q = Vf + size_t(j + 1) * w.ldv;
        e = apply_B(g, o.b_kind, vj, &w.st->inv_norm, true, w.ob, w.tvol, stop, s);
        if (e == cudaSuccess) e = launch_plane_copies(g, w.tvol, nullptr, nullptr, w.ob.Xc, w.ob.Yc, stop, s);
        if (e == cudaSuccess) e = launch_project_A(g, w.ob.Xc, w.ob.Yc, q, plain_layout(g), stop, s);
        if (e == cudaSuccess) e = arnoldi_orthogonalise(w, q, j, k, m, o, s);
    }
    if (e == cudaSuccess) e = backsolve(w.R, w.g, w.y, &w.st->iters, k, s);
    // u = V y (data space) into the last basis slot, then x = B u
    float *u = Vf + size_t(k) * w.ldv;
    if (e == cudaSuccess) e = combine(Vf, w.ldv, k, m, w.y, &w.st->iters, u, s);
    if (e == cudaSuccess) e = apply_B(g, o.b_kind, u, nullptr, false, w.ob, x, nullptr, s);
    if (e != cudaSuccess) {
        arena_close(ar);
        return cuda_error(e, "ct_abgmres_solve launch");
    }
    rc = finish_solve(w.st, w.resid, k, resid_hist, iters_done, s, "ct_abgmres_solve");
    arena_close(ar);
    return rc;
}

// ---------------------------------------------------------------------------
// Gradient through a converged BA-GMRES solve.  x = (BA)^{-1} B b, so for a
// scalar loss L(x) with gx = dL/dx:  dL/db = B^T (BA)^{-T} gx = B^T z with
// (A^T B^T) z = gx.  z comes from GMRES on A^T B^T (image-space basis, built
// afresh: the forward basis is not kept), each step applying B^T (voxel
// splatting, then F^T for B_FBP) and A^T (ray scatter).
// ---------------------------------------------------------------------------
struct VjpWs {
    GmresWs gm;
    float *t = nullptr, *tf = nullptr;   // sinogram-space temporaries
    float *acc = nullptr;                // A^T's accumulators
    float *bt_acc = nullptr;             // B_un^T's accumulators
};

static void carve_vjp(Arena &ar, const GeomDev &g, int k, int b_kind, VjpWs &w)
{
    const size_t n = size_t(g.nx) * g.ny * g.nz;
    const size_t m = size_t(g.n_views) * g.nv * g.nu;
    w.gm.ldv = round_ld(n);
    w.gm.V = ar.take<float>(w.gm.ldv * size_t(k + 1));
    w.t = ar.take<float>(m);
    w.tf = b_kind == CT_B_FBP ? ar.take<float>(m) : nullptr;
    w.acc = ar.take<float>(at_scratch_floats(g, at_scatter(g)));
    w.bt_acc = ar.take<float>(bt_scratch_floats(g, bt_scatter(g)));
    const size_t ld = size_t(k) + 1;
    w.gm.H = ar.take<double>(ld * k);
    w.gm.H2 = ar.take<double>(ld);
    w.gm.R = ar.take<double>(ld * k);
    w.gm.cs = ar.take<double>(k);
    w.gm.sn = ar.take<double>(k);
    w.gm.g = ar.take<double>(ld);
    w.gm.resid = ar.take<double>(ld);
    w.gm.y = ar.take<double>(k);
    w.gm.partials = ar.take<double>(partials_count());
    w.gm.slots = ar.take<unsigned long long>(slots_count());
    w.gm.st = ar.take<SolverState>(1);
}

static size_t vjp_bytes(const GeomDev &g, int k, int b_kind)
{
    Arena ar;
    ar.size = ~size_t(0) >> 1;
    VjpWs w;
    carve_vjp(ar, g, k, b_kind, w);
    return ar.used;
}

__global__ void scale_vec_kernel(float *__restrict__ v, size_t len, const double *__restrict__ scale,
                                 const int *__restrict__ stop)
{
    if (stop && *stop) return;
    const float sc = float(*scale);
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < len; i += size_t(gridDim.x) * blockDim.x)
        v[i] *= sc;
}

// out_sino = B^T vol (plain layout); b_kind B_UN or B_FBP
static cudaError_t apply_Bt(const GeomDev &g, int b_kind, const float *vol, float *t, float *bt_acc, float *out,
                            const int *stop, cudaStream_t s)
{
    cudaError_t e = launch_voxel_Bt(g, bt_scatter(g), vol, b_kind == CT_B_FBP ? t : out, bt_acc, stop, s);
    if (e == cudaSuccess && b_kind == CT_B_FBP) e = launch_ramp(g, t, out, plain_layout(g), true, stop, s);
    return e;
}

static ct_status bagmres_vjp(const ct_geom *geom, const float *gx, int k, float *gb, double *resid_hist,
                             const ct_solve_opts &o, int *iters_done, cudaStream_t s)
{
    if (o.b_kind == CT_B_AT)
        return set_error(CT_EINVAL, "ct_bagmres_vjp: b_kind must be CT_B_UN or CT_B_FBP");
    const GeomDev &g = geom->g;
    const size_t n = geom->n;
    ct_status rc = o.b_kind == CT_B_FBP ? check_ramp(g, "ct_bagmres_vjp") : CT_OK;
    if (rc != CT_OK) return rc;
    Arena ar;
    rc = open_ws(ar, vjp_bytes(g, k, o.b_kind), o, s);
    if (rc != CT_OK) return rc;
    VjpWs w;
    carve_vjp(ar, g, k, o.b_kind, w);
    GmresWs &gm = w.gm;
    const int *stop = &gm.st->status;
    const unsigned vb = red_blocks(n);
    float *Vf = static_cast<float *>(gm.V);   // image-space basis, FP32
    float *sino = o.b_kind == CT_B_FBP ? w.tf : w.t;   // B^T v lands here
    cudaError_t e = gmres_state_reset(gm, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(Vf, gx, n * sizeof(float), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess)
        e = mgs_pass(o.dot_mode, Vf, nullptr, nullptr, nullptr, n, gm.partials, &gm.st->counter, nullptr,
                     &gm.st->sumsq, nullptr, nullptr, s);
    if (e == cudaSuccess) {
        { ProfScope prof(PK_SMALL, s); gmres_init_kernel<<<1, 1, 0, s>>>(gm.st, gm.g, gm.resid, k); }
        e = cudaGetLastError();
    }
    for (int j = 0; j < k && e == cudaSuccess; ++j) {
        NvtxRange iter_range("adjoint GMRES iteration");
        float *vj = Vf + size_t(j) * gm.ldv;
        float *q = Vf + size_t(j + 1) * gm.ldv;
        {
            ProfScope prof(PK_CGLS_VEC, s);
            scale_vec_kernel<<<vb, RED_BLOCK, 0, s>>>(vj, n, &gm.st->inv_norm, stop);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = apply_Bt(g, o.b_kind, vj, w.t, w.bt_acc, sino, stop, s);
        if (e == cudaSuccess) e = launch_project_At(g, at_scatter(g), sino, q, w.acc, stop, s);
        if (e == cudaSuccess) e = arnoldi_orthogonalise(gm, q, j, k, n, o, s);
    }
    if (e == cudaSuccess) e = backsolve(gm.R, gm.g, gm.y, &gm.st->iters, k, s);
    float *z = Vf + size_t(k) * gm.ldv;
    if (e == cudaSuccess) e = combine(Vf, gm.ldv, k, n, gm.y, &gm.st->iters, z, s);
    if (e == cudaSuccess) e = apply_Bt(g, o.b_kind, z, w.t, w.bt_acc, gb, nullptr, s);
    if (e != cudaSuccess) {
        arena_close(ar);
        return cuda_error(e, "ct_bagmres_vjp launch");
    }
    rc = finish_solve(gm.st, gm.resid, k, resid_hist, iters_done, s, "ct_bagmres_vjp");
    arena_close(ar);
    return rc;
}

// ---------------------------------------------------------------------------
// CGLS with back-projector B
// ---------------------------------------------------------------------------
struct CglsWs {
    OpBufs ob;
    float *r = nullptr, *s = nullptr, *p = nullptr, *q = nullptr, *ax = nullptr;
    double *resid = nullptr, *partials = nullptr;
    SolverState *st = nullptr;
};

static void carve_cgls(Arena &ar, const GeomDev &g, int k, int b_kind, bool data_resid, CglsWs &w)
{
    const size_t n = size_t(g.nx) * g.ny * g.nz;
    const size_t m = size_t(g.n_views) * g.nv * g.nu;
    take_op_bufs(ar, g, w.ob, false, b_kind == CT_B_AT);
    w.r = ar.take<float>(m);
    w.q = ar.take<float>(m);
    w.s = ar.take<float>(n);
    w.p = ar.take<float>(n);
    w.ax = data_resid ? ar.take<float>(m) : nullptr;
    w.resid = ar.take<double>(size_t(k) + 1);
    w.partials = ar.take<double>(partials_count());
    w.st = ar.take<SolverState>(1);
}

static size_t cgls_ws_bytes(const GeomDev &g, int k, int b_kind, bool data_resid)
{
    Arena ar;
    ar.size = ~size_t(0) >> 1;
    CglsWs w;
    carve_cgls(ar, g, k, b_kind, data_resid, w);
    return ar.used;
}

static ct_status cgls(const ct_geom *geom, const float *b, int k, float *x, double *resid_hist,
                      const ct_solve_opts &o, int *iters_done, cudaStream_t s)
{
    const GeomDev &g = geom->g;
    const size_t n = geom->n, m = geom->m;
    const bool data = o.record_data_resid != 0;
    Arena ar;
    ct_status rc = open_ws(ar, cgls_ws_bytes(g, k, o.b_kind, data), o, s);
    if (rc != CT_OK) return rc;
    CglsWs w;
    carve_cgls(ar, g, k, o.b_kind, data, w);
    SolverState *st = w.st;
    const int *stop = &st->status;
    unsigned *ctr = &st->counter;
    const unsigned vb = red_blocks(std::max(n, m));
    cudaError_t e = cudaMemsetAsync(st, 0, sizeof(SolverState), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(w.ob.ypad, 0, padded_sino_floats(g) * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(x, 0, n * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w.r, b, m * sizeof(float), cudaMemcpyDeviceToDevice, s);
    // rr = ||r||^2, s = B r, gamma = ||s||^2, p = s
    if (e == cudaSuccess)
        e = mgs_pass(1, w.r, nullptr, nullptr, nullptr, m, w.partials, ctr, nullptr, &st->rr, nullptr, nullptr, s);
    if (e == cudaSuccess) e = apply_B(g, o.b_kind, w.r, nullptr, false, w.ob, w.s, nullptr, s);
    if (e == cudaSuccess)
        e = mgs_pass(1, w.s, nullptr, nullptr, nullptr, n, w.partials, ctr, nullptr, &st->gamma, nullptr, nullptr, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w.p, w.s, n * sizeof(float), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) {
        { ProfScope prof(PK_SMALL, s); cgls_init_kernel<<<1, 1, 0, s>>>(st, w.resid, k); }
        e = cudaGetLastError();
    }
    for (int j = 1; j <= k && e == cudaSuccess; ++j) {
        NvtxRange iter_range("CGLS iteration");
        // q = A p ; delta = ||q||^2
        e = launch_plane_copies(g, w.p, nullptr, nullptr, w.ob.Xc, w.ob.Yc, stop, s);
        if (e == cudaSuccess) e = launch_project_A(g, w.ob.Xc, w.ob.Yc, w.q, plain_layout(g), stop, s);
        if (e == cudaSuccess) e = fault_poison(w.q, j, stop, s);
        if (e == cudaSuccess)
            e = mgs_pass(1, w.q, nullptr, nullptr, nullptr, m, w.partials, ctr, nullptr, &st->delta, stop, nullptr, s);
        if (e == cudaSuccess) {
            { ProfScope prof(PK_SMALL, s); cgls_check_kernel<<<1, 1, 0, s>>>(st, 0); }
            e = cudaGetLastError();
        }
        // x += alpha p ; r -= alpha q (alpha = gamma / delta) ; rr = ||r||^2
        if (e == cudaSuccess) {
            ProfScope prof(PK_CGLS_VEC, s);
            axpy_ratio_kernel<<<vb, RED_BLOCK, 0, s>>>(x, w.p, &st->gamma, &st->delta, 1.0f, n, w.partials,
                                                       ctr, nullptr, stop);
            axpy_ratio_kernel<<<vb, RED_BLOCK, 0, s>>>(w.r, w.q, &st->gamma, &st->delta, -1.0f, m, w.partials,
                                                       ctr, &st->rr, stop);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && data) {
            e = launch_plane_copies(g, x, nullptr, nullptr, w.ob.Xc, w.ob.Yc, stop, s);
            if (e == cudaSuccess) e = launch_project_A(g, w.ob.Xc, w.ob.Yc, w.ax, plain_layout(g), stop, s);
            if (e == cudaSuccess) {
                { ProfScope prof(PK_CGLS_VEC, s); diff_sumsq_kernel<<<vb, RED_BLOCK, 0, s>>>(b, w.ax, m, w.partials, ctr, &st->data_rr, stop); }
                e = cudaGetLastError();
            }
        }
        // s = B r ; gamma_new = ||s||^2 ; p = s + (gamma_new/gamma) p ; gamma = gamma_new
        if (e == cudaSuccess) e = apply_B(g, o.b_kind, w.r, nullptr, false, w.ob, w.s, stop, s);
        if (e == cudaSuccess)
            e = mgs_pass(1, w.s, nullptr, nullptr, nullptr, n, w.partials, ctr, nullptr, &st->gamma_new, stop,
                         nullptr, s);
        if (e == cudaSuccess) {
            { ProfScope prof(PK_SMALL, s); cgls_record_kernel<<<1, 1, 0, s>>>(st, w.resid, j, data ? 1 : 0, o.tol); }
            { ProfScope prof(PK_CGLS_VEC, s); xpby_ratio_kernel<<<vb, RED_BLOCK, 0, s>>>(w.p, w.s, &st->gamma_new, &st->gamma, n, stop); }
            { ProfScope prof(PK_SMALL, s); cgls_shift_kernel<<<1, 1, 0, s>>>(st); }
            e = cudaGetLastError();
        }
    }
    if (e != cudaSuccess) {
        arena_close(ar);
        return cuda_error(e, "ct_cgls_solve launch");
    }
    rc = finish_solve(st, w.resid, k, resid_hist, iters_done, s, "ct_cgls_solve");
    arena_close(ar);
    return rc;
}

// ---------------------------------------------------------------------------
// Persistent BA-GMRES state: the workspace of one solve kept between calls,
// so a finished solve can be extended by more iterations, saved to a file
// and restored (the paper keeps its growing Krylov basis on disk, Sec. II).
// The basis lives in device memory or in page-locked host memory that the
// kernels read and write in place (on Grace-Blackwell over NVLink-C2C).
// ---------------------------------------------------------------------------
struct StateFileHeader {
    char magic[8];            // "CTGMRS01"
    int version;              // 1
    int vbf16;                // basis storage: 1 = bf16, 0 = float
    ct_geom_desc desc;        // the geometry the state belongs to
    int b_kind, dot_mode, reorth;
    int k_done;               // iterations done
    unsigned long long n;     // basis vector length
    SolverState st;           // device solver state at the save
};

}  // namespace ct

struct ct_gmres_state {
    const ct_geom *geom = nullptr;
    ct_solve_opts o{};
    int kmax = 0;
    int basis = CT_BASIS_DEVICE;
    void *dev_mem = nullptr;      // cudaMalloc'ed workspace (all but a host basis)
    void *host_basis = nullptr;   // cudaHostAlloc'ed basis (CT_BASIS_HOST)
    void *stage_mem = nullptr;    // cudaMalloc'ed ring and newest-vector buffers (CT_BASIS_HOST)
    ct::Stager stager;            // streams a host basis through stage_mem (CT_BASIS_HOST)
    ct::GmresWs w;
    int started = 0;
    int k_done = 0;               // iterations done, as of the last synchronising call
    int status = 0;               // device status word, as of the last synchronising call
};

namespace ct {

static void state_free(ct_gmres_state *st)
{
    if (!st) return;
    Stager &sg = st->stager;
    if (sg.cs) cudaStreamSynchronize(sg.cs);
    for (cudaEvent_t e : sg.ev)
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : sg.ready)
        if (e) cudaEventDestroy(e);
    if (sg.vnew_free) cudaEventDestroy(sg.vnew_free);
    if (sg.cs) cudaStreamDestroy(sg.cs);
    if (st->dev_mem) cudaFree(st->dev_mem);
    if (st->stage_mem) cudaFree(st->stage_mem);
    if (st->host_basis) cudaFreeHost(st->host_basis);
    delete st;
}

// The copy stream, events and device buffers of a staged host basis.
static cudaError_t stager_init(ct_gmres_state *st)
{
    Stager &sg = st->stager;
    const GmresWs &w = st->w;
    const size_t esz = w.vbf16 ? 2 : 4;
    sg.vbytes = st->geom->n * esz;
    sg.vbytes_ld = w.ldv * esz;
    const size_t slot = Arena::align(sg.vbytes);
    cudaError_t e = cudaMalloc(&st->stage_mem, 4 * slot);
    if (e != cudaSuccess) return e;
    char *base = static_cast<char *>(st->stage_mem);
    for (int i = 0; i < 3; ++i) sg.ring[i] = base + i * slot;
    sg.vnew = base + 3 * slot;
    sg.host = static_cast<char *>(st->host_basis);
    e = cudaStreamCreateWithFlags(&sg.cs, cudaStreamNonBlocking);
    for (int i = 0; i < 8 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&sg.ev[i], cudaEventDisableTiming);
    for (int i = 0; i < 3 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&sg.ready[i], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&sg.vnew_free, cudaEventDisableTiming);
    return e;
}

__global__ void __launch_bounds__(RED_BLOCK) basis_axpy_kernel_f32(float *__restrict__ x, const float *__restrict__ v,
                                                                   const double *__restrict__ y, int i, size_t len)
{
    const float yi = float(y[i]);
    for (size_t e = blockIdx.x * size_t(RED_BLOCK) + threadIdx.x; e < len; e += size_t(gridDim.x) * RED_BLOCK)
        x[e] = fmaf(yi, v[e], i == 0 ? 0.0f : x[e]);
}

__global__ void __launch_bounds__(RED_BLOCK) basis_axpy_kernel_bf16(float *__restrict__ x,
                                                                    const __nv_bfloat16 *__restrict__ v,
                                                                    const double *__restrict__ y, int i, size_t len)
{
    const float yi = float(y[i]);
    for (size_t e = blockIdx.x * size_t(RED_BLOCK) + threadIdx.x; e < len; e += size_t(gridDim.x) * RED_BLOCK)
        x[e] = fmaf(yi, __bfloat162float(v[e]), i == 0 ? 0.0f : x[e]);
}

// x = sum_{i < count} y_i V_i over a staged basis, one vector at a time in
// the order (and with the FMA rounding) of combine_kernel, so the result is
// the same bits.
static cudaError_t staged_combine(Stager &sg, bool vbf16, int count, const double *y, size_t len, float *x,
                                  cudaStream_t s)
{
    if (count <= 0) return cudaMemsetAsync(x, 0, len * sizeof(float), s);
    cudaError_t e = sg.fetch(0, s);
    if (e == cudaSuccess && 1 < count) e = sg.fetch(1, s);
    const unsigned blocks = unsigned(std::max<size_t>(1, std::min((len + RED_BLOCK - 1) / RED_BLOCK,
                                                                  size_t(num_sms()) * 8)));
    for (int i = 0; i < count && e == cudaSuccess; ++i) {
        const void *v = sg.vector(i, -1, s);
        {
            ProfScope prof(PK_COMBINE, s);
            if (vbf16)
                basis_axpy_kernel_bf16<<<blocks, RED_BLOCK, 0, s>>>(x, static_cast<const __nv_bfloat16 *>(v), y, i,
                                                                      len);
            else
                basis_axpy_kernel_f32<<<blocks, RED_BLOCK, 0, s>>>(x, static_cast<const float *>(v), y, i, len);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess && i + 2 < count) e = sg.fetch(i + 2, s);
    }
    return e;
}

static ct_status state_alloc(const ct_geom *geom, int kmax, int basis, const ct_solve_opts &o, ct_gmres_state **out)
{
    const GeomDev &g = geom->g;
    const bool host = basis == CT_BASIS_HOST;
    ct_gmres_state *st = new (std::nothrow) ct_gmres_state;
    if (!st) return set_error(CT_ENOMEM, "ct_bagmres_state: out of host memory");
    st->geom = geom;
    st->o = o;
    st->o.tol = 0.0;   // the state runs exactly the iterations asked for
    st->o.workspace = nullptr;
    st->o.workspace_bytes = 0;
    st->kmax = kmax;
    st->basis = basis;
    const size_t bytes = gmres_bytes(g, kmax, false, o.b_kind, host);
    cudaError_t e = cudaMalloc(&st->dev_mem, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        st->dev_mem = nullptr;
        state_free(st);
        return set_error(CT_ENOMEM, "ct_bagmres_state: cudaMalloc(%zu bytes) failed", bytes);
    }
    Arena ar;
    ar.base = static_cast<char *>(st->dev_mem);
    ar.size = bytes;
    carve_gmres(ar, g, kmax, false, o.b_kind, st->w, host);
    if (host) {
        const size_t vb = basis_bytes(g, kmax, false);
        e = cudaHostAlloc(&st->host_basis, vb, cudaHostAllocMapped | cudaHostAllocPortable);
        if (e != cudaSuccess) {
            cudaGetLastError();
            st->host_basis = nullptr;
            state_free(st);
            return set_error(CT_ENOMEM, "ct_bagmres_state: cudaHostAlloc(%zu bytes) for the basis failed", vb);
        }
        // the kernels see only the device staging buffers; the host pointer
        // serves the copies (and save/load)
        st->w.V = st->host_basis;
        e = stager_init(st);
        if (e != cudaSuccess) {
            cudaGetLastError();
            state_free(st);
            return set_error(CT_ENOMEM, "ct_bagmres_state: the device staging buffers of a host basis failed");
        }
    }
    *out = st;
    return CT_OK;
}

static ct_status state_check_device(const ct_geom *geom, const char *who)
{
    int dev = -1;
    CT_CUDA(cudaGetDevice(&dev));
    if (dev != geom->device)
        return set_error(CT_EINVAL, "%s: the geometry lives on device %d but device %d is current", who,
                         geom->device, dev);
    return CT_OK;
}

static bool same_desc(const ct_geom_desc &a, const ct_geom_desc &b)
{
    return a.kind == b.kind && a.nx == b.nx && a.ny == b.ny && a.nz == b.nz && a.voxel_mm == b.voxel_mm &&
           a.n_views == b.n_views && a.angle_start_rad == b.angle_start_rad &&
           a.angle_span_rad == b.angle_span_rad && a.nu == b.nu && a.nv == b.nv && a.du_mm == b.du_mm &&
           a.dv_mm == b.dv_mm && a.sod_mm == b.sod_mm && a.sdd_mm == b.sdd_mm && a.vol_dtype == b.vol_dtype &&
           a.sino_dtype == b.sino_dtype && a.projector == b.projector;
}

}  // namespace ct

using namespace ct;

static ct_solve_opts resolve_opts(const ct_solve_opts *opts)
{
    ct_solve_opts o;
    ct_solve_opts_default(&o);
    if (opts) o = *opts;
    return o;
}

extern "C" {

size_t ct_workspace_bytes(const ct_geom *geom, int k, int solver, const ct_solve_opts *opts)
{
    if (!geom || k < 1) return 0;
    ct_solve_opts o = resolve_opts(opts);
    switch (solver) {
    case CT_SOLVER_BA: return gmres_bytes(geom->g, k, false, o.b_kind);
    case CT_SOLVER_AB: return gmres_bytes(geom->g, k, true, o.b_kind);
    case CT_SOLVER_CGLS: return cgls_ws_bytes(geom->g, k, o.b_kind, o.record_data_resid != 0);
    case CT_SOLVER_BA_VJP: return vjp_bytes(geom->g, k, o.b_kind);
    default: return 0;
    }
}

ct_status ct_bagmres_solve(const ct_geom *geom, const float *b_dev, int k, float *x_out_dev,
                           double *resid_hist, const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_bagmres_solve");
    ct_solve_opts o = resolve_opts(opts);
    ct_status rc = check_common(geom, b_dev, k, x_out_dev, &o);
    if (rc != CT_OK) return rc;
    return bagmres(geom, b_dev, k, x_out_dev, resid_hist, o, iters_done, static_cast<cudaStream_t>(stream));
}

ct_status ct_bagmres_solve_host(const ct_geom *geom, const float *b_host, int k, float *x_out_host,
                                double *resid_hist, const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_bagmres_solve_host");
    ct_solve_opts o = resolve_opts(opts);
    ct_status rc = check_common(geom, b_host, k, x_out_host, &o);
    if (rc != CT_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t mb = geom->m * sizeof(float), nb = geom->n * sizeof(float);
    void *bd = nullptr, *xd = nullptr;
    cudaError_t e = scratch_alloc(&bd, mb, s);
    if (e == cudaSuccess) e = scratch_alloc(&xd, nb, s);
    if (e != cudaSuccess) {
        if (bd) cudaFreeAsync(bd, s);
        cudaGetLastError();
        return set_error(CT_ENOMEM, "ct_bagmres_solve_host: device buffers of %zu + %zu bytes: %s", mb, nb,
                         cudaGetErrorString(e));
    }
    e = cudaMemcpyAsync(bd, b_host, mb, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        rc = bagmres(geom, static_cast<const float *>(bd), k, static_cast<float *>(xd), resid_hist, o, iters_done, s);
        if (rc == CT_OK || rc == CT_BREAKDOWN_LUCKY) {
            e = cudaMemcpyAsync(x_out_host, xd, nb, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        }
    }
    cudaFreeAsync(xd, s);
    cudaFreeAsync(bd, s);
    if (e != cudaSuccess) return cuda_error(e, "ct_bagmres_solve_host copy");
    return rc;
}

ct_status ct_bagmres_solve_err(const ct_geom *geom, const float *b_dev, int k, float *x_out_dev,
                               const float *x_ref_dev, double *resid_hist, double *err_hist,
                               const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_bagmres_solve_err");
    ct_solve_opts o = resolve_opts(opts);
    ct_status rc = check_common(geom, b_dev, k, x_out_dev, &o);
    if (rc != CT_OK) return rc;
    if (!x_ref_dev || !err_hist) return set_error(CT_EINVAL, "ct_bagmres_solve_err: NULL x_ref or err_hist");
    return bagmres(geom, b_dev, k, x_out_dev, resid_hist, o, iters_done, static_cast<cudaStream_t>(stream),
                   x_ref_dev, err_hist);
}

ct_status ct_bagmres_restarted(const ct_geom *geom, const float *b_dev, int m, int cycles, float *x_out_dev,
                               double *resid_hist, const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_bagmres_restarted");
    ct_solve_opts o = resolve_opts(opts);
    ct_status rc = check_common(geom, b_dev, m, x_out_dev, &o);
    if (rc != CT_OK) return rc;
    if (cycles < 1 || size_t(m) * cycles > 1u << 20)
        return set_error(CT_EINVAL, "ct_bagmres_restarted: cycles must be >= 1 and m * cycles <= 2^20");
    return bagmres_restarted(geom, b_dev, m, cycles, x_out_dev, resid_hist, o, iters_done,
                             static_cast<cudaStream_t>(stream));
}

ct_status ct_abgmres_solve(const ct_geom *geom, const float *b_dev, int k, float *x_out_dev,
                           double *resid_hist, const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_abgmres_solve");
    ct_solve_opts o = resolve_opts(opts);
    ct_status rc = check_common(geom, b_dev, k, x_out_dev, &o);
    if (rc != CT_OK) return rc;
    return abgmres(geom, b_dev, k, x_out_dev, resid_hist, o, iters_done, static_cast<cudaStream_t>(stream));
}

ct_status ct_cgls_solve(const ct_geom *geom, const float *b_dev, int k, float *x_out_dev,
                        double *resid_hist, const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_cgls_solve");
    ct_solve_opts o = resolve_opts(opts);
    ct_status rc = check_common(geom, b_dev, k, x_out_dev, &o);
    if (rc != CT_OK) return rc;
    return cgls(geom, b_dev, k, x_out_dev, resid_hist, o, iters_done, static_cast<cudaStream_t>(stream));
}

ct_status ct_bagmres_vjp(const ct_geom *geom, const float *gx_dev, int k, float *gb_dev, double *resid_hist,
                         const ct_solve_opts *opts, int *iters_done, void *stream)
{
    NvtxRange call_range("ct_bagmres_vjp");
    ct_solve_opts o = resolve_opts(opts);
    if (!geom || !gx_dev || !gb_dev) return set_error(CT_EINVAL, "ct_bagmres_vjp: NULL argument");
    if (k < 1 || k > 4096) return set_error(CT_EINVAL, "ct_bagmres_vjp: k must be in [1, 4096] (got %d)", k);
    if (o.dot_mode != 0 && o.dot_mode != 1) return set_error(CT_EINVAL, "ct_bagmres_vjp: dot_mode must be 0 or 1");
    if (!(o.tol >= 0.0)) return set_error(CT_EINVAL, "ct_bagmres_vjp: tol must be >= 0");
    return bagmres_vjp(geom, gx_dev, k, gb_dev, resid_hist, o, iters_done, static_cast<cudaStream_t>(stream));
}

ct_status ct_bagmres_state_create(const ct_geom *geom, int kmax, int basis, const ct_solve_opts *opts,
                                  ct_gmres_state **out)
{
    NvtxRange call_range("ct_bagmres_state_create");
    if (out) *out = nullptr;
    if (!geom || !out) return set_error(CT_EINVAL, "ct_bagmres_state_create: NULL argument");
    if (kmax < 1 || kmax > 4096)
        return set_error(CT_EINVAL, "ct_bagmres_state_create: kmax must be in 1..4096 (got %d)", kmax);
    if (basis != CT_BASIS_DEVICE && basis != CT_BASIS_HOST)
        return set_error(CT_EINVAL, "ct_bagmres_state_create: unknown basis location %d", basis);
    ct_solve_opts o = resolve_opts(opts);
    if (o.b_kind != CT_B_UN && o.b_kind != CT_B_FBP && o.b_kind != CT_B_AT)
        return set_error(CT_EINVAL, "ct_bagmres_state_create: unknown b_kind %d", o.b_kind);
    if (o.dot_mode != 0 && o.dot_mode != 1)
        return set_error(CT_EINVAL, "ct_bagmres_state_create: dot_mode must be 0 or 1");
    ct_status rc = state_check_device(geom, "ct_bagmres_state_create");
    if (rc != CT_OK) return rc;
    return state_alloc(geom, kmax, basis, o, out);
}

void ct_gmres_state_destroy(ct_gmres_state *state)
{
    if (!state) return;
    cudaDeviceSynchronize();   // no kernel of the state may still run
    state_free(state);
}

int ct_gmres_state_iters(const ct_gmres_state *state) { return state ? state->k_done : -1; }

size_t ct_gmres_state_basis_bytes(const ct_geom *geom, int kmax)
{
    if (!geom || kmax < 1) return 0;
    return basis_bytes(geom->g, kmax, false);
}

ct_status ct_bagmres_state_start(ct_gmres_state *state, const float *b_dev, void *stream)
{
    NvtxRange call_range("ct_bagmres_state_start");
    if (!state || !b_dev) return set_error(CT_EINVAL, "ct_bagmres_state_start: NULL argument");
    ct_status rc = state_check_device(state->geom, "ct_bagmres_state_start");
    if (rc == CT_OK && state->o.b_kind == CT_B_FBP) rc = check_ramp(state->geom->g, "ct_bagmres_state_start");
    if (rc != CT_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = ba_start(state->geom->g, state->w, b_dev, state->kmax, state->geom->n, state->o, s);
    if (e != cudaSuccess) return cuda_error(e, "ct_bagmres_state_start launch");
    state->started = 1;
    state->k_done = 0;
    state->status = ST_RUN;
    return CT_OK;
}

ct_status ct_bagmres_state_extend(ct_gmres_state *state, int k, float *x_out_dev, double *resid_hist,
                                  int *iters_done, void *stream)
{
    NvtxRange call_range("ct_bagmres_state_extend");
    if (!state || !x_out_dev) return set_error(CT_EINVAL, "ct_bagmres_state_extend: NULL argument");
    if (!state->started) return set_error(CT_EINVAL, "ct_bagmres_state_extend: the state has not been started");
    if (k < 1 || k > state->kmax)
        return set_error(CT_EINVAL, "ct_bagmres_state_extend: k must be in 1..%d (the state's kmax), got %d",
                         state->kmax, k);
    ct_status rc = state_check_device(state->geom, "ct_bagmres_state_extend");
    if (rc != CT_OK) return rc;
    const GeomDev &g = state->geom->g;
    const size_t n = state->geom->n;
    GmresWs &w = state->w;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    Stager *sg = state->basis == CT_BASIS_HOST ? &state->stager : nullptr;
    if (state->status == ST_RUN)
        for (int j = state->k_done; j < k && e == cudaSuccess; ++j)
            e = ba_iteration(g, w, j, state->kmax, n, state->o, s, sg);
    // x = V_c y_c with c = min(k, iterations done)
    if (e == cudaSuccess) {
        {
            ProfScope prof(PK_SMALL, s);
            iterate_upto_kernel<<<1, 1, 0, s>>>(w.st, k, w.cnt);
        }
        e = backsolve(w.R, w.g, w.y, w.cnt, state->kmax, s);
    }
    SolverState hst;
    std::vector<double> hres(size_t(k) + 1);
    if (e == cudaSuccess && sg) {
        // a staged basis streams exactly the vectors the iterate needs: learn
        // how many first
        e = cudaMemcpyAsync(&hst, w.st, sizeof(SolverState), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e == cudaSuccess) e = staged_combine(*sg, w.vbf16, hst.iters < k ? hst.iters : k, w.y, n, x_out_dev, s);
    } else if (e == cudaSuccess) {
        e = w.vbf16 ? combine_t(static_cast<const __nv_bfloat16 *>(w.V), w.ldv, state->kmax, n, w.y, w.cnt,
                                x_out_dev, s)
                    : combine(static_cast<const float *>(w.V), w.ldv, state->kmax, n, w.y, w.cnt, x_out_dev, s);
    }
    if (e != cudaSuccess) return cuda_error(e, "ct_bagmres_state_extend launch");
    CT_CUDA(cudaMemcpyAsync(&hst, w.st, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
    CT_CUDA(cudaMemcpyAsync(hres.data(), w.resid, sizeof(double) * (k + 1), cudaMemcpyDeviceToHost, s));
    CT_CUDA(cudaStreamSynchronize(s));
    if (sg) CT_CUDA(cudaStreamSynchronize(sg->cs));   // the host basis holds every vector on return
    state->k_done = hst.iters;
    state->status = hst.status;
    if (resid_hist) std::copy(hres.begin(), hres.end(), resid_hist);
    if (iters_done) *iters_done = hst.iters < k ? hst.iters : k;
    if (hst.status == ST_NONFINITE)
        return set_error(CT_ENONFINITE, "ct_bagmres_state_extend: a norm became NaN/Inf after %d iterations",
                         hst.iters);
    if (hst.status == ST_TIMEOUT)
        return set_error(CT_ETIMEOUT, "ct_bagmres_state_extend: a wait between blocks ran out after %d iterations",
                         hst.iters);
    if (hst.status == ST_LUCKY) return CT_BREAKDOWN_LUCKY;
    return CT_OK;
}

ct_status ct_gmres_state_save(const ct_gmres_state *state, const char *path, void *stream)
{
    NvtxRange call_range("ct_gmres_state_save");
    if (!state || !path) return set_error(CT_EINVAL, "ct_gmres_state_save: NULL argument");
    if (!state->started) return set_error(CT_EINVAL, "ct_gmres_state_save: the state has not been started");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const GmresWs &w = state->w;
    const size_t n = state->geom->n;
    const int kd = state->k_done;
    const size_t ld = size_t(state->kmax) + 1;
    StateFileHeader h;
    std::memset(&h, 0, sizeof(h));
    std::memcpy(h.magic, "CTGMRS01", 8);
    h.version = 1;
    h.vbf16 = w.vbf16 ? 1 : 0;
    h.desc = state->geom->desc;
    h.b_kind = state->o.b_kind;
    h.dot_mode = state->o.dot_mode;
    h.reorth = state->o.reorth;
    h.k_done = kd;
    h.n = n;
    CT_CUDA(cudaStreamSynchronize(s));
    if (state->stager.cs) CT_CUDA(cudaStreamSynchronize(state->stager.cs));
    CT_CUDA(cudaMemcpy(&h.st, w.st, sizeof(SolverState), cudaMemcpyDeviceToHost));
    if (h.st.iters != kd) return set_error(CT_EINVAL, "ct_gmres_state_save: the state changed since its last call");
    // the first kd columns of H and R (rows 0..kd), cs, sn, g and resid (kd + 1)
    const size_t rows = size_t(kd) + 1;
    std::vector<double> H(rows * kd), R(rows * kd), cs(kd), sn(kd), gv(rows), res(rows);
    for (int j = 0; j < kd; ++j) {
        CT_CUDA(cudaMemcpy(H.data() + j * rows, w.H + j * ld, rows * sizeof(double), cudaMemcpyDeviceToHost));
        CT_CUDA(cudaMemcpy(R.data() + j * rows, w.R + j * ld, rows * sizeof(double), cudaMemcpyDeviceToHost));
    }
    if (kd > 0) {
        CT_CUDA(cudaMemcpy(cs.data(), w.cs, kd * sizeof(double), cudaMemcpyDeviceToHost));
        CT_CUDA(cudaMemcpy(sn.data(), w.sn, kd * sizeof(double), cudaMemcpyDeviceToHost));
    }
    CT_CUDA(cudaMemcpy(gv.data(), w.g, rows * sizeof(double), cudaMemcpyDeviceToHost));
    CT_CUDA(cudaMemcpy(res.data(), w.resid, rows * sizeof(double), cudaMemcpyDeviceToHost));
    std::vector<float> q(n);
    CT_CUDA(cudaMemcpy(q.data(), w.q, n * sizeof(float), cudaMemcpyDeviceToHost));
    FILE *f = std::fopen(path, "wb");
    if (!f) return set_error(CT_EINVAL, "ct_gmres_state_save: cannot open %s for writing", path);
    bool ok = std::fwrite(&h, sizeof(h), 1, f) == 1;
    auto put = [&](const void *p, size_t bytes) { ok = ok && (bytes == 0 || std::fwrite(p, bytes, 1, f) == 1); };
    put(H.data(), H.size() * sizeof(double));
    put(R.data(), R.size() * sizeof(double));
    put(cs.data(), cs.size() * sizeof(double));
    put(sn.data(), sn.size() * sizeof(double));
    put(gv.data(), gv.size() * sizeof(double));
    put(res.data(), res.size() * sizeof(double));
    put(q.data(), n * sizeof(float));
    // the kd basis vectors, one at a time
    const size_t esz = w.vbf16 ? 2 : 4;
    std::vector<char> vbuf(n * esz);
    for (int i = 0; i < kd && ok; ++i) {
        cudaError_t e = cudaMemcpy(vbuf.data(), w.vec(i), n * esz, cudaMemcpyDefault);
        if (e != cudaSuccess) {
            std::fclose(f);
            return cuda_error(e, "ct_gmres_state_save: basis copy");
        }
        put(vbuf.data(), n * esz);
    }
    ok = (std::fclose(f) == 0) && ok;
    if (!ok) return set_error(CT_EINVAL, "ct_gmres_state_save: writing %s failed", path);
    return CT_OK;
}

ct_status ct_gmres_state_load(const ct_geom *geom, const char *path, int kmax, int basis, ct_gmres_state **out,
                              void *stream)
{
    NvtxRange call_range("ct_gmres_state_load");
    if (out) *out = nullptr;
    if (!geom || !path || !out) return set_error(CT_EINVAL, "ct_gmres_state_load: NULL argument");
    if (basis != CT_BASIS_DEVICE && basis != CT_BASIS_HOST)
        return set_error(CT_EINVAL, "ct_gmres_state_load: unknown basis location %d", basis);
    ct_status rc = state_check_device(geom, "ct_gmres_state_load");
    if (rc != CT_OK) return rc;
    FILE *f = std::fopen(path, "rb");
    if (!f) return set_error(CT_EINVAL, "ct_gmres_state_load: cannot open %s", path);
    StateFileHeader h;
    bool ok = std::fread(&h, sizeof(h), 1, f) == 1;
    const size_t n = geom->n;
    if (!ok || std::memcmp(h.magic, "CTGMRS01", 8) != 0 || h.version != 1) {
        std::fclose(f);
        return set_error(CT_EINVAL, "ct_gmres_state_load: %s is not a saved solver state", path);
    }
    if (!same_desc(h.desc, geom->desc) || h.n != n || h.vbf16 != (geom->g.vol_bf16 ? 1 : 0)) {
        std::fclose(f);
        return set_error(CT_EINVAL, "ct_gmres_state_load: %s belongs to another geometry", path);
    }
    const int kd = h.k_done;
    if (kd < 0 || kd > 4096 || kmax < kd || kmax < 1 || kmax > 4096) {
        std::fclose(f);
        return set_error(CT_EINVAL, "ct_gmres_state_load: kmax %d must be in %d..4096 (the iterations saved)",
                         kmax, kd > 1 ? kd : 1);
    }
    ct_solve_opts o;
    ct_solve_opts_default(&o);
    o.b_kind = h.b_kind;
    o.dot_mode = h.dot_mode;
    o.reorth = h.reorth;
    ct_gmres_state *st = nullptr;
    rc = state_alloc(geom, kmax, basis, o, &st);
    if (rc != CT_OK) {
        std::fclose(f);
        return rc;
    }
    const size_t rows = size_t(kd) + 1, ld = size_t(kmax) + 1;
    std::vector<double> H(rows * kd), R(rows * kd), cs(kd), sn(kd), gv(rows), res(rows);
    auto get = [&](void *p, size_t bytes) { ok = ok && (bytes == 0 || std::fread(p, bytes, 1, f) == 1); };
    get(H.data(), H.size() * sizeof(double));
    get(R.data(), R.size() * sizeof(double));
    get(cs.data(), cs.size() * sizeof(double));
    get(sn.data(), sn.size() * sizeof(double));
    get(gv.data(), gv.size() * sizeof(double));
    get(res.data(), res.size() * sizeof(double));
    std::vector<float> q(n);
    get(q.data(), n * sizeof(float));
    GmresWs &w = st->w;
    cudaError_t e = cudaSuccess;
    // H, R, g zero beyond what was saved; resid -1 after the iterations done
    std::vector<double> res_full(ld, -1.0);
    std::copy(res.begin(), res.end(), res_full.begin());
    e = cudaMemset(w.H, 0, sizeof(double) * ld * kmax);
    if (e == cudaSuccess) e = cudaMemset(w.R, 0, sizeof(double) * ld * kmax);
    if (e == cudaSuccess) e = cudaMemset(w.g, 0, sizeof(double) * ld);
    if (e == cudaSuccess) e = cudaMemset(w.ob.ypad, 0, padded_sino_floats(geom->g) * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(w.slots, 0xff, slots_count() * sizeof(unsigned long long));
    for (int j = 0; j < kd && e == cudaSuccess; ++j) {
        e = cudaMemcpy(w.H + j * ld, H.data() + j * rows, rows * sizeof(double), cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(w.R + j * ld, R.data() + j * rows, rows * sizeof(double), cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess && kd > 0) e = cudaMemcpy(w.cs, cs.data(), kd * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && kd > 0) e = cudaMemcpy(w.sn, sn.data(), kd * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w.g, gv.data(), rows * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w.resid, res_full.data(), ld * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w.q, q.data(), n * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w.st, &h.st, sizeof(SolverState), cudaMemcpyHostToDevice);
    const size_t esz = w.vbf16 ? 2 : 4;
    std::vector<char> vbuf(n * esz);
    for (int i = 0; i < kd && ok && e == cudaSuccess; ++i) {
        get(vbuf.data(), n * esz);
        if (ok) e = cudaMemcpy(w.vec(i), vbuf.data(), n * esz, cudaMemcpyDefault);
    }
    std::fclose(f);
    if (e == cudaSuccess) e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (!ok || e != cudaSuccess) {
        state_free(st);
        if (e != cudaSuccess) return cuda_error(e, "ct_gmres_state_load: upload");
        return set_error(CT_EINVAL, "ct_gmres_state_load: %s is truncated", path);
    }
    st->started = 1;
    st->k_done = kd;
    st->status = h.st.status;
    *out = st;
    return CT_OK;
}

ct_status ct_mgs_sweep(const float *V_dev, size_t ldv, int j, size_t len, float *q_dev, double *h_dev,
                       int dot_mode, void *stream)
{
    NvtxRange call_range("ct_mgs_sweep");
    if (!q_dev || !h_dev || (j > 0 && !V_dev)) return set_error(CT_EINVAL, "ct_mgs_sweep: NULL argument");
    if (j < 0 || len == 0 || (j > 0 && ldv < len))
        return set_error(CT_EINVAL, "ct_mgs_sweep: bad sizes (j=%d len=%zu ldv=%zu)", j, len, ldv);
    if (dot_mode != 0 && dot_mode != 1) return set_error(CT_EINVAL, "ct_mgs_sweep: dot_mode must be 0 or 1");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Arena ar;
    const size_t bytes = Arena::align(partials_count() * sizeof(double)) + Arena::align(sizeof(unsigned));
    ct_status rc = arena_open(ar, bytes, nullptr, 0, s);
    if (rc != CT_OK) return rc;
    double *partials = ar.take<double>(partials_count());
    unsigned *ctr = ar.take<unsigned>(1);
    cudaError_t e = cudaMemsetAsync(ctr, 0, sizeof(unsigned), s);
    for (int i = 0; i <= j && e == cudaSuccess; ++i) {
        const float *vprev = i > 0 ? V_dev + size_t(i - 1) * ldv : nullptr;
        const double *hprev = i > 0 ? h_dev + (i - 1) : nullptr;
        const float *vcur = i < j ? V_dev + size_t(i) * ldv : nullptr;
        double *odot = i < j ? h_dev + i : nullptr;
        double *oss = i == j ? h_dev + j : nullptr;
        e = mgs_pass(dot_mode, q_dev, vprev, hprev, vcur, len, partials, ctr, odot, oss, nullptr, nullptr, s);
    }
    // h[j] = sqrt(||q||^2)
    if (e == cudaSuccess) {
        { ProfScope prof(PK_SMALL, s); sqrt_inplace_kernel<<<1, 1, 0, s>>>(h_dev + j); }
        e = cudaGetLastError();
    }
    arena_close(ar);
    if (e != cudaSuccess) return cuda_error(e, "ct_mgs_sweep launch");
    return CT_OK;
}

ct_status ct_basis_combine(const float *V_dev, size_t ldv, int k, size_t len, const double *y_dev,
                           float *x_dev, void *stream)
{
    NvtxRange call_range("ct_basis_combine");
    if (!V_dev || !y_dev || !x_dev) return set_error(CT_EINVAL, "ct_basis_combine: NULL argument");
    if (k < 1 || len == 0 || ldv < len) return set_error(CT_EINVAL, "ct_basis_combine: bad sizes");
    if (k > 4096) return set_error(CT_EINVAL, "ct_basis_combine: k must be <= 4096");
    cudaError_t e = combine(V_dev, ldv, k, len, y_dev, nullptr, x_dev, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_error(e, "ct_basis_combine launch");
    return CT_OK;
}

}  // extern "C"
