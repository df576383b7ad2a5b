// Ray-driven Joseph projector A and its exact transpose A^T.
//
// A (Sec. I Eq. 1, Sec. III): every detector ray walks the voxel-centre
// planes of its dominant axis (x when |d_x| >= |d_y|, else y); on each plane
// it takes the bilinear interpolation of the four neighbouring voxels in
// that plane (neighbours outside the grid are zero), and the sum is scaled
// by the step length vox |d| / |d_a|.
//
// GPU layout.  The gathers run against two plane-major copies of the volume
// with a zero border of PAD_A voxels around the in-plane and z axes:
//   Xc[zp][x][yp]  for x-dominant rays (planes along x, in-plane axis y fastest),
//   Yc[zp][y][xp]  for y-dominant rays (planes along y, in-plane axis x fastest).
// Neighbouring rays of a detector row then read neighbouring words, and each
// ray's plane range is clipped up front so that the unrolled inner loop has no
// bounds tests.  Building the copies reads the volume once and is also where
// the Arnoldi step normalises its newest basis vector.
//
// Ray coordinates.  The sample position on plane p is affine in p:
//   f_b(p) = fbc + (p - c_a) gb,  f_z(p) = fzc + (p - c_a) gz
// with the value at the central plane computed from the cross product
// (S x d)_z rather than from S + t d, which in FP32 would cancel two terms of
// the size of the source distance; (S x d)_z = sod*u exactly for this
// geometry, so the intercept keeps full relative precision.
#include <algorithm>
#include <mutex>

#include "ct_internal.cuh"

namespace ct {

// Narrows [p0, p1] to the planes whose f(p) = fc + (p - ca) g lies in
// [lo - 0.5, hi + 0.5].  Every sample with f in [lo, hi) stays inside; every
// kept sample has floor(f) in [lo - 1, hi], inside the zero border.
__device__ __forceinline__ void clip_planes(float fc, float g, float lo, float hi, float ca, int Na,
                                            int &p0, int &p1)
{
    if (fabsf(g) < 1e-20f) {
        if (!(fc >= lo - 0.5f && fc <= hi + 0.5f)) p1 = -1;
        return;
    }
    float ig = 1.0f / g;
    float t1 = (lo - 0.5f - fc) * ig + ca;
    float t2 = (hi + 0.5f - fc) * ig + ca;
    // both ends are held to [-1, Na]: a ray nearly parallel to a grid side that
    // passes beside it has t of 1e17, and plane numbers that saturate would
    // overflow in the kernels' sums (a warp's share is added to p0)
    float tl = fminf(fmaxf(fminf(t1, t2), -1.0f), float(Na));
    float th = fmaxf(fminf(fmaxf(t1, t2), float(Na)), -1.0f);
    p0 = max(p0, int(ceilf(tl)));
    p1 = min(p1, int(floorf(th)));
}

// Planes on which some ray of a run of rays has its coordinate f inside
// [lo, hi] (with clip_planes's half-voxel margin), the run's rays lying
// between its first ray (fc_f, g_f) and its last (fc_l, g_l) on every plane
// (f is linear in the ray's row, and the rows run in order).  On a plane the
// run covers [min(f_f, f_l), max(f_f, f_l)], so the plane is needed when one
// end ray is above lo and one end ray is below hi.  Each condition holds on a
// union of two half-lines of planes; its hull is taken (exact when one end
// ray stays above the other over the grid, as when the source lies outside
// the grid's plane range; otherwise a superset, whose extra planes add
// zeros).  Joining the two end rays' own plane ranges instead misses the far
// planes of the rays between them when the end rays leave through opposite
// faces (a short volume under a tall detector).
__device__ __forceinline__ void clip_planes_run(float fc_f, float g_f, float fc_l, float g_l, float lo, float hi,
                                                float ca, int Na, int &p0, int &p1)
{
    constexpr float BIG = 3.0e38f;
    auto hull = [](int a0, int a1, int b0, int b1, int &h0, int &h1) {
        if (a0 > a1) {
            h0 = b0;
            h1 = b1;
        } else if (b0 > b1) {
            h0 = a0;
            h1 = a1;
        } else {
            h0 = min(a0, b0);
            h1 = max(a1, b1);
        }
    };
    int a0 = 0, a1 = Na - 1, b0 = 0, b1 = Na - 1, u0, u1, w0, w1;
    clip_planes(fc_f, g_f, lo, BIG, ca, Na, a0, a1);   // first ray above lo
    clip_planes(fc_l, g_l, lo, BIG, ca, Na, b0, b1);   // last ray above lo
    hull(a0, a1, b0, b1, u0, u1);
    a0 = 0, a1 = Na - 1, b0 = 0, b1 = Na - 1;
    clip_planes(fc_f, g_f, -BIG, hi, ca, Na, a0, a1);  // first ray below hi
    clip_planes(fc_l, g_l, -BIG, hi, ca, Na, b0, b1);  // last ray below hi
    hull(a0, a1, b0, b1, w0, w1);
    p0 = max(p0, max(u0, w0));
    p1 = min(p1, min(u1, w1));
}

// ---------------------------------------------------------------------------
// Plane-major zero-bordered copies.  One block handles a 32x32 (x, y) tile
// of one padded z slice, read with a one-voxel halo so that bf16 pairs
// (b, b+1) can be formed; Yc rows are written straight from the tile, Xc
// rows from its transpose in shared memory.  When a basis slot is given the
// scaled volume is stored there too (each voxel by the tile that owns it).
// ---------------------------------------------------------------------------
template <bool BF>
__global__ void __launch_bounds__(256) plane_copies_kernel(GeomDev g, const float *__restrict__ vol,
                                                           const double *__restrict__ scale,
                                                           void *__restrict__ basis_out,
                                                           float *__restrict__ Xc, float *__restrict__ Yc,
                                                           const int *__restrict__ stop)
{
    if (stop && *stop) return;
    __shared__ float tile[33][33];
    const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
    const int tid = ty * 32 + tx;
    const int xp0 = blockIdx.x * 32, yp0 = blockIdx.y * 32;  // padded tile origin
    const int zp = blockIdx.z;
    const int z = zp - PAD_A;
    const float sc = scale ? float(*scale) : 1.0f;
    const bool zin = z >= 0 && z < g.nz;
    for (int i = tid; i < 33 * 33; i += 256) {
        const int r = i / 33, c = i - r * 33;
        const int x = xp0 + c - PAD_A, y = yp0 + r - PAD_A;
        float val = 0.0f;
        if (zin && x >= 0 && x < g.nx && y >= 0 && y < g.ny) {
            const size_t idx = (size_t(z) * g.ny + y) * g.nx + x;
            val = vol[idx] * sc;
            if (basis_out && r < 32 && c < 32) {
                if (BF)
                    static_cast<__nv_bfloat16 *>(basis_out)[idx] = __float2bfloat16_rn(val);
                else
                    static_cast<float *>(basis_out)[idx] = val;
            }
        }
        tile[r][c] = val;
    }
    __syncthreads();
    // Yc[zp][y][xp] for y in the grid, xp over the padded row
    for (int r = ty; r < 32; r += 8) {
        const int y = yp0 + r - PAD_A, xp = xp0 + tx;
        if (y >= 0 && y < g.ny && xp < g.pitchY) {
            const size_t o = (size_t(zp) * g.ny + y) * g.pitchY + xp;
            if (BF)
                reinterpret_cast<uint32_t *>(Yc)[o] = pack_bf16x2(tile[r][tx], tile[r][tx + 1]);
            else
                Yc[o] = tile[r][tx];
        }
    }
    // Xc[zp][x][yp] for x in the grid, yp over the padded row
    for (int r = ty; r < 32; r += 8) {
        const int x = xp0 + r - PAD_A, yp = yp0 + tx;
        if (x >= 0 && x < g.nx && yp < g.pitchX) {
            const size_t o = (size_t(zp) * g.nx + x) * g.pitchX + yp;
            if (BF)
                reinterpret_cast<uint32_t *>(Xc)[o] = pack_bf16x2(tile[tx][r], tile[tx + 1][r]);
            else
                Xc[o] = tile[tx][r];
        }
    }
}

cudaError_t launch_plane_copies(const GeomDev &g, const float *vol, const double *scale, void *basis_out,
                                float *Xc, float *Yc, const int *stop, cudaStream_t st)
{
    ProfScope prof(PK_PLANE_COPIES, st);
    dim3 block(32, 8);
    dim3 grid((g.nx + 2 * PAD_A + 31) / 32, (g.ny + 2 * PAD_A + 31) / 32, g.nzp);
    if (g.vol_bf16)
        plane_copies_kernel<true><<<grid, block, 0, st>>>(g, vol, scale, basis_out, Xc, Yc, stop);
    else
        plane_copies_kernel<false><<<grid, block, 0, st>>>(g, vol, scale, basis_out, Xc, Yc, stop);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// y = A x.
//
// One thread walks VR rays of one detector column: same view and u,
// consecutive v.  On a flat detector those rays share d_x, d_y and the cross
// product, hence the dominant axis and the in-plane coordinate f_b(p) of every
// plane; only z differs, f_z(p, v) = cz + gz(v) (p - c_a - S_a/vox), with
// gz(v) = v dzv / d_a.  Per plane the thread interpolates along b once per
// z-row it needs.  Lanes are consecutive u of one detector row
// segment and walk a warp-uniform plane range, so a warp's loads of one plane
// fall in a few consecutive sectors.  Samples outside a ray's own range have
// their row / column clamped into the zero border and add exactly zero.
// ---------------------------------------------------------------------------
constexpr int A_BLOCK = 128;

// What the rays iv0 .. iv0 + VR - 1 of one detector column share.
struct ColumnA {
    bool xdom;            // planes along x
    int Na, Nb, p0, p1;   // planes, cells per plane row, warp-uniform inclusive plane range
    float ca, gb, fbc;    // central plane; in-plane coordinate: slope per plane, value at ca
    float Sv;             // source coordinate along the axis, in voxels
    float gz0, gz_step;   // z slope of the first ray, and its change from ray to ray
    float dxy2, inv_da, dzv;
};

// In-plane direction (d_x, d_y) of detector column iu of view s.
__device__ __forceinline__ float2 column_dir(const GeomDev &g, int s, int iu)
{
    const float4 a = __ldg(reinterpret_cast<const float4 *>(g.viewA + s));   // (dx0, dxu, dy0, dyu)
    const float u = (float(iu) - g.cu) * g.du;
    return make_float2(fmaf(u, a.y, a.x), fmaf(u, a.w, a.z));
}

// The column's rays walked along x (xdom) or y.  All lanes of the warp call
// it; lanes that are not live do not widen the range.
template <int VR>
__device__ __forceinline__ ColumnA column_A(const GeomDev &g, int s, int iv0, int iu, bool live, bool xdom)
{
    const float4 b = __ldg(reinterpret_cast<const float4 *>(g.viewA + s) + 1);   // (dzv, crossu, sx, sy)
    const float2 d = column_dir(g, s, iu);
    const float dx = d.x, dy = d.y;
    const float cross = (float(iu) - g.cu) * g.du * b.y;
    ColumnA c;
    c.xdom = xdom;
    const float da = c.xdom ? dx : dy;
    c.inv_da = 1.0f / da;
    c.Na = c.xdom ? g.nx : g.ny;
    c.Nb = c.xdom ? g.ny : g.nx;
    c.ca = c.xdom ? g.cx : g.cy;
    c.gb = (c.xdom ? dy : dx) * c.inv_da;
    const float cterm = cross * c.inv_da * g.inv_vox;
    c.fbc = c.xdom ? g.cy - cterm : g.cx + cterm;
    c.Sv = (c.xdom ? b.z : b.w) * g.inv_vox;
    c.gz_step = g.dv * b.x * c.inv_da;
    c.gz0 = (float(iv0) - g.cv) * c.gz_step;
    c.dxy2 = fmaf(dx, dx, dy * dy);
    c.dzv = b.x;

    // plane range: the b range of the column met with the planes on which
    // any of its rays is inside the grid in z, then joined over the warp
    int p0 = 0, p1 = c.Na - 1;
    clip_planes(c.fbc, c.gb, -1.0f, float(c.Nb), c.ca, c.Na, p0, p1);
    const float gzl = (float(min(iv0 + VR - 1, g.nv - 1)) - g.cv) * c.gz_step;
    clip_planes_run(fmaf(-c.Sv, c.gz0, g.cz), c.gz0, fmaf(-c.Sv, gzl, g.cz), gzl, -1.0f, float(g.nz), c.ca, c.Na, p0,
                    p1);
    if (!live) {
        p0 = c.Na;
        p1 = -1;
    }
    c.p0 = __reduce_min_sync(0xffffffffu, p0);
    // lanes of one warp can differ in axis (views near 45 degrees); each stays
    // inside its own plane count
    c.p1 = min(__reduce_max_sync(0xffffffffu, p1), c.Na - 1);
    return c;
}

// The same along the column's dominant axis.
template <int VR>
__device__ __forceinline__ ColumnA column_A(const GeomDev &g, int s, int iv0, int iu, bool live)
{
    const float2 d = column_dir(g, s, iu);
    return column_A<VR>(g, s, iv0, iu, live, fabsf(d.x) >= fabsf(d.y));
}

// Step length vox |d| / |d_a| of ray iv of a column.
__device__ __forceinline__ float step_weight(const GeomDev &g, const ColumnA &c, int iv)
{
    const float dz = (float(iv) - g.cv) * g.dv * c.dzv;
    return g.vox * sqrtf(fmaf(dz, dz, c.dxy2)) * fabsf(c.inv_da);
}

// b-interpolated value of one plane row: (1 - wb) V[b0] + wb V[b0+1], read as
// two floats or as one packed bf16 pair
template <bool BF>
__device__ __forceinline__ float row_lerp(const float *p, float wb)
{
    if (BF) {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(p));
        const float v0 = bf16_lo(w), v1 = bf16_hi(w);
        return fmaf(wb, v1 - v0, v0);
    }
    const float v0 = __ldg(p), v1 = __ldg(p + 1);
    return fmaf(wb, v1 - v0, v0);
}

// The walk of detectors with one row (2D scans above all).  A scan has few
// rays (8550 of them for 64 x 64 pixels and 90 views: two warps an SM), so
// what bounds it is one ray's chain of loads.  `split` (1, 2, 4 or 8) of a
// block's 8 warps share the planes of a ray and add their sums, and a thread
// fetches a batch of planes before it adds any: a loop that steps by `split`
// is not unrolled into one by the compiler (1000 x 100 pixels with 90 views:
// 196 us without batches, at any unroll factor).  FLAT: a 2D scan, whose rays
// stay in its one slice.  DIRECT: small images are read where they are (Xc is
// the volume; cells off the grid read as zero, bf16 storage rounds what it
// reads), without copies.
// Registers for 4 blocks an SM: ptxas then keeps a batch's loads together (512 x
// 512, 720 views 190 us without a bound, 162 us for 2 to 4 blocks, 175 for 6).
// Calls with copies, two interpolated rows a plane and one warp a ray against
// this: 512 x 512 with 720 views 325 -> 162 us, 1024 x 1024 with 360 views 622 ->
// 310 us, 1000 x 100 with 90 views 129 -> 28 us (bf16 84 -> 29 us).
template <bool FLAT, bool BF, bool DIRECT>
__global__ void __launch_bounds__(256, 4) joseph_A_row_kernel(GeomDev g, const float *__restrict__ Xc,
                                                           const float *__restrict__ Yc, float *__restrict__ y,
                                                           SinoLayout lay, int split,
                                                           const int *__restrict__ stop)
{
    if (stop && *stop) return;
    // planes a batch (8 of bf16 pairs, whose one load a row is half as long a chain, are slower)
    constexpr int BATCH = BF ? 4 : 8;
    __shared__ float part[8][32];
    const int w = threadIdx.y, wp = w % split;   // the warp's share of its rays' planes
    const int lane_u = (blockIdx.x * (8 / split) + w / split) * 32 + threadIdx.x;
    const int s = blockIdx.z;
    const bool live = lane_u < g.nu;
    const ColumnA c = column_A<1>(g, s, 0, min(lane_u, g.nu - 1), live);
    const int pitch = c.xdom ? g.pitchX : g.pitchY;
    const int zstride = c.Na * pitch;
    // (z = 0, plane 0, b = 0) in the padded copy
    const float *__restrict__ base = (c.xdom ? Xc : Yc) + PAD_A * zstride + PAD_A;
    struct Sample {
        float wb, wz;
        float lo[2], hi[2];   // the two cells of the sample's row and of the row above (bf16 copies: a pair in the first)
    };
    auto fetch = [&](int p) {
        Sample t;
        const float pm = float(p) - c.ca;
        const float fb = fmaf(pm, c.gb, c.fbc);
        const float b0f = floorf(fb);
        const int b0 = min(max(int(b0f), -PAD_A), c.Nb);
        t.wb = fb - b0f;
        if (DIRECT) {
            const float *v = Xc + (c.xdom ? b0 * g.nx + p : p * g.nx + b0);
            t.lo[0] = b0 >= 0 && b0 < c.Nb ? __ldg(v) : 0.0f;
            t.lo[1] = b0 + 1 >= 0 && b0 + 1 < c.Nb ? __ldg(v + (c.xdom ? g.nx : 1)) : 0.0f;
        } else {
            const float *r = base + p * pitch + b0;
            if (!FLAT) {
                const float fz = fmaf(c.gz0, pm - c.Sv, g.cz);
                const float z0f = floorf(fz);
                t.wz = fz - z0f;
                r += min(max(int(z0f), -PAD_A), g.nz) * zstride;
                t.hi[0] = __ldg(r + zstride);
                if (!BF) t.hi[1] = __ldg(r + zstride + 1);
            }
            t.lo[0] = __ldg(r);
            if (!BF) t.lo[1] = __ldg(r + 1);
        }
        return t;
    };
    auto lerp = [&](const float (&v)[2], float wb) {   // (1 - wb) V[b0] + wb V[b0 + 1]
        float v0 = v[0], v1 = v[1];
        if (BF && DIRECT) {
            v0 = __bfloat162float(__float2bfloat16_rn(v0));
            v1 = __bfloat162float(__float2bfloat16_rn(v1));
        } else if (BF) {
            v0 = bf16_lo(__float_as_uint(v[0]));
            v1 = bf16_hi(__float_as_uint(v[0]));
        }
        return fmaf(wb, v1 - v0, v0);
    };
    auto value = [&](const Sample &t) {
        const float lo = lerp(t.lo, t.wb);
        return FLAT ? lo : fmaf(t.wz, lerp(t.hi, t.wb) - lo, lo);
    };
    float acc = 0.0f;
    int p = c.p0 + wp;
    for (; p + (BATCH - 1) * split <= c.p1; p += BATCH * split) {
        Sample t[BATCH];
#pragma unroll
        for (int k = 0; k < BATCH; ++k) t[k] = fetch(p + k * split);
#pragma unroll
        for (int k = 0; k < BATCH; ++k) acc += value(t[k]);
    }
    for (; p <= c.p1; p += split) acc += value(fetch(p));
    part[w][threadIdx.x] = acc;
    __syncthreads();
    if (wp > 0 || !live) return;
    for (int i = 1; i < split; ++i) acc += part[w + i][threadIdx.x];
    store_sino(y, lay, s, 0, lane_u, acc * step_weight(g, c, 0));
}

// ---------------------------------------------------------------------------
// The walk of cone-beam detectors, two neighbouring rays an instruction.
// What bounds the walk is issue slots (76 % busy) and, for its floors and
// float-to-int conversions, the XU pipe (66 %: each takes it 8 cycles a
// warp).  sm_103a's packed FP32 operations (add, sub, fma .f32x2) do the
// arithmetic of two values in one issue slot, at the same rate a value.  The
// floor comes from them too: t = z + 1.5 2^23 rounded down holds floor(z) in
// its low mantissa bits, so a row's address is one wide multiply-add of t's
// bits (the constant's share is folded into the base pointer) and nothing
// runs on the XU pipe.
//
// WINDOW: every ray of a column moves up at most one z row per detector row
// (a_window), so the low row of a sample is the low or the high row of the
// ray before: one new row a ray instead of two.
//
// Needs |z| < 2^22: the copies' grid takes 65531 slices at most, and the clamped
// form bounds z before the floor.  The values and their rounding are those of a
// walk of one ray at a time.
// ---------------------------------------------------------------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2_down(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
constexpr float FLOOR_MAGIC = 12582912.0f;   // 1.5 2^23
constexpr unsigned FLOOR_MAGIC_BITS = 0x4b400000u;

// Registers for 4 resident blocks (128) and a plane loop unrolled by 4: at
// 256^3 4.32 ms (bf16 copies 4.41 ms); unrolled by 2, 4.38 ms (4.57 ms); 5
// blocks unrolled by 2, 4.42 ms; 6 and 8 blocks, 4.80 and 5.51 ms (ptxas then
// keeps fewer row loads in flight); 8 rays a thread, 4.65-4.74 ms.  The plain
// walk over a two-row window took 5.04 ms (bf16 5.41 ms).  On bf16 copies with the
// clamp (a detector taller than the slices) 4 planes at a time need more registers
// than there are: 74 x 143 x 24, 21 views 93 us against 83 by 3 (plain walk 82), 31 x
// 68 x 42, 18 views 52 against 45 (47); by 2, 5 % slower on few views.  Left after it:
// 11.9 instructions a sample (16.8 before), the FMA pipe 52-55 % and issue 55-58
// % busy, the rest latency of the row loads (a third of them miss L1).
constexpr int kAPlaneUnroll = 4;
constexpr int kAPlaneUnrollClampedBF = 3;
constexpr int kAMinBlocks = 4;

template <int VR, bool WINDOW, bool ZCLAMP, bool BF>
__global__ void __launch_bounds__(A_BLOCK, kAMinBlocks)
    joseph_A_pairs_kernel(GeomDev g, const float *__restrict__ Xc, const float *__restrict__ Yc,
                          float *__restrict__ y, SinoLayout lay, const int *__restrict__ stop)
{
    static_assert(VR % 2 == 0, "rays are walked in pairs");
    if (stop && *stop) return;
    const int lane_u = blockIdx.x * 32 + (threadIdx.x & 31);
    const int iv0 = (blockIdx.y * (A_BLOCK / 32) + (threadIdx.x >> 5)) * VR;
    const int s = blockIdx.z;
    const bool live = lane_u < g.nu && iv0 < g.nv;
    const ColumnA c = column_A<VR>(g, s, iv0, min(lane_u, g.nu - 1), live);
    const int pitch = c.xdom ? g.pitchX : g.pitchY;
    const int zstride = c.Na * pitch;
    const unsigned zs4 = unsigned(zstride) * 4u;
    // (z = 0, plane 0, b = 0), less the floor constant's share of a row address
    const char *__restrict__ base = reinterpret_cast<const char *>(c.xdom ? Xc : Yc) +
                                    4 * (ptrdiff_t(PAD_A) * zstride + PAD_A) -
                                    ptrdiff_t(FLOOR_MAGIC_BITS) * ptrdiff_t(zs4);

    f32x2 acc[VR / 2];
#pragma unroll
    for (int i = 0; i < VR / 2; ++i) acc[i] = pack2(0.0f, 0.0f);
    const f32x2 magic = pack2(FLOOR_MAGIC, FLOOR_MAGIC);

#pragma unroll (BF && ZCLAMP ? kAPlaneUnrollClampedBF : kAPlaneUnroll)
    for (int p = c.p0; p <= c.p1; ++p) {
        const float pm = float(p) - c.ca;
        const float fb = fmaf(pm, c.gb, c.fbc);
        const float b0f = floorf(fb);
        const float wb = fb - b0f;
        const int b0 = min(max(int(b0f), -PAD_A), c.Nb);
        const char *rowp = base + 4 * ptrdiff_t(p * pitch + b0);
        const float q = pm - c.Sv;
        const float fz0 = fmaf(c.gz0, q, g.cz);   // z of the first ray
        const float dzr = c.gz_step * q;          // z step from ray to ray
        const f32x2 fz02 = pack2(fz0, fz0), dzr2 = pack2(dzr, dzr), wb2 = pack2(wb, wb);
        float lo_prev = 0.0f, hi_prev = 0.0f, t_prev = 0.0f;
#pragma unroll
        for (int i = 0; i < VR; i += 2) {
            f32x2 fz = fma2(pack2(float(i), float(i + 1)), dzr2, fz02);
            if (ZCLAMP) {   // a sample off the grid takes both rows from the zero border
                float f0, f1;
                unpack2(fz, f0, f1);
                fz = pack2(fminf(fmaxf(f0, -float(PAD_A)), float(g.nz)), fminf(fmaxf(f1, -float(PAD_A)), float(g.nz)));
            }
            const f32x2 t = add2_down(fz, magic);
            const f32x2 wz = sub2(fz, sub2(t, magic));
            float t0, t1;
            unpack2(t, t0, t1);
            unsigned m0 = __float_as_uint(t0), m1 = __float_as_uint(t1);   // floor(z) + FLOOR_MAGIC_BITS
            const int z0 = int(m0 - FLOOR_MAGIC_BITS), z1 = int(m1 - FLOOR_MAGIC_BITS);   // checked builds only
            if (!CT_IN_BOUNDS(g, z0 >= -PAD_A && z0 <= g.nz + PAD_A - 2, BS_A_Z, s, z0)) m0 = FLOOR_MAGIC_BITS - PAD_A;
            if (!CT_IN_BOUNDS(g, z1 >= -PAD_A && z1 <= g.nz + PAD_A - 2, BS_A_Z, s, z1)) m1 = FLOOR_MAGIC_BITS - PAD_A;
            if (WINDOW) {
                const int zp = int(__float_as_uint(t_prev) - FLOOR_MAGIC_BITS);
                (void)CT_IN_BOUNDS(g, z1 == z0 || z1 == z0 + 1, BS_A_WINDOW, s, z1 - z0);
                if (i > 0) (void)CT_IN_BOUNDS(g, z0 == zp || z0 == zp + 1, BS_A_WINDOW, s, z0 - zp);
                (void)zp;
            }
            const float *r0 = reinterpret_cast<const float *>(rowp + (unsigned long long)m0 * zs4);
            const float *r1 = reinterpret_cast<const float *>(rowp + (unsigned long long)m1 * zs4);
            // high rows of the two samples
            f32x2 hi;
            if (BF) {
                const uint32_t w0 = __ldg(reinterpret_cast<const uint32_t *>(r0 + zstride));
                const uint32_t w1 = __ldg(reinterpret_cast<const uint32_t *>(r1 + zstride));
                const f32x2 v0 = pack2(bf16_lo(w0), bf16_lo(w1)), v1 = pack2(bf16_hi(w0), bf16_hi(w1));
                hi = fma2(wb2, sub2(v1, v0), v0);
            } else {
                const f32x2 v0 = pack2(__ldg(r0 + zstride), __ldg(r1 + zstride));
                const f32x2 v1 = pack2(__ldg(r0 + zstride + 1), __ldg(r1 + zstride + 1));
                hi = fma2(wb2, sub2(v1, v0), v0);
            }
            float h0, h1, lo0, lo1;
            unpack2(hi, h0, h1);
            if (WINDOW) {
                lo0 = i == 0 ? row_lerp<BF>(r0, wb) : (t0 == t_prev ? lo_prev : hi_prev);
                lo1 = t1 == t0 ? lo0 : h0;
            } else {
                lo0 = row_lerp<BF>(r0, wb);
                lo1 = row_lerp<BF>(r1, wb);
            }
            const f32x2 lo = pack2(lo0, lo1);
            acc[i / 2] = add2(acc[i / 2], fma2(wz, sub2(hi, lo), lo));
            lo_prev = lo1;
            hi_prev = h1;
            t_prev = t1;
        }
    }
    if (!live) return;
#pragma unroll
    for (int i = 0; i < VR; i += 2) {
        float a0, a1;
        unpack2(acc[i / 2], a0, a1);
        if (iv0 + i < g.nv) store_sino(y, lay, s, iv0 + i, lane_u, a0 * step_weight(g, c, iv0 + i));
        if (iv0 + i + 1 < g.nv) store_sino(y, lay, s, iv0 + i + 1, lane_u, a1 * step_weight(g, c, iv0 + i + 1));
    }
}

// Warps that share the planes of a one-row detector's rays: as many as keep the
// grid within 32 warps an SM, and on to 128, about four waves, while a share is 32
// planes or more: rays leave the image after different numbers of planes, and more
// and shorter shares even out (9 x 1000 pixels, 90 views: 114 us with 32 warps an
// SM, 36 us with 96; 512 x 512, 360 views 99 us with 96, 90 us with 128; the
// transpose of 1024 x 1024, 90 views 320 us with 32, 232 us with 96).
static int row_split(const GeomDev &g, int limit)
{
    const size_t warps = size_t((g.nu + 31) / 32) * g.n_views, sms = num_sms();
    int split = 1;
    while (split < limit && (warps * split * 2 <= sms * 32 ||
                             (warps * split * 2 <= sms * 128 && std::max(g.nx, g.ny) >= split * 2 * 32)))
        split *= 2;
    return split;
}

template <bool FLAT, bool BF, bool DIRECT>
static void launch_joseph_A_row(const GeomDev &g, const float *Xc, const float *Yc, float *y, SinoLayout lay,
                                const int *stop, cudaStream_t st)
{
    const int tiles = (g.nu + 31) / 32, split = row_split(g, 8);
    const dim3 block(32, 8), grid((tiles * split + 7) / 8, 1, g.n_views);
    joseph_A_row_kernel<FLAT, BF, DIRECT><<<grid, block, 0, st>>>(g, Xc, Yc, y, lay, split, stop);
}

template <bool BF>
static void launch_joseph_A_t(const GeomDev &g, const float *Xc, const float *Yc, float *y, SinoLayout lay,
                              const int *stop, cudaStream_t st)
{
    constexpr int WPB = A_BLOCK / 32, VR = A_VR;
    if (g.nv == 1) {
        if (g.kind == CT_PARALLEL_2D)
            launch_joseph_A_row<true, BF, false>(g, Xc, Yc, y, lay, stop, st);
        else
            launch_joseph_A_row<false, BF, false>(g, Xc, Yc, y, lay, stop, st);
        return;
    }
    dim3 grid((g.nu + 31) / 32, (g.nv + WPB * VR - 1) / (WPB * VR), g.n_views);
    if (g.a_window && g.a_zsafe)
        joseph_A_pairs_kernel<VR, true, false, BF><<<grid, A_BLOCK, 0, st>>>(g, Xc, Yc, y, lay, stop);
    else if (g.a_window)
        joseph_A_pairs_kernel<VR, true, true, BF><<<grid, A_BLOCK, 0, st>>>(g, Xc, Yc, y, lay, stop);
    else
        joseph_A_pairs_kernel<VR, false, true, BF><<<grid, A_BLOCK, 0, st>>>(g, Xc, Yc, y, lay, stop);
}

cudaError_t launch_project_A(const GeomDev &g, const float *Xc, const float *Yc, float *y,
                            SinoLayout lay, const int *stop, cudaStream_t st)
{
    ProfScope prof(PK_JOSEPH_A, st);
    if (g.siddon) return launch_siddon_A(g, Xc, Yc, y, lay, stop, st);
    if (g.vol_bf16)
        launch_joseph_A_t<true>(g, Xc, Yc, y, lay, stop, st);
    else
        launch_joseph_A_t<false>(g, Xc, Yc, y, lay, stop, st);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// x = A^T y, the exact transpose of the projector above: the same column
// walk (A_VR rays of one detector column per thread, warp-uniform plane
// range, the same sample positions and bilinear weights), scattering
// instead of gathering.  Contributions go with FP32 reductions into
// plane-major accumulators laid out like the projector's copies
// (X[zp][x][yp] for x-dominant rays, Y[zp][y][xp]), so the lanes of a
// warp (consecutive u) add to neighbouring words of one row.  Within a
// thread the rays of a column add to a two-row window per plane, as the
// projector reads one: contributions to the same row are summed in
// registers and a row is flushed when the window moves past it.
//
// A flush adds to two neighbouring cells, b0 and b0 + 1: as two requests, or
// (PAIRS) as one to one of an orientation's two accumulators (add_pair; the
// rule and both sides' times stand at at_scatter).  Samples on the zero border
// add to the border or are skipped (they are zero entries of A); a last pass
// adds the accumulators up.  Small scans were bound by a warp's chain of planes,
// which `p_split` warps share: 44^3 0.121 -> 0.039 ms, 64 x 64 30 -> 19 us.
// ---------------------------------------------------------------------------
static size_t at_floats(const GeomDev &g, bool x)
{
    return pair_acc_floats(size_t(g.nzp) * (x ? size_t(g.nx) * g.pitchX : size_t(g.ny) * g.pitchY));
}

size_t at_scratch_floats(const GeomDev &g, Scatter how)
{
    return how == SCATTER_DIRECT ? 0 : (how == SCATTER_PAIRS ? 2 : 1) * (at_floats(g, true) + at_floats(g, false));
}

Scatter at_scatter_lean(const GeomDev &g) { return g.siddon ? SCATTER_DIRECT : SCATTER_SINGLE; }

// What each way costs beside its scattered adds: zeroing the accumulators and
// adding them up.  Measured (dense data; one way and the other):
// - Pairs halve the requests and double what the adds touch.  While the four
//   accumulators fit L2 (129 MB), they win: 128^3, 128 views 0.89 against 1.10 ms,
//   192^3 3.4 against 4.0 ms.  Past it single accumulators do: 256^3, 358 views
//   11.7 against 12.2 ms, 320^3 28 against 51 ms, 512^3, 64 views 25 against 40 ms.
// - Nor do they win where few rays cross a voxel (100^3 with one view 31 against
//   33 us), or on large one-row scans (1024 x 1024, 128 views or more, 1 % either
//   way, but 10 views 47 against 52 us).
// - The line-intersection transpose straight into the volume saves two launches
//   (16^3 9 against 15 us; not where hundreds of rays cross each voxel: 21 x 46 x
//   3, 180 views 43 against 29 us), wins where few rays cross a voxel of a tall
//   volume (214 x 131 x 296, 3 views, 82 against 105 us), and where dozens of
//   columns fall on a voxel (44^3, 1320 columns 18 against 21 ms).
Scatter at_scatter(const GeomDev &g)
{
    const double planes = double(g.n_views) * g.nu * g.nv * std::max(g.nx, g.ny);   // of all rays
    const double per_voxel = planes / (double(g.nx) * g.ny * g.nz);
    if (g.siddon)
        return (planes < 2.5e6 && per_voxel < 200.0) || (planes < 6e6 && per_voxel < 25.0) ||
                       (per_voxel < 10.0 && g.nv < g.nz) || g.nu > 20 * std::max(g.nx, g.ny)
                   ? SCATTER_DIRECT : SCATTER_SINGLE;
    const double bytes = 4.0 * at_scratch_floats(g, SCATTER_PAIRS);
    if (g.nv == 1) return bytes <= 50e6 ? SCATTER_PAIRS : SCATTER_SINGLE;
    return bytes <= 128e6 && (per_voxel >= 10.0 || bytes <= 12e6) ? SCATTER_PAIRS : SCATTER_SINGLE;
}

template <int VR, bool WINDOW, bool ZCLAMP, bool PAIRS>
__global__ void __launch_bounds__(A_BLOCK) joseph_At_kernel(GeomDev g, const float *__restrict__ y,
                                                            float *__restrict__ X, size_t x_odd,
                                                            float *__restrict__ Y, size_t y_odd, int v_tiles,
                                                            int p_split, const int *__restrict__ stop)
{
    if (stop && *stop) return;
    const int lane_u = blockIdx.x * 32 + (threadIdx.x & 31);
    const int job = blockIdx.y * (A_BLOCK / 32) + (threadIdx.x >> 5);   // (tile of VR rows, share of the planes)
    const int iv0 = (job / p_split) * VR, share = job % p_split;
    const int s = blockIdx.z;
    const bool live = lane_u < g.nu && job < v_tiles * p_split;
    const int iu = min(lane_u, g.nu - 1);
    float2 d = column_dir(g, s, iu);
    ColumnA c = column_A<VR>(g, s, iv0, iu, live, fabsf(d.x) >= fabsf(d.y));

    // each ray's value times its step weight (zero past nv and for idle lanes)
    float val[VR];
    bool any = false;
#pragma unroll
    for (int i = 0; i < VR; ++i) {
        val[i] = 0.0f;
        if (live && iv0 + i < g.nv) val[i] = y[(size_t(s) * g.nv + iv0 + i) * g.nu + iu] * step_weight(g, c, iv0 + i);
        any = any || val[i] != 0.0f;
    }
    if (!__any_sync(0xffffffffu, any)) return;
    // lanes with nothing to add do not widen the warp's range
    c = column_A<VR>(g, s, iv0, iu, any, c.xdom);
    if (!any) return;   // after the warp-wide reductions
    const int each = (max(c.p1 - c.p0 + 1, 0) + p_split - 1) / p_split;
    const int pa = c.p0 + share * each, pb = min(pa + each - 1, c.p1);

    float *__restrict__ base = c.xdom ? X : Y;
    const size_t odd = c.xdom ? x_odd : y_odd;
    const int pitch = c.xdom ? g.pitchX : g.pitchY;
    const unsigned zstride = unsigned(c.Na) * pitch;
    const int zmax = g.nz;

    for (int p = pa; p <= pb; ++p) {
        const float pm = float(p) - c.ca;
        const float fb = fmaf(pm, c.gb, c.fbc);
        const float b0f = floorf(fb);
        const float wb = fb - b0f;
        const int b0 = min(max(int(b0f), -PAD_A), c.Nb);
        if (b0 < -1 || b0 >= c.Nb) continue;   // both cells on the border
        const unsigned row0 = PAD_A * zstride + unsigned(p) * pitch + b0 + PAD_A;   // (z = 0, plane p, b0)
        const float q = pm - c.Sv;
        const float fz0 = fmaf(c.gz0, q, g.cz);
        const float dzr = c.gz_step * q;
        // adds a row's summed contribution r to cells b0, b0 + 1 of grid row z
        auto flush = [&](int z, float r) {
            if (r == 0.0f || z < 0 || z >= zmax) return;
            const unsigned e = row0 + unsigned(z) * zstride;
            if (PAIRS) {
                add_pair(base, odd, e, r * (1.0f - wb), r * wb);
            } else {
                if (b0 >= 0) atomicAdd(base + e, r * (1.0f - wb));
                if (b0 + 1 < c.Nb) atomicAdd(base + e + 1, r * wb);
            }
        };
        int zc = 0;
        float acc_lo = 0.0f, acc_hi = 0.0f;   // rows zc and zc + 1
#pragma unroll
        for (int i = 0; i < VR; ++i) {
            const float fz = fmaf(float(i), dzr, fz0);
            const float z0f = floorf(fz);
            const float wz = fz - z0f;
            const int z0 = ZCLAMP ? min(max(int(z0f), -PAD_A), zmax) : int(z0f);
            const float c_lo = val[i] * (1.0f - wz), c_hi = val[i] * wz;
            if (!WINDOW) {
                flush(z0, c_lo);
                flush(z0 + 1, c_hi);
            } else if (i == 0) {
                zc = z0;
                acc_lo = c_lo;
                acc_hi = c_hi;
            } else if (z0 == zc) {
                acc_lo += c_lo;
                acc_hi += c_hi;
            } else {   // z0 == zc + 1: row zc is complete
                (void)CT_IN_BOUNDS(g, z0 == zc + 1, BS_AT_WINDOW, s, z0 - zc);
                flush(zc, acc_lo);
                zc = z0;
                acc_lo = acc_hi + c_lo;
                acc_hi = c_hi;
            }
        }
        if (WINDOW) {
            flush(zc, acc_lo);
            flush(zc + 1, acc_hi);
        }
    }
}

// x[z][y][x] = X[z][x][y] + Y[z][y][x] over the grid (padded indices), each from its two copies (PAIRS) or its one
template <bool PAIRS>
__global__ void __launch_bounds__(256) unplane_kernel(GeomDev g, const float *__restrict__ X, size_t x_odd,
                                                      const float *__restrict__ Y, size_t y_odd,
                                                      float *__restrict__ x, const int *__restrict__ stop)
{
    if (stop && *stop) return;
    __shared__ float tile[32][33];
    const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (int z = blockIdx.z; z < g.nz; z += gridDim.z) {
        const size_t zp = size_t(z) + PAD_A;
        __syncthreads();
        // tile[xl][yl] = X[zp][x0 + xl][y0 + yl + PAD_A], read along y
        for (int r = ty; r < 32; r += 8) {
            const int xx = x0 + r, yy = y0 + tx;
            const size_t e = (zp * g.nx + xx) * g.pitchX + yy + PAD_A;
            tile[r][tx] = (xx < g.nx && yy < g.ny) ? (PAIRS ? X[e] + X[x_odd + e + 1] : X[e]) : 0.0f;
        }
        __syncthreads();
        for (int r = ty; r < 32; r += 8) {
            const int yy = y0 + r, xx = x0 + tx;
            const size_t e = (zp * g.ny + yy) * g.pitchY + xx + PAD_A;
            if (xx < g.nx && yy < g.ny)
                x[(size_t(z) * g.ny + yy) * g.nx + xx] = tile[tx][r] + (PAIRS ? Y[e] + Y[y_odd + e + 1] : Y[e]);
        }
    }
}

template <bool PAIRS>
static void launch_joseph_At(const GeomDev &g, const float *y, float *X, size_t x_odd, float *Y, size_t y_odd,
                             const int *stop, cudaStream_t st)
{
    constexpr int WPB = A_BLOCK / 32;
    const int u_tiles = (g.nu + 31) / 32, v_tiles = g.nv == 1 ? 1 : (g.nv + A_VR - 1) / A_VR;
    // small scans: warps share a tile's planes until the grid has 32 warps an SM
    const size_t most = size_t(num_sms()) * 32;
    int split = 1;
    while (split < 16 && size_t(u_tiles) * v_tiles * g.n_views * split * 2 <= most) split *= 2;
    if (g.nv == 1) split = row_split(g, 16);
    const dim3 grid(u_tiles, (v_tiles * split + WPB - 1) / WPB, g.n_views);
    if (g.nv == 1)
        joseph_At_kernel<1, false, true, PAIRS><<<grid, A_BLOCK, 0, st>>>(g, y, X, x_odd, Y, y_odd, v_tiles, split, stop);
    else if (g.a_window && g.a_zsafe)
        joseph_At_kernel<A_VR, true, false, PAIRS><<<grid, A_BLOCK, 0, st>>>(g, y, X, x_odd, Y, y_odd, v_tiles, split, stop);
    else if (g.a_window)
        joseph_At_kernel<A_VR, true, true, PAIRS><<<grid, A_BLOCK, 0, st>>>(g, y, X, x_odd, Y, y_odd, v_tiles, split, stop);
    else
        joseph_At_kernel<A_VR, false, true, PAIRS><<<grid, A_BLOCK, 0, st>>>(g, y, X, x_odd, Y, y_odd, v_tiles, split, stop);
}

cudaError_t launch_project_At(const GeomDev &g, Scatter how, const float *y, float *x, float *acc, const int *stop,
                             cudaStream_t st)
{
    ProfScope prof(PK_JOSEPH_AT, st);
    const bool direct = how == SCATTER_DIRECT, pairs = how == SCATTER_PAIRS;
    const size_t x_odd = at_floats(g, true), y_odd = at_floats(g, false);
    float *X = direct ? x : acc, *Y = direct ? nullptr : acc + (pairs ? 2 : 1) * x_odd;
    const size_t zeroed = direct ? size_t(g.nx) * g.ny * g.nz : at_scratch_floats(g, how);
    cudaError_t e = cudaMemsetAsync(X, 0, sizeof(float) * zeroed, st);
    if (e != cudaSuccess) return e;
    if (g.siddon)
        e = launch_siddon_At(g, y, X, Y, stop, st);
    else if (pairs)
        launch_joseph_At<true>(g, y, X, x_odd, Y, y_odd, stop, st);
    else
        launch_joseph_At<false>(g, y, X, x_odd, Y, y_odd, stop, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess || direct) return e;
    const dim3 ublock(32, 8), ugrid((g.nx + 31) / 32, (g.ny + 31) / 32, std::min(g.nz, 65535));
    if (pairs)
        unplane_kernel<true><<<ugrid, ublock, 0, st>>>(g, X, x_odd, Y, y_odd, x, stop);
    else
        unplane_kernel<false><<<ugrid, ublock, 0, st>>>(g, X, x_odd, Y, y_odd, x, stop);
    return cudaGetLastError();
}

}  // namespace ct

using namespace ct;

// 2D images that are projected without copies: one launch instead of two.  Small
// ones (96 x 96 pixels), while a call is short: a sample costs more than one
// from the copies, whose lanes always read along a row, and most where rows are
// multiples of 64 bytes, since a column of the image then lies in few of L1's
// sets.  Samples (rays times planes) at which the two cross: 64 x 64 4e6, 96 x 96
// between 1.2e6 and 5e6, 128 x 72 between 2e6 and 7e6, against 72 x 128 over 3e7,
// 60 x 150 over 4e7, 9 x 1000 1e8.  Direct and with copies: 64 x 64 pixels, 90
// views 7.2 and 11.0 us; 96 x 96, 90 views 10.1 and 12.4; 96 x 96, 1500 views 82 and 36.
static bool reads_in_place(const GeomDev &g)
{
    const double samples = double(g.n_views) * g.nu * std::max(g.nx, g.ny);
    return g.kind == CT_PARALLEL_2D && !g.siddon && size_t(g.nx) * g.ny <= 96 * 96 &&
           samples <= (g.nx % 16 ? 3e7 : 4e6);
}

extern "C" ct_status ct_project_A(const ct_geom *geom, const float *x_dev, float *y_dev, void *stream)
{
    NvtxRange call_range("ct_project_A");
    if (!geom || !x_dev || !y_dev) return set_error(CT_EINVAL, "ct_project_A: NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const GeomDev &g = geom->g;
    if (reads_in_place(g)) {
        ProfScope prof(PK_JOSEPH_A, st);
        if (g.vol_bf16)
            launch_joseph_A_row<true, true, true>(g, x_dev, x_dev, y_dev, plain_layout(g), nullptr, st);
        else
            launch_joseph_A_row<true, false, true>(g, x_dev, x_dev, y_dev, plain_layout(g), nullptr, st);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? CT_OK : cuda_error(e, "ct_project_A launch");
    }
    Arena ar;
    ct_status rc = arena_open(ar, plane_copies_bytes(g), nullptr, 0, st);
    if (rc != CT_OK) return rc;
    float *Xc = ar.take<float>(size_t(g.nzp) * g.nx * g.pitchX);
    float *Yc = ar.take<float>(size_t(g.nzp) * g.ny * g.pitchY);
    cudaError_t e = launch_plane_copies(g, x_dev, nullptr, nullptr, Xc, Yc, nullptr, st);
    if (e == cudaSuccess) e = launch_project_A(g, Xc, Yc, y_dev, plain_layout(g), nullptr, st);
    arena_close(ar);
    if (e != cudaSuccess) return cuda_error(e, "ct_project_A launch");
    return CT_OK;
}

extern "C" ct_status ct_adjoint_At(const ct_geom *geom, const float *y_dev, float *x_dev, void *stream)
{
    NvtxRange call_range("ct_adjoint_At");
    if (!geom || !y_dev || !x_dev) return set_error(CT_EINVAL, "ct_adjoint_At: NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const GeomDev &g = geom->g;
    Arena ar;
    Scatter how = at_scatter(g);
    ct_status rc = arena_open(ar, Arena::align(at_scratch_floats(g, how) * sizeof(float)), nullptr, 0, st);
    if (rc == CT_ENOMEM && how != at_scatter_lean(g)) {   // short of memory: the way that takes less
        how = at_scatter_lean(g);
        rc = arena_open(ar, Arena::align(at_scratch_floats(g, how) * sizeof(float)), nullptr, 0, st);
    }
    if (rc != CT_OK) return rc;
    cudaError_t e = launch_project_At(g, how, y_dev, x_dev, ar.take<float>(at_scratch_floats(g, how)), nullptr, st);
    arena_close(ar);
    if (e != cudaSuccess) return cuda_error(e, "ct_adjoint_At launch");
    return CT_OK;
}

// ---------------------------------------------------------------------------
// Projector without allocation: the plane copies live in a fixed device
// array instead of stream-ordered scratch (see ct_project_A_noalloc in ct.h).
// ---------------------------------------------------------------------------
namespace {
constexpr size_t kNoallocFloats = CT_NOALLOC_SCRATCH_BYTES / sizeof(float);
__device__ __align__(256) float g_noalloc_scratch[kNoallocFloats];

constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mu;
float *g_noalloc_addr[kNoallocMaxDevices] = {};  // device address of the array, per device
}  // namespace

extern "C" ct_status ct_project_A_noalloc(const ct_geom *geom, const float *x_dev, float *y_dev,
                                          void *stream)
{
    if (!geom || !x_dev || !y_dev) return set_error(CT_EINVAL, "ct_project_A_noalloc: NULL argument");
    const GeomDev &g = geom->g;
    const size_t xc_bytes = Arena::align(size_t(g.nzp) * g.nx * g.pitchX * sizeof(float));
    const size_t yc_bytes = Arena::align(size_t(g.nzp) * g.ny * g.pitchY * sizeof(float));
    if (xc_bytes + yc_bytes > size_t(CT_NOALLOC_SCRATCH_BYTES))
        return set_error(CT_EINVAL,
                         "ct_project_A_noalloc: this volume needs %zu bytes of projector scratch, more than "
                         "the %zu-byte fixed scratch; use ct_project_A",
                         xc_bytes + yc_bytes, size_t(CT_NOALLOC_SCRATCH_BYTES));
    int dev = -1;
    CT_CUDA(cudaGetDevice(&dev));
    if (dev != geom->device)
        return set_error(CT_EINVAL, "ct_project_A_noalloc: the geometry lives on device %d but device %d is current",
                         geom->device, dev);
    if (dev < 0 || dev >= kNoallocMaxDevices)
        return set_error(CT_EINVAL, "ct_project_A_noalloc: device index %d is out of range", dev);
    float *base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(projector scratch)");
            g_noalloc_addr[dev] = static_cast<float *>(p);
        }
        base = g_noalloc_addr[dev];
    }
    float *Xc = base;
    float *Yc = base + xc_bytes / sizeof(float);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = launch_plane_copies(g, x_dev, nullptr, nullptr, Xc, Yc, nullptr, st);
    if (e == cudaSuccess) e = launch_project_A(g, Xc, Yc, y_dev, plain_layout(g), nullptr, st);
    if (e != cudaSuccess) return cuda_error(e, "ct_project_A_noalloc launch");
    return CT_OK;
}
