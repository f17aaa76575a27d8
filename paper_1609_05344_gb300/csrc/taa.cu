// taa.cu -- reprojection motion and the temporal anti-aliasing resolve
// (Sec. 3.2: jittered frames are accumulated by Playdead-style TAA).
//
// Streaming passes over 32-pixel-wide tiles of 32x8 threads, several vertically
// adjacent pixels a thread, 16-byte RGBA loads/stores (8-byte for FP16 history).
// The current frame's 3x3 neighbourhoods come from a shared-memory tile, the 2x2
// history footprint through L1; each pixel's own current value, history, motion
// and output are the compulsory traffic.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <mutex>

#include "common.cuh"

namespace cloudvol {

struct MotionParams {
    // current camera, camera-space ray slopes: a = a0 + x ax, b = b0 + y by;
    // the ray is (a, b, 1) in (right, up, forward) coordinates
    float a0, ax, b0, by;
    float rz, uz, fz;      // world z of the current right, up, forward
    float zlo, zhi, tmax;  // slab_lo - o_z, slab_hi - o_z, far clip
    // previous camera: q = dlt + lambda (I + G) (a, b, 1), G = R' R^T - I,
    // dlt = R' (o - o'); projections compared as differences of slopes
    float G[3][3], dlt[3];
    float kx, ky, kx1, ky1;  // aT'/aT, T'/T, and the same minus 1
    float sx, sy;            // W / (2 aT'), H / (2 T')
    int width, height;
    // double-float restatement of the world-space ray for near-tie layer-entry
    // decisions: v(x, y) = v00 + x vx + y vy (vx, vy split so that x * hi is
    // exact), slab_lo - o_z, slab_hi - o_z and the far clip
    float v00h[3], v00l[3], vxh[3], vxl[3], vyh[3], vyl[3];
    float zlo_h, zlo_l, zhi_h, zhi_l, tmax_h, tmax_l;
    unsigned *check;  // status word of the checked build, else nullptr
};

// Reprojection depth parameter lambda (t / |v|) of the layer entry point, or
// of the far clip when the ray does not enter the layer ahead of the camera,
// in double-float FP32 (about 48 bits, the layer clip of the raymarch): for the
// rays whose entry FP32 cannot decide.
__device__ __noinline__ float entry_lambda_exact(const MotionParams &p, int x, int y) {
    const float xf = (float)x, yf = (float)y;
    df r[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        df a = {p.v00h[k], p.v00l[k] + fmaf(xf, p.vxl[k], yf * p.vyl[k])};
        a = df_addf(a, xf * p.vxh[k]);  // exact products
        r[k] = df_addf(a, yf * p.vyh[k]);
    }
    const df n2 = df_add(df_add(df_mul(r[0], r[0]), df_mul(r[1], r[1])), df_mul(r[2], r[2]));
    const df rn = df_rsqrt(n2);  // 1 / |v|
    const df lam_max = df_mul({p.tmax_h, p.tmax_l}, rn);
    if (fabsf(r[2].hi) * rn.hi < 1e-8f) return lam_max.hi;  // horizontal ray
    const df inv = df_recip(r[2]);
    const df ll = df_mul({p.zlo_h, p.zlo_l}, inv), lh = df_mul({p.zhi_h, p.zhi_l}, inv);
    const df zero = {0.0f, 0.0f};
    const df l0 = df_max(df_min(ll, lh), zero), l1 = df_min(df_max(ll, lh), lam_max);
    return (df_gt(l1, l0) && df_gt(l0, zero)) ? l0.hi : lam_max.hi;
}

// Motion of one pixel.  The motion is a small difference of nearly equal
// pixel positions; it is computed directly as a difference of camera-space
// slopes (no large terms cancel), so FP32 keeps it to ~1e-6 pixel.  Split in
// three parts so that a thread can share the column terms between pixels and
// interleave the arithmetic of several pixels: the column terms, the depth
// parameter of the layer entry (FP32, with a flag for the near ties that the
// double-float restatement decides), and the projection into the previous
// camera.
//
// Two rows of a column at a time, on packed FP32x2 operations (the arithmetic is
// what bounds the motion: 118 instructions a pixel one at a time).
struct MotionCol {
    float a, n2x, vzx, gx0, gx1, gx2, akx, nx0;
};
__device__ __forceinline__ MotionCol motion_col(const MotionParams &p, int x) {
    MotionCol c;
    c.a = fmaf((float)x, p.ax, p.a0);
    c.n2x = fmaf(c.a, c.a, 1.0f);
    c.vzx = fmaf(c.a, p.rz, p.fz);
    c.gx0 = fmaf(p.G[0][0], c.a, p.G[0][2]);
    c.gx1 = fmaf(p.G[1][0], c.a, p.G[1][2]);
    c.gx2 = fmaf(p.G[2][0], c.a, p.G[2][2]);
    c.akx = c.a * p.kx;
    c.nx0 = fmaf(c.akx, p.dlt[2], -p.dlt[0]);
    return c;
}
// Slopes of rows y and y + 1.
__device__ __forceinline__ float2 motion_rows(const MotionParams &p, int y) {
    return make_float2(fmaf((float)y, p.by, p.b0), fmaf((float)(y + 1), p.by, p.b0));
}
// Depth parameter lambda (t / |v|) of the layer entry, or of the far clip;
// *exact is set when FP32 cannot call the entry (the caller then takes
// entry_lambda_exact).
__device__ __forceinline__ float motion_entry(const MotionParams &p, float lmax, float ll, float lh,
                                              bool horizontal, bool *exact) {
    const float l0 = fmaxf(fminf(ll, lh), 0.0f), l1 = fminf(fmaxf(ll, lh), lmax);
    *exact = !horizontal && fabsf(l1 - l0) <= 1e-5f * fmaxf(l1, l0);  // too close to call in FP32
    return !horizontal && l1 > l0 && l0 > 0.0f ? l0 : lmax;
}
// Both rows' lambda; b: the rows' slopes.
__device__ __forceinline__ float2 motion_lambda(const MotionParams &p, const MotionCol &c, float2 b,
                                                bool *exact0, bool *exact1) {
    const float2 n2 = __ffma2_rn(b, b, both(c.n2x));
    const float2 vz = __ffma2_rn(b, both(p.uz), both(c.vzx));
    // divisions by hardware reciprocals (relative error ~1e-7, far below the
    // 1e-5 margin of the near-tie test and the motion's own accuracy) of normal
    // numbers, without the scaling of subnormal ones
    const float2 lmax = __fmul2_rn(both(p.tmax), make_float2(rsqrt_norm(n2.x), rsqrt_norm(n2.y)));
    const float2 vz2 = __fmul2_rn(vz, vz), lim = __fmul2_rn(n2, both(1e-16f));
    const float2 ivz = make_float2(rcp_norm(vz.x), rcp_norm(vz.y));
    const float2 ll = __fmul2_rn(both(p.zlo), ivz), lh = __fmul2_rn(both(p.zhi), ivz);
    // horizontal: |d_z| < 1e-8
    return make_float2(motion_entry(p, lmax.x, ll.x, lh.x, !(vz2.x >= lim.x), exact0),
                       motion_entry(p, lmax.y, ll.y, lh.y, !(vz2.y >= lim.y), exact1));
}
// Both rows' motion: (x, y) of row y, then of row y + 1.
__device__ __forceinline__ float4 motion_project(const MotionParams &p, const MotionCol &c, float2 b,
                                                 float2 lam) {
    const float2 g0 = __ffma2_rn(both(p.G[0][1]), b, both(c.gx0));
    const float2 g1 = __ffma2_rn(both(p.G[1][1]), b, both(c.gx1));
    const float2 g2 = __ffma2_rn(both(p.G[2][1]), b, both(c.gx2));
    const float2 qz = __ffma2_rn(lam, __fadd2_rn(both(1.0f), g2), both(p.dlt[2]));
    // a kx qz - qx and qy - b ky qz, expanded so the O(lambda) terms cancel exactly
    const float2 nbky = __fmul2_rn(b, both(-p.ky));
    const float2 nx = __ffma2_rn(lam, __ffma2_rn(both(c.a), both(p.kx1), __ffma2_rn(both(c.akx), g2, neg2(g0))),
                                 both(c.nx0));
    const float2 ny = __ffma2_rn(lam, __ffma2_rn(b, both(-p.ky1), __ffma2_rn(nbky, g2, g1)),
                                 __ffma2_rn(nbky, both(p.dlt[2]), both(p.dlt[1])));
    const float2 iq = make_float2(rcp_norm(qz.x), rcp_norm(qz.y));
    const float2 mx = __fmul2_rn(__fmul2_rn(both(p.sx), nx), iq);
    const float2 my = __fmul2_rn(__fmul2_rn(both(p.sy), ny), iq);
    const bool on0 = qz.x > 0.0f, on1 = qz.y > 0.0f;  // not behind the previous camera
    return make_float4(on0 ? mx.x : 1e9f, on0 ? my.x : 1e9f, on1 ? mx.y : 1e9f, on1 ? my.y : 1e9f);
}
// Motions of kRows (even) vertically adjacent pixels of column x from row y0 on.
template <int kRows>
__device__ __forceinline__ void motion_column(const MotionParams &p, int x, int y0, float2 (&m)[kRows]) {
    const MotionCol col = motion_col(p, x);
    float2 b[kRows / 2], lam[kRows / 2];
    bool ex[kRows], any = false;
#pragma unroll
    for (int r = 0; r < kRows; r += 2) {
        b[r / 2] = motion_rows(p, y0 + r);
        lam[r / 2] = motion_lambda(p, col, b[r / 2], &ex[r], &ex[r + 1]);
        any = any || ex[r] || ex[r + 1];
    }
    if (any) {  // rare
#pragma unroll
        for (int r = 0; r < kRows; ++r)
            if (ex[r]) (r & 1 ? lam[r / 2].y : lam[r / 2].x) = entry_lambda_exact(p, x, y0 + r);
    }
#pragma unroll
    for (int r = 0; r < kRows; r += 2) {
        const float4 q = motion_project(p, col, b[r / 2], lam[r / 2]);
        m[r] = make_float2(q.x, q.y);
        m[r + 1] = make_float2(q.z, q.w);
    }
}

// Motions of kMotionRows vertically adjacent pixels of one column per thread:
// the column terms are computed once and the rows' dependent chains (a
// reciprocal square root and two reciprocals in series each) overlap; stores
// stay coalesced along x.  Four rows (1920x1080 5.8 us), or two where tiles of four
// would leave SMs without a CTA (128x128: 1.6 us, with four 1.85).
template <int kMotionRows>
__global__ void __launch_bounds__(256) motion_kernel(const __grid_constant__ MotionParams p,
                                                     float2 *__restrict__ motion) {
    const int x = blockIdx.x * 32 + threadIdx.x;
    const int y0 = (blockIdx.y * 8 + threadIdx.y) * kMotionRows;
    if (x >= p.width || y0 >= p.height) return;
    float2 m[kMotionRows];
    motion_column<kMotionRows>(p, x, y0, m);
#pragma unroll
    for (int r = 0; r < kMotionRows; ++r)
        if (y0 + r < p.height) motion[(size_t)(y0 + r) * p.width + x] = m[r];
}

__device__ __forceinline__ float4 load_hist(const float4 *h, size_t i) { return __ldg(h + i); }
__device__ __forceinline__ float4 load_hist(const uint2 *h, size_t i) {
    const uint2 r = __ldg(h + i);
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&r.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&r.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store_hist(float4 *h, size_t i, float4 v) { h[i] = v; }
__device__ __forceinline__ void store_hist(uint2 *h, size_t i, float4 v) {
    const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
    uint2 r;
    r.x = *reinterpret_cast<const uint32_t *>(&a);
    r.y = *reinterpret_cast<const uint32_t *>(&b);
    h[i] = r;
}

__device__ __forceinline__ float4 fmin4(float4 a, float4 b) {
    return make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), fminf(a.w, b.w));
}
__device__ __forceinline__ float4 fmax4(float4 a, float4 b) {
    return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
}
// Three-input minimum / maximum (sm_100+ PTX min/max with three sources),
// per channel; exact, like every min/max.
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float4 min3_4(float4 a, float4 b, float4 c) {
    return make_float4(min3f(a.x, b.x, c.x), min3f(a.y, b.y, c.y), min3f(a.z, b.z, c.z), min3f(a.w, b.w, c.w));
}
__device__ __forceinline__ float4 max3_4(float4 a, float4 b, float4 c) {
    return make_float4(max3f(a.x, b.x, c.x), max3f(a.y, b.y, c.y), max3f(a.z, b.z, c.z), max3f(a.w, b.w, c.w));
}
// a + t (b - a) on packed FP32x2 lanes (each lane rounds like the scalar form)
__device__ __forceinline__ float2 lerp2(float2 a, float2 b, float t) {
    return __ffma2_rn(make_float2(t, t), __fadd2_rn(b, make_float2(-a.x, -a.y)), a);
}
// Bilinear filter of four RGBA texels: x on both rows, then y.
__device__ __forceinline__ float4 bil4(float fx, float fy, float4 h00, float4 h01, float4 h10, float4 h11) {
    const float2 xy = lerp2(lerp2(make_float2(h00.x, h00.y), make_float2(h01.x, h01.y), fx),
                            lerp2(make_float2(h10.x, h10.y), make_float2(h11.x, h11.y), fx), fy);
    const float2 zw = lerp2(lerp2(make_float2(h00.z, h00.w), make_float2(h01.z, h01.w), fx),
                            lerp2(make_float2(h10.z, h10.w), make_float2(h11.z, h11.w), fx), fy);
    return make_float4(xy.x, xy.y, zw.x, zw.y);
}
// TAA blend h + b (c - h) of the clamped history towards the current value
__device__ __forceinline__ float4 blend4(float4 h, float4 c, float b) {
    const float2 xy = lerp2(make_float2(h.x, h.y), make_float2(c.x, c.y), b);
    const float2 zw = lerp2(make_float2(h.z, h.w), make_float2(c.z, c.w), b);
    return make_float4(xy.x, xy.y, zw.x, zw.y);
}

// Reprojection and TAA resolve fused (Sec. 3.2): each pixel's motion is
// computed in registers (the motion kernel's arithmetic, bitwise) instead
// of being written and read back; the current frame's 3x3 neighbourhoods come
// from a shared-memory tile with a clamped one-pixel halo, brought in by one
// TMA bulk tensor copy while the motion is computed; each thread resolves
// ResolvePix<H> vertically adjacent pixels, whose 3x3 windows share rows, and
// filters their history footprints before it waits for the tile.
#ifndef CLOUDVOL_TAA_PIX_F32
#define CLOUDVOL_TAA_PIX_F32 4  // pixels per thread, FP32 history (78 registers)
#endif
#ifndef CLOUDVOL_TAA_PIX_F16
#define CLOUDVOL_TAA_PIX_F16 2  // pixels per thread, FP16 history
#endif
template <typename H>
struct ResolvePix {
    static constexpr int value = CLOUDVOL_TAA_PIX_F32;
    static constexpr int rows = 8 * value;  // pixel rows of a tile
};
template <>
struct ResolvePix<uint2> {
    static constexpr int value = CLOUDVOL_TAA_PIX_F16;
    static constexpr int rows = 8 * value;
};
constexpr int kTW = 32;  // pixel tile of a 32x8-thread CTA: 32 x ResolvePix<H>::rows
#ifndef CLOUDVOL_TAA_MIN_BLOCKS
#define CLOUDVOL_TAA_MIN_BLOCKS 3  // CTAs per SM the fused kernel is compiled for
#endif

// Waits that gave up (a bulk copy that did not complete in time): counted on
// the device, read by cloud_device_wait_timeouts; a launch may also be given a
// counter of its own (`status`, device or mapped host memory) that its caller
// reads.  Every wait below is bounded.  The first wait polls `first_polls`
// times (kWaitPolls by default; cloud_debug_set_wait_polls changes it for
// tests); after a give-up one thread waits once more, at most kDrainPolls
// polls with a short sleep between them (about 0.1 s), for the copy already
// issued, so that it lands before the block exits.
__device__ unsigned int g_wait_timeouts = 0;
constexpr int kWaitPolls = 1 << 16;
constexpr int kDrainPolls = 1 << 20;
std::atomic<int> g_first_polls{kWaitPolls};

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// Bounded wait for phase `parity` of an mbarrier: at most `polls` polls
// (with a sleep of `sleep_ns` between them); false when it gave up.
__device__ __forceinline__ bool mbar_wait(const uint64_t *bar, unsigned parity, int polls,
                                          unsigned sleep_ns = 0) {
    const unsigned a = smem_addr(bar);
    for (int it = 0; it < polls; ++it) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if (sleep_ns) __nanosleep(sleep_ns);
    }
    return false;
}

// 16 bytes from global to shared memory, asynchronously (cp.async).
__device__ __forceinline__ void copy_async16(void *smem, const void *global) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(smem)), "l"(global)
                 : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void *p) {
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
}

// The history footprints of a thread's kPix vertically adjacent pixels, filtered
// bilinearly: the off-screen test, then the texels around each sample position.
template <typename H, int kPix>
struct Footprints {
    bool use[kPix];    // the pixel has history on screen
    float4 hf[kPix];   // its filtered value

    // mot(r) gives the motion of pixel (x, y0 + r)
    template <typename Motion>
    __device__ __forceinline__ void gather(const H *__restrict__ hist, int x, int y0, int W, int Hh,
                                           unsigned *check, const Motion &mot) {
        float fxs[kPix], fys[kPix];
        float4 h00[kPix], h01[kPix], h10[kPix], h11[kPix];
#pragma unroll
        for (int r = 0; r < kPix; ++r) {
            use[r] = false;
            const int y = y0 + r;
            if (y >= Hh) continue;
            const float2 m = mot(r);
            const float xc = (float)x + 0.5f, yc = (float)y + 0.5f;
            // q = centre - m outside [0,W] x [0,H]: exact comparisons in FP32
            if ((m.x > xc) || (m.x < xc - (float)W) || (m.y > yc) || (m.y < yc - (float)Hh)) continue;
            // sample position (x - m.x, y - m.y) in texel-centre coordinates,
            // split into integer and fraction without rounding
            const float nx = -m.x, ny = -m.y;
            const float flx = floorf(nx), fly = floorf(ny);
            fxs[r] = nx - flx;
            fys[r] = ny - fly;
            const int ix = x + (int)flx, iy = y + (int)fly;
            const int xa = min(max(ix, 0), W - 1), xb = min(max(ix + 1, 0), W - 1);
            const int ya = min(max(iy, 0), Hh - 1), yb = min(max(iy + 1, 0), Hh - 1);
            if (!in_range(check, xa >= 0 && xb < W && ya >= 0 && yb < Hh, kChkHistory)) continue;
            const H *ra = hist + (size_t)ya * W, *rb = hist + (size_t)yb * W;
            h00[r] = load_hist(ra, xa);
            h01[r] = load_hist(ra, xb);
            h10[r] = load_hist(rb, xa);
            h11[r] = load_hist(rb, xb);
            use[r] = true;
        }
#pragma unroll
        for (int r = 0; r < kPix; ++r)
            if (use[r]) hf[r] = bil4(fxs[r], fys[r], h00[r], h01[r], h10[r], h11[r]);
    }
};

template <int kPix>
using ResolveTile = float4[8 * kPix + 2][kTW + 2];

// The end of a resolved tile: 3x3 ranges from the kPix + 2 tile rows the
// thread's windows cover (three-input min/max): each row's three texels reduced
// once, each pixel combines three row results as soon as its last row is in;
// clamp the filtered history, blend, store.
template <typename H, int kPix>
__device__ __forceinline__ void resolve_pixels(const ResolveTile<kPix> &tile, const Footprints<H, kPix> &f,
                                               H *__restrict__ out, float blend, int x, int y0, int W,
                                               int Hh, unsigned *check) {
    constexpr int kTH = 8 * kPix;
    const int tx = threadIdx.x, ty = threadIdx.y;
    if (x >= W) return;
    if (!in_range(check, tx + 2 < kTW + 2 && kPix * ty + kPix + 1 < kTH + 2, kChkTile)) return;
    float4 rmn[kPix + 2], rmx[kPix + 2], cen[kPix + 2];
#pragma unroll
    for (int j = 0; j < kPix + 2; ++j) {
        const float4 a = tile[kPix * ty + j][tx], b = tile[kPix * ty + j][tx + 1],
                     d = tile[kPix * ty + j][tx + 2];
        rmn[j] = min3_4(a, b, d);
        rmx[j] = max3_4(a, b, d);
        cen[j] = b;
        if (j < 2) continue;
        const int r = j - 2;  // the pixel whose window ends at row j
        const int y = y0 + r;
        if (y >= Hh) continue;
        const float4 c = cen[r + 1];
        float4 res = c;
        if (f.use[r]) {
            const float4 mn = min3_4(rmn[r], rmn[r + 1], rmn[r + 2]);
            const float4 mx = max3_4(rmx[r], rmx[r + 1], rmx[r + 2]);
            res = blend4(fmin4(fmax4(f.hf[r], mn), mx), c, blend);
        }
        if (in_range(check, y >= 0 && x >= 0, kChkPixel)) store_hist(out, (size_t)y * W + x, res);
    }
}

// One tile (bx, by) of 32 x ResolvePix<H>::rows pixels of the fused resolve: the
// body of both the single-view kernel and the multi-view kernel.  tile_map
// points to the current frame's tensor map (kernel parameter or global memory),
// tile and bar are the block's shared memory.
template <typename H>
__device__ __forceinline__ void resolve_tile(const CUtensorMap *tile_map, const MotionParams &mp,
                                             const H *__restrict__ hist, H *__restrict__ out,
                                             float blend, int bx, int by, ResolveTile<ResolvePix<H>::value> &tile,
                                             uint64_t &bar, int first_polls, unsigned int *status) {
    constexpr int kPix = ResolvePix<H>::value, kTH = ResolvePix<H>::rows;
    const int W = mp.width, Hh = mp.height;
    const int x0 = bx * kTW, y0 = by * kTH;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = x0 + tx;
    const int tid = ty * 32 + tx;
    // 1. current-frame tile with a one-pixel halo (34 x kTH + 2 texels), one TMA
    //    bulk copy issued by one thread, landing while the motion is computed.
    //    The box starts at texel (x0 - 1, y0 - 1): its x offset in bytes is
    //    16 (x0 - 1), a multiple of 16; texels outside the frame arrive as
    //    zeros and are replaced by their clamped neighbours below.
    //    Thread 0 initialises the barrier and issues the copy; the other
    //    threads only touch the barrier after the __syncthreads below, so the
    //    motion arithmetic starts at once.
    if (hist && x < W) {
#pragma unroll
        for (int r = 0; r < kPix; ++r)
            if (y0 + kPix * ty + r < Hh) prefetch_l2(hist + (size_t)(y0 + kPix * ty + r) * W + x);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        constexpr unsigned kTileBytes = (kTH + 2) * (kTW + 2) * 16;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                     ::"r"(smem_addr(&bar)), "r"(kTileBytes) : "memory");
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3}], [%4];\n"
            ::"r"(smem_addr(&tile[0][0])), "l"(tile_map), "r"(4 * (x0 - 1)), "r"(y0 - 1),
              "r"(smem_addr(&bar))
            : "memory");
    }
    // 2. motion (registers only) and the history footprint of the thread's
    //    pixels (rows kPix ty .. kPix ty + kPix - 1 of the tile): column terms
    //    once, the pixels' arithmetic interleaved, the rare near-tie calls
    //    after; filtered before the wait for the tile
    Footprints<H, kPix> f;
#pragma unroll
    for (int r = 0; r < kPix; ++r) f.use[r] = false;
    if (hist && x < W) {
        float2 m[kPix];
        motion_column<kPix>(mp, x, y0 + kPix * ty, m);
        f.gather(hist, x, y0 + kPix * ty, W, Hh, mp.check, [&](int r) { return m[r]; });
    }
    __syncthreads();  // the barrier's initialisation is visible to every thread
    const bool landed = mbar_wait(&bar, 0, first_polls);
    if (!__syncthreads_and(landed)) {
        // the copy did not complete within the bounded wait: count it (globally
        // and in the launch's own counter), leave the outputs of this tile
        // unwritten, and give the copy already issued one more bounded wait
        // (about 0.1 s) before the block exits; if that wait also gives up the
        // copy may still be pending, which counts a second time
        if (tid == 0) {
            atomicAdd(&g_wait_timeouts, 1u);
            if (status) atomicAdd_system(status, 1u);
            if (!mbar_wait(&bar, 0, kDrainPolls, 100)) {
                atomicAdd(&g_wait_timeouts, 1u);
                if (status) atomicAdd_system(status, 1u);
            }
        }
        return;
    }
    // texels outside the frame: clamp to the edge (border tiles only); every
    // source is an in-frame texel of the tile and every target an outside one
    const int r_lo = max(0, 1 - y0), r_hi = min(kTH + 1, Hh - y0);
    const int c_lo = max(0, 1 - x0), c_hi = min(kTW + 1, W - x0);
    if (r_lo > 0 || c_lo > 0 || r_hi < kTH + 1 || c_hi < kTW + 1) {
        for (int i = tid; i < (kTH + 2) * (kTW + 2); i += 256) {
            const int r = i / (kTW + 2), c = i - r * (kTW + 2);
            const int rr = min(max(r, r_lo), r_hi), cc = min(max(c, c_lo), c_hi);
            if (!in_range(mp.check, rr >= 0 && rr < kTH + 2 && cc >= 0 && cc < kTW + 2, kChkTile)) continue;
            if (rr != r || cc != c) tile[r][c] = tile[rr][cc];
        }
        __syncthreads();
    }
    // 3. 3x3 ranges, clamp, blend
    resolve_pixels<H, kPix>(tile, f, out, blend, x, y0 + kPix * ty, W, Hh, mp.check);
}

// TAA resolve of a first frame: the current frame in the history's format.  A plain
// copy, bound by memory; the resolve's tile and its halo would read 19 % more and
// wait for the tile (1920x1080 FP32 11.7 us against 17.9, FP16 9.8 against 15.9).
template <typename H>
__global__ void __launch_bounds__(256) first_frame_kernel(const float4 *__restrict__ cur, H *__restrict__ out,
                                                          int n) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) store_hist(out, i, __ldg(cur + i));
}

// TAA resolve (Sec. 3.2) with a given motion field: the pixel code of the fused
// resolve; the current frame's tile, its halo clamped to the frame's edge, is
// copied to shared memory asynchronously (cp.async) while the motion and then
// the history footprints are read.  Bound by the latency of those two dependent
// reads, so the motion is asked for first, the history's lines are prefetched
// into the L2 without waiting for it (motion is a few pixels), and the smaller
// tile of two pixels a thread lets four CTAs overlap: 1920x1080 FP32, motion
// kernel included, 32.8 us against 40.6 us for one pixel a thread with its
// neighbours read through L1.  Two pixels and 4 / 5 CTAs 34.7 / 34.6
// us with the motion, four pixels and 3 CTAs 38.0, one pixel and 6 CTAs 38.1
// (before the prefetch).  One pixel a thread (kPix) where tiles of two would leave
// SMs without a CTA: 128x128 FP16 2.1 us, with two 2.65.
constexpr int kTaaBlocks = 4;
template <typename H, int kPix>
__global__ void __launch_bounds__(256, kTaaBlocks)
    taa_kernel(const H *__restrict__ hist, const float4 *__restrict__ cur,
               const float2 *__restrict__ mot, H *__restrict__ out, int W, int Hh, float blend,
               unsigned *check) {
    constexpr int kTH = 8 * kPix;
    __shared__ __align__(128) ResolveTile<kPix> tile;
    const int x0 = blockIdx.x * kTW, y0 = blockIdx.y * kTH;
    const int x = x0 + threadIdx.x, y = y0 + kPix * threadIdx.y;
    float2 m[kPix];
#pragma unroll
    for (int r = 0; r < kPix; ++r)
        m[r] = x < W && y + r < Hh ? __ldg(mot + (size_t)(y + r) * W + x) : make_float2(0.0f, 0.0f);
    if (x < W) {
#pragma unroll
        for (int r = 0; r < kPix; ++r)
            if (y + r < Hh) prefetch_l2(hist + (size_t)(y + r) * W + x);
    }
    // row by row, a warp a row: texels -1 .. 30 of the row, then lanes 0 and 1
    // the two to the right
    const int xl = min(max(x - 1, 0), W - 1), xr = min(x + kTW - 1, W - 1);
#pragma unroll
    for (int k = 0; k <= kPix; ++k) {
        const int r = threadIdx.y + 8 * k;
        if (r >= kTH + 2) break;
        const int yy = min(max(y0 + r - 1, 0), Hh - 1);
        if (!in_range(check, xl < W && xr >= 0 && yy >= 0 && yy < Hh, kChkHistory)) continue;
        const float4 *row = cur + (size_t)yy * W;
        copy_async16(&tile[r][threadIdx.x], row + xl);
        if (threadIdx.x < 2) copy_async16(&tile[r][threadIdx.x + kTW], row + xr);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    Footprints<H, kPix> f;
#pragma unroll
    for (int r = 0; r < kPix; ++r) f.use[r] = false;
    if (x < W) f.gather(hist, x, y, W, Hh, check, [&](int r) { return m[r]; });
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    resolve_pixels<H, kPix>(tile, f, out, blend, x, y, W, Hh, check);
}

template <typename H>
__global__ void __launch_bounds__(256, CLOUDVOL_TAA_MIN_BLOCKS)
    taa_reproject_kernel(const __grid_constant__ CUtensorMap tile_map,
                         const __grid_constant__ MotionParams mp, const H *__restrict__ hist,
                         H *__restrict__ out, float blend, int first_polls, unsigned int *status) {
    __shared__ __align__(128) ResolveTile<ResolvePix<H>::value> tile;
    __shared__ __align__(8) uint64_t bar;
    resolve_tile<H>(&tile_map, mp, hist, out, blend, blockIdx.x, blockIdx.y, tile, bar, first_polls,
                    status);
}

// Many views' resolves in one launch (the render server's batches): block b
// is tile b of the concatenated views' tile lists; its view is found by
// binary search over the views' first tiles and its motion constants staged
// in shared memory.  Each tile is computed exactly as by taa_reproject_kernel.
struct alignas(128) ResolveView {  // the tensor map's own alignment
    CUtensorMap map;  // the view's current frame
    MotionParams mp;
    const void *hist;
    void *out;
    float blend;
    int tiles_x, tile_begin;
};

template <typename H>
__global__ void __launch_bounds__(256, CLOUDVOL_TAA_MIN_BLOCKS)
    taa_reproject_batch_kernel(const ResolveView *__restrict__ views, int n_views, int first_polls,
                               unsigned int *status) {
    __shared__ __align__(128) ResolveTile<ResolvePix<H>::value> tile;
    __shared__ __align__(8) uint64_t bar;
    __shared__ MotionParams smp;
    __shared__ int s_view;
    const int t = blockIdx.x, tid = threadIdx.y * 32 + threadIdx.x;
    if (tid == 0) {
        int lo = 0, hi = n_views - 1;  // last view with tile_begin <= t
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (views[mid].tile_begin <= t) lo = mid;
            else hi = mid - 1;
        }
        s_view = lo;
    }
    __syncthreads();
    const ResolveView &rv = views[s_view];
    const int *src = reinterpret_cast<const int *>(&rv.mp);
    int *dst = reinterpret_cast<int *>(&smp);
    for (int i = tid; i < (int)(sizeof(MotionParams) / 4); i += 256) dst[i] = src[i];
    __syncthreads();
    const int local = t - rv.tile_begin;
    if (!in_range(smp.check, s_view >= 0 && s_view < n_views && local >= 0, kChkView)) return;
    resolve_tile<H>(&rv.map, smp, (const H *)rv.hist, (H *)rv.out, rv.blend, local % rv.tiles_x,
                    local / rv.tiles_x, tile, bar, first_polls, status);
}

int build_motion_params(const cloud_volume *vol, const cloud_params *prm, const cloud_camera *prev,
                        const cloud_camera *cur, int width, int height, MotionParams *p) {
    if (width < 1 || height < 1 || width > CLOUD_MAX_DIM || height > CLOUD_MAX_DIM)
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_motion: width/height outside [1, 16384]");
    if (!(cur->tan_half_fovy > 0.0) || !(prev->tan_half_fovy > 0.0) || !(prm->t_max_m > 0.0))
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_motion: bad camera or t_max");
    *p = MotionParams{};
    const double aspect = (double)width / (double)height;
    const double aT = aspect * cur->tan_half_fovy, aTp = aspect * prev->tan_half_fovy;
    const double T = cur->tan_half_fovy, Tp = prev->tan_half_fovy;
    p->a0 = (float)((1.0 / width - 1.0) * aT);
    p->ax = (float)(2.0 * aT / width);
    p->b0 = (float)((1.0 - 1.0 / height) * T);
    p->by = (float)(-2.0 * T / height);
    p->rz = (float)cur->right[2];
    p->uz = (float)cur->up[2];
    p->fz = (float)cur->forward[2];
    p->zlo = (float)(vol->desc.slab_lo_m - cur->pos[2]);
    p->zhi = (float)(vol->desc.slab_hi_m - cur->pos[2]);
    p->tmax = (float)prm->t_max_m;
    // rows of R (current) and R' (previous): right, up, forward
    const double *R[3] = {cur->right, cur->up, cur->forward};
    const double *Rp[3] = {prev->right, prev->up, prev->forward};
    for (int i = 0; i < 3; ++i) {
        double dl = 0.0;
        for (int k = 0; k < 3; ++k) dl += Rp[i][k] * (cur->pos[k] - prev->pos[k]);
        p->dlt[i] = (float)dl;
        for (int j = 0; j < 3; ++j) {
            double mij = 0.0;  // (R' R^T)_ij = Rp_i . R_j
            for (int k = 0; k < 3; ++k) mij += Rp[i][k] * R[j][k];
            p->G[i][j] = (float)(mij - (i == j ? 1.0 : 0.0));
        }
    }
    p->kx = (float)(aTp / aT);
    p->ky = (float)(Tp / T);
    p->kx1 = (float)((aTp - aT) / aT);
    p->ky1 = (float)((Tp - T) / T);
    p->sx = (float)(width / (2.0 * aTp));
    p->sy = (float)(height / (2.0 * Tp));
    p->width = width;
    p->height = height;
    const double a0 = (1.0 / width - 1.0) * aT, ax = 2.0 * aT / width;
    const double b0 = (1.0 - 1.0 / height) * T, by = -2.0 * T / height;
    for (int k = 0; k < 3; ++k) {
        split_df(cur->forward[k] + a0 * cur->right[k] + b0 * cur->up[k], &p->v00h[k], &p->v00l[k]);
        split_df10(ax * cur->right[k], &p->vxh[k], &p->vxl[k]);
        split_df10(by * cur->up[k], &p->vyh[k], &p->vyl[k]);
    }
    split_df(vol->desc.slab_lo_m - cur->pos[2], &p->zlo_h, &p->zlo_l);
    split_df(vol->desc.slab_hi_m - cur->pos[2], &p->zhi_h, &p->zhi_l);
    split_df(prm->t_max_m, &p->tmax_h, &p->tmax_l);
    p->check = check_word();
    return CLOUD_OK;
}

int launch_motion(const cloud_volume *vol, const cloud_params *prm, const cloud_camera *prev,
                  const cloud_camera *cur, int width, int height, float *motion, cudaStream_t s) {
    if (!vol || !prm || !prev || !cur || !motion)
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_motion: null pointer");
    if (!aligned(motion, 8)) return set_error(CLOUD_ERR_INVALID_ARG, "cloud_motion: motion not 8-byte aligned");
    MotionParams p;
    if (int rc = build_motion_params(vol, prm, prev, cur, width, height, &p)) return rc;
    const int columns = (width + 31) / 32, rows = columns * ((height + 31) / 32) < sm_count() ? 2 : 4;
    const dim3 grid(columns, (height + 8 * rows - 1) / (8 * rows)), block(32, 8);
    if (rows == 2)
        motion_kernel<2><<<grid, block, 0, s>>>(p, (float2 *)motion);
    else
        motion_kernel<4><<<grid, block, 0, s>>>(p, (float2 *)motion);
    return check_launch("motion_kernel");
}

template <typename H>
static void launch_taa_kernel(const void *history, const float *current, const float *motion,
                              void *history_out, int width, int height, int pix, float blend, cudaStream_t s) {
    const dim3 grid((width + kTW - 1) / kTW, (height + 8 * pix - 1) / (8 * pix)), block(32, 8);
    const auto kernel = pix == 1 ? taa_kernel<H, 1> : taa_kernel<H, 2>;
    kernel<<<grid, block, 0, s>>>((const H *)history, (const float4 *)current, (const float2 *)motion,
                                  (H *)history_out, width, height, blend, check_word());
}

int launch_taa(const void *history, const float *current, const float *motion, void *history_out,
               int width, int height, int fmt, float blend, cudaStream_t s) {
    if (!current || !motion || !history_out)
        return set_error(CLOUD_ERR_INVALID_ARG, "taa_resolve: null pointer");
    if (width < 1 || height < 1 || width > CLOUD_MAX_DIM || height > CLOUD_MAX_DIM)
        return set_error(CLOUD_ERR_INVALID_ARG, "taa_resolve: width/height outside [1, 16384]");
    if (fmt != CLOUD_HISTORY_FP32 && fmt != CLOUD_HISTORY_FP16)
        return set_error(CLOUD_ERR_INVALID_ARG, "taa_resolve: bad history format");
    if (!(blend >= 0.0f && blend <= 1.0f))
        return set_error(CLOUD_ERR_INVALID_ARG, "taa_resolve: blend outside [0, 1]");
    const size_t px = (size_t)width * height, eb = fmt == CLOUD_HISTORY_FP32 ? 16 : 8;
    if (!aligned(current, 16) || !aligned(motion, 8) || !aligned(history_out, eb) ||
        (history && !aligned(history, eb)))
        return set_error(CLOUD_ERR_INVALID_ARG, "taa_resolve: misaligned buffer");
    if (history) {
        const char *a = (const char *)history, *b = (const char *)history_out;
        if (a < b + px * eb && b < a + px * eb)
            return set_error(CLOUD_ERR_INVALID_ARG, "taa_resolve: history and history_out overlap");
    }
    if (!history) {
        const int n = width * height, blocks = (n + 255) / 256;
        if (fmt == CLOUD_HISTORY_FP32)
            first_frame_kernel<float4><<<blocks, 256, 0, s>>>((const float4 *)current, (float4 *)history_out, n);
        else
            first_frame_kernel<uint2><<<blocks, 256, 0, s>>>((const float4 *)current, (uint2 *)history_out, n);
        return check_launch("first_frame_kernel");
    }
    const int columns = (width + kTW - 1) / kTW, pix = columns * ((height + 15) / 16) < sm_count() ? 1 : 2;
    if (fmt == CLOUD_HISTORY_FP32)
        launch_taa_kernel<float4>(history, current, motion, history_out, width, height, pix, blend, s);
    else
        launch_taa_kernel<uint2>(history, current, motion, history_out, width, height, pix, blend, s);
    return check_launch("taa_kernel");
}

// Tensor map of the current frame for the resolve's tile copy: the frame as
// a 2-D FP32 array of 4 W x H elements (row stride 16 W bytes), box 4 (kTW + 2)
// x (rows + 2) elements, zero fill outside.  The encoder is the driver's,
// fetched through the runtime once.
static int current_tile_map(const float *current, int width, int height, int rows, CUtensorMap *map) {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    std::call_once(once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    if (!encode) return set_error(CLOUD_ERR_CUDA, "cloud_taa_reproject: cuTensorMapEncodeTiled unavailable");
    const cuuint64_t dims[2] = {4ull * (cuuint64_t)width, (cuuint64_t)height};
    const cuuint64_t strides[1] = {16ull * (cuuint64_t)width};
    const cuuint32_t box[2] = {4u * (kTW + 2), (cuuint32_t)(rows + 2)};
    const cuuint32_t elem[2] = {1u, 1u};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(current), dims,
                              strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(CLOUD_ERR_CUDA, "cloud_taa_reproject: tensor map rejected");
    return CLOUD_OK;
}

int launch_taa_reproject(const cloud_volume *vol, const cloud_params *prm, const cloud_camera *prev,
                         const cloud_camera *cur, const void *history, const float *current,
                         void *history_out, int width, int height, int fmt, float blend,
                         unsigned int *status, cudaStream_t s) {
    if (!vol || !prm || !cur || !current || !history_out || (history && !prev))
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_taa_reproject: null pointer");
    if (fmt != CLOUD_HISTORY_FP32 && fmt != CLOUD_HISTORY_FP16)
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_taa_reproject: bad history format");
    if (!(blend >= 0.0f && blend <= 1.0f))
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_taa_reproject: blend outside [0, 1]");
    MotionParams p;
    if (int rc = build_motion_params(vol, prm, history ? prev : cur, cur, width, height, &p)) return rc;
    const size_t px = (size_t)width * height, eb = fmt == CLOUD_HISTORY_FP32 ? 16 : 8;
    if (!aligned(current, 16) || !aligned(history_out, eb) || (history && !aligned(history, eb)))
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_taa_reproject: misaligned buffer");
    if (history) {
        const char *a = (const char *)history, *b = (const char *)history_out;
        if (a < b + px * eb && b < a + px * eb)
            return set_error(CLOUD_ERR_INVALID_ARG, "cloud_taa_reproject: history and history_out overlap");
    }
    const int rows = fmt == CLOUD_HISTORY_FP32 ? ResolvePix<float4>::rows : ResolvePix<uint2>::rows;
    CUtensorMap map;
    if (int rc = current_tile_map(current, width, height, rows, &map)) return rc;
    const dim3 grid((width + kTW - 1) / kTW, (height + rows - 1) / rows), block(32, 8);
    const int polls = g_first_polls.load();
    if (fmt == CLOUD_HISTORY_FP32)
        taa_reproject_kernel<float4><<<grid, block, 0, s>>>(map, p, (const float4 *)history,
                                                            (float4 *)history_out, blend, polls,
                                                            status);
    else
        taa_reproject_kernel<uint2><<<grid, block, 0, s>>>(map, p, (const uint2 *)history,
                                                           (uint2 *)history_out, blend, polls,
                                                           status);
    return check_launch("taa_reproject_kernel");
}

int launch_taa_reproject_batch(const cloud_volume *vol, const cloud_params *prm,
                               const ResolveRequest *reqs, int n, int fmt, float blend,
                               void *h_table_v, void *d_table_v, unsigned int *status,
                               cudaStream_t s) {
    if (!vol || !prm || !reqs || n < 1 || !h_table_v || !d_table_v)
        return set_error(CLOUD_ERR_INVALID_ARG, "resolve batch: bad arguments");
    if (fmt != CLOUD_HISTORY_FP32 && fmt != CLOUD_HISTORY_FP16)
        return set_error(CLOUD_ERR_INVALID_ARG, "resolve batch: bad history format");
    if (!(blend >= 0.0f && blend <= 1.0f))
        return set_error(CLOUD_ERR_INVALID_ARG, "resolve batch: blend outside [0, 1]");
    ResolveView *h_table = static_cast<ResolveView *>(h_table_v);
    int next = 0;
    const size_t eb = fmt == CLOUD_HISTORY_FP32 ? 16 : 8;
    const int rows = fmt == CLOUD_HISTORY_FP32 ? ResolvePix<float4>::rows : ResolvePix<uint2>::rows;
    for (int i = 0; i < n; ++i) {
        const ResolveRequest &r = reqs[i];
        if (!r.cur || !r.current || !r.out || (r.history && !r.prev))
            return set_error(CLOUD_ERR_INVALID_ARG, "resolve batch: null pointer");
        ResolveView &v = h_table[i];
        if (int rc = build_motion_params(vol, prm, r.history ? r.prev : r.cur, r.cur, r.width,
                                         r.height, &v.mp))
            return rc;
        const size_t px = (size_t)r.width * r.height;
        if (!aligned(r.current, 16) || !aligned(r.out, eb) || (r.history && !aligned(r.history, eb)))
            return set_error(CLOUD_ERR_INVALID_ARG, "resolve batch: misaligned buffer");
        if (r.history) {
            const char *a = (const char *)r.history, *b = (const char *)r.out;
            if (a < b + px * eb && b < a + px * eb)
                return set_error(CLOUD_ERR_INVALID_ARG, "resolve batch: history and output overlap");
        }
        if (int rc = current_tile_map(r.current, r.width, r.height, rows, &v.map)) return rc;
        v.hist = r.history;
        v.out = r.out;
        v.blend = blend;
        v.tiles_x = (r.width + kTW - 1) / kTW;
        v.tile_begin = next;
        next += v.tiles_x * ((r.height + rows - 1) / rows);
    }
    if (int rc = check_cuda(cudaMemcpyAsync(d_table_v, h_table, sizeof(ResolveView) * n,
                                            cudaMemcpyHostToDevice, s),
                            "resolve batch: upload table"))
        return rc;
    const ResolveView *d_table = static_cast<const ResolveView *>(d_table_v);
    const int polls = g_first_polls.load();
    if (fmt == CLOUD_HISTORY_FP32)
        taa_reproject_batch_kernel<float4><<<next, dim3(32, 8), 0, s>>>(d_table, n, polls, status);
    else
        taa_reproject_batch_kernel<uint2><<<next, dim3(32, 8), 0, s>>>(d_table, n, polls, status);
    return check_launch("taa_reproject_batch_kernel");
}

size_t resolve_view_bytes() { return sizeof(ResolveView); }

// Composite (Sec. 3.2): the low-resolution cloud buffer, resampled
// bilinearly to the display size, laid over the background (premultiplied
// "over").  Streaming: the background is read and the result written once
// (32 B per pixel); the small cloud buffer is served by L1/L2.
// Source texel coordinate of output pixel x: u = (2x + 1) sw / (2 dw) - 1/2,
// split into floor(u) and frac(u) with integer arithmetic so that the texel
// choice is exact and frac is one correctly rounded division.
__device__ __forceinline__ void src_coord(int x, int sw, int dw, int &i0, float &f) {
    const int num = (2 * x + 1) * sw - dw, den = 2 * dw;  // < 2^31 for sizes <= 16384
    const int q = num >= 0 ? num / den : -1;              // num >= -dw > -den
    f = (float)(num - q * den) / (float)den;
    i0 = q;
}

template <typename H>
__global__ void __launch_bounds__(256) composite_kernel(const H *__restrict__ cloud, int sw, int sh,
                                                        const float4 *__restrict__ bg, float4 *out,
                                                        int dw, int dh, unsigned *check) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
    if (x >= dw || y >= dh) return;
    int u0, v0;
    float fx, fy;
    src_coord(x, sw, dw, u0, fx);
    src_coord(y, sh, dh, v0, fy);
    const int xa = max(u0, 0), xb = min(u0 + 1, sw - 1);
    const int ya = max(v0, 0), yb = min(v0 + 1, sh - 1);
    if (!in_range(check, xa < sw && xb >= 0 && ya < sh && yb >= 0, kChkHistory)) return;
    const float4 c00 = load_hist(cloud, (size_t)ya * sw + xa), c01 = load_hist(cloud, (size_t)ya * sw + xb);
    const float4 c10 = load_hist(cloud, (size_t)yb * sw + xa), c11 = load_hist(cloud, (size_t)yb * sw + xb);
    const float4 c = bil4(fx, fy, c00, c01, c10, c11);
    const size_t i = (size_t)y * dw + x;
    const float4 b = __ldg(bg + i);
    const float t = 1.0f - c.w;
    out[i] = make_float4(fmaf(t, b.x, c.x), fmaf(t, b.y, c.y), fmaf(t, b.z, c.z), fmaf(t, b.w, c.w));
}

int launch_composite(const void *cloud, int fmt, int sw, int sh, const float *bg, float *out, int dw,
                     int dh, cudaStream_t s) {
    if (!cloud || !bg || !out) return set_error(CLOUD_ERR_INVALID_ARG, "cloud_composite: null pointer");
    if (sw < 1 || sh < 1 || dw < 1 || dh < 1 || sw > CLOUD_MAX_DIM || sh > CLOUD_MAX_DIM ||
        dw > CLOUD_MAX_DIM || dh > CLOUD_MAX_DIM)
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_composite: sizes outside [1, 16384]");
    if (fmt != CLOUD_HISTORY_FP32 && fmt != CLOUD_HISTORY_FP16)
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_composite: bad cloud format");
    if (!aligned(cloud, fmt == CLOUD_HISTORY_FP32 ? 16 : 8) || !aligned(bg, 16) || !aligned(out, 16))
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_composite: misaligned buffer");
    const dim3 grid((dw + 31) / 32, (dh + 7) / 8), block(32, 8);
    if (fmt == CLOUD_HISTORY_FP32)
        composite_kernel<float4><<<grid, block, 0, s>>>((const float4 *)cloud, sw, sh, (const float4 *)bg,
                                                        (float4 *)out, dw, dh, check_word());
    else
        composite_kernel<uint2><<<grid, block, 0, s>>>((const uint2 *)cloud, sw, sh, (const float4 *)bg,
                                                       (float4 *)out, dw, dh, check_word());
    return check_launch("composite_kernel");
}

}  // namespace cloudvol

using namespace cloudvol;

extern "C" int cloud_motion(const cloud_volume *vol, const cloud_params *prm,
                            const cloud_camera *prev, const cloud_camera *cur, int width,
                            int height, float *motion, void *stream) {
    clear_error();
    return launch_motion(vol, prm, prev, cur, width, height, motion, (cudaStream_t)stream);
}

extern "C" int taa_resolve(const void *history, const float *current, const float *motion,
                           void *history_out, int width, int height, int history_fmt, float blend,
                           void *stream) {
    clear_error();
    return launch_taa(history, current, motion, history_out, width, height, history_fmt, blend,
                      (cudaStream_t)stream);
}

extern "C" int cloud_taa_reproject(const cloud_volume *vol, const cloud_params *prm,
                                   const cloud_camera *prev, const cloud_camera *cur,
                                   const void *history, const float *current, void *history_out,
                                   int width, int height, int history_fmt, float blend,
                                   void *stream) {
    clear_error();
    return launch_taa_reproject(vol, prm, prev, cur, history, current, history_out, width, height,
                                history_fmt, blend, nullptr, (cudaStream_t)stream);
}

extern "C" int cloud_composite(const void *cloud, int cloud_fmt, int cloud_width, int cloud_height,
                               const float *background, float *out, int width, int height,
                               void *stream) {
    clear_error();
    return launch_composite(cloud, cloud_fmt, cloud_width, cloud_height, background, out, width,
                            height, (cudaStream_t)stream);
}

extern "C" int cloud_device_wait_timeouts(unsigned int *count, int reset) {
    clear_error();
    if (!count) return set_error(CLOUD_ERR_INVALID_ARG, "cloud_device_wait_timeouts: null pointer");
    if (int rc = check_cuda(cudaMemcpyFromSymbol(count, g_wait_timeouts, sizeof(unsigned int)),
                            "cloud_device_wait_timeouts"))
        return rc;
    if (reset) {
        const unsigned int zero = 0;
        return check_cuda(cudaMemcpyToSymbol(g_wait_timeouts, &zero, sizeof(unsigned int)),
                          "cloud_device_wait_timeouts");
    }
    return CLOUD_OK;
}

extern "C" int cloud_debug_set_wait_polls(int first_polls) {
    clear_error();
    if (first_polls > (1 << 30))
        return set_error(CLOUD_ERR_INVALID_ARG, "cloud_debug_set_wait_polls: more than 2^30 polls");
    g_first_polls.store(first_polls < 0 ? kWaitPolls : first_polls);
    return CLOUD_OK;
}
