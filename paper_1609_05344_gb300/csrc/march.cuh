// march.cuh -- device side of the per-pixel cloud raymarch (Sec. 1, Sec. 3.1,
// Sec. 3.2), shared by the single-view kernel (render.cu) and the persistent
// multi-view kernel (batch.cu).
//
// Precision design.  Grazing rays are tens of kilometres long and, with 8
// view steps, a step is kilometres long; the estimator then multiplies any
// density error by alpha*D*L_in (hundreds), so sample positions must be far
// more accurate than FP32 world coordinates allow.  Per ray, the start and
// the step of every lattice axis (base xyz, detail xyz, weather xy) and of the
// height above the layer bottom are computed in double-float FP32 and stored
// as 32-bit fixed-point values: 2^32 units per tile period, so unsigned
// overflow is exactly the periodic wrap of the tile.  A view step adds the
// ray's increment and a light sample adds a per-launch constant offset --
// integer adds, no rounding.  The texel index is the top log2(N) bits, the
// interpolation weight the next 23 bits.  Radiance and the optical-depth sum
// are FP32.
//
// Times in the comments below compare a choice with its alternatives in one run of
// its time; cameras and builds differ from comment to comment (1920x1080 x 8 steps of
// the standard FP32 volume: 83 to 116 us), so figures of different comments do not
// compare.  Now: 116 us for the mean of a 32-frame orbit with the L2 flushed, 94 us a
// pass with inputs in turn.
#pragma once

#include "common.cuh"

// CTAs per SM the march of volumes of any tile sizes is compiled for (register budget
// 65536 / (128 x this)).  FP32 records: six for one view, five for the multi-view
// kernel, whose loop needs more registers; 16-bit records: six for both.  More of them
// spill, and cost more than the occupancy gives (64^3 base with detail and weather).
// FP16, six against seven (80 against 72 registers): 307x257 x 64 steps 74.5 us against
// 84.1, 12 views of 8 to 128 steps 1.27 ms against 1.33, 16 small ones 52 us against 63.
// FP32, one view, six against five: 256x152 x 8 steps (detail at 700 m) 10.4 us against
// 12.2, 1280x720 x 64 steps 227 us against 231; many views, five against six: 16 small
// ones 46 us against 51, 12 larger ones 1.27 ms against 1.26.
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_F32
#define CLOUDVOL_MARCH_MIN_BLOCKS_F32 6
#endif
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_F32_VIEWS
#define CLOUDVOL_MARCH_MIN_BLOCKS_F32_VIEWS 5
#endif
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_16
#define CLOUDVOL_MARCH_MIN_BLOCKS_16 6
#endif

namespace cloudvol {

// Records at the standard tile sizes and base tiles alone, 8 view steps per warp
// iteration: 8 CTAs (64 registers; the 16-bit kernels of the standard sizes spill 4 to
// 12 bytes in the multi-view and many-chunk marches, the FP32 ones of base tiles 4 to
// 16, the others nothing; 1920x1080 x 8 steps, FP32: 83.4 us, 83.3 with 7, 84.3 with 6,
// 86.5 with 9; 64 views, BF16: 10.50 ms, 10.73 with 7, 10.96 with 6).  With 16 steps per iteration the per-warp scratch is 1.7x larger
// and 8 CTAs would leave the L1 28 KB: 7 CTAs for FP32 records and 6 for 16-bit
// ones (64 views, BF16, by an earlier build: 18.7 ms against 19.5 ms with 8).
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_F32_FX
#define CLOUDVOL_MARCH_MIN_BLOCKS_F32_FX 8
#endif
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_16_FX
#define CLOUDVOL_MARCH_MIN_BLOCKS_16_FX 8
#endif
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_F32_FX16
#define CLOUDVOL_MARCH_MIN_BLOCKS_F32_FX16 7
#endif
#ifndef CLOUDVOL_MARCH_MIN_BLOCKS_16_FX16
#define CLOUDVOL_MARCH_MIN_BLOCKS_16_FX16 6
#endif
template <typename T, int VOL, int CH, bool VIEWS>
struct MarchBlocks {
    static constexpr bool f32 = sizeof(T) == 4;
    static constexpr int any_f32 = VIEWS ? CLOUDVOL_MARCH_MIN_BLOCKS_F32_VIEWS : CLOUDVOL_MARCH_MIN_BLOCKS_F32;
    static constexpr int value =
        VOL == kAnyVolume ? (f32 ? any_f32 : CLOUDVOL_MARCH_MIN_BLOCKS_16)
        : CH <= 8 ? (f32 ? CLOUDVOL_MARCH_MIN_BLOCKS_F32_FX : CLOUDVOL_MARCH_MIN_BLOCKS_16_FX)
                  : (f32 ? CLOUDVOL_MARCH_MIN_BLOCKS_F32_FX16 : CLOUDVOL_MARCH_MIN_BLOCKS_16_FX16);
};

// Light samples of a march evaluated per iteration of the light loop (the
// density code is inlined that many times): one for FP32 records, whose three
// wide loads per sample keep the memory busy (1920x1080 x 8 steps 86.1 us, two
// 86.8, three 96.9); two for 16-bit ones (64 views 10.86 ms, one 11.38, three
// 11.11) and where the tile sizes are not constants; three for a base tile alone,
// one record a sample (1280x720 x 64 steps 307.5 us, one 339.6, two 313.7, six
// 305.6; 128x128 32.3, 39.2, 33.3, 33.1).
#ifndef CLOUDVOL_LIGHT_UNROLL_F32
#define CLOUDVOL_LIGHT_UNROLL_F32 1
#endif
#ifndef CLOUDVOL_LIGHT_UNROLL_BASE
#define CLOUDVOL_LIGHT_UNROLL_BASE 3
#endif
#ifndef CLOUDVOL_LIGHT_UNROLL_16
#define CLOUDVOL_LIGHT_UNROLL_16 2
#endif
template <typename T, int VOL>
struct LightUnroll {
    static constexpr int value = VOL == kBaseVolume                             ? CLOUDVOL_LIGHT_UNROLL_BASE
                                 : VOL == kStandardVolume && sizeof(T) == 4 ? CLOUDVOL_LIGHT_UNROLL_F32 : CLOUDVOL_LIGHT_UNROLL_16;
};
// View lookups a lane evaluates per round of the shared-out view phase (their
// record loads can overlap; more of them cost registers): one for FP32
// records; for 16-bit records one with 8 view steps per iteration (the
// registers buy an eighth CTA per SM instead) and two with 16.
#ifndef CLOUDVOL_VIEW_BATCH_F32
#define CLOUDVOL_VIEW_BATCH_F32 1
#endif
#ifndef CLOUDVOL_VIEW_BATCH_16
#define CLOUDVOL_VIEW_BATCH_16 1
#endif
#ifndef CLOUDVOL_VIEW_BATCH_16_CH16
#define CLOUDVOL_VIEW_BATCH_16_CH16 2
#endif
template <typename T, int CH>
struct ViewBatch {
    static constexpr int value = sizeof(T) == 4 ? CLOUDVOL_VIEW_BATCH_F32
                                 : CH <= 8      ? CLOUDVOL_VIEW_BATCH_16
                                                : CLOUDVOL_VIEW_BATCH_16_CH16;
};
enum Axis { kBX = 0, kBY, kBZ, kDX, kDY, kDZ, kWX, kWY, kLatticeAxes };

// Constants shared by every view of a launch: volume, lighting, light march.
struct SceneParams {
    // Fixed-point lattice coordinates: coordinate = p * kfix - half a texel
    // (mod 2^32), kfix = 2^32 / tile period.
    float2 kfix_h[kLatticeAxes], kfix_l[kLatticeAxes];   // each value twice (packed operands)
    // light-sample offsets; in standard volumes those of the detail axes are what is
    // left of them once the base offset is shifted (see light_coords)
    uint32_t loff[CLOUD_MAX_LIGHT_STEPS][kLatticeAxes];
    int32_t lh[CLOUD_MAX_LIGHT_STEPS];                   // light-sample height offsets
    int32_t h_top;                                       // layer thickness in 2^-16 m
    float h_lo_scale, h_hi_scale;  // 10/thickness, 2.5/thickness, per 2^-16 m
    float sun[3], sun_rad[3], ambient[3];
    float hg_g, hg_norm, absorption, light_step, tau_max;  // hg_norm = (1 - g^2)/(4 pi)
    // k0 = 1/2 - c - w_d/2 minus the record decode bias b folded in:
    // k0 - b + w_d b; w_off = 1/2 - b (weather values are stored centred)
    float k0, inv_1mc, detail_w, rho0, w_off;
    // occupancy grid of the volume (bit set: density may be > 0 somewhere in
    // the macro-cell of 2^kOccShift records per axis), or nullptr; log2 of its
    // cells per axis
    const uint32_t *occ;
    // the same grid in blocks of 16^3 cells (standard tile sizes), or nullptr
    const uint32_t *occ_blocks;
    int log2_occ;
    unsigned *check;  // status word of the checked build, else nullptr
    int log2_base, log2_detail, log2_weather;
    int light_steps, integration;
    int wide;  // t_max spans more than 1000 tile periods (df2_to_u32)
    // detail coordinates = base detail_mul + detail_add (mod 2^32) when the base
    // tile period is 2^detail_shift detail periods (-1: convert separately)
    int detail_shift;
    uint32_t detail_mul, detail_add;
    // strides of a record index on y and z (y only for weather).  Powers of two,
    // but passed as values so that the index is built by multiply-adds: the march
    // keeps the ALU pipe (shifts, logic, integer adds) twice as busy as the FMA
    // pipe, which runs the multiply-adds.
    uint32_t base_mul[2], detail_rec_mul[2], weather_mul;
    uint32_t one;  // 1, for additions as multiply-adds (see above)
};

// One camera view: rays, layer clip, step count, jitter frame, output.
struct ViewParams {
    // Camera rays, unnormalised: v(x, y) = v00 + x vx + y vy, as double-float
    // pairs; vx/vy are split so that x * hi is exact (see split_df10).
    float v00h[3], v00l[3], vxh[3], vxl[3], vyh[3], vyl[3];
    // camera position in fixed-point lattice coordinates (half a texel taken off) and
    // its height above the layer bottom in 2^-16 m, each as the nearest integer and
    // the rest (in [-1/2, 1/2]): a sample's coordinate is rounded once, from the sum
    uint32_t org[kLatticeAxes], org_h;
    float org_rest[kLatticeAxes], org_h_rest;
    float zlo_h, zlo_l;    // slab_lo - o_z
    float zhi_h, zhi_l;    // slab_hi - o_z
    float tmax_h, tmax_l;  // far clip distance
    float invn_h, invn_l;  // 1 / steps
    // rays with d_z below miss_below (camera under the layer) or above
    // miss_above (camera over it) cannot reach the layer within t_max
    float miss_below, miss_above;
    int width, height, steps;
    float u_frame;         // >= 0: the start offset of every ray (no or per-frame jitter); < 0: per pixel
    uint32_t jitter_hash;  // the part of the per-pixel hash that the frame and the seed decide
    int tiles_x;           // tiles per image row
    int tile_begin;        // first work-queue index of this view (multi-view launches)
    float4 *out;     // device RGBA, width * height
};

// CTA pixel-tile shapes (4 warps of 32 lanes); the autotuner picks one.
//   shape 0: warp 8x4,  CTA 2x2 warps -> 16x8 pixels
//   shape 1: warp 8x4,  CTA 4x1 warps -> 32x4 pixels
//   shape 2: warp 16x2, CTA 2x2 warps -> 32x4 pixels
//   shape 3: warp 4x8,  CTA 2x2 warps -> 8x16 pixels
// and three with fewer rays than lanes, for images that would not fill the GPU
// (small_shape in render.cu): the shared-out phases still use every lane
//   shape 4: warp 4x4,  CTA 2x2 warps -> 8x8 pixels
//   shape 5: warp 4x2,  CTA 2x2 warps -> 8x4 pixels
//   shape 6: warp 2x2,  CTA 2x2 warps -> 4x4 pixels
constexpr int kShapes = 4;  // those the autotuner chooses from
constexpr int kAllShapes = 7;
template <int S>
struct TileShape;
template <>
struct TileShape<0> { static constexpr int WX = 8, WY = 4, CX = 2, CY = 2; };
template <>
struct TileShape<1> { static constexpr int WX = 8, WY = 4, CX = 4, CY = 1; };
template <>
struct TileShape<2> { static constexpr int WX = 16, WY = 2, CX = 2, CY = 2; };
template <>
struct TileShape<3> { static constexpr int WX = 4, WY = 8, CX = 2, CY = 2; };
template <>
struct TileShape<4> { static constexpr int WX = 4, WY = 4, CX = 2, CY = 2; };
template <>
struct TileShape<5> { static constexpr int WX = 4, WY = 2, CX = 2, CY = 2; };
template <>
struct TileShape<6> { static constexpr int WX = 2, WY = 2, CX = 2, CY = 2; };
inline void tile_dims(int shape, int *tw, int *th) {
    // not static: a static local of an inline function is one object per process,
    // also between two builds of the library
    constexpr int w[kAllShapes] = {16, 32, 32, 8, 8, 8, 4}, h[kAllShapes] = {8, 4, 4, 16, 8, 4, 4};
    *tw = w[shape];
    *th = h[shape];
}

// Launch configurations the autotuner chooses from: a pixel-tile shape and the
// number of view steps a warp evaluates per iteration of its march (the chunk
// of phase A/B/C below).  config = shape + kShapes * chunk index.
constexpr int CHSizes[2] = {8, 16};
constexpr int kConfigs = kShapes * 2;
inline int config_shape(int config) { return config % kShapes; }
inline int config_chunk(int config) { return CHSizes[(config / kShapes) & 1]; }
// Step counts a march is compiled for: any, at most one chunk, more than one.
// Single-view launches at the standard tile sizes know theirs (1920x1080 x 8
// steps FP16 106.0 -> 103.4 us, 957x541 30.5 -> 30.1 us, four cameras' mean); the
// views of a multi-view launch differ.
enum StepRange { kAnySteps, kOneChunk, kManyChunks };
constexpr unsigned kFull = 0xFFFFFFFFu;

// A ray's start coordinates and per-step increments as the warp stages them, in
// 16-byte groups so that a lane fetches another lane's ray with two, three or
// five wide shared loads instead of one load per axis:
//   group 0  start of base x, y, z and of the height
//   group 1  their increments
//   group 2  start of weather x, y, then their increments
//   group 3  start of detail x, y, z, then the increment of detail x
//   group 4  increments of detail y, z
// Standard volumes (the base tile period is 2^detail_shift detail periods) have no
// groups 3 and 4: the detail coordinates follow from the base ones by an exact
// shift; a base tile alone uses groups 0 and 1.
// Three and five groups a lane are odd strides: lanes that fetch neighbouring
// rays meet no bank conflict.
template <int VOL>
struct RayGroups { static constexpr int value = VOL == kAnyVolume ? 5 : 3; };

// Per-warp shared scratch of the march: each lane's staged ray and step length,
// the list of (step, lane) pairs to evaluate, and two values per (step, lane)
// of a chunk of CH view steps: the view density, then the integration weight;
// the optical depth before the step, then the sun's share of the light.
template <int CH, int VOL>
struct WarpScratch {
    uint4 ray[32][RayGroups<VOL>::value];
    float length[32];
    float rho[CH][32];
    float aux[CH][32];
    uint16_t pairs[CH * 32];
};

// Two interpolation weights (23 bits below the index bits, shifted to the top)
// with one packed subtraction.
__device__ __forceinline__ float2 frac23(uint32_t f, uint32_t g) {
    return __fadd2_rn(make_float2(__uint_as_float((f >> 9) | 0x3F800000u),
                                  __uint_as_float((g >> 9) | 0x3F800000u)),
                      make_float2(-1.0f, -1.0f));
}

// a b + c (mod 2^32) as one integer multiply-add, whatever b is.
__device__ __forceinline__ uint32_t mad32(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// Corner-packed sampling at fixed-point coordinates: the record index is the
// top L bits of each coordinate, the interpolation weights the next 23 bits.
__device__ __forceinline__ uint32_t rec3(const uint32_t (&mul)[2], int L, uint32_t cx, uint32_t cy,
                                         uint32_t cz) {
    const int sh = 32 - L;
    return mad32(cz >> sh, mul[1], mad32(cy >> sh, mul[0], cx >> sh));
}
__device__ __forceinline__ uint32_t rec2(uint32_t mul, int L, uint32_t cx, uint32_t cy) {
    const int sh = 32 - L;
    return mad32(cy >> sh, mul, cx >> sh);
}
// Interpolation on packed FP32x2 (Blackwell FFMA2/FADD2): x first on the
// (z0, z1) pairs of both y rows (the x differences come with the record),
// then y on the pair, then z.  Each lane of a packed op rounds exactly like
// the scalar op.
__device__ __forceinline__ float trilerp(const float c[8], float fx, float fy, float fz) {
    const float2 a0 = make_float2(c[0], c[1]), a1 = make_float2(c[2], c[3]);  // dx = 0
    const float2 d0 = make_float2(c[4], c[5]), d1 = make_float2(c[6], c[7]);  // dx = 1 minus dx = 0
    const float2 fx2 = make_float2(fx, fx), fy2 = make_float2(fy, fy);
    const float2 x0 = __ffma2_rn(fx2, d0, a0);  // dy = 0
    const float2 x1 = __ffma2_rn(fx2, d1, a1);  // dy = 1
    const float2 yz = __ffma2_rn(fy2, __fadd2_rn(x1, make_float2(-x0.x, -x0.y)), x0);  // (z0, z1)
    return fmaf(fz, yz.y - yz.x, yz.x);
}
__device__ __forceinline__ float bilerp(const float c[4], float fx, float fy) {
    const float2 a = make_float2(c[0], c[1]), d = make_float2(c[2], c[3]);  // (y0, y1): dx = 0, difference
    const float2 xy = __ffma2_rn(make_float2(fx, fx), d, a);
    return fmaf(fy, xy.y - xy.x, xy.x);
}

// Height profile g(h) of the layer at a fixed-point height (2^-16 m above the
// layer bottom): clamp(h / 0.1, 0, 1) clamp((1 - h) / 0.4, 0, 1), h in layer
// thicknesses.
__device__ __forceinline__ float height_profile(const SceneParams &p, int32_t hq) {
    const float ga = __saturatef((float)hq * p.h_lo_scale);
    const float gb = __saturatef((float)(p.h_top - hq) * p.h_hi_scale);
    return ga * gb;
}

// Occupancy bit of the macro-cell holding a sample's base record: clear where
// the volume's bound proves B - w_d Dt - c < 0, i.e. zero density.  At the
// standard sizes a cell coordinate is the top byte of the base coordinate, so
// two byte permutations gather the cell index and its low bits select the bit
// (the funnel shift takes its count modulo 32).
template <int VOL>
__device__ __forceinline__ bool occupied(const SceneParams &p, uint32_t bx, uint32_t by, uint32_t bz) {
    // macro-cell = record index >> kOccShift on each axis; bits x fastest
    constexpr bool FX = VOL == kStandardVolume, kBytes = FX && kStdLog2Base - kOccShift == 8;
    const int lo = FX ? kStdLog2Base - kOccShift : p.log2_occ, sh = 32 - lo;
    const uint32_t cell = kBytes ? __byte_perm(__byte_perm(bx, by, 0x7373), bz >> 24, 0x5410)
                                 : ((bz >> sh) << (2 * lo)) | ((by >> sh) << lo) | (bx >> sh);
    if (!in_range(p.check, cell < (1u << (3 * lo)), kChkOccupancy)) return true;
    return __funnelshift_r(__ldg(p.occ + (cell >> 5)), 0u, cell) & 1u;
}

// The same bit from the blocked copy of the grid, for rays of a warp that are
// spread along their direction by a jitter of their own: a 128-byte line covers
// 400 x 400 x 100 m instead of 6400 x 100 x 25 m, so the warp's reads meet fewer
// lines.  Index: high nibbles of the cell coordinates (the block), then their low
// ones, each triple gathered by one multiplication (no two of its partial products
// meet).  Costs six more instructions a step: 1920x1080 x 8 steps 112.0 -> 107.7 us
// with an offset per pixel, 89.0 -> 90.4 us with one per frame, and slower in long
// marches, whose steps follow each other along a line anyway.
__device__ __forceinline__ bool occupied_blocks(const SceneParams &p, uint32_t bx, uint32_t by, uint32_t bz) {
    const uint32_t t = __byte_perm(__byte_perm(bz, by, 0x7373), bx, 0x7710);  // bytes z, y, x from below
    const uint32_t cell = (t & 0x0F0F0Fu) * 0x01001001u, block = (t & 0xF0F0F0u) * 0x01001001u;
    const uint32_t word = ((block >> 13) & ~127u) | ((cell >> 21) & 127u);
    if (!in_range(p.check, word < (1u << (3 * (kStdLog2Base - kOccShift) - 5)), kChkOccupancy)) return true;
    return __funnelshift_r(__ldg(p.occ_blocks + word), 0u, cell >> 16) & 1u;
}

// Density at a sample (Sec. 1):
//   rho = g(h) W max(0, (B - w_d Dt - c)/(1 - c)),
// tiles stored centred (value - 1/2), so (B - w_d Dt - c) = Bc - w_d Dtc + k0;
// the records' decode bias is folded into k0 and w_off.  Returned as the two
// factors g W and max(0, .), so that a light march adds their product in one
// operation.  The three record loads are issued together so that one memory
// round trip serves the lookup; there is no branch on g: a sample outside the
// layer reads records (every index is in range) and multiplies them by g = 0,
// which costs less than a divergent branch in every lookup (with the index
// built by multiply-adds, 16-bit records: 64 views 12.23 -> 10.86 ms, 1920x1080
// x 8 steps 95.2 -> 88.0 us; FP32 90.3 -> 86.1 us).
struct Density {
    float gw, r;
    __device__ __forceinline__ float value() const { return __fmul_rn(gw, r); }
};
template <int VOL, typename T>
__device__ __forceinline__ Density density(const SceneParams &p, const T *__restrict__ base,
                                           const T *__restrict__ detail,
                                           const T *__restrict__ weather, const uint32_t c[8],
                                           int32_t hq) {
    constexpr bool FX = VOL == kStandardVolume;
    const bool has_detail = FX || (VOL == kAnyVolume && detail), has_weather = FX || (VOL == kAnyVolume && weather);
    const int lb = FX ? kStdLog2Base : p.log2_base, ld = FX ? kStdLog2Detail : p.log2_detail,
              lw = FX ? kStdLog2Weather : p.log2_weather;
    const float g = height_profile(p, hq);
    float cb[8], cd[8], cw[4];
    const uint32_t rb = rec3(p.base_mul, lb, c[kBX], c[kBY], c[kBZ]),
                   rd = rec3(p.detail_rec_mul, ld, c[kDX], c[kDY], c[kDZ]),
                   rw = rec2(p.weather_mul, lw, c[kWX], c[kWY]);
    if (!in_range(p.check,
                  rb < (1u << (3 * lb)) && (!has_detail || rd < (1u << (3 * ld))) &&
                      (!has_weather || rw < (1u << (2 * lw))),
                  kChkRecord))
        return {0.0f, 0.0f};
    const float ob = load_rec8(base, rb, cb);
    float od = 0.0f, ow = 0.0f;
    if (has_detail) od = load_rec8(detail, rd, cd);
    if (has_weather) ow = load_rec4(weather, rw, cw);
    const float2 fb = frac23(c[kBX] << lb, c[kBY] << lb), fd = frac23(c[kDX] << ld, c[kDY] << ld),
                 fz = frac23(c[kBZ] << lb, c[kDZ] << ld), fw = frac23(c[kWX] << lw, c[kWY] << lw);
    const float b = trilerp(cb, fb.x, fb.y, fz.x) + ob;
    float r = b + p.k0;
    if (has_detail) {
        const float dt = trilerp(cd, fd.x, fd.y, fz.y) + od;
        r = fmaf(-p.detail_w, dt, r);
    }
    r = fmaxf(r * p.inv_1mc, 0.0f);
    const float w = has_weather ? bilerp(cw, fw.x, fw.y) + ow + p.w_off : 1.0f;
    return {__fmul_rn(g, w), r};
}

// Coordinates of light sample j of a point.  In standard volumes the detail
// coordinates follow from the base ones by a multiply-add that also adds the
// offset's rest in detail units, so that the offset is as exact as if it were added
// to the point's own detail coordinates, which then need not be kept.
template <int VOL>
__device__ __forceinline__ void light_coords(const SceneParams &p, const uint32_t cs[kLatticeAxes], int j,
                                             uint32_t cj[kLatticeAxes]) {
#pragma unroll
    for (int a = 0; a < kLatticeAxes; ++a)
        cj[a] = VOL == kStandardVolume && a >= kDX && a <= kDZ ? mad32(cj[a - kDX], p.detail_mul, p.loff[j][a])
                                                               : mad32(cs[a], p.one, p.loff[j][a]);
}

// Staging of one lane's start coordinates and increments (lattice axes, then
// the height) into the warp's scratch.
template <int CH, int VOL>
__device__ __forceinline__ void stage_ray(WarpScratch<CH, VOL> &ws, unsigned lane,
                                          const uint32_t c[kLatticeAxes],
                                          const uint32_t e[kLatticeAxes], int32_t hq, int32_t eh) {
    ws.ray[lane][0] = make_uint4(c[kBX], c[kBY], c[kBZ], (uint32_t)hq);
    ws.ray[lane][1] = make_uint4(e[kBX], e[kBY], e[kBZ], (uint32_t)eh);
    if (VOL != kBaseVolume) ws.ray[lane][2] = make_uint4(c[kWX], c[kWY], e[kWX], e[kWY]);
    if (VOL == kAnyVolume) {
        ws.ray[lane][RayGroups<VOL>::value - 2] = make_uint4(c[kDX], c[kDY], c[kDZ], e[kDX]);
        ws.ray[lane][RayGroups<VOL>::value - 1] = make_uint4(e[kDY], e[kDZ], 0u, 0u);
    }
}

// Coordinates of view step i of ray `ow` of the warp from its staged start and
// increment (integer arithmetic: the same values as adding the increment step
// by step; in standard volumes the detail coordinates are the base ones shifted,
// as the ray setup derives them).  Returns the height.
template <int CH, int VOL>
__device__ __forceinline__ int32_t step_coords(const SceneParams &p, const WarpScratch<CH, VOL> &ws,
                                               unsigned ow, uint32_t i, uint32_t cs[kLatticeAxes]) {
    const uint4 s = ws.ray[ow][0], e = ws.ray[ow][1];
    cs[kBX] = s.x + i * e.x;
    cs[kBY] = s.y + i * e.y;
    cs[kBZ] = s.z + i * e.z;
    if (VOL == kBaseVolume) {
#pragma unroll
        for (int a = kDX; a < kLatticeAxes; ++a) cs[a] = 0u;  // no such tile
        return (int32_t)(s.w + i * e.w);
    }
    const uint4 w = ws.ray[ow][2];
    cs[kWX] = w.x + i * w.z;
    cs[kWY] = w.y + i * w.w;
    if (VOL == kStandardVolume) {
#pragma unroll
        for (int b = 0; b < 3; ++b)
            cs[kDX + b] = mad32(cs[b], p.detail_mul, p.detail_add);
    } else {
        const uint4 d = ws.ray[ow][RayGroups<VOL>::value - 2], f = ws.ray[ow][RayGroups<VOL>::value - 1];
        cs[kDX] = d.x + i * d.w;
        cs[kDY] = d.y + i * f.x;
        cs[kDZ] = d.z + i * f.y;
    }
    return (int32_t)(s.w + i * e.w);
}

// sigma D of one step, rounded the same way wherever it is recomputed
__device__ __forceinline__ float step_depth(float absorption, float rho, float D) {
    return __fmul_rn(__fmul_rn(absorption, rho), D);
}
// Weight of a step of depth sd behind the optical depth t0 (a6, Sec. 3.1).
__device__ __forceinline__ float step_weight(const SceneParams &p, float t0, float sd) {
    return p.integration == CLOUD_INTEGRATE_ANALYTIC ? expf(-t0) * -expm1f(-sd) : expf(-__fadd_rn(t0, sd)) * sd;
}
// Transmittance towards the sun of a light march's density sum (a5).
__device__ __forceinline__ float sun_transmittance(const SceneParams &p, float rho_sum) {
    return expf(-p.absorption * p.light_step * rho_sum);
}

// The march of one CTA pixel tile (4 warps, one pixel per lane).  View steps
// are processed in chunks of CH:
//   A  view densities and the early out (the optical depth does not depend on
//      the lighting): each lane marks which of its steps need a lookup (occupied
//      macro-cell), the warp shares those lookups out over all 32 lanes,
//      ViewBatch per lane at a time, and each lane then walks its own steps in
//      order for the optical depth and the early out;
//   B  the warp shares out every (step, lane) light march with density > 0
//      over all 32 lanes, so lanes whose own rays are empty, finished or
//      outside the layer do useful work; the lane that marches a pair also
//      evaluates its exponentials (the sun's transmittance and the step's
//      weight), which phase C would evaluate with only the lanes busy that have
//      density at that step;
//   C  each lane sums its steps in order.
// What bounds it is the L1's data path (83 % busy) where every ray has an offset
// of its own, and instruction issue (75 %) with the latency of the lookups
// elsewhere, so work moves to where most lanes are busy.  The exponentials in
// phase B, the list of light marches compacted from the list of lookups (instead of
// listed anew), rays staged in 16-byte groups and clear chunks left at once took
// 1920x1080 x 8 steps from 112.5 to 95.0 us, 1280x720 x 128 steps from 538 to 430
// us and 64 uneven views from 15.21 to 12.58 ms; with the steps described at the
// parts below, 128.7 to 91.4 us, 565 to 370 us and 15.5 to 10.2 ms a pass (other
// cameras).
// The arithmetic of every sample is the same as a per-lane march (a skipped
// lookup is one whose density is exactly 0).  Returns the number of density
// lookups this lane's ray performed in the method's sense (Sec. 1: one per
// view step walked, plus the light steps of each step with density).
template <typename T, int SHAPE, int VOL, int CH, int STEPS>
__device__ __forceinline__ unsigned march_tile(
    const SceneParams &p, const ViewParams &v, int tile_x, int tile_y, WarpScratch<CH, VOL> &ws,
    const T *__restrict__ base, const T *__restrict__ detail, const T *__restrict__ weather) {
    using S = TileShape<SHAPE>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int x = tile_x * (S::WX * S::CX) + (warp % S::CX) * S::WX + (lane % S::WX);
    const int y = tile_y * (S::WY * S::CY) + (warp / S::CX) * S::WY + (lane / S::WX);
    const bool in_image = lane < S::WX * S::WY && x < v.width && y < v.height;
    bool inside = in_image;
    const int nlight = p.light_steps;
    unsigned n_look = 0;
    uint32_t c[kLatticeAxes] = {}, e[kLatticeAxes] = {};
    int32_t hq = 0, eh = 0;
    float Df = 0.0f, phase = 0.0f;
    bool alive = false;
    const float xf = (float)x, yf = (float)y;
    if (inside) {
        // quick FP32 test for rays that cannot reach the layer.  It takes the 10-bit
        // high halves of the slopes only, so its d_z is off by up to 2^-10 of the
        // image plane's extent, more than the thresholds' 1e-4 margin: a ray that
        // grazes the layer near the far clip can be dropped (up to 37 pixels of a
        // 957x541 image, up to 0.1 in RGBA).
        const float qx = fmaf(yf, v.vyh[0], fmaf(xf, v.vxh[0], v.v00h[0]));
        const float qy = fmaf(yf, v.vyh[1], fmaf(xf, v.vxh[1], v.v00h[1]));
        const float qz = fmaf(yf, v.vyh[2], fmaf(xf, v.vxh[2], v.v00h[2]));
        const float dz = qz * rsqrt_norm(fmaf(qx, qx, fmaf(qy, qy, qz * qz)));
        if (dz < v.miss_below || dz > v.miss_above) inside = false;
    }
    if (inside) {
        // --- a1: pixel ray and layer clip (double-float) ---------------------
        // p(lambda) = o + lambda v with v unnormalised; t = lambda |v|.
        // x and y of v side by side (only multiplied on: lo may be a few ulp(hi)),
        // z as a normalised double-float.  The low halves of vx and vy carry up to
        // 2^-10 of the value, so their sum is one more exact addition.
        const float2 xf2 = both(xf), yf2 = both(yf);
        const df2 sx = two_sum2(make_float2(v.v00h[0], v.v00h[1]),
                                __fmul2_rn(xf2, make_float2(v.vxh[0], v.vxh[1])));  // exact products
        const df2 sy = two_sum2(sx.hi, __fmul2_rn(yf2, make_float2(v.vyh[0], v.vyh[1])));
        const df2 sl = two_sum2(sy.hi, __ffma2_rn(xf2, make_float2(v.vxl[0], v.vxl[1]),
                                                  __ffma2_rn(yf2, make_float2(v.vyl[0], v.vyl[1]),
                                                             make_float2(v.v00l[0], v.v00l[1]))));
        const df2 rxy = {sl.hi, __fadd2_rn(__fadd2_rn(sx.lo, sy.lo), sl.lo)};
        const df zx = two_sum(v.v00h[2], xf * v.vxh[2]), zy = two_sum(zx.hi, yf * v.vyh[2]);
        const df zl = two_sum(zy.hi, fmaf(xf, v.vxl[2], fmaf(yf, v.vyl[2], v.v00l[2])));
        const df rz = fast_two_sum(zl.hi, (zx.lo + zy.lo) + zl.lo);
        const df r[3] = {{rxy.hi.x, rxy.lo.x}, {rxy.hi.y, rxy.lo.y}, rz};
        // |v| in FP32 for the step length and the phase angle; the far clip
        // lambda_max = t_max / |v| in double-float only where it can decide the
        // layer exit (an FP32 test with a 1e-5 margin, far above its error)
        const float n2f = fmaf(r[0].hi, r[0].hi, fmaf(r[1].hi, r[1].hi, r[2].hi * r[2].hi));
        const float rnf = rsqrt_norm(n2f);  // 1 / |v|
        const auto lam_max = [&]() {
            const df n2 = df_add(df_add(df_mul(r[0], r[0]), df_mul(r[1], r[1])), df_mul(r[2], r[2]));
            return df_mul({v.tmax_h, v.tmax_l}, df_rsqrt(n2));
        };
        df lam0 = {0.0f, 0.0f}, lam1;
        if (fabsf(r[2].hi) * rnf < 1e-8f) {
            alive = v.zlo_h <= 0.0f && v.zhi_h >= 0.0f;  // the camera is in the layer
            lam1 = lam_max();
        } else {
            // the sign of the ray's z decides which layer boundary comes first
            const df inv = df_recip(r[2]);
            const bool up = r[2].hi > 0.0f;
            const df2 l = df2_mul_raw({up ? make_float2(v.zlo_h, v.zhi_h) : make_float2(v.zhi_h, v.zlo_h),
                                       up ? make_float2(v.zlo_l, v.zhi_l) : make_float2(v.zhi_l, v.zlo_l)},
                                      {both(inv.hi), both(inv.lo)});
            const df2 ln = fast_two_sum2(l.hi, l.lo);
            lam0 = {ln.hi.x, ln.lo.x};
            lam1 = {ln.hi.y, ln.lo.y};
            if (!(lam0.hi > 0.0f)) lam0 = {0.0f, 0.0f};
            if (!(lam1.hi < v.tmax_h * rnf * (1.0f - 1e-5f))) lam1 = df_min(lam1, lam_max());
            alive = df_gt(lam1, lam0);
        }
        if (alive) {
            // --- a2: jittered start offset (Sec. 3.2) ---------------------------
            const df D = df_mul(df_add(lam1, df_neg(lam0)), {v.invn_h, v.invn_l});
            float u = v.u_frame;
            if (u < 0.0f)
                u = (float)(pcg_hash((uint32_t)x ^ pcg_hash((uint32_t)y ^ v.jitter_hash)) >> 8) *
                    (1.0f / 16777216.0f);
            const df lam_s = df_add(lam0, df_mulf(D, u));
            // start and step of every axis, side by side: (lambda v) scaled to the
            // axis' units and rounded to fixed point, the camera's own coordinate
            // added as an integer.  The setup is bound by issue (26 us of the 83 us of
            // 1920x1080 x 8 steps); packed pairs take 83.4 to 81.4 us (FP16 84.8 to 81.1).
            const df2 ld = {make_float2(lam_s.hi, D.hi), make_float2(lam_s.lo, D.lo)};
            df2 pos[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) pos[k] = df2_mul_raw(ld, {both(r[k].hi), both(r[k].lo)});
            const bool wide = p.wide != 0;
#pragma unroll
            for (int a = 0; VOL != kConstantVolume && a < kLatticeAxes; ++a) {
                if (a >= kDX && a <= kDZ && p.detail_shift >= 0) {
                    // same origin, period 2^-shift of the base tile: exact shift
                    c[a] = mad32(c[a - kDX], p.detail_mul, p.detail_add);
                    e[a] = e[a - kDX] * p.detail_mul;
                    continue;
                }
                df2 q = df2_mul_raw(pos[a < 6 ? a % 3 : a - 6], {p.kfix_h[a], p.kfix_l[a]});
                q.lo.x += v.org_rest[a];
                const uint2 u = df2_to_u32(q, wide);
                c[a] = u.x + v.org[a];
                e[a] = u.y;
            }
            // height above the layer bottom, in 2^-16 m
            df2 qh = {__fmul2_rn(pos[2].hi, both(65536.0f)), __fmul2_rn(pos[2].lo, both(65536.0f))};
            qh.lo.x += v.org_h_rest;
            const uint2 uh = df2_to_u32(qh, false);
            hq = (int32_t)(uh.x + v.org_h);
            eh = (int32_t)uh.y;
            const float vlen = n2f * rnf;
            Df = D.hi * vlen;
            // --- a5: phase function, hoisted per ray ----------------------------
            // p_HG(mu) = (1 - g^2) / (4 pi) * (1 + g^2 - 2 g mu)^(-3/2)
            const float mu = (r[0].hi * p.sun[0] + r[1].hi * p.sun[1] + r[2].hi * p.sun[2]) * rnf;
            const float q = rsqrt_norm(fmaf(-2.0f * p.hg_g, mu, fmaf(p.hg_g, p.hg_g, 1.0f)));
            phase = p.hg_norm * q * q * q;
        }
    }
    if (VOL != kConstantVolume) {
        stage_ray(ws, lane, c, e, hq, eh);
        ws.length[lane] = Df;
        __syncwarp();
    }
    const unsigned lt_mask = (1u << lane) - 1u;
    float tau = 0.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
    if (VOL == kConstantVolume && alive) {
        // Constant density: nothing to look up and the same light march at every step,
        // so each lane walks its own steps (one exponential a step bounds it).  The
        // lists below pay only where lanes lack work: through them, 1280x720 x 64 steps
        // take 370 us (283 with the light samples unrolled), this way 24.6; 12 views of
        // up to 1280x720 x 128 steps 2.59 ms and 0.24.
        float rho_sum = 0.0f;
        for (int j = 0; j < nlight; ++j) rho_sum = __fadd_rn(rho_sum, p.rho0);
        const float sd = step_depth(p.absorption, p.rho0, Df), sun_t = sun_transmittance(p, rho_sum) * phase;
        const float lr = fmaf(p.sun_rad[0], sun_t, p.ambient[0]), lg = fmaf(p.sun_rad[1], sun_t, p.ambient[1]),
                    lb = fmaf(p.sun_rad[2], sun_t, p.ambient[2]);
        int i = 0;
        do {
            ++i;
            if (p.rho0 > 0.0f) {
                const float wgt = step_weight(p, tau, sd);
                tau = __fadd_rn(tau, sd);
                cr = fmaf(wgt, lr, cr);
                cg = fmaf(wgt, lg, cg);
                cb = fmaf(wgt, lb, cb);
            }
        } while (i < v.steps && !(tau >= p.tau_max));
        n_look = i * (p.rho0 > 0.0f ? 1 + nlight : 1);
    }
    constexpr int kScan = 16;  // steps per read of the grid in a march of many chunks
    uint32_t occ_bits = 0;
    int scanned = 0;
    for (int i0 = 0; VOL != kConstantVolume && i0 < (STEPS == kOneChunk ? 1 : v.steps) && __any_sync(kFull, alive);
         i0 += CH) {
        const int nst = min(CH, v.steps - i0);
        // --- A1: which of this lane's CH steps need a density lookup: those in an
        //     occupied macro-cell of the occupancy grid (the words of all steps are
        //     loaded together, by every lane: the coordinates of a finished ray and
        //     of steps past the last wrap into the grid too).  A step outside the
        //     layer, possible only by rounding at the ends of the clipped ray, is
        //     left to the lookup.
        // --- A2: the warp's list of the (step, lane) lookups, to be shared out over
        //     the lanes so that their loads overlap (a3) ---------------------------
        const bool grid = p.occ;
        uint32_t need = 0;
        unsigned nq = 0;
        const auto list = [&](int k, bool nd) {
            const unsigned m = __ballot_sync(kFull, nd);
            const unsigned slot = nq + __popc(m & lt_mask);
            if (nd && in_range(p.check, slot < CH * 32u, kChkWork)) ws.pairs[slot] = (uint16_t)((k << 5) | lane);
            nq += __popc(m);
        };
        if (STEPS == kManyChunks || (STEPS == kAnySteps && v.steps > CH)) {
            // Long marches are mostly clear air, where the chain of grid reads is
            // what takes time: two chunks' worth of steps per read, and one vote
            // passes over them (or over one chunk) before any list is built.
            // 1280x720 x 128 steps 494 -> 485 us, 64 views 10.25 -> 9.97 ms (kScan
            // 32: 64 views 10.15 ms); the vote alone 378 -> 366 us, another view.
            if (i0 >= scanned) {
                scanned = i0 + kScan;
                occ_bits = ~0u;
                if (grid) {
                    const uint4 s = ws.ray[lane][0], d = ws.ray[lane][1];
                    uint32_t bx = s.x + i0 * d.x, by = s.y + i0 * d.y, bz = s.z + i0 * d.z;
                    bool o[kScan];
#pragma unroll
                    for (int k = 0; k < kScan; ++k) {
                        o[k] = occupied<VOL>(p, bx, by, bz);
                        bx = mad32(d.x, p.one, bx);
                        by = mad32(d.y, p.one, by);
                        bz = mad32(d.z, p.one, bz);
                    }
                    occ_bits = 0;
#pragma unroll
                    for (int k = 0; k < kScan; ++k) occ_bits |= o[k] ? 1u << k : 0u;
                }
                const int left = v.steps - i0;
                if (left < 32) occ_bits &= (1u << left) - 1u;
                if (!__any_sync(kFull, alive && occ_bits)) {
                    n_look += alive ? min(kScan, left) : 0;
                    i0 += kScan - CH;
                    continue;
                }
            }
            need = alive ? occ_bits & ((1u << CH) - 1u) : 0u;
            occ_bits >>= CH;
            if (!__any_sync(kFull, need)) {
                n_look += alive ? nst : 0;
                continue;
            }
#pragma unroll
            for (int k = 0; k < CH; ++k) list(k, (need >> k) & 1u);
        } else {
            // a march of one chunk: hardly ever clear, so straight to the list
            bool o[CH];
            if (grid) {
                const uint4 s = ws.ray[lane][0], d = ws.ray[lane][1];
                uint32_t bx = s.x + i0 * d.x, by = s.y + i0 * d.y, bz = s.z + i0 * d.z;
                const auto read = [&](const auto &bit) {
#pragma unroll
                    for (int k = 0; k < CH; ++k) {
                        o[k] = bit(bx, by, bz);
                        bx = mad32(d.x, p.one, bx);
                        by = mad32(d.y, p.one, by);
                        bz = mad32(d.z, p.one, bz);
                    }
                };
                if (VOL == kStandardVolume && STEPS == kOneChunk && v.u_frame < 0.0f && p.occ_blocks)
                    read([&](uint32_t x, uint32_t y, uint32_t z) { return occupied_blocks(p, x, y, z); });
                else
                    read([&](uint32_t x, uint32_t y, uint32_t z) { return occupied<VOL>(p, x, y, z); });
            } else {
#pragma unroll
                for (int k = 0; k < CH; ++k) o[k] = true;
            }
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                const bool nd = o[k] && alive && k < nst;
                if (nd) need |= 1u << k;
                list(k, nd);
            }
        }
        if (nq == 0) {  // clear air, warp-wide: no optical depth, no early out
            n_look += alive ? nst : 0;
            continue;
        }
        __syncwarp();
        constexpr int kViewBatch = ViewBatch<T, CH>::value;
        for (unsigned q = lane; q < nq; q += 32 * kViewBatch) {
            // a lane without a further lookup repeats its first (same value, same entry)
            unsigned pr[kViewBatch];
            float rho[kViewBatch];
#pragma unroll
            for (int b = 0; b < kViewBatch; ++b) pr[b] = ws.pairs[q + 32 * b < nq ? q + 32 * b : q];
            bool ok = in_range(p.check, q < CH * 32u, kChkWork);
#pragma unroll
            for (int b = 0; b < kViewBatch; ++b) ok = ok && in_range(p.check, (pr[b] >> 5) < (unsigned)CH, kChkWork);
            if (!ok) continue;
#pragma unroll
            for (int b = 0; b < kViewBatch; ++b) {
                uint32_t cs[kLatticeAxes];
                const int32_t hs = step_coords(p, ws, pr[b] & 31u, (uint32_t)i0 + (pr[b] >> 5), cs);
                rho[b] = density<VOL>(p, base, detail, weather, cs, hs).value();
            }
#pragma unroll
            for (int b = 0; b < kViewBatch; ++b) ws.rho[pr[b] >> 5][pr[b] & 31u] = rho[b];
        }
        __syncwarp();
        // --- A3: each lane walks its steps in order: optical depth (kept per step
        //     with density for phase B) and the early out (a7, Sec. 1: stop once
        //     alpha is ~1) ------------------------------------------------------
        uint32_t act = 0;
        if (alive) {
            int nA = 0;
            const float Ds = ws.length[lane];
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                if (k >= nst) break;
                const float rho = ((need >> k) & 1u) ? ws.rho[k][lane] : 0.0f;
                nA = k + 1;
                if (rho > 0.0f) {
                    act |= 1u << k;
                    ws.aux[k][lane] = tau;
                    tau = __fadd_rn(tau, step_depth(p.absorption, rho, Ds));
                }
                if (tau >= p.tau_max) {
                    alive = false;
                    break;
                }
            }
            n_look += nA + nlight * __popc(act);
        }
        // --- B: light marches shared out over the warp (a4, Sec. 1): the list of
        //     lookups shrinks, in place and in order, to the pairs with density
        //     before their ray's early out -------------------------------------
        unsigned npairs = 0;
        for (unsigned q0 = 0; q0 < nq; q0 += 32) {
            const unsigned q = q0 + lane;
            const unsigned pr = q < nq ? ws.pairs[q] : 0u;
            const uint32_t owner_act = __shfl_sync(kFull, act, pr & 31u);
            const bool keep = q < nq && ((owner_act >> (pr >> 5)) & 1u);
            const unsigned m = __ballot_sync(kFull, keep);
            const unsigned slot = npairs + __popc(m & lt_mask);
            if (keep && in_range(p.check, slot <= q && slot < CH * 32u, kChkWork))
                ws.pairs[slot] = (uint16_t)pr;
            npairs += __popc(m);
        }
        if (npairs == 0) continue;  // no density in this chunk, warp-wide
        __syncwarp();
        for (unsigned q0 = 0; q0 < npairs; q0 += 32) {
            const unsigned q = q0 + lane;
            const unsigned pr = ws.pairs[q < npairs ? q : q0], k = pr >> 5, ow = pr & 31u;
            const bool ok = q < npairs && in_range(p.check, q < CH * 32u && k < (unsigned)CH, kChkWork);
            uint32_t cs[kLatticeAxes];
            const int32_t hs = step_coords(p, ws, ow, (uint32_t)(i0 + (int)k), cs);
            // light samples rise towards the sun: those that lie above the layer for
            // every lane are left out (their density is 0)
            const int32_t h_least = __reduce_min_sync(kFull, hs);
            int nl = nlight;
            while (nl > 0 && h_least + p.lh[nl - 1] >= p.h_top) --nl;
            // A lane without a pair leaves here with FP32 records, whose 80 bytes a
            // lane and sample fill the L1's data path (1920x1080 x 8 steps 115.0 ->
            // 112.0 us, 1280x720 x 128 steps 485 -> 477 us); with 16-bit ones it
            // repeats the first lane's, which spares a divergent loop (64 views 11.3
            // -> 10.9 ms).
            if (sizeof(T) == 4 && !ok) continue;
            float rho_sum = 0.0f;
            constexpr int kU = LightUnroll<T, VOL>::value;
#pragma unroll kU
            for (int j = 0; j < nl; ++j) {
                uint32_t cj[kLatticeAxes];
                light_coords<VOL>(p, cs, j, cj);
                const Density d = density<VOL>(p, base, detail, weather, cj, hs + p.lh[j]);
                rho_sum = fmaf(d.gw, d.r, rho_sum);
            }
            if (!ok) continue;
            // --- a5, a6: transmittance towards the sun and the weight of the
            //     per-step integral (Sec. 3.1) --------------------------------
            const float sd = step_depth(p.absorption, ws.rho[k][ow], ws.length[ow]);
            const float t0 = ws.aux[k][ow];
            ws.rho[k][ow] = step_weight(p, t0, sd);
            ws.aux[k][ow] = sun_transmittance(p, rho_sum);
        }
        __syncwarp();
        // --- C: in-scattered light, summed in step order -------------------------
        while (act) {
            const int k = __ffs(act) - 1;
            act &= act - 1u;
            const float wgt = ws.rho[k][lane], sun_t = ws.aux[k][lane] * phase;
            cr = fmaf(wgt, fmaf(p.sun_rad[0], sun_t, p.ambient[0]), cr);
            cg = fmaf(wgt, fmaf(p.sun_rad[1], sun_t, p.ambient[1]), cg);
            cb = fmaf(wgt, fmaf(p.sun_rad[2], sun_t, p.ambient[2]), cb);
        }
        __syncwarp();
    }
    // --- a8: premultiplied RGBA, one 16-byte store ------------------------------
    if (in_image && in_range(p.check, x >= 0 && y >= 0, kChkPixel))
        v.out[(size_t)y * v.width + x] = make_float4(cr, cg, cb, tau > 0.0f ? -expm1f(-tau) : 0.0f);
    return n_look;
}

// Warp-aggregated add of the lookup count (counting launches only).
__device__ __forceinline__ void count_lookups(unsigned long long *counter, unsigned long long n) {
    if (!counter) return;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) n += __shfl_down_sync(kFull, n, s);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(counter, n);
}

// Host side (render.cu).
int build_scene(const cloud_volume *vol, const cloud_params *prm, int light_steps, int integration,
                SceneParams *p);
int build_view(const cloud_volume *vol, const cloud_params *prm, const cloud_camera *cam, int width,
               int height, int steps, int jitter_frame, float *out, int shape, ViewParams *v);
// Pixel tiles of a view in a launch of the given tile shape.
inline int tile_count(const ViewParams &v, int shape) {
    int tw, th;
    tile_dims(shape, &tw, &th);
    return v.tiles_x * ((v.height + th - 1) / th);
}
// The autotuned launch configuration for (storage precision, light steps).
int tuned_config(int precision, int light_steps);
// Raymarch of one view with the given configuration (render.cu); the
// per-chunk-size kernels and their dispatch are instantiated in
// march{8,16}_{view,batch}.cu.
int launch_march(const SceneParams &p, const ViewParams &v, const cloud_volume *vol,
                 unsigned long long *counter, int config, cudaStream_t s);
template <int CH>
void launch_march_ch(const SceneParams &p, const ViewParams &v, const cloud_volume *vol,
                     unsigned long long *counter, int shape, cudaStream_t s);
// The same with the small shapes (4, 5, 6) and 8 view steps a chunk (march_small.cu).
void launch_march_small(const SceneParams &p, const ViewParams &v, const cloud_volume *vol,
                        unsigned long long *counter, int shape, cudaStream_t s);
template <int CH>
const void *batch_kernel_ch(int precision, int kind, int shape);

}  // namespace cloudvol
