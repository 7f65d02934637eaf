// Internal declarations shared by the libstitch translation units (device structs, planner
// output, launch helpers).  Nothing here is part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "stitch.h"

#define MAXL STITCH_MAX_LEVELS
#define MAXC STITCH_MAX_CAMERAS

// Half-open rectangle of one pyramid level, in that level's canvas coordinates.
struct Rect {
    int x0, x1, y0, y1;
    __host__ __device__ int w() const { return x1 - x0; }
    __host__ __device__ int h() const { return y1 - y0; }
    __host__ __device__ bool empty() const { return x1 <= x0 || y1 <= y0; }
    __host__ __device__ bool contains(int x, int y) const { return x >= x0 && x < x1 && y >= y0 && y < y1; }
    __host__ __device__ long long area() const { return empty() ? 0 : (long long)w() * h(); }
};

// Per-camera descriptor, resident in device memory for the life of a rig.
struct CamDev {
    double A[9];     // canvas -> camera homography, a33 = +1 or -1
    int W, H;        // source frame size
    float gain;
    int visible;     // 0 when the camera's footprint misses the canvas
    Rect V;          // level-0 bounding box of the validity region (empty when !visible)
    Rect Om[MAXL];   // Omega^l: region on which the camera's pyramid is evaluated
    Rect Z[MAXL];    // Z^l: region where the camera's weight pyramid can be non-zero
    // plain path buffers
    float4* G[MAXL];   // Gaussian pyramid (r, g, b, weight) on Om[l], row pitch Om[l].w()
    // fused path buffers
    void* FG[MAXL];    // Gaussian pyramid (r, g, b, weight) on Om[l] for l >= 1 (FP32 or FP16)
};

// Rig-wide sizes passed by value to kernels.
struct RigGeom {
    int ncam, levels;
    int seam;  // level-0 weights: 0 feather, 1 seam owner masks
    int cyl;   // canvas: 0 planar (homographies), 1 cylindrical (focal length cf, centre ccx, ccy)
    double cf, ccx, ccy;
    int nx[MAXL], ny[MAXL];  // canvas size of every level (nx[l+1] = ceil(nx[l] / 2))
};

// Device frame pointers of one call, passed by value.
struct FramePtrs {
    const uint8_t* p[MAXC];
    long long pitch[MAXC];
};

// Output descriptor of one call.
struct OutDesc {
    void* ptr;
    long long pitch;  // bytes
    int is_float;
};

// ------------------------------------------------------------------------------------------------
// debug build (STITCH_DEBUG): index checks that record the first failure in a device word of the
// translation unit and let the caller skip the access (no trap, so the context stays usable), and
// guard bands around every rig allocation.  Release builds compile the checks to `true`.

#ifdef STITCH_DEBUG
constexpr bool kStitchDebug = true;
#define STITCH_DCHECK(cond, code, val) ((cond) ? true : (stitch_dcheck_fail((code), (long long)(val)), false))
#else
constexpr bool kStitchDebug = false;
#define STITCH_DCHECK(cond, code, val) true
#endif

// Guard band around each rig allocation in the debug build: this many bytes before and after,
// filled with the quiet-NaN word kGuardWord.
constexpr size_t kGuardBytes = 256;
constexpr uint32_t kGuardWord = 0x7FC0DEADu;

// ------------------------------------------------------------------------------------------------
// Programmatic dependent launch: the kernels of a call's sequence are launched so that the next one
// may start as soon as every block of the previous one has started (pdl_trigger), and each of their
// blocks waits for the previous one's completion (pdl_wait) before its first access to anything but
// the rig's constant tables, and before it returns.  As that kernel has waited for the one before
// it, all earlier work of the stream is complete behind pdl_wait.  Without the launch attribute both
// are no-ops.  The read-only path (__ldg, and loads through `const __restrict__` pointers, which the
// compiler may turn into it) is for the rig's constant tables: its loads are promised not to change while
// the kernel runs, which begins before pdl_wait, and the compiler may move them above it.  What earlier
// work wrote is read by plain loads, __ldca or __ldcg, through pointers without `__restrict__`: the
// previous kernels' results, and the frames, whose producer may be a kernel that triggers early itself.

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// stream_launch: with the attribute (early) or without it.  The attribute relaxes a launch's dependency on
// the stream's previous kernel only, so a call on the caller's stream begins with it whatever the caller
// queued before.  Where the library itself has just queued an event wait or a copy, the first launch goes
// without: there is no kernel for it to overlap with.
template <typename... P, typename... A>
inline void stream_launch(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
inline void pdl_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A&... args) {
    stream_launch(true, kernel, grid, block, smem, s, args...);
}

// ------------------------------------------------------------------------------------------------
// small device helpers

// reflect-101 border folding on a grid of n samples: ... 2 1 | 0 1 2 ... n-1 | n-2 n-3 ...
__host__ __device__ __forceinline__ int fold101(int i, int n) {
    if (i >= 0 && i < n) return i;
    if (n == 1) return 0;
    const int period = 2 * n - 2;
    int r = i % period;
    if (r < 0) r += period;
    return r < n ? r : period - r;
}

// Accurate per-tile parameterisation of a homography.  With (X, Y) the tile anchor and
// U0 = round(u(X, Y)), the offset u - U0 = (pu0 + pu1 dx + pu2 dy) / (q0 + q1 dx + q2 dy) is
// small, so single precision keeps ~1e-5 px accuracy anywhere on a 24000-px canvas; the
// coefficients are formed in double precision once per tile.
struct TileMap {
    int U0, V0;
    float pu0, pu1, pu2, pv0, pv1, pv2, q0, q1, q2;
};

__host__ __device__ __forceinline__ TileMap make_tile_map(const double* A, int X, int Y) {
    const double x = (double)X, y = (double)Y;
    const double n0 = A[0] * x + A[1] * y + A[2];
    const double m0 = A[3] * x + A[4] * y + A[5];
    const double d0 = A[6] * x + A[7] * y + A[8];
    double u0 = n0 / d0, v0 = m0 / d0;
    u0 = fmin(fmax(u0, -1.0e8), 1.0e8);
    v0 = fmin(fmax(v0, -1.0e8), 1.0e8);
    const double U = rint(u0), V = rint(v0);
    TileMap t;
    t.U0 = (int)U;
    t.V0 = (int)V;
    t.pu0 = (float)(n0 - U * d0);
    t.pu1 = (float)(A[0] - U * A[6]);
    t.pu2 = (float)(A[1] - U * A[7]);
    t.pv0 = (float)(m0 - V * d0);
    t.pv1 = (float)(A[3] - V * A[6]);
    t.pv2 = (float)(A[4] - V * A[7]);
    t.q0 = (float)d0;
    t.q1 = (float)A[6];
    t.q2 = (float)A[7];
    return t;
}

// Source position of canvas point (anchor + (dx, dy)) as integer part + fraction in [0, 1).
struct SrcPos {
    int iu, iv;
    float fu, fv;
    float den;
};

__device__ __forceinline__ SrcPos map_point(const TileMap& t, float dx, float dy) {
    SrcPos s;
    s.den = fmaf(t.q2, dy, fmaf(t.q1, dx, t.q0));
    // approximate reciprocal (2 ulp): the offsets it scales are below ~100 px, so the error in
    // the source position stays near 1e-5 px
    const float rden = __fdividef(1.0f, s.den);
    float ru = fmaf(t.pu2, dy, fmaf(t.pu1, dx, t.pu0)) * rden;
    float rv = fmaf(t.pv2, dy, fmaf(t.pv1, dx, t.pv0)) * rden;
    ru = fminf(fmaxf(ru, -1.0e7f), 1.0e7f);
    rv = fminf(fmaxf(rv, -1.0e7f), 1.0e7f);
    const float flu = floorf(ru), flv = floorf(rv);
    s.iu = t.U0 + (int)flu;
    s.iv = t.V0 + (int)flv;
    s.fu = ru - flu;
    s.fv = rv - flv;
    return s;
}

// Raw feather weight: distance (source px) to the nearest border of the validity rectangle
// [-0.5, W-0.5) x [-0.5, H-0.5), zero outside it or behind the camera.
__device__ __forceinline__ float feather_weight(const SrcPos& s, int W, int H) {
    if (!(s.den > 0.0f)) return 0.0f;
    const bool okx = (s.iu >= 0 || (s.iu == -1 && s.fu >= 0.5f)) && (s.iu <= W - 2 || (s.iu == W - 1 && s.fu < 0.5f));
    const bool oky = (s.iv >= 0 || (s.iv == -1 && s.fv >= 0.5f)) && (s.iv <= H - 2 || (s.iv == H - 1 && s.fv < 0.5f));
    if (!(okx && oky)) return 0.0f;
    const float u = (float)s.iu + s.fu, v = (float)s.iv + s.fv;
    float m = fminf(fminf(u + 0.5f, v + 0.5f), fminf(((float)W - 0.5f) - u, ((float)H - 0.5f) - v));
    return fmaxf(m, 0.0f);
}

// The canvas point (x, y) as the vector the camera matrix A acts on: (x, y, 1) on the planar
// canvas; on the cylindrical canvas the ray (sin t, (y - cy)/f, cos t) with t = (x - cx)/f.
__host__ __device__ inline void canvas_ray(const RigGeom& g, double x, double y, double r[3]) {
    if (g.cyl) {
        const double t = (x - g.ccx) / g.cf;
        r[0] = sin(t);
        r[1] = (y - g.ccy) / g.cf;
        r[2] = cos(t);
    } else {
        r[0] = x;
        r[1] = y;
        r[2] = 1.0;
    }
}

// Source point of canvas point (x, y) in camera c, FP64: (u, v) and w (> 0 in front).
__host__ __device__ inline double source_point64(const CamDev& c, const RigGeom& g, double x, double y, double* u,
                                                 double* v) {
    double r[3];
    canvas_ray(g, x, y, r);
    const double w = c.A[6] * r[0] + c.A[7] * r[1] + c.A[8] * r[2];
    *u = (c.A[0] * r[0] + c.A[1] * r[1] + c.A[2] * r[2]) / w;
    *v = (c.A[3] * r[0] + c.A[4] * r[1] + c.A[5] * r[2]) / w;
    return w;
}

// S2 feather weight of camera c at canvas point (x, y) in FP64: distance from the source point to
// the border of the pixel-edge rectangle [-0.5, W-0.5) x [-0.5, H-0.5), 0 outside it or behind
// the camera.
__host__ __device__ inline double feather_weight64(const CamDev& c, const RigGeom& g, double x, double y) {
    double u, v;
    const double w = source_point64(c, g, x, y, &u, &v);
    if (!(w > 0.0)) return 0.0;
    if (!(u >= -0.5 && u < c.W - 0.5 && v >= -0.5 && v < c.H - 0.5)) return 0.0;
    const double m = fmin(fmin(u + 0.5, v + 0.5), fmin(c.W - 0.5 - u, c.H - 0.5 - v));
    return m > 0.0 ? m : 0.0;
}

// SrcPos of canvas pixel (x, y) in camera c from the FP64 map (see map_pos64).
__device__ inline SrcPos map_point64(const CamDev& c, const RigGeom& g, int x, int y) {
    double u, v;
    const double w = source_point64(c, g, (double)x, (double)y, &u, &v);
    u = fmin(fmax(u, -1.0e7), 1.0e7);
    v = fmin(fmax(v, -1.0e7), 1.0e7);
    const double fu = floor(u), fv = floor(v);
    SrcPos s;
    s.iu = (int)fu;
    s.iv = (int)fv;
    s.fu = (float)(u - fu);
    s.fv = (float)(v - fv);
    s.den = w > 0.0 ? 1.0f : -1.0f;
    return s;
}

// Seam owner of canvas point (x, y) among n cameras given in ascending camera order by cam_at(k)
// (which must include every camera whose validity box contains the point): the first position k
// whose feather weight is > 0 and >= (1 - 1e-9) times the largest, -1 when no weight is > 0.
// Decided in FP64, so that the binary masks do not depend on the FP32 tile anchoring.
template <class CamAt>
__device__ inline int seam_owner(const RigGeom& g, int n, const CamAt& cam_at, int x, int y) {
    double wmax = 0.0;
    for (int k = 0; k < n; ++k) {
        const CamDev& c = cam_at(k);
        if (c.V.contains(x, y)) wmax = fmax(wmax, feather_weight64(c, g, (double)x, (double)y));
    }
    if (!(wmax > 0.0)) return -1;
    for (int k = 0; k < n; ++k) {
        const CamDev& c = cam_at(k);
        if (!c.V.contains(x, y)) continue;
        const double w = feather_weight64(c, g, (double)x, (double)y);
        if (w > 0.0 && w >= (1.0 - 1e-9) * wmax) return k;
    }
    return -1;
}

// Clamped texel coordinates and fractions of a bilinear sample.
struct Tap {
    int i0, i1, j0, j1;
    float fx, fy;
};

__device__ __forceinline__ Tap clamp_tap(const SrcPos& s, int W, int H) {
    Tap t;
    if (s.iu < 0) { t.i0 = 0; t.fx = 0.0f; }
    else if (s.iu >= W - 1) { t.i0 = W - 1; t.fx = 0.0f; }
    else { t.i0 = s.iu; t.fx = s.fu; }
    if (s.iv < 0) { t.j0 = 0; t.fy = 0.0f; }
    else if (s.iv >= H - 1) { t.j0 = H - 1; t.fy = 0.0f; }
    else { t.j0 = s.iv; t.fy = s.fv; }
    t.i1 = min(t.i0 + 1, W - 1);
    t.j1 = min(t.j0 + 1, H - 1);
    return t;
}

// packed single-precision pairs (f32x2: two IEEE binary32 lanes, each rounded exactly as the
// scalar operation), used where the path computes on pairs of channels

__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b as a + (-1) b: the product is exact, so this is the rounded difference, bit for bit
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2add_rm(float2 a, float2 b) { return __fadd2_rd(a, b); }  // toward -infinity

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

// Byte j of w as a float, exactly: the bits 0x4B000000 | b encode 2^23 + b.
__device__ __forceinline__ float byte_f(uint32_t w, uint32_t j) {
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440u | j)) - 8388608.0f;
}

// 2^23 + byte j of w, as a float (exact)
__device__ __forceinline__ float byte_f23(uint32_t w, uint32_t j) {
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440u | j));
}

// The four texels of a bilinear sample (R, G, B in bytes 0 to 2 of a word), a and b the addresses of the
// left one in both rows, i0 its column; the right ones repeat the left ones in the last column.  Two
// neighbouring texels are 6 bytes at any offset: where base and pitch are multiples of 4 bytes (words)
// and three words from the first one's on lie in the row, they are two or three aligned loads and a
// funnel shift instead of six byte loads.
struct Texels {
    uint32_t t00, t01, t10, t11;
};
__device__ __forceinline__ Texels load_texels(const uint8_t* a, const uint8_t* b, int i0, int W,
                                              bool words) {
    Texels o;
    const int off = (3 * i0) & 3;
    if (words && 3 * i0 - off + 12 <= 3 * W) {
        const uint32_t* wa = reinterpret_cast<const uint32_t*>(a - off);
        const uint32_t* wb = reinterpret_cast<const uint32_t*>(b - off);
        const uint32_t a0 = __ldca(wa), a1 = __ldca(wa + 1), b0 = __ldca(wb), b1 = __ldca(wb + 1);
        uint32_t a2 = 0u, b2 = 0u;
        if (off == 3) {
            a2 = __ldca(wa + 2);
            b2 = __ldca(wb + 2);
        }
        o.t00 = __funnelshift_r(a0, a1, 8 * off);
        o.t01 = __byte_perm(o.t00, __funnelshift_r(a1, a2, 8 * off), 0x0543);
        o.t10 = __funnelshift_r(b0, b1, 8 * off);
        o.t11 = __byte_perm(o.t10, __funnelshift_r(b1, b2, 8 * off), 0x0543);
    } else {
        const int di = i0 + 1 < W ? 3 : 0;
        auto texel = [](const uint8_t* p) {
            return (uint32_t)__ldca(p) | (uint32_t)__ldca(p + 1) << 8 | (uint32_t)__ldca(p + 2) << 16;
        };
        o.t00 = texel(a);
        o.t01 = texel(a + di);
        o.t10 = texel(b);
        o.t11 = texel(b + di);
    }
    return o;
}
__device__ __forceinline__ bool word_aligned(const uint8_t* px, long long pitch) {
    return (((uint32_t)reinterpret_cast<uintptr_t>(px) | (uint32_t)pitch) & 3u) == 0u;
}

// Exact float of an 8-bit value with one integer OR and one add: the bits 0x4B000000 | b encode
// 2^23 + b, so subtracting 2^23 leaves b (IEEE-754 single precision, no rounding).
__device__ __forceinline__ float u8_to_f(uint32_t b) { return __int_as_float(0x4B000000u | b) - 8388608.0f; }

// Bilinear RGB sample of an 8-bit frame of width W, scaled by `scale` (= gain / 255).  WORDS: taps from word
// loads (load_texels) where they are possible, otherwise byte by byte.
template <bool WORDS = true>
__device__ __forceinline__ float3 bilinear_rgb(const uint8_t* px, long long pitch, int W, const Tap& t,
                                               float scale) {
    const uint8_t *r0 = px + (long long)t.j0 * pitch, *r1 = px + (long long)t.j1 * pitch;
    Texels q{};
    if (WORDS) q = load_texels(r0 + 3 * t.i0, r1 + 3 * t.i0, t.i0, W, word_aligned(px, pitch));
    float3 o;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float p00 = WORDS ? byte_f(q.t00, c) : u8_to_f(__ldca(r0 + 3 * t.i0 + c));
        const float p01 = WORDS ? byte_f(q.t01, c) : u8_to_f(__ldca(r0 + 3 * t.i1 + c));
        const float p10 = WORDS ? byte_f(q.t10, c) : u8_to_f(__ldca(r1 + 3 * t.i0 + c));
        const float p11 = WORDS ? byte_f(q.t11, c) : u8_to_f(__ldca(r1 + 3 * t.i1 + c));
        const float top = fmaf(t.fx, p01 - p00, p00);
        const float bot = fmaf(t.fx, p11 - p10, p10);
        const float v = fmaf(t.fy, bot - top, top) * scale;
        if (c == 0) o.x = v; else if (c == 1) o.y = v; else o.z = v;
    }
    return o;
}

// Anchor for a camera's tile map: the tile origin clamped into the camera's validity box, where
// w > 0 is guaranteed by the planner.
__host__ __device__ __forceinline__ void tile_anchor(const Rect& V, int X, int Y, int* ax, int* ay) {
    *ax = min(max(X, V.x0), V.x1 - 1);
    *ay = min(max(Y, V.y0), V.y1 - 1);
}

// ------------------------------------------------------------------------------------------------
// lean per-sample helpers used by the fused kernels


// One camera's mapping of canvas point anchor + (dx, dy): fraction-exact source position,
// float source coordinates for the weight, and the sign of w.
struct Pos {
    int iu, iv;    // floor of the source coordinates
    float fu, fv;  // fractions in [0, 1)
    float u, v;    // source coordinates (for validity and weight)
    float den;     // w, positive in front of the camera
};

// map_pos with the column terms (the anchored numerators and denominator at row dy = 0) given:
// fmaf(t.pu1, dx, t.pu0) etc. on the planar canvas, a host-built column table on the cylindrical
// canvas (where a column is an angle); t.pu2, t.pv2, t.q2 are the per-row slopes on both.
__device__ __forceinline__ Pos map_pos_col(const TileMap& t, float fU0, float fV0, float nuc, float nvc, float dqc,
                                           float dy) {
    Pos p;
    p.den = fmaf(t.q2, dy, dqc);
    const float rden = __fdividef(1.0f, p.den);
    float ru = fmaf(t.pu2, dy, nuc) * rden;
    float rv = fmaf(t.pv2, dy, nvc) * rden;
    ru = fminf(fmaxf(ru, -1.0e7f), 1.0e7f);
    rv = fminf(fmaxf(rv, -1.0e7f), 1.0e7f);
    const float flu = floorf(ru), flv = floorf(rv);
    p.iu = t.U0 + (int)flu;
    p.iv = t.V0 + (int)flv;
    p.fu = ru - flu;
    p.fv = rv - flv;
    p.u = fU0 + ru;
    p.v = fV0 + rv;
    return p;
}

// Position of canvas pixel (x, y) in camera c from the FP64 map (paths that are not per-frame
// hot: GENERAL tiles and the plain path on the cylindrical canvas).
__device__ inline Pos map_pos64(const CamDev& c, const RigGeom& g, int x, int y) {
    double u, v;
    const double w = source_point64(c, g, (double)x, (double)y, &u, &v);
    Pos p;
    u = fmin(fmax(u, -1.0e7), 1.0e7);
    v = fmin(fmax(v, -1.0e7), 1.0e7);
    const double fu = floor(u), fv = floor(v);
    p.iu = (int)fu;
    p.iv = (int)fv;
    p.fu = (float)(u - fu);
    p.fv = (float)(v - fv);
    p.u = (float)u;
    p.v = (float)v;
    p.den = w > 0.0 ? 1.0f : -1.0f;
    return p;
}

__device__ __forceinline__ Pos map_pos(const TileMap& t, float fU0, float fV0, float dx, float dy) {
    Pos p;
    p.den = fmaf(t.q2, dy, fmaf(t.q1, dx, t.q0));
    const float rden = __fdividef(1.0f, p.den);
    float ru = fmaf(t.pu2, dy, fmaf(t.pu1, dx, t.pu0)) * rden;
    float rv = fmaf(t.pv2, dy, fmaf(t.pv1, dx, t.pv0)) * rden;
    ru = fminf(fmaxf(ru, -1.0e7f), 1.0e7f);
    rv = fminf(fmaxf(rv, -1.0e7f), 1.0e7f);
    const float flu = floorf(ru), flv = floorf(rv);
    p.iu = t.U0 + (int)flu;
    p.iv = t.V0 + (int)flv;
    p.fu = ru - flu;
    p.fv = rv - flv;
    p.u = fU0 + ru;
    p.v = fV0 + rv;
    return p;
}

// Raw feather weight from float source coordinates; Wm = W - 0.5, Hm = H - 0.5.  Within ~1e-4 px
// of a validity border the float test may differ from the exact one (those pixels are the
// coverage-boundary set that parity excludes); everywhere else it is the same decision.
__device__ __forceinline__ float weight_of(const Pos& p, float Wm, float Hm) {
    const float m = fminf(fminf(p.u + 0.5f, p.v + 0.5f), fminf(Wm - p.u, Hm - p.v));
    const bool ok = (p.den > 0.0f) & (p.u >= -0.5f) & (p.u < Wm) & (p.v >= -0.5f) & (p.v < Hm);
    return ok ? fmaxf(m, 0.0f) : 0.0f;
}

// Bilinear RGB sample with clamped coordinates, scaled by `scale` (= gain / 255).
__device__ __forceinline__ float3 sample_rgb(const uint8_t* px, long long pitch, const Pos& p, int W,
                                             int H, float scale) {
    int i0, j0;
    float fx, fy;
    if (p.iu < 0) { i0 = 0; fx = 0.0f; }
    else if (p.iu >= W - 1) { i0 = W - 1; fx = 0.0f; }
    else { i0 = p.iu; fx = p.fu; }
    if (p.iv < 0) { j0 = 0; fy = 0.0f; }
    else if (p.iv >= H - 1) { j0 = H - 1; fy = 0.0f; }
    else { j0 = p.iv; fy = p.fv; }
    const int di = (i0 + 1 < W) ? 3 : 0;
    const long long dj = (j0 + 1 < H) ? pitch : 0;
    const uint8_t* a = px + (long long)j0 * pitch + 3 * i0;
    const uint8_t* b = a + dj;
    float3 o;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float p00 = u8_to_f(__ldca(a + c)), p01 = u8_to_f(__ldca(a + di + c));
        const float p10 = u8_to_f(__ldca(b + c)), p11 = u8_to_f(__ldca(b + di + c));
        const float top = fmaf(fx, p01 - p00, p00);
        const float bot = fmaf(fx, p11 - p10, p10);
        const float v = fmaf(fy, bot - top, top) * scale;
        if (c == 0) o.x = v; else if (c == 1) o.y = v; else o.z = v;
    }
    return o;
}

// v already clamped to [0, 1]: 2^23 + 255 v rounded once to nearest even in the addition of one
// fused multiply-add, whose low byte is round-half-even(255 v)
__device__ __forceinline__ uint32_t quantize_bits(float v) { return __float_as_uint(fmaf(v, 255.0f, 8388608.0f)); }
__device__ __forceinline__ unsigned char quantize_u8(float v) { return (unsigned char)(quantize_bits(v) & 0xffu); }

// ------------------------------------------------------------------------------------------------
// index-range planning on one axis (host)

struct Span {
    int lo, hi;  // half-open [lo, hi); empty when lo >= hi
    bool empty() const { return hi <= lo; }
};

inline Span span_union(Span a, Span b) {
    if (a.empty()) return b;
    if (b.empty()) return a;
    return {std::min(a.lo, b.lo), std::max(a.hi, b.hi)};
}

// finer-level samples read by REDUCE outputs in `c` (finer level of size n)
inline Span reduce_reads(Span c, int n) {
    if (c.empty()) return {0, 0};
    int lo = n, hi = -1;
    for (int k = c.lo; k < c.hi; ++k)
        for (int m = -2; m <= 2; ++m) {
            const int i = fold101(2 * k + m, n);
            lo = std::min(lo, i);
            hi = std::max(hi, i);
        }
    return {lo, hi + 1};
}

// coarser-level samples read by EXPAND outputs in `f` (coarser level of size n)
inline Span expand_reads(Span f, int n) {
    if (f.empty()) return {0, 0};
    int lo = n, hi = -1;
    for (int x = f.lo; x < f.hi; ++x) {
        const int k0 = (x % 2 == 0) ? x / 2 - 1 : (x - 1) / 2;
        const int k1 = (x % 2 == 0) ? x / 2 + 1 : (x + 1) / 2;
        for (int k = k0; k <= k1; ++k) {
            const int i = fold101(k, n);
            lo = std::min(lo, i);
            hi = std::max(hi, i);
        }
    }
    return {lo, hi + 1};
}

// coarser-level outputs (level size nc) whose REDUCE support meets the finer span `f` (size nf)
inline Span reduce_touch(Span f, int nf, int nc) {
    if (f.empty()) return {0, 0};
    int lo = nc, hi = -1;
    for (int k = 0; k < nc; ++k) {
        bool hit = false;
        for (int m = -2; m <= 2 && !hit; ++m) {
            const int i = fold101(2 * k + m, nf);
            hit = i >= f.lo && i < f.hi;
        }
        if (hit) {
            lo = std::min(lo, k);
            hi = std::max(hi, k);
        }
    }
    return hi < lo ? Span{0, 0} : Span{lo, hi + 1};
}

inline Rect make_rect(Span x, Span y) {
    if (x.empty() || y.empty()) return Rect{0, 0, 0, 0};
    return Rect{x.lo, x.hi, y.lo, y.hi};
}


// ------------------------------------------------------------------------------------------------
// host side

struct KernelStat {
    const char* name;
    double ms;
    long long launches;
};

struct ProfMark {
    const char* name;  // kernel that starts at this event (nullptr: end marker)
    cudaEvent_t ev;
};

struct stitch_rig {
    int device = 0;
    int sms = 0;  // of the device (plain path)
    stitch_rig_desc desc{};
    std::vector<stitch_camera> cams;
    RigGeom geom{};
    CamDev hcam[MAXC]{};
    CamDev* dcam = nullptr;
    float4* Bl[MAXL]{};  // plain path: collapsed R^l of level l >= 1 (full level grid)
    std::vector<void*> allocs;
    std::vector<std::pair<uint32_t*, size_t>> guards;  // debug build: guard bands (words)
    long long scratch_bytes = 0;
    long long roi_pixels = 0;
    int kernels_per_frame = 0;

    // fused path state
    void* fused = nullptr;

    // backward state
    void* bw = nullptr;

    // host staging for stitch_frames_host, and the overlapped pipeline of stitch_frames_host_async
    uint8_t* stage_frames[MAXC]{};
    void* stage_out = nullptr;
    void* pipe = nullptr;

    // profiling
    bool prof = false;
    std::vector<cudaEvent_t> ev_pool;
    size_t ev_used = 0;
    std::vector<ProfMark> marks;
    std::vector<KernelStat> stats;
};

// Validate one camera and plan its regions; adds its level-0 region area to *roi.
stitch_status plan_camera_geometry(const stitch_camera& c, const RigGeom& g, CamDev& d, long long* roi);

// Record a profiling mark before a launch (name) or at the end of a call (nullptr).
void prof_mark(stitch_rig* r, const char* name, cudaStream_t s);

// Device allocation owned by the rig.
void* rig_alloc(stitch_rig* r, size_t bytes);

// Path entry points (one translation unit each).
stitch_status plain_plan(stitch_rig* r);
stitch_status plain_frames(stitch_rig* r, const FramePtrs& fp, const OutDesc& od, cudaStream_t s, bool early);
stitch_status fused_plan(stitch_rig* r);
stitch_status fused_frames(stitch_rig* r, const FramePtrs& fp, const OutDesc& od, cudaStream_t s, bool early);
// stitch_frames with the choice whether its first launch carries the programmatic attribute (stream_launch)
stitch_status rig_frames(stitch_rig* r, const uint8_t* const* frames, const int64_t* pitches, void* out, int64_t out_pitch,
                         cudaStream_t s, bool early);
void fused_release(stitch_rig* r);
void fused_tile_counts(const stitch_rig* r, int counts[8]);
stitch_status backward_plan(stitch_rig* r);
stitch_status backward_run(stitch_rig* r, const FramePtrs& fp, const double* params, double* loss, double* grad,
                           cudaStream_t s);
void backward_release(stitch_rig* r);
void pipeline_release(stitch_rig* r);
stitch_status fused_precompute(stitch_rig* r);  // geometry-only tables, after the camera upload
stitch_status fused_batch_create(stitch_rig* const* rigs, int n, void** out);
stitch_status fused_batch_frames(void* b, const uint8_t* const* const* frames, const int64_t* const* pitches,
                                 void* const* outs, const int64_t* out_pitches, cudaStream_t s);
void fused_batch_destroy(void* b);
stitch_status fused_batch_info(void* b, int32_t* order, int32_t* grid, int64_t* ntasks);
stitch_status fused_batch_wait_test(void* b, int spin_limit, int rig);
stitch_status fused_batch_status(void* b);
// debug build: the fused path's first failed index check (code << 48 | value), 0 when none; reset
long long fused_debug_take(int device);

#define STITCH_CUDA_TRY(expr)                         \
    do {                                              \
        cudaError_t _e = (expr);                      \
        if (_e != cudaSuccess) return STITCH_ECUDA;   \
    } while (0)

static inline stitch_status launch_status() {
    return cudaGetLastError() == cudaSuccess ? STITCH_OK : STITCH_ECUDA;
}
