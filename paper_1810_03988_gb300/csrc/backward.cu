// S7 (an extension beyond the paper, which fixes its homographies by feature matching, Sec. 4.2,
// Algorithm 4 step 5): overlap photometric loss and its gradient with respect to each camera's
// canvas->camera homography entries a11..a32 (a33 = +-1 fixed by the rig) and gain.
//
//   loss = sum_x sum_{i<j} v_i(x) v_j(x) |I_i(x) - I_j(x)|^2,  I = gain * bilinear(frame, A x) / 255
//
// with validity masks held constant.  For camera i at pixel x with k valid cameras,
// dloss/dI_i = 2 r_i, r_i = k I_i - sum_j I_j, and by the chain rule through u = nu/w, v = nv/w:
//   d/da11 = gu x/w, d/da12 = gu y/w, d/da13 = gu/w, d/da2k likewise with gv,
//   d/da31 = -(gu u + gv v) x/w, d/da32 = -(gu u + gv v) y/w, d/dgain = 2 r . bilinear/255,
// where gu = 2 r . dI/du and gv = 2 r . dI/dv (bilinear derivative inside the cell, zero along a
// clamped axis).  Sample coordinates are recomputed per pixel, never stored.
//
// Sums run in local coordinates x' = x - c_i (c_i a fixed point of camera i's footprint) so the
// single-precision terms stay small: with S(f) = sum f, d/da11 = S(gu x'/w) + c_x S(gu/w) etc.,
// applied in double precision at the end.  Per pixel and camera the 10 terms are reduced by warp
// shuffles and a block tree to one partial per (tile, camera slot); a last kernel sums each
// camera's partials with compensated (TwoSum) single-precision arithmetic and applies the chain
// rule to canvas coordinates in double precision.
//
// Launches: k_backward_maps (every slot's tile map, in double precision), k_backward for the tiles of
// at most 2 and at most 4 candidate cameras, k_backward_many for the others, k_backward_final.
#include "stitch_internal.cuh"

namespace {

constexpr int BW_TX = 64, BW_TY = 8;  // canvas pixels per tile
constexpr int BW_THREADS = 256;
constexpr int BW_PPT = BW_TX * BW_TY / BW_THREADS;  // 2 pixels per thread
constexpr int BW_SLOTS = 4;                          // cameras accumulated per pass
constexpr int BW_NV = 10;                            // values per camera
constexpr int BW_MARGIN = 64;                        // px: how far params may move footprints

struct BwTile {
    int x0, y0, first, count;  // canvas origin, candidate cameras (range in the camera list)
    int id;                    // position of the tile's loss partial
};

// A (tile, candidate camera) slot: the camera's map anchored in the tile, from the call's parameters.
struct __align__(16) BwMap {
    TileMap tm;
    float fu0, fv0;  // U0, V0
    float ox, oy;    // tile origin minus anchor: dx, dy are taken from the anchor
    float gain;
    int cam, W, H;
    float wm, hm;    // W - 0.5, H - 0.5
    int cx, cy;      // tile origin minus the camera's local origin
    int pos;         // position of the slot's partials: the slots of a camera in a row, in tile order
    int active;      // 0: no pixel of the tile can lie in the camera's image
    int pad[3];
};
constexpr int BW_MAP_WORDS = sizeof(BwMap) / 16;
static_assert(sizeof(BwMap) == 112, "read as 16-byte words");

// One camera's sample at a pixel: bilinear value and its derivatives (before gain, in [0,1] units).
struct GSample {
    float b[3], bu[3], bv[3];
};

// The source position lies in the camera's image (and in front of the camera).
__device__ __forceinline__ bool gvalid(const Pos& p, const BwMap& m) {
    return (p.den > 0.f) & (p.u >= -0.5f) & (p.u < m.wm) & (p.v >= -0.5f) & (p.v < m.hm);
}

// The sample at p.  The texel values enter as 2^23 + byte, whose differences are those of the bytes,
// R and G as one pair.
__device__ __forceinline__ void gsample(const uint8_t* px, long long pitch, const BwMap& m, const Pos& p,
                                        GSample& s) {
    int i0, j0;
    float fx, fy;
    bool cu = false, cv = false;
    if (p.iu < 0) { i0 = 0; fx = 0.f; cu = true; }
    else if (p.iu >= m.W - 1) { i0 = m.W - 1; fx = 0.f; cu = true; }
    else { i0 = p.iu; fx = p.fu; }
    if (p.iv < 0) { j0 = 0; fy = 0.f; cv = true; }
    else if (p.iv >= m.H - 1) { j0 = m.H - 1; fy = 0.f; cv = true; }
    else { j0 = p.iv; fy = p.fv; }
    // an exact integer u = W-1 sits on the last texel: one-sided derivative there is 0 as well
    const uint8_t* a = px + (long long)j0 * pitch + 3 * i0;
    const Texels q = load_texels(a, a + (j0 + 1 < m.H ? pitch : 0), i0, m.W, word_aligned(px, pitch));
    constexpr float K23 = 8388608.0f, k255 = 1.0f / 255.0f;
    {
        const float2 a00 = make_float2(byte_f23(q.t00, 0), byte_f23(q.t00, 1)), a01 = make_float2(byte_f23(q.t01, 0), byte_f23(q.t01, 1));
        const float2 a10 = make_float2(byte_f23(q.t10, 0), byte_f23(q.t10, 1)), a11 = make_float2(byte_f23(q.t11, 0), byte_f23(q.t11, 1));
        const float2 d0 = f2sub(a01, a00), d1 = f2sub(a11, a10);
        const float2 top = f2fma(f2(fx), d0, f2sub(a00, f2(K23))), bot = f2fma(f2(fx), d1, f2sub(a10, f2(K23)));
        const float2 dv = f2sub(bot, top);
        const float2 b = f2mul(f2fma(f2(fy), dv, top), f2(k255)), bu = f2mul(f2fma(f2(fy), f2sub(d1, d0), d0), f2(k255)),
                     bv = f2mul(dv, f2(k255));
        s.b[0] = b.x;
        s.b[1] = b.y;
        s.bu[0] = cu ? 0.f : bu.x;
        s.bu[1] = cu ? 0.f : bu.y;
        s.bv[0] = cv ? 0.f : bv.x;
        s.bv[1] = cv ? 0.f : bv.y;
    }
    const float b00 = byte_f23(q.t00, 2), b01 = byte_f23(q.t01, 2), b10 = byte_f23(q.t10, 2), b11 = byte_f23(q.t11, 2);
    const float d0 = b01 - b00, d1 = b11 - b10;
    const float top = fmaf(fx, d0, b00 - K23), bot = fmaf(fx, d1, b10 - K23);
    s.b[2] = fmaf(fy, bot - top, top) * k255;
    s.bu[2] = cu ? 0.f : fmaf(fy, d1 - d0, d0) * k255;
    s.bv[2] = cv ? 0.f : (bot - top) * k255;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The tile map of every slot, one thread each.  FP64 runs at two lanes per clock and SM whether a
// warp has one lane active or 32, so this work in the first threads of every tile's block (60 double
// operations in 2 to 4 lanes) cost the 8150 tiles of 4 x 1080p about 50 us of the FP64 pipe; with full warps
// it is 7 us for all of them.
__global__ void __launch_bounds__(64) k_backward_maps(const CamDev* __restrict__ cams, const double* params,
                                                      const int4* __restrict__ slots, int nslots,
                                                      const int* __restrict__ centers, int canvas_w, int canvas_h,
                                                      BwMap* maps) {
    pdl_trigger();
    pdl_wait();
    const int q = blockIdx.x * 64 + threadIdx.x;
    if (q >= nslots) return;
    const int4 sl = slots[q];  // tile origin, camera, position of the partials
    const int c = sl.z;
    const double* p = params + 9 * c;
    const double A[9] = {p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], cams[c].A[8]};
    // anchor at the tile origin clamped into the canvas; w > 0 there for every candidate is
    // not guaranteed, so anchor where w is largest among the tile corners
    BwMap m;
    int ax = sl.x, ay = sl.y;
    double best = -1e300;
    for (int k = 0; k < 4; ++k) {
        const int x = min(sl.x + (k & 1) * (BW_TX - 1), canvas_w - 1);
        const int y = min(sl.y + (k >> 1) * (BW_TY - 1), canvas_h - 1);
        const double w = A[6] * x + A[7] * y + A[8];
        if (w > best) {
            best = w;
            ax = x;
            ay = y;
        }
    }
    m.tm = make_tile_map(A, ax, ay);
    m.fu0 = (float)m.tm.U0;
    m.fv0 = (float)m.tm.V0;
    m.ox = (float)(sl.x - ax);
    m.oy = (float)(sl.y - ay);
    m.gain = (float)p[8];
    m.cam = c;
    m.W = cams[c].W;
    m.H = cams[c].H;
    m.wm = (float)m.W - 0.5f;
    m.hm = (float)m.H - 0.5f;
    m.cx = sl.x - centers[2 * c];
    m.cy = sl.y - centers[2 * c + 1];
    m.pos = sl.w;
    // the tile maps to the hull of its corners' images where w stays well away from 0: beyond one side
    // of the image by half a pixel more than validity asks, none of its pixels is valid
    float wlo = 3e38f, whi = 0.f, ulo = 3e38f, uhi = -3e38f, vlo = 3e38f, vhi = -3e38f;
    for (int k = 0; k < 4; ++k) {
        const Pos c4 = map_pos(m.tm, m.fu0, m.fv0, m.ox + (float)((k & 1) * (BW_TX - 1)), m.oy + (float)((k >> 1) * (BW_TY - 1)));
        wlo = fminf(wlo, c4.den);
        whi = fmaxf(whi, c4.den);
        ulo = fminf(ulo, c4.u);
        uhi = fmaxf(uhi, c4.u);
        vlo = fminf(vlo, c4.v);
        vhi = fmaxf(vhi, c4.v);
    }
    const bool out = wlo > 0.25f * whi && (uhi < -1.f || ulo > m.wm + 0.5f || vhi < -1.f || vlo > m.hm + 0.5f);
    m.active = out ? 0 : 1;
    m.pad[0] = m.pad[1] = m.pad[2] = 0;
    maps[q] = m;
}

// The 10 gradient terms of a camera's sample at a pixel added to acc; r is the residual of the pixel.
__device__ __forceinline__ void grad_terms(const GSample& s, const Pos& p, const float r[3], float g, float xl, float yl,
                                           float acc[BW_NV]) {
    const float gu = 2.f * g * (r[0] * s.bu[0] + r[1] * s.bu[1] + r[2] * s.bu[2]);
    const float gv = 2.f * g * (r[0] * s.bv[0] + r[1] * s.bv[1] + r[2] * s.bv[2]);
    const float gg = 2.f * (r[0] * s.b[0] + r[1] * s.b[1] + r[2] * s.b[2]);
    const float iw = 1.0f / p.den;
    const float q = -(gu * p.u + gv * p.v) * iw;
    const float guw = gu * iw, gvw = gv * iw;
    acc[0] = fmaf(guw, xl, acc[0]);
    acc[1] = fmaf(guw, yl, acc[1]);
    acc[2] += guw;
    acc[3] = fmaf(gvw, xl, acc[3]);
    acc[4] = fmaf(gvw, yl, acc[4]);
    acc[5] += gvw;
    acc[6] = fmaf(q, xl, acc[6]);
    acc[7] = fmaf(q, yl, acc[7]);
    acc[8] += q;
    acc[9] += gg;
}

// Sums over the warp of M values per lane, M halved at each step: in step xor k a lane keeps one half
// of the values and gets its partner's sums of them for its own of the other half.  Every sum adds
// the same pairs as warp_sum (the lanes 16, 8, 4, 2, 1 apart), so the results are bit-identical, with
// about M instead of 5 M shuffles.  Value index(i) of lane l's results v[0 .. left) is sum index(i).
template <int M, int K>
struct WarpSums {
    static constexpr int HALF = (M + 1) / 2;
    static constexpr int LEFT = WarpSums<HALF, K / 2>::LEFT;
    __device__ __forceinline__ static void run(float* v, int lane) {
        const bool up = lane & K;
#pragma unroll
        for (int i = 0; i < HALF; ++i) {
            const float hi = i + HALF < M ? v[i + HALF] : 0.f;
            const float keep = up ? hi : v[i], send = up ? v[i] : hi;
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, K);
        }
        WarpSums<HALF, K / 2>::run(v, lane);
    }
    // which of the M sums lane's result i is, or -1
    __device__ __forceinline__ static int index(int i, int lane) {
        const int q = WarpSums<HALF, K / 2>::index(i, lane);
        if (q < 0) return -1;
        const int r = q + (lane & K ? HALF : 0);
        return r < M ? r : -1;
    }
};
template <int M>
struct WarpSums<M, 0> {
    static constexpr int LEFT = M;
    __device__ __forceinline__ static void run(float*, int) {}
    __device__ __forceinline__ static int index(int i, int) { return i; }
};

// A tile with at most N candidate cameras: validity from the positions first, then one sample per
// valid camera of the pixels that at least two see, kept in registers for both the sum and the
// gradient.  Bound by instruction issue: 56 + 75 us for the 4727 + 3423 tiles of 4 x 1080p, against 227 us when
// every candidate was sampled twice at every pixel, from byte loads, with 5 shuffles for each of 40 sums.
template <int N>
__global__ void __launch_bounds__(BW_THREADS, N == 2 ? 4 : 2) k_backward(const FramePtrs fp, const BwMap* maps,
                                                                        const BwTile* __restrict__ tiles, int canvas_w,
                                                                        int canvas_h, float* partials, int nslots,
                                                                        float* loss_partials) {
    __shared__ __align__(16) BwMap m[N];
    __shared__ float red[BW_THREADS / 32][N * BW_NV + 1];
    const BwTile tl = tiles[blockIdx.x];
    const int n = tl.count, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    pdl_trigger();
    pdl_wait();
    if (t < BW_MAP_WORDS * n) reinterpret_cast<int4*>(m)[t] = reinterpret_cast<const int4*>(maps + tl.first)[t];
    __syncthreads();
    auto no_overlap = [&]() {  // only zeros: no two cameras see a pixel of the tile
        if (t < n * BW_NV) partials[(long long)(t % BW_NV) * nslots + m[t / BW_NV].pos] = 0.f;
        if (t == 0) loss_partials[tl.id] = 0.f;
    };
    int seen = 0;
#pragma unroll
    for (int a = 0; a < N; ++a) seen += a < n && m[a].active;
    if (seen < 2) {
        no_overlap();
        return;
    }
    float loss = 0.f;
    float acc[N * BW_NV];
#pragma unroll
    for (int v = 0; v < N * BW_NV; ++v) acc[v] = 0.f;
    bool some = false;
#pragma unroll 1
    for (int k = 0; k < BW_PPT; ++k) {
        const int dx = t % BW_TX, dy = t / BW_TX + k * (BW_THREADS / BW_TX), x = tl.x0 + dx, y = tl.y0 + dy;
        const float fdx = (float)dx, fdy = (float)dy;
        Pos p[N];
        bool ok[N];
        int kv = 0;
#pragma unroll
        for (int a = 0; a < N; ++a) {
            ok[a] = false;
            if (a < n && m[a].active) {
                p[a] = map_pos(m[a].tm, m[a].fu0, m[a].fv0, m[a].ox + fdx, m[a].oy + fdy);
                ok[a] = gvalid(p[a], m[a]);
            }
            kv += ok[a];
        }
        if (kv < 2 || x >= canvas_w || y >= canvas_h) continue;
        some = true;
        GSample s[N];
        float S[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < N; ++a) {
            if (!ok[a]) continue;
            const int c = m[a].cam;
            const uint8_t* px = fp.p[c];
            const long long pitch = fp.pitch[c];
            gsample(px, pitch, m[a], p[a], s[a]);
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) S[ch] = fmaf(m[a].gain, s[a].b[ch], S[ch]);
        }
#pragma unroll
        for (int a = 0; a < N; ++a) {
            if (!ok[a]) continue;
            const float g = m[a].gain;
            float r[3];
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) r[ch] = (float)kv * (g * s[a].b[ch]) - S[ch];
            // with the mean m = S/k, sum_{i<j} |I_i - I_j|^2 = k sum_i |I_i - m|^2
            // = sum_i |r_i|^2 / k; r_i is small and accurate, so no cancellation
            loss += (r[0] * r[0] + r[1] * r[1] + r[2] * r[2]) / (float)kv;
            grad_terms(s[a], p[a], r, g, (float)(m[a].cx + dx), (float)(m[a].cy + dy), acc + a * BW_NV);
        }
    }
    // block reduction: warp sums, then a tree over warps; a tile (or warp) that no two cameras see has
    // only zeros
    if (!__syncthreads_or(some)) {
        no_overlap();
        return;
    }
    using Sums = WarpSums<N * BW_NV, 16>;
    if (__any_sync(0xffffffffu, some)) {
        Sums::run(acc, lane);
#pragma unroll
        for (int i = 0; i < Sums::LEFT; ++i) {
            const int v = Sums::index(i, lane);
            if (v >= 0) red[warp][v] = acc[i];
        }
        const float lw = warp_sum(loss);
        if (lane == 0) red[warp][N * BW_NV] = lw;
    } else {
        for (int v = lane; v <= N * BW_NV; v += 32) red[warp][v] = 0.f;
    }
    __syncthreads();
    if (t <= N * BW_NV) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < BW_THREADS / 32; ++w) sum += red[w][t];
        if (t == N * BW_NV) loss_partials[tl.id] = sum;
        else if (t < n * BW_NV) partials[(long long)(t % BW_NV) * nslots + m[t / BW_NV].pos] = sum;
    }
}

// Tiles with more candidates (up to MAXC), in groups of BW_SLOTS cameras: samples are taken again for
// the gradient, as registers do not hold them all.
__global__ void __launch_bounds__(BW_THREADS) k_backward_many(const FramePtrs fp, const BwMap* maps,
                                                              const BwTile* __restrict__ tiles, int canvas_w, int canvas_h,
                                                              float* partials, int nslots,
                                                              float* loss_partials) {
    __shared__ __align__(16) BwMap m[MAXC];
    __shared__ float red[BW_THREADS / 32][BW_SLOTS * BW_NV + 1];
    const BwTile tl = tiles[blockIdx.x];
    const int n = tl.count;  // <= MAXC
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    pdl_trigger();
    pdl_wait();
    static_assert(BW_MAP_WORDS * MAXC <= BW_THREADS, "one 16-byte word per thread");
    if (t < BW_MAP_WORDS * n) reinterpret_cast<int4*>(m)[t] = reinterpret_cast<const int4*>(maps + tl.first)[t];
    __syncthreads();
    auto pos_of = [&](int a, int dx, int dy) {
        return map_pos(m[a].tm, m[a].fu0, m[a].fv0, m[a].ox + (float)dx, m[a].oy + (float)dy);
    };
    auto sample = [&](int a, const Pos& p, GSample& s) {
        const uint8_t* px = fp.p[m[a].cam];
        const long long pitch = fp.pitch[m[a].cam];
        gsample(px, pitch, m[a], p, s);
    };
    float loss = 0.f;
    for (int g0 = 0; g0 < n; g0 += BW_SLOTS) {
        float acc[BW_SLOTS][BW_NV];
#pragma unroll
        for (int s = 0; s < BW_SLOTS; ++s)
#pragma unroll
            for (int v = 0; v < BW_NV; ++v) acc[s][v] = 0.f;
#pragma unroll
        for (int k = 0; k < BW_PPT; ++k) {
            const int dx = t % BW_TX, dy = t / BW_TX + k * (BW_THREADS / BW_TX);
            if (tl.x0 + dx >= canvas_w || tl.y0 + dy >= canvas_h) continue;
            // pass 1: number of valid cameras and the sum of their intensities
            int kv = 0;
            float S[3] = {0.f, 0.f, 0.f};
            for (int a = 0; a < n; ++a) {
                if (!m[a].active) continue;
                const Pos p = pos_of(a, dx, dy);
                if (!gvalid(p, m[a])) continue;
                GSample s;
                sample(a, p, s);
                ++kv;
#pragma unroll
                for (int c = 0; c < 3; ++c) S[c] = fmaf(m[a].gain, s.b[c], S[c]);
            }
            if (kv < 2) continue;
            // pass 2: loss (first group only) and gradient terms of this group's cameras
            for (int a = 0; a < n; ++a) {
                const int slot = a - g0;
                if (g0 > 0 && (slot < 0 || slot >= BW_SLOTS)) continue;
                if (!m[a].active) continue;
                const Pos p = pos_of(a, dx, dy);
                if (!gvalid(p, m[a])) continue;
                GSample s;
                sample(a, p, s);
                const float g = m[a].gain;
                float r[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) r[c] = (float)kv * (g * s.b[c]) - S[c];
                if (g0 == 0) loss += (r[0] * r[0] + r[1] * r[1] + r[2] * r[2]) / (float)kv;
                // unrolled slot selection keeps the accumulators in registers
#pragma unroll
                for (int ss = 0; ss < BW_SLOTS; ++ss)
                    if (ss == slot) grad_terms(s, p, r, g, (float)(m[a].cx + dx), (float)(m[a].cy + dy), acc[ss]);
            }
        }
        // block reduction of this group's slots: warp sums, then a tree over warps
        using Sums = WarpSums<BW_SLOTS * BW_NV, 16>;
        Sums::run(&acc[0][0], lane);
#pragma unroll
        for (int i = 0; i < Sums::LEFT; ++i) {
            const int v = Sums::index(i, lane);
            if (v >= 0) red[warp][v] = acc[0][i];
        }
        __syncthreads();
        if (t < BW_SLOTS * BW_NV) {
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < BW_THREADS / 32; ++w) sum += red[w][t];
            const int a = g0 + t / BW_NV;
            if (a < n) partials[(long long)(t % BW_NV) * nslots + m[a].pos] = sum;
        }
        __syncthreads();
    }
    const float lw = warp_sum(loss);
    if (lane == 0) red[warp][BW_SLOTS * BW_NV] = lw;
    __syncthreads();
    if (t == 0) {
        float sum = 0.f;
        for (int w = 0; w < BW_THREADS / 32; ++w) sum += red[w][BW_SLOTS * BW_NV];
        loss_partials[tl.id] = sum;
    }
}

// Error-free sum of two floats (Knuth's TwoSum): a + b = s + e exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Compensated sums of NS runs x[v * stride + lo .. v * stride + hi) by a block of 256 threads: thread t
// adds every 256th value from lo + t on, a tree adds the threads' pairs.  The loads of 8 values per
// run are in flight before their additions.
template <int NS>
__device__ __forceinline__ void block_csums(const float* x, long long stride, int lo, int hi, double S[NS]) {
    __shared__ float sh_s[NS][256], sh_c[NS][256];
    constexpr int D = 8;
    const int t = threadIdx.x;
    float s[NS], c[NS];
#pragma unroll
    for (int v = 0; v < NS; ++v) s[v] = c[v] = 0.f;
    for (int k0 = lo + t; k0 < hi; k0 += D * 256) {
        float r[NS][D];
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int v = 0; v < NS; ++v) r[v][d] = k0 + d * 256 < hi ? __ldcg(x + v * stride + k0 + d * 256) : 0.f;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            if (k0 + d * 256 >= hi) break;
#pragma unroll
            for (int v = 0; v < NS; ++v) {
                float ns, ne;
                two_sum(s[v], r[v][d], ns, ne);
                s[v] = ns;
                c[v] += ne;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < NS; ++v) {
        sh_s[v][t] = s[v];
        sh_c[v][t] = c[v];
    }
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (t < h) {
#pragma unroll
            for (int v = 0; v < NS; ++v) {
                float ns, ne;
                two_sum(sh_s[v][t], sh_s[v][t + h], ns, ne);
                sh_s[v][t] = ns;
                sh_c[v][t] += sh_c[v][t + h] + ne;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int v = 0; v < NS; ++v) S[v] = (double)sh_s[v][0] + (double)sh_c[v][0];
}

// Blocks (group, camera): the terms 3 g .. 3 g + 2 of the camera (group 3: the gain's term), so that four
// blocks share its walk over the partials; a further block (0, ncam) sums the loss.  A chain of
// latencies: 8 us for the 8150 tiles of 4 x 1080p, against 29 us with a block per camera that
// reached each slot's terms through an index.
__global__ void __launch_bounds__(256) k_backward_final(int ncam, const float* partials, int nslots,
                                                         const float* loss_partials, int ntiles,
                                                         const int* __restrict__ cam_slot_start,
                                                         const int* __restrict__ centers, double* __restrict__ loss,
                                                         double* __restrict__ grad) {
    pdl_trigger();
    pdl_wait();
    const int b = blockIdx.y, g = blockIdx.x;
    double S[3];
    if (b == ncam) {
        if (g != 0) return;
        block_csums<1>(loss_partials, 0, 0, ntiles, S);
        if (threadIdx.x == 0) *loss = S[0];
        return;
    }
    if (!grad) return;
    const int lo = cam_slot_start[b], hi = cam_slot_start[b + 1];
    double* gr = grad + 9 * b;
    if (g == 3) {
        block_csums<1>(partials + 9LL * nslots, 0, lo, hi, S);
        if (threadIdx.x == 0) gr[8] = S[0];
        return;
    }
    block_csums<3>(partials + 3LL * g * nslots, nslots, lo, hi, S);
    if (threadIdx.x == 0) {
        gr[3 * g] = S[0] + centers[2 * b] * S[2];
        gr[3 * g + 1] = S[1] + centers[2 * b + 1] * S[2];
        if (g < 2) gr[3 * g + 2] = S[2];
    }
}

// tiles by candidate count: at most 2, at most 4, more
constexpr int BW_CLASSES = 3;

struct BwState {
    BwTile* tiles = nullptr;  // class by class
    int ntiles = 0, nclass[BW_CLASSES] = {}, nslots = 0;
    int4* slots = nullptr;    // per slot: tile origin, camera, position of its partials
    BwMap* maps = nullptr;
    int* centers = nullptr;
    int* cam_slot_start = nullptr;
    float* partials = nullptr;  // [BW_NV][nslots]
    float* loss_partials = nullptr;
};

template <typename V>
stitch_status upload_bw(stitch_rig* r, const std::vector<V>& v, V** out) {
    *out = nullptr;
    if (v.empty()) return STITCH_OK;
    *out = (V*)rig_alloc(r, sizeof(V) * v.size());
    if (!*out) return STITCH_ENOMEM;
    STITCH_CUDA_TRY(cudaMemcpy(*out, v.data(), sizeof(V) * v.size(), cudaMemcpyHostToDevice));
    return STITCH_OK;
}

}  // namespace

// Candidate tiles: canvas tiles met by the footprint boxes (grown by BW_MARGIN px) of at least two
// cameras; parameters that move a footprint further than that leave pixels uncounted.
stitch_status backward_plan(stitch_rig* r) {
    const RigGeom& g = r->geom;
    BwState* bs = new (std::nothrow) BwState();
    if (!bs) return STITCH_ENOMEM;
    r->bw = bs;
    std::vector<BwTile> tiles[BW_CLASSES];
    std::vector<int> camlist, centers(2 * g.ncam, 0);
    std::vector<int4> sl;
    std::vector<std::vector<int>> slots(g.ncam);
    for (int i = 0; i < g.ncam; ++i) {
        const Rect v = r->hcam[i].V;
        centers[2 * i] = r->hcam[i].visible ? (v.x0 + v.x1) / 2 : 0;
        centers[2 * i + 1] = r->hcam[i].visible ? (v.y0 + v.y1) / 2 : 0;
    }
    const int Wc = g.nx[0], Hc = g.ny[0];
    for (int y0 = 0; y0 < Hc; y0 += BW_TY)
        for (int x0 = 0; x0 < Wc; x0 += BW_TX) {
            const int x1 = std::min(x0 + BW_TX, Wc), y1 = std::min(y0 + BW_TY, Hc);
            BwTile t{x0, y0, (int)camlist.size(), 0, bs->ntiles};
            for (int i = 0; i < g.ncam; ++i) {
                const CamDev& c = r->hcam[i];
                if (!c.visible) continue;
                const Rect v = c.V;
                if (v.x0 - BW_MARGIN < x1 && v.x1 + BW_MARGIN > x0 && v.y0 - BW_MARGIN < y1 && v.y1 + BW_MARGIN > y0) {
                    camlist.push_back(i);
                    ++t.count;
                }
            }
            if (t.count < 2) {
                camlist.resize(t.first);
                continue;
            }
            for (int k = 0; k < t.count; ++k) {
                slots[camlist[t.first + k]].push_back(t.first + k);
                sl.push_back(make_int4(x0, y0, camlist[t.first + k], 0));
            }
            tiles[t.count <= 2 ? 0 : t.count <= 4 ? 1 : 2].push_back(t);
            ++bs->ntiles;
        }
    // a camera's partials lie in a row, in tile order
    std::vector<int> start(g.ncam + 1, 0);
    for (int i = 0; i < g.ncam; ++i) {
        start[i + 1] = start[i] + (int)slots[i].size();
        for (size_t k = 0; k < slots[i].size(); ++k) sl[slots[i][k]].w = start[i] + (int)k;
    }
    std::vector<BwTile> all;
    for (int k = 0; k < BW_CLASSES; ++k) {
        bs->nclass[k] = (int)tiles[k].size();
        all.insert(all.end(), tiles[k].begin(), tiles[k].end());
    }
    bs->nslots = (int)sl.size();
    stitch_status st;
    if ((st = upload_bw(r, all, &bs->tiles)) != STITCH_OK) return st;
    if ((st = upload_bw(r, sl, &bs->slots)) != STITCH_OK) return st;
    if ((st = upload_bw(r, centers, &bs->centers)) != STITCH_OK) return st;
    if ((st = upload_bw(r, start, &bs->cam_slot_start)) != STITCH_OK) return st;
    bs->maps = (BwMap*)rig_alloc(r, sizeof(BwMap) * std::max(bs->nslots, 1));
    bs->partials = (float*)rig_alloc(r, sizeof(float) * BW_NV * std::max(bs->nslots, 1));
    bs->loss_partials = (float*)rig_alloc(r, sizeof(float) * std::max(bs->ntiles, 1));
    if (!bs->maps || !bs->partials || !bs->loss_partials) return STITCH_ENOMEM;
    return STITCH_OK;
}

stitch_status backward_run(stitch_rig* r, const FramePtrs& fp, const double* params, double* loss, double* grad,
                           cudaStream_t s) {
    BwState* bs = (BwState*)r->bw;
    if (!bs) return STITCH_EINVAL;
    const RigGeom& g = r->geom;
    if (bs->ntiles > 0) {
        prof_mark(r, "backward_maps", s);
        pdl_launch(k_backward_maps, (bs->nslots + 63) / 64, 64, 0, s, r->dcam, params, bs->slots, bs->nslots, bs->centers,
                   g.nx[0], g.ny[0], bs->maps);
        const BwTile* tl = bs->tiles;
        for (int k = 0; k < BW_CLASSES; tl += bs->nclass[k++]) {
            if (bs->nclass[k] == 0) continue;
            prof_mark(r, "backward", s);
            auto fn = k == 0 ? k_backward<2> : k == 1 ? k_backward<4> : k_backward_many;
            pdl_launch(fn, bs->nclass[k], BW_THREADS, 0, s, fp, bs->maps, tl, g.nx[0], g.ny[0], bs->partials, bs->nslots,
                       bs->loss_partials);
        }
    }
    prof_mark(r, "backward_final", s);
    pdl_launch(k_backward_final, dim3(4, g.ncam + 1), 256, 0, s, g.ncam, bs->partials, bs->nslots, bs->loss_partials,
               bs->ntiles, bs->cam_slot_start, bs->centers, loss, grad);
    return launch_status();
}

void backward_release(stitch_rig* r) {
    delete (BwState*)r->bw;
    r->bw = nullptr;
}
