// Plain path: the steps of the stitching definition (Algorithm 4, step 6, with the multi-band fusion of
// Sec. 1) written out, FP32 intermediates in HBM.  It is the comparison path for the fused
// implementation and what stitch_frames_static runs:
//   warp+weights (S1, S2) of every camera -> REDUCE per level (S3) -> per level, top down: Laplacian
//   bands (S4), their normalised blend on the canvas grid (S5), collapse and output (S6).
// A launch covers all cameras; on the small rigs of stitch_frames_static the path is a chain of
// sub-wave launches, so their number sets its time.  Two 640 x 360 cameras, 4 levels: 8 launches,
// 59 us per call, against 22 launches (each camera, step and level its own) and 185 us.
#include "stitch_internal.cuh"

namespace {

constexpr int BX = 32, BY = 8;

__device__ __forceinline__ float4 ld4(const float4* p) { return *p; }

// The blocks of one launch over a rectangle per camera: camera i has blocks first[i] .. first[i + 1] - 1,
// bx[i] to a row.
struct CamGrid {
    int first[MAXC + 1], bx[MAXC];
};

// Camera of this block and its block position.
__device__ __forceinline__ int grid_cam(const CamGrid& cg, int ncam, int* bx, int* by) {
    int i = 0;
    while (i + 1 < ncam && (int)blockIdx.x >= cg.first[i + 1]) ++i;
    const int q = blockIdx.x - cg.first[i];
    *by = q / cg.bx[i];
    *bx = q - *by * cg.bx[i];
    return i;
}

// S1 + S2: level 0 of every camera on its Om[0]: (I_i rgb, What_i).
//
// Each block anchors the maps of the cameras that meet it (make_tile_map) in FP64, of which this part
// issues one instruction per warp and scheduler in 64 cycles: a thread per camera ran 60 of them in
// the first warp of every block, all on the same scheduler of an SM (38 us a camera, of which the pixels
// take 2).  Here a map takes three lanes (the rows of A: u, v, w), which do the same operations side
// by side, about 18 instructions, in a warp that changes from one wave of blocks to the next.
//
// CYL, SEAM: the cylindrical canvas and seam weights, which work in FP64 per pixel, are kernels of
// their own: compiled as run-time choices, loop-invariant parts of their FP64 arithmetic ran for every
// pixel of the planar feather path too (74 % of the FP64 pipe; 68 us for two 640 x 360 cameras, 19 us now).
template <bool CYL, bool SEAM>
__global__ void __launch_bounds__(BX* BY) k_plain_warp(const CamDev* cams, int ncam,
                                                        const __grid_constant__ CamGrid cg, const __grid_constant__ FramePtrs fp,
                                                        const __grid_constant__ RigGeom g, int sms) {
    __shared__ TileMap tm[MAXC];
    __shared__ int list[MAXC], s_n;
    __shared__ int ax[MAXC], ay[MAXC];
    pdl_trigger();
    pdl_wait();
    int bx, by;
    const int i = grid_cam(cg, ncam, &bx, &by);
    const CamDev& ci = cams[i];
    const Rect om = ci.Om[0];
    const int X = om.x0 + bx * BX, Y = om.y0 + by * BY;
    if (threadIdx.y == (blockIdx.x / (unsigned)sms) % BY) {
        const int t = threadIdx.x;
        bool a = false;
        if (t < ncam) {
            const CamDev& cj = cams[t];
            const Rect v = cj.V;
            // camera t matters for this block if it is camera i or its validity box meets the block
            a = cj.visible && (t == i || (v.x0 < X + BX && v.x1 > X && v.y0 < Y + BY && v.y1 > Y));
        }
        const unsigned m = __ballot_sync(0xffffffffu, a);
        if (a) list[__popc(m & ((1u << t) - 1u))] = t;
        const int n = __popc(m);
        if (t == 0) s_n = n;
        __syncwarp();
        for (int k0 = 0; k0 < (CYL ? 0 : n); k0 += 8) {
            // lane 4 k + q: row q of the map of camera k (q = 2 serves w; lane 4 k + 3 repeats it)
            const int k = min(k0 + t / 4, n - 1), q = min(t % 4, 2);
            const CamDev& cj = cams[list[k]];
            int px, py;
            tile_anchor(cj.V, X, Y, &px, &py);
            const double* B = cj.A + 3 * q;
            const double x = (double)px, y = (double)py;
            const double n0 = B[0] * x + B[1] * y + B[2];
            const double d0 = __shfl_sync(0xffffffffu, n0, (t & ~3) + 2);
            double u0 = n0 / d0;
            u0 = fmin(fmax(u0, -1.0e8), 1.0e8);
            const double U = q < 2 ? rint(u0) : 0.0;
            const float p0 = (float)(n0 - U * d0), p1 = (float)(B[0] - U * cj.A[6]), p2 = (float)(B[1] - U * cj.A[7]);
            if (k0 + t / 4 < n && t % 4 < 3) {
                TileMap& o = tm[k];
                if (q == 0) {
                    o.U0 = (int)U;
                    o.pu0 = p0;
                    o.pu1 = p1;
                    o.pu2 = p2;
                    ax[k] = px;
                    ay[k] = py;
                } else if (q == 1) {
                    o.V0 = (int)U;
                    o.pv0 = p0;
                    o.pv1 = p1;
                    o.pv2 = p2;
                } else {
                    o.q0 = p0;
                    o.q1 = p1;
                    o.q2 = p2;
                }
            }
        }
    }
    __syncthreads();
    const int x = X + threadIdx.x, y = Y + threadIdx.y;
    if (x >= om.x1 || y >= om.y1) return;
    float3 rgb = make_float3(0.f, 0.f, 0.f);
    float wi = 0.f, ws = 0.f;
    // seam weights: the pixel's owner among all cameras (FP64 decision)
    const int own = SEAM ? seam_owner(g, ncam, [&](int k) -> const CamDev& { return cams[k]; }, x, y) : -1;
    for (int k = 0; k < s_n; ++k) {
        const int j = list[k];
        const CamDev& cj = cams[j];
        const SrcPos s = CYL ? map_point64(cj, g, x, y) : map_point(tm[k], (float)(x - ax[k]), (float)(y - ay[k]));
        const float w = SEAM ? (own == j ? 1.f : 0.f) : (cj.V.contains(x, y) ? feather_weight(s, cj.W, cj.H) : 0.f);
        ws += w;
        if (j == i) {
            wi = w;
            rgb = bilinear_rgb(fp.p[i], fp.pitch[i], cj.W, clamp_tap(s, cj.W, cj.H), cj.gain * (1.0f / 255.0f));
        }
    }
    const float what = ws > 0.f ? wi / ws : 0.f;
    ci.G[0][(long long)(y - om.y0) * om.w() + (x - om.x0)] = make_float4(rgb.x, rgb.y, rgb.z, what);
}

// S3: G^{l+1} = REDUCE(G^l) on Om[l+1] (all four channels) of every camera, 25 taps read straight from
// HBM/L2, all in flight.
__global__ void __launch_bounds__(BX* BY) k_plain_reduce(const CamDev* cams, int ncam, int l,
                                                          const __grid_constant__ CamGrid cg, const __grid_constant__ RigGeom g) {
    pdl_trigger();
    pdl_wait();
    int bx, by;
    const CamDev& c = cams[grid_cam(cg, ncam, &bx, &by)];
    const Rect oc = c.Om[l + 1], of = c.Om[l];
    const int k = oc.x0 + bx * BX + threadIdx.x, j = oc.y0 + by * BY + threadIdx.y;
    if (k >= oc.x1 || j >= oc.y1) return;
    const float w5[5] = {1.f / 16, 4.f / 16, 6.f / 16, 4.f / 16, 1.f / 16};
    int xo[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) xo[m] = fold101(2 * k + m - 2, g.nx[l]) - of.x0;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int n = 0; n < 5; ++n) {
        const float4* src = c.G[l] + (long long)(fold101(2 * j + n - 2, g.ny[l]) - of.y0) * of.w();
        float4 row = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const float4 v = ld4(src + xo[m]);
            const float wm = w5[m];
            row.x = fmaf(wm, v.x, row.x);
            row.y = fmaf(wm, v.y, row.y);
            row.z = fmaf(wm, v.z, row.z);
            row.w = fmaf(wm, v.w, row.w);
        }
        const float wn = w5[n];
        acc.x = fmaf(wn, row.x, acc.x);
        acc.y = fmaf(wn, row.y, acc.y);
        acc.z = fmaf(wn, row.z, acc.z);
        acc.w = fmaf(wn, row.w, acc.w);
    }
    c.G[l + 1][(long long)(j - oc.y0) * oc.w() + (k - oc.x0)] = acc;
}

// EXPAND of a coarse buffer (rect r of a level of size nxc x nyc) at fine (x, y), rgb only: taps
// k - 1, k, k + 1 with weights 1/8, 3/4, 1/8 at even positions 2k and k, k + 1 with 1/2, 1/2 at odd ones.  A
// warp's lanes take the same 9 loads (those an odd position has no use for are kept inside the buffer); the
// taps that it does not have are left out, not multiplied by 0, which a value out of range would survive.
__device__ __forceinline__ float3 expand_rgb(const float4* buf, const Rect& r, int nxc, int nyc, int x,
                                             int y) {
    const bool ox = x & 1, oy = y & 1;
    const float wx[3] = {ox ? 0.f : 0.125f, ox ? 0.5f : 0.75f, ox ? 0.5f : 0.125f};
    const float wy[3] = {oy ? 0.f : 0.125f, oy ? 0.5f : 0.75f, oy ? 0.5f : 0.125f};
    int xo[3], yo[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        xo[a] = min(max(fold101((x >> 1) + a - 1, nxc) - r.x0, 0), r.w() - 1);
        yo[a] = min(max(fold101((y >> 1) + a - 1, nyc) - r.y0, 0), r.h() - 1);
    }
    float4 v[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) v[a][b] = ld4(buf + (long long)yo[a] * r.w() + xo[b]);
    float3 acc = make_float3(0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float3 row = make_float3(0.f, 0.f, 0.f);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (b == 0 && ox) continue;
            row.x = fmaf(wx[b], v[a][b].x, row.x);
            row.y = fmaf(wx[b], v[a][b].y, row.y);
            row.z = fmaf(wx[b], v[a][b].z, row.z);
        }
        if (a == 0 && oy) continue;
        acc.x = fmaf(wy[a], row.x, acc.x);
        acc.y = fmaf(wy[a], row.y, acc.y);
        acc.z = fmaf(wy[a], row.z, acc.z);
    }
    return acc;
}

// S4 - S6 on one level of the canvas: B^l = sum_i G^l(What_i) L^l_i / S^l with L^l_i = G^l_i -
// EXPAND(G^{l+1}_i) (the top level: G^l_i), R^l = B^l + EXPAND(R^{l+1}); at level 0 mask, clamp, output.
__global__ void __launch_bounds__(BX* BY) k_plain_level(const CamDev* cams, int l, const __grid_constant__ RigGeom g,
                                                         float4* Bl, const float4* Rc, OutDesc od) {
    pdl_trigger();
    pdl_wait();
    const int x = blockIdx.x * BX + threadIdx.x, y = blockIdx.y * BY + threadIdx.y;
    if (x >= g.nx[l] || y >= g.ny[l]) return;
    const bool top = l == g.levels - 1;
    float nr = 0.f, ng = 0.f, nb = 0.f, s = 0.f;
    for (int i = 0; i < g.ncam; ++i) {
        const CamDev& c = cams[i];
        if (!c.visible || !c.Z[l].contains(x, y)) continue;
        const Rect o = c.Om[l];
        float4 v = ld4(c.G[l] + (long long)(y - o.y0) * o.w() + (x - o.x0));
        if (!top) {
            const float3 e = expand_rgb(c.G[l + 1], c.Om[l + 1], g.nx[l + 1], g.ny[l + 1], x, y);
            v.x -= e.x;
            v.y -= e.y;
            v.z -= e.z;
        }
        nr = fmaf(v.w, v.x, nr);
        ng = fmaf(v.w, v.y, ng);
        nb = fmaf(v.w, v.z, nb);
        s += v.w;
    }
    float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
    if (s > 1e-12f) {
        b.x = nr / s;
        b.y = ng / s;
        b.z = nb / s;
    }
    if (!top) {
        const Rect rc{0, g.nx[l + 1], 0, g.ny[l + 1]};
        const float3 e = expand_rgb(Rc, rc, g.nx[l + 1], g.ny[l + 1], x, y);
        b.x += e.x;
        b.y += e.y;
        b.z += e.z;
    }
    if (l > 0) {
        Bl[(long long)y * g.nx[l] + x] = b;
        return;
    }
    const bool cov = s > 0.f;
    const float r = cov ? __saturatef(b.x) : 0.f, gg = cov ? __saturatef(b.y) : 0.f, bb = cov ? __saturatef(b.z) : 0.f;
    if (od.is_float) {
        float* o = (float*)((char*)od.ptr + (long long)y * od.pitch) + 3 * x;
        o[0] = r;
        o[1] = gg;
        o[2] = bb;
    } else {
        unsigned char* o = (unsigned char*)od.ptr + (long long)y * od.pitch + 3 * x;
        o[0] = quantize_u8(r);
        o[1] = quantize_u8(gg);
        o[2] = quantize_u8(bb);
    }
}

// Blocks over level l's Om of every visible camera; the total in *n.
CamGrid cam_grid(const stitch_rig* r, int l, int* n) {
    CamGrid cg{};
    *n = 0;
    for (int i = 0; i < r->geom.ncam; ++i) {
        const CamDev& c = r->hcam[i];
        cg.first[i] = *n;
        cg.bx[i] = 1;
        if (c.visible && !c.Om[l].empty()) {
            cg.bx[i] = (c.Om[l].w() + BX - 1) / BX;
            *n += cg.bx[i] * ((c.Om[l].h() + BY - 1) / BY);
        }
        cg.first[i + 1] = *n;
    }
    return cg;
}

}  // namespace

stitch_status plain_plan(stitch_rig* r) {
    const RigGeom& g = r->geom;
    for (int i = 0; i < g.ncam; ++i) {
        CamDev& c = r->hcam[i];
        if (!c.visible) continue;
        for (int l = 0; l < g.levels; ++l) {
            c.G[l] = (float4*)rig_alloc(r, sizeof(float4) * (size_t)c.Om[l].area());
            if (!c.G[l]) return STITCH_ENOMEM;
        }
    }
    for (int l = 1; l < g.levels; ++l) {
        r->Bl[l] = (float4*)rig_alloc(r, sizeof(float4) * (size_t)g.nx[l] * g.ny[l]);
        if (!r->Bl[l]) return STITCH_ENOMEM;
    }
    int kernels = g.levels;
    for (int l = 0; l < g.levels; ++l) {
        int n;
        cam_grid(r, l, &n);
        kernels += n > 0;
    }
    r->kernels_per_frame = kernels;
    return STITCH_OK;
}

stitch_status plain_frames(stitch_rig* r, const FramePtrs& fp, const OutDesc& od, cudaStream_t s, bool early) {
    const RigGeom& g = r->geom;
    const dim3 blk(BX, BY);
    const auto put = [&](auto kernel, dim3 grid, const auto&... args) {
        stream_launch(early, kernel, grid, blk, 0, s, args...);
        early = true;
    };
    for (int l = 0; l < g.levels; ++l) {
        int n;
        const CamGrid cg = cam_grid(r, l, &n);
        if (n == 0) continue;
        prof_mark(r, l == 0 ? "plain_warp" : "plain_reduce", s);
        if (l == 0) {
            auto warp = g.cyl ? (g.seam ? k_plain_warp<true, true> : k_plain_warp<true, false>)
                              : (g.seam ? k_plain_warp<false, true> : k_plain_warp<false, false>);
            put(warp, n, r->dcam, g.ncam, cg, fp, g, std::max(r->sms, 1));
        } else {
            put(k_plain_reduce, n, r->dcam, g.ncam, l - 1, cg, g);
        }
    }
    for (int l = g.levels - 1; l >= 0; --l) {
        prof_mark(r, "plain_level", s);
        const dim3 grid((g.nx[l] + BX - 1) / BX, (g.ny[l] + BY - 1) / BY);
        put(k_plain_level, grid, r->dcam, l, g, r->Bl[l], l + 1 < g.levels ? r->Bl[l + 1] : nullptr, od);
    }
    return launch_status();
}
