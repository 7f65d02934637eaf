// L-ORB feature extraction (Sec. 4.1, Algorithms 1 and 2) on the GPU, in exact integer
// arithmetic so that every decision (FAST, threshold, non-maximum suppression, top-N, BRIEF
// bits) is the one of the definition:
//   gray = (77 R + 150 G + 29 B + 128) >> 8; candidates inside the detection areas and at least
//   LORB_MARGIN px from the image border; FAST-9 on the radius-3 circle with threshold t;
//   Ix, Iy central differences; A, B, C their products weighted by the binomial [1,4,6,4,1]^2
//   (the sigma = 1 Gaussian, unnormalised); R' = 25 (AB - C^2) - (A + B)^2 = 25 R with
//   alpha = 0.04, kept when R' > t_h; non-maximum suppression over the 8-neighbourhood with ties
//   to the lower index y W + x; the N strongest (R' descending, index ascending); BRIEF bits
//   [S(x + p_k) > S(x + q_k)] of the binomial-smoothed image S for 256 given point pairs.
//
// Kernels: lorb_detect (gray, FAST, Harris and non-maximum suppression of a tile on chip; survivors
// appended, their order being irrelevant since the selection below is exact, and counted in a
// histogram of coarse response bins), lorb_prune (the survivors in the bins that can hold the N
// strongest; when those are too many to rank, its last block selects the N strongest itself) and
// lorb_rank_brief (rank by counting, then the BRIEF bits from the point's patch of the frame).
#include "stitch_internal.cuh"

namespace {

constexpr int LORB_MARGIN = 18;
constexpr int LORB_MAX_AREAS = 64;
constexpr int LORB_MAX_POINTS = 2048;
constexpr int SEL_THREADS = 1024;

struct LorbAreas {
    int n;
    int r[LORB_MAX_AREAS][4];  // x0, y0, x1, y1 clipped to the margin, half-open
};

struct LorbPattern {
    char4 p[256];  // ax, ay, bx, by
};

struct Cand {
    long long r;
    int idx, pad;
};

__device__ __forceinline__ bool in_areas(const LorbAreas& a, int x, int y) {
    for (int k = 0; k < a.n; ++k)
        if (x >= a.r[k][0] && x < a.r[k][2] && y >= a.r[k][1] && y < a.r[k][3]) return true;
    return false;
}

__device__ __forceinline__ unsigned gray_of(unsigned r, unsigned g, unsigned b) { return (77u * r + 150u * g + 29u * b + 128u) >> 8; }

// gray of the four pixels in the bytes R G B R | G B R G | B R G B of a, b, c
__device__ __forceinline__ void gray4(unsigned a, unsigned b, unsigned c, unsigned o[4]) {
    o[0] = __dp4a(a, 0x001D964Du, 128u) >> 8;
    o[1] = __dp4a(b, 0x00001D96u, __dp4a(a, 0x4D000000u, 128u)) >> 8;
    o[2] = __dp4a(c, 0x0000001Du, __dp4a(b, 0x964D0000u, 128u)) >> 8;
    o[3] = __dp4a(c, 0x1D964D00u, 128u) >> 8;
}

// Coarse, monotone (non-decreasing in R') bin of a response: the position of its leading bit and
// the 4 bits below it; R' <= 0 in bin 0.  The N strongest candidates all lie in the bins at or above
// the bin where the count from the top reaches N.
constexpr int LORB_BINS = 1024;
__device__ __forceinline__ int lorb_bin(long long r) {
    if (r <= 0) return 0;
    const int e = 64 - __clzll(r);  // 1 .. 63
    const int m = e > 5 ? (int)((r >> (e - 5)) & 15) : (int)(r & 15);
    return 16 * e + m;
}

// Counters of a call, zero between calls but for n2 (lorb_prune's last block clears them; after a sequence
// that a refused launch cut short, the next call does): survivors, finished lorb_prune blocks, pruned
// candidates, survivors per response bin.
struct LorbCount {
    int n, done, n2, pad;
    int hist[LORB_BINS];
    char4 pat[256];  // the call's BRIEF pattern
};

// lorb_detect: gray, FAST, Harris response and non-maximum suppression of one tile, appending the
// survivors to cand (their order is irrelevant) and counting them in the bin histogram.
//
// A block of 256 threads evaluates 64 x 32 pixels and owns the inner 60 x 30: the ring around them
// gives the suppression its neighbours, so no response ever leaves the chip.  What bounds it is
// instruction issue: 8.3 MPix of a 4K view cost about 30 instructions each (reading the 25 MB takes
// 4 us).  Hence:
//  - the tile's gray is staged as words that hold a pixel and the one below it (16 bits each), so one
//    32-bit load and one 16-bit-pair minimum or maximum serve two pixels, at any offset;
//  - a pair is tested on its 4 compass pixels first (an arc of 9 of the 16 circle pixels holds two
//    neighbouring ones).  The pairs that pass are gathered for the block, so the 16-pixel test and
//    then the Harris response of the corners run with full warps instead of under a branch that nearly
//    every warp takes for a few lanes, and spread over all warps however the corners lie.
// One 3840 x 2160 view: 34 us (of which 18 us are issue slots; 35 us and a quarter more instructions with
// lists per warp) against 134 us for gray and smoothed maps, response map (8 bytes per pixel written and
// read back) and suppression as three kernels.
constexpr int DT_EX = 64, DT_EY = 32;   // evaluated pixels
constexpr int DT_OX = 60, DT_OY = 30;   // owned pixels: columns 2 .. 61, rows 1 .. 30
constexpr int DT_PX = 72, DT_PY = 39;   // gray words: 18 groups of 4 columns, 13 strips of 3 rows
constexpr int DT_PAIRS = DT_EX * DT_EY / 2;

// whether either of the two pixels p (16 bits each) has an arc value above it (mb: the largest of the
// arcs' smallest values) or below it (md) by more than the threshold; lim = threshold + 256
__device__ __forceinline__ unsigned fast_excess(unsigned p, unsigned mb, unsigned md) {
    return __vmaxu2((mb + 0x01000100u) - p, (p + 0x01000100u) - md);
}

__global__ void __launch_bounds__(256, 5) lorb_detect(const uint8_t* frame, long long pitch, int W, int H,
                                                      int ox, int oy, const __grid_constant__ LorbAreas areas, int lim,
                                                      long long harris_t, Cand* cand, int* ncand,
                                                      int cap, int* hist, int* n2) {
    __shared__ __align__(16) unsigned P[DT_PX * DT_PY];
    __shared__ long long R[DT_EX * DT_EY];
    __shared__ unsigned mask[DT_EY][2];  // which pixels of a row have a response
    __shared__ uint16_t pairs[DT_PAIRS], corners[2 * DT_PAIRS];
    __shared__ int s_np, s_nc, s_n, s_base;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    pdl_trigger();
    pdl_wait();
    // owned pixels start at (bx, by); bx is 1 modulo 4, so the staged columns start at a multiple of 4
    const int bx = ox + DT_OX * blockIdx.x, by = oy + DT_OY * blockIdx.y;
    if (blockIdx.x == 0 && blockIdx.y == 0 && t == 0) *n2 = 0;
    bool any = false;
    for (int k = 0; k < areas.n; ++k)
        any |= bx < areas.r[k][2] && bx + DT_OX > areas.r[k][0] && by < areas.r[k][3] && by + DT_OY > areas.r[k][1];
    if (!any) return;
    if (t < 2 * DT_EY) mask[t >> 1][t & 1] = 0u;
    if (t == 0) s_np = s_nc = s_n = 0;
    if (t < 18 * 13) {
        const int j = t % 18, st = t / 18, gx0 = bx - 5 + 4 * j;
        const bool words = ((reinterpret_cast<uintptr_t>(frame) | (uintptr_t)pitch) & 3) == 0 && gx0 + 3 < W;
        unsigned g[4][4];
        if (words) {
            unsigned v[4][3];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int y = min(by - 4 + 3 * st + k, H - 1);
                const unsigned* q = reinterpret_cast<const unsigned*>(frame + (long long)y * pitch + 3LL * gx0);
                v[k][0] = __ldca(q);
                v[k][1] = __ldca(q + 1);
                v[k][2] = __ldca(q + 2);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) gray4(v[k][0], v[k][1], v[k][2], g[k]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint8_t* row = frame + (long long)min(by - 4 + 3 * st + k, H - 1) * pitch;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint8_t* q = row + 3LL * min(gx0 + i, W - 1);
                    g[k][i] = gray_of(__ldca(q), __ldca(q + 1), __ldca(q + 2));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
            *reinterpret_cast<uint4*>(P + (3 * st + k) * DT_PX + 4 * j) =
                make_uint4(g[k][0] | g[k + 1][0] << 16, g[k][1] | g[k + 1][1] << 16, g[k][2] | g[k + 1][2] << 16,
                           g[k][3] | g[k + 1][3] << 16);
    }
    __syncthreads();
    // evaluated pixel (ex, ey) is image pixel (bx - 2 + ex, by - 1 + ey), staged at P[ey + 3][ex + 3]
    constexpr int fo[16] = {-3 * DT_PX,     -3 * DT_PX + 1, -2 * DT_PX + 2, -DT_PX + 3, 3,  DT_PX + 3,  2 * DT_PX + 2,  3 * DT_PX + 1,
                            3 * DT_PX,      3 * DT_PX - 1,  2 * DT_PX - 2,  DT_PX - 3,  -3, -DT_PX - 3, -2 * DT_PX - 2, -3 * DT_PX - 1};
    const unsigned below = (1u << lane) - 1u;
    // appends v of the lanes with `keep` to a list of the block
    auto append = [&](bool keep, int v, uint16_t* list, int* n) {
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (m == 0u) return;
        int base = 0;
        if (lane == 0) base = atomicAdd(n, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (keep) list[base + __popc(m & below)] = (uint16_t)v;
    };
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int ey = 4 * w + 2 * (it >> 1), ex = 32 * (it & 1) + lane;
        const unsigned* c = P + (ey + 3) * DT_PX + ex + 3;
        const unsigned p = c[0], n = c[fo[0]], e = c[fo[4]], s = c[fo[8]], o = c[fo[12]];
        const unsigned x = fast_excess(p, __vminu2(__vmaxu2(n, s), __vmaxu2(e, o)), __vmaxu2(__vminu2(n, s), __vminu2(e, o)));
        const bool pass = ((int)(x & 0xffffu) > lim || (int)(x >> 16) > lim) && ex >= 1 && ex <= 62;
        append(pass, ey * DT_EX + ex, pairs, &s_np);
    }
    __syncthreads();
    const int np = s_np;
    for (int i0 = 32 * w; i0 < np; i0 += 256) {
        bool lo = false, hi = false;
        int at = 0;
        if (i0 + lane < np) {
            at = pairs[i0 + lane];
            const int ex = at & (DT_EX - 1), ey = at / DT_EX;
            const unsigned* c = P + (ey + 3) * DT_PX + ex + 3;
            unsigned v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = c[fo[k]];
            unsigned mb, md;
            {
                unsigned m3[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) m3[k] = __vimin3_u16x2(v[k], v[(k + 1) & 15], v[(k + 2) & 15]);
                mb = __vimin3_u16x2(m3[0], m3[3], m3[6]);
#pragma unroll
                for (int k = 1; k < 16; ++k) mb = __vmaxu2(mb, __vimin3_u16x2(m3[k], m3[(k + 3) & 15], m3[(k + 6) & 15]));
            }
            {
                unsigned m3[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) m3[k] = __vimax3_u16x2(v[k], v[(k + 1) & 15], v[(k + 2) & 15]);
                md = __vimax3_u16x2(m3[0], m3[3], m3[6]);
#pragma unroll
                for (int k = 1; k < 16; ++k) md = __vminu2(md, __vimax3_u16x2(m3[k], m3[(k + 3) & 15], m3[(k + 6) & 15]));
            }
            const unsigned x = fast_excess(c[0], mb, md);
            const int ix = bx - 2 + ex, iy = by - 1 + ey;
            lo = (int)(x & 0xffffu) > lim && in_areas(areas, ix, iy);
            hi = (int)(x >> 16) > lim && in_areas(areas, ix, iy + 1);
        }
        append(lo, at, corners, &s_nc);
        append(hi, at + DT_EX, corners, &s_nc);
    }
    __syncthreads();
    const int nc = s_nc;
    for (int i = t; i < nc; i += 256) {
        const int at = corners[i], ex = at & (DT_EX - 1), ey = at / DT_EX;
        const uint16_t* c = reinterpret_cast<const uint16_t*>(P + (ey + 3) * DT_PX + ex + 3);  // the pixel's own half
        const int b5[5] = {1, 4, 6, 4, 1};
        int A = 0, B = 0, C = 0;  // at most 256 * 255 * 255
#pragma unroll
        for (int r = -2; r <= 2; ++r) {
            int sxx = 0, syy = 0, sxy = 0;
#pragma unroll
            for (int k = -2; k <= 2; ++k) {
                const int ix = (int)c[2 * (r * DT_PX + k + 1)] - (int)c[2 * (r * DT_PX + k - 1)];
                const int iy = (int)c[2 * ((r + 1) * DT_PX + k)] - (int)c[2 * ((r - 1) * DT_PX + k)];
                sxx += b5[k + 2] * ix * ix;
                syy += b5[k + 2] * iy * iy;
                sxy += b5[k + 2] * ix * iy;
            }
            A += b5[r + 2] * sxx;
            B += b5[r + 2] * syy;
            C += b5[r + 2] * sxy;
        }
        const long long tr = (long long)A + B, rr = 25 * ((long long)A * B - (long long)C * C) - tr * tr;
        if (rr > harris_t) {
            R[at] = rr;
            atomicOr(&mask[ey][ex >> 5], 1u << (ex & 31));
        }
    }
    __syncthreads();
    // non-maximum suppression (ties to the lower index), survivors into the pair list's memory: no two
    // are neighbours, so at most a quarter of the evaluated pixels
    uint16_t* surv = pairs;
    static_assert(DT_PAIRS >= (DT_OX / 2) * (DT_OY / 2), "room for the survivors");
    for (int i0 = 32 * w; i0 < nc; i0 += 256) {
        bool keep = false;
        int at = 0;
        if (i0 + lane < nc) {
            at = corners[i0 + lane];
            const int ex = at & (DT_EX - 1), ey = at / DT_EX;
            if (ex >= 2 && ex < 2 + DT_OX && ey >= 1 && ey < 1 + DT_OY && (mask[ey][ex >> 5] >> (ex & 31) & 1u)) {
                const long long r = R[at];
                keep = true;
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy) {
                    const unsigned long long m = mask[ey + dy][0] | (unsigned long long)mask[ey + dy][1] << 32;
                    const unsigned nb = (unsigned)(m >> (ex - 1)) & 7u;
#pragma unroll
                    for (int dx = -1; dx <= 1; ++dx) {
                        if ((dx || dy) && (nb >> (dx + 1) & 1u)) {
                            const long long o = R[at + dy * DT_EX + dx];
                            keep &= r > o || (r == o && (dy > 0 || (dy == 0 && dx > 0)));
                        }
                    }
                }
            }
        }
        append(keep, at, surv, &s_n);
    }
    __syncthreads();
    if (t == 0) s_base = s_n ? atomicAdd(ncand, s_n) : 0;
    __syncthreads();
    for (int i = t; i < s_n; i += 256) {
        const int at = surv[i], pos = s_base + i;
        const long long r = R[at];
        if (pos < cap) {
            cand[pos] = Cand{r, (by - 1 + at / DT_EX) * W + bx - 2 + (at & (DT_EX - 1)), 0};
            atomicAdd(&hist[lorb_bin(r)], 1);
        }
    }
}

// key order: R' descending, index ascending == (u, ~idx) descending with u = R' with the sign
// bit flipped
__device__ __forceinline__ unsigned long long ukey(long long r) { return (unsigned long long)r ^ (1ull << 63); }

// Threshold digit of one radix-selection pass over the 256-bin histogram (threads 0..255 take a
// bin each; every thread of the block calls this): from the top, the bin b where the count of the
// bins from the top down to b first reaches `need` (the largest keys); from the bottom, the same
// counting up (the smallest indices).  Returns b and leaves in `need` what is still wanted among
// the keys of bin b.  If the count never reaches `need`, the last bin and the remainder, as a
// sequential scan would leave them.
__device__ __forceinline__ int select_digit(const int* hist, int* wsum, int& need, bool from_top, int* s_out) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const bool act = t < 256;
    const int b = from_top ? 255 - t : t;
    const int own = act ? hist[b] : 0;
    int v = own;  // inclusive prefix over the bins in scan order
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    if (act && lane == 31) wsum[w] = v;
    const int nd = need;
    __syncthreads();
    int S = v;
    if (act)
        for (int k = 0; k < w; ++k) S += wsum[k];
    if (t == 255) {  // the last bin in scan order: the fallback
        s_out[0] = b;
        s_out[1] = nd - (S - own);
    }
    __syncthreads();
    if (act && t < 255 && S >= nd && S - own < nd) {
        s_out[0] = b;
        s_out[1] = nd - (S - own);
    }
    __syncthreads();
    need = s_out[1];
    const int r = s_out[0];
    __syncthreads();
    return r;
}

// The N strongest of a crowded candidate set, sorted, by one block of SEL_THREADS threads: radix
// selection (8-bit digits, most significant first) of the N-th largest u; survivors above it are
// taken, and among those equal to it the lowest indices (a second radix selection on the index);
// then a bitonic sort.
struct SelectSmem {
    Cand win[LORB_MAX_POINTS];
    int hist[256], wsum[32], pick[2];
    unsigned long long prefix;
    int need, nwin;
};

__device__ void lorb_select(const Cand* cand, int n, int npts, int W, int* out_xy,
                            long long* out_resp, SelectSmem& sm) {
    int* hist = sm.hist;
    Cand* win = sm.win;
    unsigned long long& s_prefix = sm.prefix;
    int &s_need = sm.need, &s_nwin = sm.nwin;
    int *s_wsum = sm.wsum, *s_pick = sm.pick;
    const int t = threadIdx.x;
    const int want = min(n, npts);
    if (t == 0) {
        s_prefix = 0;
        s_need = want;
        s_nwin = 0;
    }
    __syncthreads();
    // radix selection of the want-th largest u (threshold value uT)
    unsigned long long mask = 0;
    for (int d = 7; d >= 0 && want > 0; --d) {
        for (int k = t; k < 256; k += SEL_THREADS) hist[k] = 0;
        __syncthreads();
        const unsigned long long prefix = s_prefix;
        for (int i = t; i < n; i += SEL_THREADS) {
            const unsigned long long u = ukey(__ldcg(&cand[i].r));
            if ((u & mask) == prefix) atomicAdd(&hist[(u >> (8 * d)) & 255], 1);
        }
        __syncthreads();
        int need = s_need;
        const int b = select_digit(hist, s_wsum, need, true, s_pick);
        if (t == 0) {
            s_prefix = prefix | ((unsigned long long)b << (8 * d));
            s_need = need;  // how many of the keys equal to the final prefix are still wanted
        }
        __syncthreads();
        mask |= 255ull << (8 * d);
    }
    const unsigned long long uT = s_prefix;
    const int need_eq = s_need;
    // the index threshold among keys equal to uT: the need_eq-th smallest index
    int iT = INT_MAX;
    if (want > 0) {
        unsigned prefix = 0, imask = 0;
        if (t == 0) s_need = need_eq;
        __syncthreads();
        for (int d = 3; d >= 0; --d) {
            for (int k = t; k < 256; k += SEL_THREADS) hist[k] = 0;
            __syncthreads();
            for (int i = t; i < n; i += SEL_THREADS) {
                if (ukey(__ldcg(&cand[i].r)) != uT) continue;
                const unsigned ix = (unsigned)__ldcg(&cand[i].idx);
                if ((ix & imask) == prefix) atomicAdd(&hist[(ix >> (8 * d)) & 255], 1);
            }
            __syncthreads();
            int need = s_need;
            const int b = select_digit(hist, s_wsum, need, false, s_pick);
            if (t == 0) {
                s_prefix = prefix | ((unsigned)b << (8 * d));
                s_need = need;
            }
            __syncthreads();
            prefix = (unsigned)s_prefix;
            imask |= 255u << (8 * d);
        }
        iT = (int)prefix;
    }
    // gather the winners: u > uT, or u == uT with index <= iT
    for (int i = t; i < n && want > 0; i += SEL_THREADS) {
        const Cand c{__ldcg(&cand[i].r), __ldcg(&cand[i].idx), 0};
        const unsigned long long u = ukey(c.r);
        if (u > uT || (u == uT && c.idx <= iT)) {
            const int pos = atomicAdd(&s_nwin, 1);
            if (pos < LORB_MAX_POINTS) win[pos] = c;
        }
    }
    __syncthreads();
    // bitonic sort of the winners (padded with the weakest key)
    int m = 1;
    while (m < want) m <<= 1;
    for (int i = want + t; i < m; i += SEL_THREADS) win[i] = Cand{LLONG_MIN, INT_MAX, 0};
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = t; i < m; i += SEL_THREADS) {
                const int l = i ^ j;
                if (l <= i) continue;
                const Cand a = win[i], b = win[l];
                // a before b when a is stronger: R' descending, index ascending
                const bool a_first = a.r > b.r || (a.r == b.r && a.idx < b.idx);
                const bool up = (i & k) == 0;
                if (up != a_first) {
                    win[i] = b;
                    win[l] = a;
                }
            }
            __syncthreads();
        }
    for (int i = t; i < want; i += SEL_THREADS) {
        out_xy[2 * i] = win[i].idx % W;
        out_xy[2 * i + 1] = win[i].idx / W;
        out_resp[i] = win[i].r;
    }
}

// The candidates in the bins at or above the threshold bin (where the count from the top reaches
// N) appended to cand2: a superset of the N strongest, typically a small one.  Grid-stride; every
// block finds the threshold bin from the histogram (a suffix sum over the bins).  The last block to
// finish (a ticket; no block waits) writes the number of points, clears the counters for the next
// call, and selects the points itself when cand2 is too crowded to be ranked by counting.
constexpr int PRUNE_THREADS = 1024, PRUNE_BLOCKS = 64;
constexpr int RANK_MAX = 8192;  // candidates that lorb_rank_brief ranks by counting
__global__ void __launch_bounds__(PRUNE_THREADS) lorb_prune(const Cand* cand, LorbCount* cnt, int cap,
                                                            int npts, Cand* cand2, int W,
                                                            const __grid_constant__ LorbPattern pat,
                                                            int* out_xy, long long* out_resp,
                                                            int* count) {
    static_assert(PRUNE_THREADS == LORB_BINS && PRUNE_THREADS == SEL_THREADS, "one bin per thread; the block also selects");
    __shared__ SelectSmem sm;
    __shared__ int wsum[32];
    __shared__ int s_b, s_last;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    pdl_trigger();
    pdl_wait();
    // the pattern to memory, where lorb_rank_brief's lanes read it side by side (lane-dependent reads of
    // the parameter space are serialised)
    if (blockIdx.x == 1 && t < 256) cnt->pat[t] = pat.p[t];
    const int n = min(cnt->n, cap), want = min(n, npts);
    const int* hist = cnt->hist;
    if (t == 0) s_b = LORB_BINS;  // want == 0: nothing
    // suffix sums: thread t takes bin 1023 - t and an inclusive prefix sum over t
    const int b = LORB_BINS - 1 - t;
    int v = hist[b];
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    if (lane == 31) wsum[w] = v;
    __syncthreads();
    if (w == 0) {
        int x = wsum[lane];
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += o;
        }
        wsum[lane] = x;
    }
    __syncthreads();
    const int S = v + (w > 0 ? wsum[w - 1] : 0);  // candidates in bins >= b
    const int S_above = S - hist[b];             // in bins > b
    if (want > 0 && S >= want && S_above < want) s_b = b;
    __syncthreads();
    const int bT = s_b;
    for (int i0 = blockIdx.x * PRUNE_THREADS; i0 < n; i0 += gridDim.x * PRUNE_THREADS) {
        const int i = i0 + t;
        Cand cv{0, 0, 0};
        bool keep = false;
        if (i < n) {
            cv = cand[i];
            keep = lorb_bin(cv.r) >= bT;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (!m) continue;
        int base = 0;
        const int leader = __ffs(m) - 1;
        if (lane == leader) base = atomicAdd(&cnt->n2, __popc(m));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (keep) cand2[base + __popc(m & ((1u << lane) - 1))] = cv;
    }
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(&cnt->done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    // every block has read n and the histogram, and appended to cand2
    cnt->hist[t] = 0;
    if (t == 0) {
        *count = want;
        cnt->n = 0;
        cnt->done = 0;
    }
    const int n2 = __ldcg(&cnt->n2);
    if (n2 > RANK_MAX) lorb_select(cand2, n2, npts, W, out_xy, out_resp, sm);
}

// A block per candidate: its rank among the pruned candidates (how many are stronger, or as strong
// with a lower index) is its place among the points; a candidate ranked below N is dropped.  Then the
// point's BRIEF bits from a 35 x 35 patch of the frame: gray, the separable [1,4,6,4,1] sums (the
// unnormalised S, at most 255 * 256), and one comparison per thread, packed by ballots.  A few
// hundred points need 0.4 MB of patches, so no smoothed map of the image is ever formed; the kernel
// is a chain of latencies (9 us for 500 points of a 4K view, against 19 us for a one-block selection
// and 11 us for BRIEF on the map, whose pattern was read from parameter space lane by lane).
constexpr int RB_P = 35, RB_W = 36, RB_S = 31;  // patch and its row pitch, positions of S
__global__ void __launch_bounds__(256) lorb_rank_brief(const uint8_t* frame, long long pitch, int W,
                                                       const Cand* cand2, const LorbCount* cnt,
                                                       const int* count, int* xy,
                                                       long long* resp, unsigned* desc) {
    __shared__ __align__(4) uint8_t g[RB_P * RB_W];
    __shared__ uint16_t hs[RB_P][RB_S + 1], S[RB_S][RB_S + 1];
    __shared__ int s_w[8];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    pdl_trigger();
    pdl_wait();
    const int n2 = cnt->n2, want = *count;
    const bool selected = n2 > RANK_MAX;  // lorb_prune has written xy and resp
    const bool words = word_aligned(frame, pitch);
    for (int i = blockIdx.x; i < (selected ? want : n2); i += gridDim.x) {
        int k = i, x, y;
        if (selected) {
            x = xy[2 * k];
            y = xy[2 * k + 1];
        } else {
            const Cand c = cand2[i];
            int c0 = 0;
            for (int j = t; j < n2; j += 256) {
                const Cand o = cand2[j];
                c0 += o.r > c.r || (o.r == c.r && o.idx < c.idx);
            }
            c0 = __reduce_add_sync(0xffffffffu, c0);
            if (lane == 0) s_w[w] = c0;
            __syncthreads();
            k = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) k += s_w[q];
            x = c.idx % W;
            y = c.idx / W;
            if (t == 0 && k < want) {
                xy[2 * k] = x;
                xy[2 * k + 1] = y;
                resp[k] = c.r;
            }
        }
        if (k < want) {  // the whole block
            // points keep 18 px from the border, so the patch and a 36th column lie inside the image
            const char4 pr = cnt->pat[t];
            const uint8_t* p0 = frame + (long long)(y - 17) * pitch + 3LL * (x - 17);
            if (words) {
                // groups of 4 pixels (12 bytes at any offset): four aligned words, shifted
                const int off = (3 * (x - 17)) & 3;
                for (int q = t; q < RB_P * (RB_W / 4); q += 256) {
                    const int r = q / (RB_W / 4), j = q - r * (RB_W / 4);
                    const unsigned* p = reinterpret_cast<const unsigned*>(p0 - off + (long long)r * pitch + 12 * j);
                    const unsigned v0 = __ldca(p), v1 = __ldca(p + 1), v2 = __ldca(p + 2), v3 = off ? __ldca(p + 3) : 0u;
                    const unsigned a = __funnelshift_r(v0, v1, 8 * off), b = __funnelshift_r(v1, v2, 8 * off),
                                   c = __funnelshift_r(v2, v3, 8 * off);
                    unsigned o[4];
                    gray4(a, b, c, o);
                    *reinterpret_cast<unsigned*>(g + r * RB_W + 4 * j) = o[0] | o[1] << 8 | o[2] << 16 | o[3] << 24;
                }
            } else {
                for (int q = t; q < RB_P * RB_P; q += 256) {
                    const int r = q / RB_P, c = q - r * RB_P;
                    const uint8_t* p = p0 + (long long)r * pitch + 3 * c;
                    g[r * RB_W + c] = (uint8_t)gray_of(__ldca(p), __ldca(p + 1), __ldca(p + 2));
                }
            }
            __syncthreads();
            for (int q = t; q < RB_P * RB_S; q += 256) {
                const int r = q / RB_S, c = q - r * RB_S;
                const uint8_t* p = g + r * RB_W + c;
                hs[r][c] = (uint16_t)(p[0] + 4 * p[1] + 6 * p[2] + 4 * p[3] + p[4]);
            }
            __syncthreads();
            for (int q = t; q < RB_S * RB_S; q += 256) {
                const int r = q / RB_S, c = q - r * RB_S;
                S[r][c] = (uint16_t)(hs[r][c] + 4 * hs[r + 1][c] + 6 * hs[r + 2][c] + 4 * hs[r + 3][c] + hs[r + 4][c]);
            }
            __syncthreads();
            const unsigned bits = __ballot_sync(0xffffffffu, S[15 + pr.y][15 + pr.x] > S[15 + pr.w][15 + pr.z]);
            if (lane == 0) desc[8 * k + w] = bits;  // bit b of the descriptor: byte b/8, bit b%8 (little endian)
        }
        __syncthreads();
    }
}

}  // namespace

struct stitch_lorb {
    int device = 0;
    int max_w = 0, max_h = 0, max_points = 0, cap = 0;
    Cand* cand = nullptr;
    Cand* cand2 = nullptr;  // the pruned candidates
    LorbCount* cnt = nullptr;
    bool stale = false;  // a refused launch left counts behind: the next call clears them
};

static void lorb_free(stitch_lorb* c) {
    if (!c) return;
    cudaFree(c->cand);
    cudaFree(c->cand2);
    cudaFree(c->cnt);
    delete c;
}

extern "C" stitch_status stitch_lorb_create(int32_t max_width, int32_t max_height, int32_t max_points, int32_t device,
                                            stitch_lorb** out) {
    if (!out) return STITCH_EINVAL;
    *out = nullptr;
    if (max_width < 2 * LORB_MARGIN + 1 || max_height < 2 * LORB_MARGIN + 1 || max_points < 1 ||
        max_points > LORB_MAX_POINTS || (long long)max_width * max_height > (1LL << 30))
        return STITCH_EINVAL;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
        cudaGetLastError();
        return STITCH_ECUDA;
    }
    if (device < 0 || device >= ndev) return STITCH_EINVAL;
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(device) != cudaSuccess) return STITCH_ECUDA;
    stitch_lorb* c = new (std::nothrow) stitch_lorb();
    if (!c) return STITCH_ENOMEM;
    c->device = device;
    c->max_w = max_width;
    c->max_h = max_height;
    c->max_points = max_points;
    c->cap = (int)(((size_t)max_width + 1) / 2 * (((size_t)max_height + 1) / 2));  // NMS survivors are never adjacent
    stitch_status st = STITCH_OK;
    if (cudaMalloc(&c->cand, (size_t)c->cap * sizeof(Cand)) != cudaSuccess ||
        cudaMalloc(&c->cand2, (size_t)c->cap * sizeof(Cand)) != cudaSuccess ||
        cudaMalloc(&c->cnt, sizeof(LorbCount)) != cudaSuccess) {
        cudaGetLastError();
        st = STITCH_ENOMEM;
    }
    if (st == STITCH_OK && cudaMemset(c->cnt, 0, sizeof(LorbCount)) != cudaSuccess) st = STITCH_ECUDA;
    if (prev >= 0) cudaSetDevice(prev);
    if (st != STITCH_OK) {
        lorb_free(c);
        return st;
    }
    *out = c;
    return STITCH_OK;
}

extern "C" void stitch_lorb_destroy(stitch_lorb* c) {
    if (!c) return;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(c->device);
    cudaDeviceSynchronize();
    lorb_free(c);
    if (prev >= 0) cudaSetDevice(prev);
}

extern "C" stitch_status stitch_lorb_detect(stitch_lorb* c, const uint8_t* frame, int32_t width, int32_t height,
                                            int64_t pitch, const int32_t* areas, int32_t n_areas,
                                            const stitch_lorb_params* params, const int8_t* pattern,
                                            int32_t* xy, int64_t* resp, uint8_t* desc, int32_t* count,
                                            void* stream) {
    if (!c || !frame || !params || !pattern || !xy || !resp || !desc || !count) return STITCH_EINVAL;
    if (width < 1 || height < 1 || width > c->max_w || height > c->max_h || pitch < 3LL * width || n_areas < 0 ||
        n_areas > LORB_MAX_AREAS || (n_areas > 0 && !areas) || params->fast_t < 0 || params->max_points < 0 ||
        params->max_points > c->max_points)
        return STITCH_EINVAL;
    LorbPattern pat;
    for (int k = 0; k < 256; ++k)
        for (int j = 0; j < 4; ++j) {
            if (pattern[4 * k + j] < -15 || pattern[4 * k + j] > 15) return STITCH_EINVAL;
        }
    memcpy(pat.p, pattern, sizeof(pat.p));
    // areas clipped to the margin; bounding box of the candidates, and of what BRIEF reads
    LorbAreas ar{};
    int bx0 = width, by0 = height, bx1 = 0, by1 = 0;
    for (int k = 0; k < n_areas; ++k) {
        const int x0 = std::max(areas[4 * k], LORB_MARGIN), y0 = std::max(areas[4 * k + 1], LORB_MARGIN);
        const int x1 = std::min(areas[4 * k + 2], width - LORB_MARGIN), y1 = std::min(areas[4 * k + 3], height - LORB_MARGIN);
        if (x1 <= x0 || y1 <= y0) continue;
        ar.r[ar.n][0] = x0;
        ar.r[ar.n][1] = y0;
        ar.r[ar.n][2] = x1;
        ar.r[ar.n][3] = y1;
        ++ar.n;
        bx0 = std::min(bx0, x0);
        by0 = std::min(by0, y0);
        bx1 = std::max(bx1, x1);
        by1 = std::max(by1, y1);
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != c->device && cudaSetDevice(c->device) != cudaSuccess) return STITCH_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    stitch_status st = STITCH_OK;
    auto ok = [&](cudaError_t e) {
        if (e != cudaSuccess && st == STITCH_OK) st = STITCH_ECUDA;
    };
    bool keep = false;
    if (c->stale) {
        // while the stream is captured the clearing is part of the graph: the next call clears too
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        ok(cudaStreamIsCapturing(s, &cap));
        keep = cap != cudaStreamCaptureStatusNone;
        ok(cudaMemsetAsync(c->cnt, 0, offsetof(LorbCount, pat), s));
    }
    if (ar.n > 0) {
        // tiles over the candidates' box, owned pixels starting at a column 1 modulo 4
        const int ox = 1 + ((bx0 - 1) & ~3), oy = by0;
        pdl_launch(lorb_detect, dim3((bx1 - ox + DT_OX - 1) / DT_OX, (by1 - oy + DT_OY - 1) / DT_OY), 256, 0, s, frame, pitch,
                   width, height, ox, oy, ar, std::min(params->fast_t, 255) + 256, (long long)params->harris_t, c->cand,
                   &c->cnt->n, c->cap, c->cnt->hist, &c->cnt->n2);
    } else {
        ok(cudaMemsetAsync(&c->cnt->n2, 0, sizeof(int), s));
    }
    pdl_launch(lorb_prune, PRUNE_BLOCKS, PRUNE_THREADS, 0, s, c->cand, c->cnt, c->cap, params->max_points, c->cand2, width,
               pat, xy, reinterpret_cast<long long*>(resp), count);
    // the pruned candidates are a few more than the points: a block each, or a few passes
    pdl_launch(lorb_rank_brief, std::min(2 * params->max_points + 64, 1216), 256, 0, s, frame, pitch, width, c->cand2, c->cnt,
               count, xy, reinterpret_cast<long long*>(resp), reinterpret_cast<unsigned*>(desc));
    ok(cudaGetLastError());
    c->stale = keep || st != STITCH_OK;
    if (prev >= 0 && prev != c->device) cudaSetDevice(prev);
    return st;
}
