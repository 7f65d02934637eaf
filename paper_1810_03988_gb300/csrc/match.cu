// Feature matching and homography estimation (Sec. 4.2, Algorithm 3) on the GPU: Multi-Probe LSH
// matching of BRIEF descriptors, then PROSAC over the matches in quality order.  Decisions are
// those of the definition in integer arithmetic (hash keys, Hamming distances, ratio test,
// ordering) and in IEEE double without contractions (every double operation below is an explicit
// round-to-nearest intrinsic, evaluated in the order of the definition), so that the PROSAC
// samples, hypotheses, inlier counts and the refit are bit-identical to a sequential evaluation:
//   M1 L tables hashing a descriptor to k given bit positions; a query probes its own bucket and
//      the k buckets at Hamming distance 1 of every table; the nearest probed descriptor (ties to
//      the lower index) is the match when its distance <= max_dist and den * d1 < num * d2 (d2:
//      nearest other probed index, none passes);
//   M2 quality order: distance ascending, query index ascending;
//   M3 PROSAC (Chum and Matas growth schedule, m = 4, T_N = 200000, its increments
//      T_{n+1} - T_n evaluated exactly as integer ceilings; the newest of the top n plus 3
//      of the top n - 1, or 4 of the top n once t > T'_n, drawn without replacement from given
//      random words); 4-point homography (h33 = 1) by 8x8 Gaussian elimination with partial
//      pivoting in coordinates normalised per image (bounding box of the matched points);
//      inliers: w > 0 and squared transfer error < (inlier_px scaled)^2; best: most inliers,
//      ties to the earlier iteration; least squares on its inliers; returned in pixels.
//
// Kernels, in launch order: mt_keys (hash keys of both images), mt_match (a warp per query against every
// descriptor of image B), mt_rank (quality order by counting, normalised coordinates, growth
// schedule), mt_hypotheses (four iterations per block: samples, 4-point solves, inlier counts, the
// best by an atomic maximum) and mt_final (inlier flags, ordered normal-equation sums, refit, back to
// pixels).  What bounds them is FP64: this part issues one double-precision instruction per warp
// and scheduler about every 64 cycles, with no gain from independent ones, so a chain costs its
// number of instructions times 64 cycles, and lanes left idle are lost.
#include <climits>

#include "stitch_internal.cuh"

namespace {

constexpr int MT_MAX_POINTS = 2048;
constexpr int MT_MAX_TABLES = 32, MT_MAX_BITS = 20;
constexpr int MT_MAX_WORDS = 32;  // key words of a descriptor

struct LshBits {
    int L, k;
    uint8_t b[MT_MAX_TABLES][MT_MAX_BITS];
};

struct Norm {
    double ca0, ca1, cb0, cb1, sa, sb;
};

__device__ __forceinline__ double dA(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dS(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dM(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dD(double a, double b) { return __ddiv_rn(a, b); }

// State of one call, set up by mt_keys.
struct MtState {
    int mn[4], mx[4];         // bounding boxes of the matched points: x, y in image A, x, y in image B
    int n;                    // matches
    int pad;
    unsigned long long best;  // (inliers + 1) << 32 | (2^32 - 1 - iteration) of the best hypothesis, 0 when none
    Norm norm;
    double t2;                // squared inlier threshold in normalised coordinates,
    float t_in, t_out;        // and a little below and above it (FastInlier)
};

constexpr float MT_EPS = 9.5367431640625e-7f;  // 2^-20, see FastInlier

// Hash keys as words whose difference is tested at once: with k <= 16 two tables share a word,
// otherwise a table has a word of its own.  Words are padded to a power of two of at least 2; unused
// words and halves differ in every bit.
__host__ __device__ __forceinline__ bool mt_packed(const LshBits& lb) { return lb.k <= 16; }
inline int mt_words(const LshBits& lb) {
    int w = 2;
    while (w < (mt_packed(lb) ? (lb.L + 1) / 2 : lb.L)) w *= 2;
    return w;
}

// One key word (blockIdx.y) of 128 descriptors of image A (blockIdx.z 0) or B; the first block also
// sets up the call's state.  The bit positions are the same for the whole block, so they come from the
// parameter space as uniform loads; the descriptors' words from shared memory.
__global__ void __launch_bounds__(128) mt_keys(const unsigned* desc_a, const int* count_a,
                                               const unsigned* desc_b, const int* count_b,
                                               const __grid_constant__ LshBits lb, int cap, unsigned* keys_a,
                                               unsigned* keys_b, MtState* st) {
    __shared__ unsigned d[8][128];
    pdl_trigger();
    pdl_wait();
    const int t = threadIdx.x, i = blockIdx.x * 128 + t, w = blockIdx.y;
    const bool isb = blockIdx.z != 0;
    if (blockIdx.x == 0 && w == 0 && !isb && t < 4) {
        st->mn[t] = INT_MAX;
        st->mx[t] = INT_MIN;
        if (t == 0) {
            st->n = 0;
            st->best = 0ull;
        }
    }
    const int n = min(isb ? *count_b : *count_a, cap);
    if (i >= n) return;
    const unsigned* src = (isb ? desc_b : desc_a) + 8 * (size_t)i;
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k][t] = __ldcg(src + k);
    auto key_of = [&](int l) {
        unsigned key = 0;
#pragma unroll 4
        for (int j = 0; j < lb.k; ++j) {
            const int bit = lb.b[l][j];
            key |= ((d[bit >> 5][t] >> (bit & 31)) & 1u) << j;
        }
        return key;
    };
    unsigned key = isb ? 0u : 0xffffffffu;
    if (mt_packed(lb)) {
        if (2 * w < lb.L) key = key_of(2 * w) | (key & 0xffff0000u);
        if (2 * w + 1 < lb.L) key = key_of(2 * w + 1) << 16 | (key & 0xffffu);
    } else if (w < lb.L) {
        key = key_of(w);
    }
    (isb ? keys_b : keys_a)[(size_t)w * cap + i] = key;
}

__device__ __forceinline__ int hamming(const unsigned* a, const unsigned* b) {
    int d = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) d += __popc(a[k] ^ b[k]);
    return d;
}

struct Top2 {
    int d1, b1, d2, b2;
};

__device__ __forceinline__ void top2_add(Top2& t, int d, int b) {
    if (d < t.d1 || (d == t.d1 && b < t.b1)) {
        if (b != t.b1) {
            t.d2 = t.d1;
            t.b2 = t.b1;
        }
        t.d1 = d;
        t.b1 = b;
    } else if (b != t.b1 && (d < t.d2 || (d == t.d2 && b < t.b2))) {
        t.d2 = d;
        t.b2 = b;
    }
}

// A warp per query, its lanes over every descriptor of image B: those that the query meets in a table
// (keys differing in at most one bit) are gathered and their distances taken 32 at a time.  Image B's
// keys pass through shared memory in chunks, so that their loads are all in flight, the query's stay in
// registers; a pair then costs some 30 instructions.  11 us for 1000 x 1000 points and 8 tables (38 us
// with the keys read from global memory pair by pair); hashing into sorted buckets and probing them
// took 32 us (a bitonic sort per table, then a chain of dependent loads per probe).
constexpr int MT_CHUNK = 8192;  // key words of a chunk
template <bool PACKED, int NW>
__global__ void __launch_bounds__(256) mt_match(const unsigned* desc_a, const int* count_a,
                                                const unsigned* desc_b, const int* count_b,
                                                const unsigned* keys_a, const unsigned* keys_b,
                                                int cap, const int* xy_a, const int* xy_b,
                                                int max_dist, int rnum, int rden, int2* best,
                                                MtState* st) {
    constexpr int CB = MT_CHUNK / NW;  // descriptors of a chunk
    __shared__ unsigned s_kb[NW][CB];
    __shared__ uint16_t s_hit[8][64];
    __shared__ int s_mn[4], s_mx[4], s_n;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31, a = blockIdx.x * 8 + w;
    const bool aligned_b = (reinterpret_cast<uintptr_t>(desc_b) & 15) == 0;
    pdl_trigger();
    pdl_wait();
    const int na = min(*count_a, cap), nb = min(*count_b, cap);
    if (blockIdx.x * 8 >= na) return;
    if (t < 4) {
        s_mn[t] = INT_MAX;
        s_mx[t] = INT_MIN;
        if (t == 0) s_n = 0;
    }
    unsigned da[8], ka[NW];
#pragma unroll
    for (int k = 0; k < 8; ++k) da[k] = a < na ? desc_a[8 * (size_t)a + k] : 0u;
#pragma unroll
    for (int k = 0; k < NW; ++k) ka[k] = a < na ? keys_a[(size_t)k * cap + a] : 0u;
    constexpr int INF = 1 << 30;
    Top2 best2{INF, -1, INF, -1};
    int nh = 0;
    auto take = [&](int n) {  // the first n gathered descriptors
        if (lane < n) {
            const int b = s_hit[w][lane];
            const uint4* q = reinterpret_cast<const uint4*>(desc_b) + 2 * (size_t)b;
            unsigned db[8];
            if (aligned_b) {
                const uint4 q0 = __ldcg(q), q1 = __ldcg(q + 1);
                db[0] = q0.x, db[1] = q0.y, db[2] = q0.z, db[3] = q0.w;
                db[4] = q1.x, db[5] = q1.y, db[6] = q1.z, db[7] = q1.w;
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) db[k] = __ldcg(desc_b + 8 * (size_t)b + k);
            }
            top2_add(best2, hamming(da, db), b);
        }
        __syncwarp();
    };
    for (int c0 = 0; c0 < nb; c0 += CB) {
        const int cn = min(CB, nb - c0);
        __syncthreads();
#pragma unroll 8
        for (int q = t; q < NW * CB; q += 256) {
            const int i = q % CB;
            if (i < cn) s_kb[q / CB][i] = __ldcg(keys_b + (size_t)(q / CB) * cap + c0 + i);
        }
        __syncthreads();
        if (a >= na) continue;
        for (int b0 = 0; b0 < cn; b0 += 32) {
            const int b = b0 + lane;
            // x & (x - 1) clears the lowest bit of x; on packed halves a borrow leaves the lower half
            // only when that half is 0, that is, when it has already met
            unsigned acc = 0xffffffffu;
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const unsigned x = ka[k] ^ s_kb[k][b];
                const unsigned z = x & (x - (PACKED ? 0x00010001u : 1u));
                acc = PACKED ? __vminu2(acc, z) : min(acc, z);
            }
            const bool hit = b < cn && (PACKED ? (acc & 0xffffu) == 0u || (acc >> 16) == 0u : acc == 0u);
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (m == 0u) continue;
            if (hit) s_hit[w][nh + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(c0 + b);
            nh += __popc(m);
            __syncwarp();
            if (nh >= 32) {
                take(32);
                nh -= 32;
                const uint16_t rest = s_hit[w][32 + lane];
                __syncwarp();
                if (lane < nh) s_hit[w][lane] = rest;
                __syncwarp();
            }
        }
    }
    if (a < na) {
        take(nh);
        // merge: the union's two nearest distinct indices are among the lanes' two nearest
        for (int off = 16; off > 0; off >>= 1) {
            Top2 o;
            o.d1 = __shfl_down_sync(0xffffffffu, best2.d1, off);
            o.b1 = __shfl_down_sync(0xffffffffu, best2.b1, off);
            o.d2 = __shfl_down_sync(0xffffffffu, best2.d2, off);
            o.b2 = __shfl_down_sync(0xffffffffu, best2.b2, off);
            if (o.b1 >= 0) top2_add(best2, o.d1, o.b1);
            if (o.b2 >= 0) top2_add(best2, o.d2, o.b2);
        }
        if (lane == 0) {
            const bool ok = best2.b1 >= 0 && best2.d1 <= max_dist &&
                            (best2.d2 == INF || (long long)rden * best2.d1 < (long long)rnum * best2.d2);
            best[a] = make_int2(ok ? best2.b1 : -1, best2.d1);
            if (ok) {
                const int v[4] = {xy_a[2 * a], xy_a[2 * a + 1], xy_b[2 * best2.b1], xy_b[2 * best2.b1 + 1]};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    atomicMin(&s_mn[k], v[k]);
                    atomicMax(&s_mx[k], v[k]);
                }
                atomicAdd(&s_n, 1);
            }
        }
    }
    __syncthreads();
    if (t < 4 && s_n > 0) {
        atomicMin(&st->mn[t], s_mn[t]);
        atomicMax(&st->mx[t], s_mx[t]);
        if (t == 0) atomicAdd(&st->n, s_n);
    }
}

// The growth schedule by one block of 256 threads.  The top n grows to n + 1 at iteration E_j
// (j = n - 4), E_0 = 1 and E_{j+1} = E_j + ceil(T_N m n (n-1) (n-2) / (N (N-1) (N-2) (N-3))) (m = 4,
// T_N = 200000: the exact increment T_{n+1} - T_n of T_n = T_N C(n, m) / C(N, m)), up to n = N.
__device__ __forceinline__ void mt_schedule(int N, long long* E) {
    __shared__ long long wsum[8];
    constexpr int PT = MT_MAX_POINTS / 256;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (N < 4) return;
    const int K = N - 4;  // growth events j = 0 .. K-1 (n = 4 + j)
    const long long Q = (long long)N * (N - 1) * (N - 2) * (N - 3);
    long long d[PT], v = 0;
#pragma unroll
    for (int e = 0; e < PT; ++e) {
        const long long n = 4 + PT * t + e;
        d[e] = PT * t + e < K ? (800000LL * n * (n - 1) * (n - 2) + Q - 1) / Q : 0;
        v += d[e];
    }
    long long s = v;  // inclusive sums over the threads
    for (int off = 1; off < 32; off <<= 1) {
        const long long o = __shfl_up_sync(0xffffffffu, s, off);
        if (lane >= off) s += o;
    }
    if (lane == 31) wsum[w] = s;
    __syncthreads();
    for (int k = 0; k < w; ++k) s += wsum[k];
    long long x = 1 + s - v;
#pragma unroll
    for (int e = 0; e < PT; ++e) {
        if (PT * t + e <= K) E[PT * t + e] = x;
        x += d[e];
    }
}

// A warp per query: an accepted match's place in quality order is the number of accepted matches
// before it.  It writes the match and its normalised coordinates (x, y, u, v), the latter also in
// single precision for the inlier tests.  The last block computes the growth schedule.
__global__ void __launch_bounds__(256) mt_rank(const int2* best, const int* count_a, int cap,
                                               const int* xy_a, const int* xy_b,
                                               MtState* st, int* matches,
                                               int* n_matches, double* xyuv,
                                               float* xyuvf, long long* E, double inlier_px) {
    pdl_trigger();
    pdl_wait();
    const int t = threadIdx.x, lane = t & 31, N = st->n;
    if (blockIdx.x == gridDim.x - 1) {
        mt_schedule(N, E);
        return;
    }
    const int a = blockIdx.x * 8 + (t >> 5), na = min(*count_a, cap);
    const bool first = blockIdx.x == 0 && t < 32;  // writes the call's results
    if (first && lane == 0) *n_matches = N;
    const int2 m = a < na ? best[a] : make_int2(-1, 0);
    if (m.x < 0 && !first) return;
    // normalisation: lane 0 .. 3 takes x, y of image A, x, y of image B
    const int l = lane & 3, q = l & 2;
    double c = 0.0, sc = 1.0;
    if (N > 0) {
        c = dM(0.5, dA((double)st->mn[l], (double)st->mx[l]));
        const int r = max(st->mx[q] - st->mn[q], st->mx[q + 1] - st->mn[q + 1]);
        sc = dD(2.0, (double)(r > 1 ? r : 1));
    }
    if (first && lane < 4) {
        double* z = &st->norm.ca0;
        z[l] = c;
        if (l == 0) st->norm.sa = sc;
        if (l == 2) {
            const double tn = dM(inlier_px, sc), t2 = dM(tn, tn);
            st->norm.sb = sc;
            st->t2 = t2;
            st->t_in = __double2float_rd(t2) * (1.0f - MT_EPS);
            st->t_out = __double2float_ru(t2) * (1.0f + MT_EPS);
        }
    }
    if (m.x < 0) return;
    int r = 0;
    for (int i = lane; i < na; i += 32) {
        const int2 o = best[i];
        r += o.x >= 0 && (o.y < m.y || (o.y == m.y && i < a));
    }
    r = __reduce_add_sync(0xffffffffu, r);
    if (lane < 3) matches[3 * r + lane] = lane == 0 ? a : lane == 1 ? m.x : m.y;
    if (lane < 4) {
        const double v = dM(dS((double)(l < 2 ? xy_a[2 * a + l] : xy_b[2 * m.x + l - 2]), c), sc);
        xyuv[4 * r + l] = v;
        xyuvf[4 * r + l] = (float)v;
    }
}

// |x| of a finite or infinite double orders like its bit pattern read as an integer.
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffll; }

__device__ __forceinline__ bool inlier(const double h[8], double x, double y, double u, double v, double t2) {
    const double w = dA(dA(dM(h[6], x), dM(h[7], y)), 1.0);
    if (!(w > 0.0)) return false;
    const double pu = dS(dD(dA(dA(dM(h[0], x), dM(h[1], y)), h[2]), w), u);
    const double pv = dS(dD(dA(dA(dM(h[3], x), dM(h[4], y)), h[5]), w), v);
    return dA(dM(pu, pu), dM(pv, pv)) < t2;
}

__device__ __forceinline__ int nth_free(int j, const int* chosen, int c) {
    int s[4];
    for (int i = 0; i < c; ++i) s[i] = chosen[i];
    for (int i = 1; i < c; ++i)
        for (int k = i; k > 0 && s[k - 1] > s[k]; --k) {
            const int tmp = s[k];
            s[k] = s[k - 1];
            s[k - 1] = tmp;
        }
    for (int i = 0; i < c; ++i)
        if (s[i] <= j) ++j;
    return j;
}

// a / b for finite b; a zero a, which half the entries of a DLT system are and which the division
// leaves to its slow path, gets its signed zero directly.
__device__ __forceinline__ double quotient(double a, double b) {
    const unsigned long long x = (unsigned long long)__double_as_longlong(a), y = (unsigned long long)__double_as_longlong(b);
    const bool zero = (x << 1) == 0ull;
    const double q = dD(zero ? 1.0 : a, b);
    return zero ? __longlong_as_double((long long)((x ^ y) & (1ull << 63))) : q;
}

// M h = r by 8 lanes (a lane per row of A = [M | r], four systems per warp): every entry receives the
// operations of the sequential elimination with partial pivoting in the same order, so h is bit-identical.
// Rows stay in their lanes; a lane keeps its row's place in the current order, and the pivot is the
// largest magnitude, ties to the first row in that order.  240 double-precision instructions for four
// systems, 8 us; a block per system with a thread per entry kept three schedulers busy for each.  False
// when a pivot is below 1e-12 in magnitude or NaN.  All 32 lanes call it; h is complete in each.
__device__ bool solve8(double A[9], double h[8]) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, group = lane & 24;
    int place = lane & 7;
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        long long v = place >= c ? abs_bits(A[c]) : -1;
        int p = place;
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) {
            const long long ov = __shfl_xor_sync(FULL, v, off);
            const int op = __shfl_xor_sync(FULL, p, off);
            if (ov > v || (ov == v && op < p)) {
                v = ov;
                p = op;
            }
        }
        ok &= v >= __double_as_longlong(1e-12) && v <= 0x7ff0000000000000ll;
        place = place == p ? c : place == c ? p : place;  // the pivot row and row c change places
        const int src = group + __ffs(__ballot_sync(FULL, place == c) >> group) - 1;
        const double f = quotient(A[c], __shfl_sync(FULL, A[c], src));
#pragma unroll
        for (int j = c + 1; j < 9; ++j) {
            const double x = __shfl_sync(FULL, A[j], src);
            if (place > c) A[j] = dS(A[j], dM(f, x));
        }
    }
    double prod[8];
#pragma unroll
    for (int c = 7; c >= 0; --c) {
        double s = A[8];
#pragma unroll
        for (int k = c + 1; k < 8; ++k) s = dS(s, prod[k]);
        const int src = group + __ffs(__ballot_sync(FULL, place == c) >> group) - 1;
        h[c] = __shfl_sync(FULL, quotient(s, place == c ? A[c] : 1.0), src);
        prod[c] = dM(A[c], h[c]);
    }
    return ok;
}

// The inlier test of a hypothesis with its decision taken in single precision wherever that is
// certain.  With (a, b) = (num_u - u w, num_v - v w), the test is w > 0 and a^2 + b^2 < t2 w^2.  All
// coordinates lie in [-1, 1], so with Mu = |h0| + |h1| + |h2|, Mv likewise and Mw = |h6| + |h7| + 1,
// rounding the inputs and evaluating in single precision moves w by less than 5 2^-24 Mw and a by less
// than 8 2^-24 (Mu + Mw); the bounds used are 2^-20 of those sums, which also covers the rounding
// of the double-precision test (2^-50 of them) and the final squares.  Between the bounds (and for
// anything not finite) the double-precision test decides, so the flags are always its own: for 1000
// hypotheses and 374 matches it runs for a few dozen warps, not 12 000.
struct FastInlier {
    float h[8], eu, ev, ew, t_in, t_out;
    // hf: the hypothesis rounded to single precision
    __device__ __forceinline__ FastInlier(const float* hf, const MtState* st) : t_in(st->t_in), t_out(st->t_out) {
#pragma unroll
        for (int k = 0; k < 8; ++k) h[k] = hf[k];
        const float E = MT_EPS;
        const float mw = fabsf(h[6]) + fabsf(h[7]) + 1.0f;
        eu = E * (fabsf(h[0]) + fabsf(h[1]) + fabsf(h[2]) + mw) + 1e-30f;
        ev = E * (fabsf(h[3]) + fabsf(h[4]) + fabsf(h[5]) + mw) + 1e-30f;
        ew = E * mw;
    }
    // 1 inlier, 0 outlier, -1 undecided
    __device__ __forceinline__ int operator()(float4 p) const {
        const float w = fmaf(h[6], p.x, fmaf(h[7], p.y, 1.0f));
        const float a = fabsf(fmaf(-p.z, w, fmaf(h[0], p.x, fmaf(h[1], p.y, h[2]))));
        const float b = fabsf(fmaf(-p.w, w, fmaf(h[3], p.x, fmaf(h[4], p.y, h[5]))));
        const float wl = w - ew, wh = fabsf(w) + ew, ah = a + eu, bh = b + ev, al = fmaxf(a - eu, 0.0f), bl = fmaxf(b - ev, 0.0f);
        if (wl > 0.0f && fmaf(ah, ah, bh * bh) < t_in * (wl * wl)) return 1;
        if (w + ew < 0.0f || fmaf(al, al, bl * bl) > fmaf(t_out, wh * wh, 1e-37f)) return 0;
        return -1;
    }
};

__device__ __forceinline__ bool mt_inlier(const FastInlier& fast, const double* h, const double* xyuv,
                                          float4 p, int i, double t2) {
    const int d = fast(p);
    if (d >= 0) return d != 0;
    return inlier(h, xyuv[4 * i], xyuv[4 * i + 1], xyuv[4 * i + 2], xyuv[4 * i + 3], t2);
}

// Four iterations per block of 4 warps.  Each warp draws the sample of one (its place in the growth
// schedule c = #{j < N - 4 : E_j <= t}, n(t) = 4 + c, uniform sampling when E_c < t), one warp solves the
// four 4-point systems, then each warp counts the inliers of one.  The solving warp is another one
// from each wave of `sms` blocks to the next, so that the blocks of an SM solve on different
// schedulers.  23 us for 1000 iterations on 374 matches, against 61 us for the two kernels with a
// block per iteration (FP64 inlier tests alone: 30 us at two lanes per clock and SM).
__global__ void __launch_bounds__(128) mt_hypotheses(int iters, const long long* E,
                                                     const unsigned* rnd, const double* xyuv,
                                                     const float* xyuvf, int sms,
                                                     double* hyp, MtState* st) {
    __shared__ int sidx[4][4];
    __shared__ double sh[4][8];
    __shared__ float shf[4][8];
    __shared__ int s_ok[4];
    __shared__ float4 pts[MT_MAX_POINTS];  // the matches, brought in by the warps that do not solve
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, it = 4 * blockIdx.x + w;
    pdl_trigger();
    pdl_wait();
    const int N = st->n;
    if (N < 4) return;
    {
        const long long t = min(it, iters - 1) + 1;
        const int K = N - 4;
        // E does not decrease: whole segments of 64 events first, then the events of the next one
        const int s = __popc(__ballot_sync(0xffffffffu, 64 * lane + 63 < K && E[min(64 * lane + 63, K)] <= t));
        const int j = 64 * s + lane;
        const int c = 64 * s + __popc(__ballot_sync(0xffffffffu, j < K && E[min(j, K)] <= t)) +
                      __popc(__ballot_sync(0xffffffffu, j + 32 < K && E[min(j + 32, K)] <= t));
        if (lane == 0) {
            const int n = 4 + c;
            const unsigned* rw = rnd + 4 * (size_t)(t - 1);
            int idx[4];
            if (E[c] < t) {
                for (int k = 0; k < 4; ++k) idx[k] = nth_free((int)(rw[k] % (unsigned)(n - k)), idx, k);
            } else {
                idx[0] = n - 1;
                int chosen[3];
                for (int k = 0; k < 3; ++k) {
                    chosen[k] = nth_free((int)(rw[k] % (unsigned)(n - 1 - k)), chosen, k);
                    idx[k + 1] = chosen[k];
                }
            }
            for (int k = 0; k < 4; ++k) sidx[w][k] = idx[k];
        }
    }
    __syncthreads();
    const int solver = (int)((blockIdx.x / (unsigned)sms) & 3u);
    if (w != solver) {
        const int k = (w - solver - 1) & 3;  // 0, 1, 2
#pragma unroll 4
        for (int i = 32 * k + lane; i < N; i += 96) pts[i] = __ldcg(reinterpret_cast<const float4*>(xyuvf) + i);
    } else {
        // rows 2k, 2k+1 of pair k: (x, y, 1, 0, 0, 0, -ux, -uy | u), (0, 0, 0, x, y, 1, -vx, -vy | v)
        const int g = lane >> 3, r = lane & 7, m = sidx[g][r >> 1];
        const bool odd = r & 1;
        const double x = xyuv[4 * m], y = xyuv[4 * m + 1], u = xyuv[4 * m + 2 + odd];
        double A[9] = {odd ? 0.0 : x, odd ? 0.0 : y, odd ? 0.0 : 1.0, odd ? x : 0.0, odd ? y : 0.0, odd ? 1.0 : 0.0,
                       -dM(u, x), -dM(u, y), u};
        double h[8];
        const bool ok = solve8(A, h);
        if (r == 0) s_ok[g] = ok;
        double mine = h[0];
#pragma unroll
        for (int k = 1; k < 8; ++k) mine = r == k ? h[k] : mine;
        sh[g][r] = mine;
        shf[g][r] = (float)mine;
        if (4 * (int)blockIdx.x + g < iters) hyp[8 * (size_t)(4 * blockIdx.x + g) + r] = mine;
    }
    __syncthreads();
    if (it >= iters || !s_ok[w]) return;
    const double t2 = st->t2;
    const FastInlier fast(shf[w], st);
    int c = 0;
    for (int i = lane; i < N; i += 32) c += mt_inlier(fast, sh[w], xyuv, pts[i], i, t2);
    c = __reduce_add_sync(0xffffffffu, c);
    // most inliers, ties to the earlier iteration
    if (lane == 0) atomicMax(&st->best, (unsigned long long)(c + 1) << 32 | (unsigned long long)(0xffffffffu - (unsigned)it));
}

// One block: the best hypothesis' inlier flags, the least-squares normal equations on them, the refit
// (the 4-point hypothesis when singular), and back to pixels, H = Tb^-1 Hn Ta with h33 = 1; identity
// and 0 inliers when there is no model.
//
// The two DLT rows of a match are row0 = (g, 0, 0, 0, a6, a7), row1 = (0, 0, 0, g, b6, b7) with
// g = (x, y, 1), a6 = -ux, a7 = -uy, b6 = -vx, b7 = -vy; M[p][q] adds row0[p] row0[q], then
// row1[p] row1[q], match by match in quality order.  A product with a structural zero adds +-0 to a sum
// that is never -0, so it is left out without changing a bit.  That leaves 24 different sums of one
// product per match and 5 of two (the first and second parts of M's and r's entries coincide, as M is
// symmetric).  A sum is a chain of additions in order, 64 cycles each whether one lane adds or 32: warp 0
// carries the 24 in its lanes, warp 1 the 5, on schedulers of their own, while the warps of the other
// two schedulers form the products of the next 64 inliers.  The longest chain is two additions per
// inlier (20 us for 333) and bounds the kernel; 45 us in all, against 61 us as three kernels.
constexpr int MF_THREADS = 512, MF_CHUNK = 64, MF_ONE = 24, MF_TWO = 5, MF_ROW = 35;
__global__ void __launch_bounds__(MF_THREADS, 1) mt_final(MtState* st, const double* hyp,
                                                       const double* xyuv, const float* xyuvf,
                                                       unsigned char* inl,
                                                       double* H, int* n_inliers) {
    __shared__ double buf[2][MF_CHUNK * MF_ROW];  // products of a chunk's inliers: 24, then 5 pairs
    __shared__ uint16_t list[MT_MAX_POINTS];      // the inliers in quality order
    __shared__ double sums[MF_ONE + MF_TWO];
    __shared__ double hb[8], Hn[9], P[9], Q[9];
    __shared__ float hf[8];
    __shared__ int wcnt[MF_THREADS / 32], s_n;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    pdl_trigger();
    pdl_wait();
    const int N = st->n;
    const unsigned long long best = st->best;
    const int bc = (int)(best >> 32) - 1;
    if (N < 4 || bc < 4) {
        for (int i = t; i < N; i += MF_THREADS) inl[i] = 0;
        if (t < 9) H[t] = t % 4 == 0 ? 1.0 : 0.0;
        if (t == 0) *n_inliers = 0;
        return;
    }
    const Norm z = st->norm;
    if (t < 8) {
        hb[t] = hyp[8 * (size_t)(0xffffffffu - (unsigned)best) + t];
        hf[t] = (float)hb[t];
    }
    if (t == 0) s_n = 0;
    __syncthreads();
    {
        const double t2 = st->t2;
        const FastInlier fast(hf, st);
        for (int i0 = 0; i0 < N; i0 += MF_THREADS) {
            const int i = i0 + t;
            const bool f = i < N && mt_inlier(fast, hb, xyuv, reinterpret_cast<const float4*>(xyuvf)[i], i, t2);
            if (i < N) inl[i] = f;
            const unsigned m = __ballot_sync(0xffffffffu, f);
            if (lane == 0) wcnt[w] = __popc(m);
            __syncthreads();
            int at = s_n + __popc(m & ((1u << lane) - 1u));
            for (int k = 0; k < w; ++k) at += wcnt[k];
            if (f) list[at] = (uint16_t)i;
            __syncthreads();
            if (t == MF_THREADS - 1) s_n = at + f;
            __syncthreads();
        }
    }
    const int n = s_n, chunks = (n + MF_CHUNK - 1) / MF_CHUNK;
    // the products of inlier q of chunk k, a lane per inlier; producer warps are those of schedulers 2, 3
    auto produce = [&](int k, int q) {
        const int j = MF_CHUNK * k + q;
        if (j >= n) return;
        const double* c = xyuv + 4 * (size_t)list[j];
        const double x = c[0], y = c[1], u = c[2], v = c[3];
        double* o = buf[k & 1] + q * MF_ROW;
        const double ux = dM(u, x), uy = dM(u, y), vx = dM(v, x), vy = dM(v, y);
        const double a6 = -ux, a7 = -uy, b6 = -vx, b7 = -vy;
        o[0] = dM(x, x);
        o[1] = dM(x, y);
        o[2] = x;
        o[3] = dM(y, y);
        o[4] = y;
        o[5] = 1.0;
        o[6] = dM(x, a6);
        o[7] = dM(y, a6);
        o[8] = a6;
        o[9] = dM(x, a7);
        o[10] = dM(y, a7);
        o[11] = a7;
        o[12] = dM(x, b6);
        o[13] = dM(y, b6);
        o[14] = b6;
        o[15] = dM(x, b7);
        o[16] = dM(y, b7);
        o[17] = b7;
        o[18] = ux;
        o[19] = uy;
        o[20] = u;
        o[21] = vx;
        o[22] = vy;
        o[23] = v;
        o[24] = dM(a6, a6);
        o[25] = dM(b6, b6);
        o[26] = dM(a6, a7);
        o[27] = dM(b6, b7);
        o[28] = dM(a7, a7);
        o[29] = dM(b7, b7);
        o[30] = dM(a6, u);
        o[31] = dM(b6, v);
        o[32] = dM(a7, u);
        o[33] = dM(b7, v);
    };
    const int prod = w == 2 ? 0 : w == 3 ? 32 : -1;
    static_assert(MF_CHUNK == 64, "two producer warps");
    if (prod >= 0) produce(0, prod + lane);
    __syncthreads();
    double acc = 0.0;
    for (int k = 0; k < chunks; ++k) {
        const int m = min(MF_CHUNK, n - MF_CHUNK * k);
        const double* b = buf[k & 1];
        if (w == 0 && lane < MF_ONE) {
#pragma unroll 8
            for (int q = 0; q < m; ++q) acc = dA(acc, b[q * MF_ROW + lane]);
        } else if (w == 1 && lane < MF_TWO) {
            b += MF_ONE + 2 * lane;
#pragma unroll 8
            for (int q = 0; q < m; ++q) acc = dA(dA(acc, b[q * MF_ROW]), b[q * MF_ROW + 1]);
        } else if (prod >= 0 && k + 1 < chunks) {
            produce(k + 1, prod + lane);
        }
        __syncthreads();
    }
    if (w == 0 && lane < MF_ONE) sums[lane] = acc;
    if (w == 1 && lane < MF_TWO) sums[MF_ONE + lane] = acc;
    __syncthreads();
    if (w != 0) return;
    {
        // row r of [M | r]: (g_p g_q sums) in the blocks of x, y, 1, then columns 6, 7 and the right-hand side
        const int r = lane & 7, p = r < 3 ? r : r - 3;
        double A[9], h[8];
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            int e = -1;  // the sum in column j, -1 for none
            if (r < 6) {
                if (j < 6) {
                    if (j / 3 == r / 3) {
                        const int q = j % 3, lo = min(p, q), hi = max(p, q);
                        e = lo == 0 ? hi : lo == 1 ? 2 + hi : 5;
                    }
                } else {
                    e = j == 8 ? 18 + r : (r < 3 ? 6 : 12) + 3 * (j - 6) + p;
                }
            } else {
                e = j < 6 ? (j < 3 ? 6 : 12) + 3 * (r - 6) + j % 3 : j == 8 ? 27 + r - 6 : 24 + (r - 6) + (j - 6);
            }
            A[j] = e >= 0 ? sums[e] : 0.0;
        }
        const bool ok = solve8(A, h);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (lane == k) Hn[k] = ok ? h[k] : hb[k];
        if (lane == 8) Hn[8] = 1.0;
    }
    __syncwarp();
    // Hn = [h0 h1 h2; h3 h4 h5; h6 h7 1], Ta = [sa 0 -sa ca0; 0 sa -sa ca1; 0 0 1],
    // Tb^-1 = [1/sb 0 cb0; 0 1/sb cb1; 0 0 1]
    const int r = lane / 3, k = lane % 3;
    if (lane < 9) {
        const double Ta[9] = {z.sa, 0.0, -dM(z.sa, z.ca0), 0.0, z.sa, -dM(z.sa, z.ca1), 0.0, 0.0, 1.0};
        P[lane] = dA(dA(dM(Hn[3 * r], Ta[k]), dM(Hn[3 * r + 1], Ta[3 + k])), dM(Hn[3 * r + 2], Ta[6 + k]));
    }
    __syncwarp();
    if (lane < 9) {
        const double isb = dD(1.0, z.sb);
        const double Tbi[9] = {isb, 0.0, z.cb0, 0.0, isb, z.cb1, 0.0, 0.0, 1.0};
        Q[lane] = dA(dA(dM(Tbi[3 * r], P[k]), dM(Tbi[3 * r + 1], P[3 + k])), dM(Tbi[3 * r + 2], P[6 + k]));
    }
    __syncwarp();
    if (lane < 9) H[lane] = dD(Q[lane], Q[8]);
    if (lane == 0) *n_inliers = bc;
}

}  // namespace

struct stitch_matcher {
    int device = 0, max_points = 0, max_iters = 0, sms = 1;
    unsigned* keys = nullptr;  // key words of image A, then of image B: [word][point]
    int2* best = nullptr;      // per query: match (or -1) and distance
    MtState* st = nullptr;
    long long* E = nullptr;    // growth schedule
    double* hyp = nullptr;
    double* xyuv = nullptr;
    float* xyuvf = nullptr;
};

static void matcher_free(stitch_matcher* c) {
    if (!c) return;
    cudaFree(c->keys);
    cudaFree(c->best);
    cudaFree(c->st);
    cudaFree(c->E);
    cudaFree(c->hyp);
    cudaFree(c->xyuv);
    cudaFree(c->xyuvf);
    delete c;
}

extern "C" stitch_status stitch_matcher_create(int32_t max_points, int32_t max_iters, int32_t device,
                                               stitch_matcher** out) {
    if (!out) return STITCH_EINVAL;
    *out = nullptr;
    if (max_points < 1 || max_points > MT_MAX_POINTS || max_iters < 0 || max_iters > (1 << 16)) return STITCH_EINVAL;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
        cudaGetLastError();
        return STITCH_ECUDA;
    }
    if (device < 0 || device >= ndev) return STITCH_EINVAL;
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(device) != cudaSuccess) return STITCH_ECUDA;
    stitch_matcher* c = new (std::nothrow) stitch_matcher();
    if (!c) return STITCH_ENOMEM;
    c->device = device;
    c->max_points = max_points;
    c->max_iters = max_iters;
    const size_t it = (size_t)std::max(max_iters, 1);
    bool okm = cudaMalloc(&c->keys, sizeof(unsigned) * 2 * MT_MAX_WORDS * max_points) == cudaSuccess &&
               cudaMalloc(&c->best, sizeof(int2) * max_points) == cudaSuccess &&
               cudaMalloc(&c->st, sizeof(MtState)) == cudaSuccess &&
               cudaMalloc(&c->E, sizeof(long long) * MT_MAX_POINTS) == cudaSuccess &&
               cudaMalloc(&c->hyp, sizeof(double) * 8 * it) == cudaSuccess &&
               cudaMalloc(&c->xyuv, sizeof(double) * 4 * max_points) == cudaSuccess &&
               cudaMalloc(&c->xyuvf, sizeof(float) * 4 * max_points) == cudaSuccess;
    if (cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || c->sms < 1) c->sms = 1;
    if (prev >= 0) cudaSetDevice(prev);
    if (!okm) {
        cudaGetLastError();
        matcher_free(c);
        return STITCH_ENOMEM;
    }
    *out = c;
    return STITCH_OK;
}

extern "C" void stitch_matcher_destroy(stitch_matcher* c) {
    if (!c) return;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(c->device);
    cudaDeviceSynchronize();
    matcher_free(c);
    if (prev >= 0) cudaSetDevice(prev);
}

extern "C" stitch_status stitch_match_homography(stitch_matcher* c, const int32_t* xy_a, const uint8_t* desc_a,
                                                 const int32_t* count_a, const int32_t* xy_b, const uint8_t* desc_b,
                                                 const int32_t* count_b, const stitch_match_params* prm,
                                                 const uint8_t* bits, const uint32_t* rnd, int32_t* matches,
                                                 int32_t* n_matches, double* H, int32_t* n_inliers, uint8_t* inlier,
                                                 void* stream) {
    if (!c || !xy_a || !desc_a || !count_a || !xy_b || !desc_b || !count_b || !prm || !bits || !matches ||
        !n_matches || !H || !n_inliers || !inlier)
        return STITCH_EINVAL;
    if (prm->tables < 1 || prm->tables > MT_MAX_TABLES || prm->bits < 1 || prm->bits > MT_MAX_BITS ||
        prm->ratio_num < 1 || prm->ratio_den < 1 || prm->iters < 0 || prm->iters > c->max_iters ||
        (prm->iters > 0 && !rnd) || !(prm->inlier_px > 0.0) ||
        ((reinterpret_cast<uintptr_t>(desc_a) | reinterpret_cast<uintptr_t>(desc_b)) & 3) != 0)
        return STITCH_EINVAL;
    LshBits lb{};
    lb.L = prm->tables;
    lb.k = prm->bits;
    for (int l = 0; l < lb.L; ++l)
        for (int j = 0; j < lb.k; ++j) lb.b[l][j] = bits[l * lb.k + j];
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != c->device && cudaSetDevice(c->device) != cudaSuccess) return STITCH_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const int cap = c->max_points;
    const unsigned* da = reinterpret_cast<const unsigned*>(desc_a);
    const unsigned* db = reinterpret_cast<const unsigned*>(desc_b);
    const int nw = mt_words(lb), iters = prm->iters;
    unsigned *ka = c->keys, *kb = c->keys + (size_t)MT_MAX_WORDS * cap;
    pdl_launch(mt_keys, dim3((cap + 127) / 128, nw, 2), 128, 0, s, da, count_a, db, count_b, lb, cap, ka, kb, c->st);
    const bool pk = mt_packed(lb);
    auto match = nw <= 2   ? (pk ? mt_match<true, 2> : mt_match<false, 2>)
                 : nw <= 4 ? (pk ? mt_match<true, 4> : mt_match<false, 4>)
                 : nw <= 8 ? (pk ? mt_match<true, 8> : mt_match<false, 8>)
                 : nw <= 16 ? (pk ? mt_match<true, 16> : mt_match<false, 16>)
                            : mt_match<false, 32>;
    pdl_launch(match, (cap + 7) / 8, 256, 0, s, da, count_a, db, count_b, ka, kb, cap, xy_a, xy_b, prm->max_dist,
               prm->ratio_num, prm->ratio_den, c->best, c->st);
    pdl_launch(mt_rank, (cap + 7) / 8 + 1, 256, 0, s, c->best, count_a, cap, xy_a, xy_b, c->st, matches, n_matches,
               c->xyuv, c->xyuvf, c->E, prm->inlier_px);
    if (iters > 0)
        pdl_launch(mt_hypotheses, (iters + 3) / 4, 128, 0, s, iters, c->E, rnd, c->xyuv, c->xyuvf, c->sms, c->hyp, c->st);
    pdl_launch(mt_final, 1, MF_THREADS, 0, s, c->st, c->hyp, c->xyuv, c->xyuvf, inlier, H, n_inliers);
    stitch_status st = cudaGetLastError() == cudaSuccess ? STITCH_OK : STITCH_ECUDA;
    if (prev >= 0 && prev != c->device) cudaSetDevice(prev);
    return st;
}
