// Offsetting by sphere unions (Section 4.2): the solid H united with (inner
// offset: minus) one sphere of radius r about every sample of its three
// LDNIs, each sphere given by its own LDNIs on H's grid.
//
// The paper applies one Boolean per sphere.  Here every ray is answered once:
// the ray's samples of H and of every sphere that meets it are ordered by
// depth and swept in one pass.  The result is the one the step-by-step
// Booleans give (without small-interval removal, which follows once):
//  - the solid is {t : H(t) or some sphere holds t} (inner: H(t) and no
//    sphere), by associativity of the set operations;
//  - where it changes state at depth d, the step-by-step Booleans keep the
//    sample of the first source in the order H, sphere 0, sphere 1, ... whose
//    own state changes at d (each Boolean keeps the accumulated solid's
//    sample at a tie), so the sweep takes that one.
//
// A sample of image a at pixel (i, j) with depth d sits at the point with
// a-coordinate d and in-plane coordinates c_u(i), c_v(j),
// c(t) = fl32(o + fl32((t + 1/2) h)), h = fl32(W / res); spheres are numbered
// in sample order (image x, y, z, each in CSR order).  The sphere about C
// meets the ray through (P_u, P_v) of image b iff q < fl32(r r) with
// q = fl32(fl32(du du) + fl32(dv dv)), du = fl32(P_u - C_u), dv likewise; its
// samples are fl32(C_b -+ t), t = sqrt(fl32(r r - q)) rounded, with outward
// normals (du / r, dv / r, -+t / r), each operation rounded to nearest.
//
// A sphere covers the interval between its two samples, so the ray's result
// is bounded by the ends of the connected components of its intervals: the
// spheres' and, for the outer offset, H's solid intervals; for the inner one
// H's gaps, the result being what lies between the components.  Intervals that
// touch belong together (the state does not change where one ends and another
// begins), empty ones do not count, and at an end of a component the sources
// that change there are exactly the intervals that end (or begin) at its
// depth, so the first of them in the order above gives the sample.
//
// Stages: sphere centres; per image, sphere lists of 8 x 8-pixel tiles
// (count, scan, fill); per ray (a warp each) the components and the count of
// its samples; the scan of the counts into the output offsets; the samples.
#include <algorithm>
#include <climits>
#include <cmath>

#include "ldni_host.h"
#include "sample_common.cuh"

namespace ldni {
namespace {

constexpr int kOffWarps = 8;      // rays (warps) per block: one pixel row of a tile
constexpr int kStagePer = 2;      // spheres of the tile's list a thread looks at per round
constexpr int kStage = kOffWarps * 32 * kStagePer;
constexpr int kMaxComp = 257;     // components a ray may keep when its intervals are merged to make room: those
                                  // of 512 samples (an inner offset's are bounded by one more than its intervals)
constexpr int kBuf = kMaxComp + 32;  // intervals of one ray held in shared memory: room for a warp's after a merge
constexpr int kMaxHSamples = 384; // H's samples on one ray
constexpr int kKept = 8;          // samples whose sources the count pass leaves to the write pass
// Rays per image up to which the three images' sources are kept side by side;
// larger images are counted and written one after another and share the space
// (32 instead of 96 bytes a pixel), where a few launches more do not show.
constexpr long long kKeptTogether = 1ll << 20;
constexpr int kTile = kOffWarps;  // pixels per side of a sphere-list tile
constexpr int kThreads = 256;

struct OffArgs {
    // H
    const int *hoff[3];
    const float *hd[3], *hx[3], *hy[3], *hz[3];
    const int *ht[3];
    long long base[3];  // first sphere of each image
    long long n[3];     // samples of each image
    long long S;        // spheres
    // grid
    float o[3];
    float h;
    int res;
    float r, r2, eps;
    float inv_h;
    float slack[3];  // pixels by which a shadow is widened, per world axis (off_bin)
    int inner;
    int img0;        // first image of the launch (counts and writes)
    // sphere centres and tile lists
    float4 *C;
    int *tcnt[3];   // per tile: spheres binned (count pass), then the fill cursor
    int *toff[3];   // tile list offsets [ntiles + 1]
    int *tlist[3];  // sphere indices
    int ntx;        // tiles per side
    // output
    int *cnt[3];    // per-ray output counts
    int *deep;      // number and list of the rows (image, tile row) with rays of more than kKept samples
    uint4 *kept[3]; // per ray, the sources of its samples (two uint4), when there are at most kKept
    int *ooff[3];
    float *od[3], *ox[3], *oy[3], *oz[3];
    int *ot[3];
    long long ocap[3];
};

__device__ __forceinline__ float pix(long long t, float o, float h) {
    return __fadd_rn(o, __fmul_rn((float)t + 0.5f, h));
}

__device__ __forceinline__ float c4(const float4 &c, int k) { return k == 0 ? c.x : (k == 1 ? c.y : c.z); }

template <class T>
__device__ __forceinline__ T pick(T const (&arr)[3], int a) {
    return a == 0 ? arr[0] : (a == 1 ? arr[1] : arr[2]);
}

// the sphere about c on the ray (pu, pv) of image b
__device__ __forceinline__ bool sphere_hit(const float4 &c, int b, float pu, float pv, float r2, float &e, float &x,
                                           float &t, float &du, float &dv) {
    du = __fsub_rn(pu, c4(c, b == 2 ? 0 : b + 1));
    dv = __fsub_rn(pv, c4(c, b == 0 ? 2 : b - 1));
    const float q = __fadd_rn(__fmul_rn(du, du), __fmul_rn(dv, dv));
    if (!(q < r2)) return false;
    t = __fsqrt_rn(__fsub_rn(r2, q));
    e = __fsub_rn(c4(c, b), t);
    x = __fadd_rn(c4(c, b), t);
    return true;
}

// sphere centres in sample order: a thread per ray of image blockIdx.y
__global__ void __launch_bounds__(kThreads) off_centres(OffArgs A) {
    const int a = blockIdx.y;
    const long long N = (long long)A.res * A.res;
    const long long p = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (p >= N) return;
    const int *off = pick(A.hoff, a);
    const float *D = pick(A.hd, a);
    const int iu = a == 2 ? 0 : a + 1, iv = a == 0 ? 2 : a - 1;
    const float cu = pix(p % A.res, A.o[iu], A.h), cv = pix(p / A.res, A.o[iv], A.h);
    const long long b0 = pick(A.base, a), na = pick(A.n, a);
    for (long long k = max(off[p], 0); k < min((long long)off[p + 1], na); ++k) {
        float v[3];
        v[a] = D[k];
        v[iu] = cu;
        v[iv] = cv;
        A.C[b0 + k] = make_float4(v[0], v[1], v[2], 0.0f);
    }
}

// Sphere s into the lists of the tiles of image blockIdx.y that its shadow
// touches: count (kFill = false) or fill.  The lists only have to hold every
// sphere that can meet a ray of the tile, so the shadow's bounds are taken in
// FP32 (this GPU runs FP64 at 1/64 of its rate) and widened by `slack` pixels,
// which covers the rounding of the bounds and of the pixel centres.
// Neighbouring samples touch the same few tiles, whose counters then take
// every lane's atomic in turn (70 us a pass for the 42,000 spheres of the
// 128^2 flower on 768 counters): the lanes of a warp that hold the same tile
// send one atomic for all (9 us, the bounds in FP32 among it).
template <bool kFill>
__global__ void __launch_bounds__(kThreads) off_bin(OffArgs A) {
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const long long s = blockIdx.x * (long long)kThreads + threadIdx.x;
    const float4 c = s < A.S ? A.C[s] : make_float4(INFINITY, INFINITY, INFINITY, 0.0f);
    const int bu = b == 2 ? 0 : b + 1, bv = b == 0 ? 2 : b - 1;
    const float rp = A.r * A.inv_h, last = (float)(A.res - 1);
    const float u = (c4(c, bu) - A.o[bu]) * A.inv_h - 0.5f, v = (c4(c, bv) - A.o[bv]) * A.inv_h - 0.5f;
    const float ru = rp + A.slack[bu], rv = rp + A.slack[bv];
    const float i0 = fmaxf(floorf(u - ru), 0.0f), i1 = fminf(ceilf(u + ru), last);
    const float j0 = fmaxf(floorf(v - rv), 0.0f), j1 = fminf(ceilf(v + rv), last);
    // (false for a sample at infinity and for a shadow that misses the image)
    const bool live = isfinite(u) && isfinite(v) && isfinite(rp) && i0 <= i1 && j0 <= j1;
    int *tc = pick(A.tcnt, b);
    const int ti0 = live ? (int)i0 / kTile : 0, tj0 = live ? (int)j0 / kTile : 0;
    const int nti = live ? (int)i1 / kTile - ti0 + 1 : 1, n = live ? nti * ((int)j1 / kTile - tj0 + 1) : 0;
    const int steps = __reduce_max_sync(0xffffffffu, n);
    int ti = 0, tj = 0;
    for (int k = 0; k < steps; ++k) {
        const int tile = k < n ? (tj0 + tj) * A.ntx + ti0 + ti : -1;
        if (++ti == nti) {
            ti = 0;
            ++tj;
        }
        const unsigned same = __match_any_sync(0xffffffffu, tile);
        const int leader = __ffs(same) - 1;
        int at = 0;
        if (lane == leader && tile >= 0) at = atomicAdd(tc + tile, __popc(same));
        if (!kFill) continue;
        at = __shfl_sync(0xffffffffu, at, leader);
        if (tile >= 0)
            pick(A.tlist, b)[pick(A.toff, b)[tile] + at + __popc(same & ((1u << lane) - 1u))] = (int)s;
    }
}

// ---- components of a ray's intervals -----------------------------------------------
//
// An interval is (first key, last key, first source, last source).  Keys order
// depths as unsigned words (-0 as +0); kLow and kHigh stand below and above
// every depth.  A source is 0 for H and s + 1 for sphere s, so the smaller one
// comes first in the order of the step-by-step Booleans.
constexpr unsigned kLow = 0u, kHigh = 0xffffffffu;
constexpr unsigned kSph = 0x40000000u;  // sample tag: sphere (2 s + leaving), else H's sample index on the ray
constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ unsigned depth_key(float d) {
    const unsigned u = __float_as_uint(__fadd_rn(d, 0.0f));
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_depth(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k ^ 0x80000000u) : ~k);
}

struct Comp {
    unsigned lo, hi, lo_src, hi_src;
};

// A lane's share of the buffer's (first key, last key) pairs: in registers
// when kRegs of them per lane are enough, else read from the buffer each time.
constexpr int kRegs = 8;

template <bool kInRegs>
struct Ends {
    const uint4 *buf;
    int nb, lane;
    uint2 v[kInRegs ? kRegs : 1];
    __device__ __forceinline__ Ends(const uint4 *buf_, int nb_, int lane_) : buf(buf_), nb(nb_), lane(lane_) {
        if constexpr (kInRegs) {
#pragma unroll
            for (int k = 0; k < kRegs; ++k)
                v[k] = 32 * k + lane < nb ? *reinterpret_cast<const uint2 *>(buf + 32 * k + lane)
                                          : make_uint2(kHigh, kHigh);
        }
    }
    template <class F>
    __device__ __forceinline__ void each(F &&f) const {
        if constexpr (kInRegs) {
#pragma unroll
            for (int k = 0; k < kRegs; ++k) f(v[k].x, v[k].y);
        } else {
            for (int i = lane; i < nb; i += 32) {
                const uint2 u = *reinterpret_cast<const uint2 *>(buf + i);
                f(u.x, u.y);
            }
        }
    }
};

// The first component that begins at or above `from`; false when there is
// none.  Whole warp; every loop moves a key strictly upwards through the
// buffer's keys, so it ends.
template <class E>
__device__ __forceinline__ bool next_comp(const E &ends, unsigned from, Comp &c) {
    unsigned lo = kHigh;
    ends.each([&](unsigned e, unsigned) { lo = e >= from ? min(lo, e) : lo; });
    lo = __reduce_min_sync(kAll, lo);
    if (lo == kHigh) return false;  // (an interval's first key is below its last)
    unsigned hi = lo;
    for (;;) {
        unsigned m = hi;
        ends.each([&](unsigned e, unsigned x) { m = e <= hi ? max(m, x) : m; });
        m = __reduce_max_sync(kAll, m);
        if (m == hi) break;
        hi = m;
    }
    unsigned lo_src = kAll, hi_src = kAll;
    int at = ends.lane;
    ends.each([&](unsigned e, unsigned x) {
        if (e == lo) lo_src = min(lo_src, ends.buf[at].z);
        if (x == hi) hi_src = min(hi_src, ends.buf[at].w);
        at += 32;
    });
    c = Comp{lo, hi, __reduce_min_sync(kAll, lo_src), __reduce_min_sync(kAll, hi_src)};
    return true;
}

// Turns the entries [first, nb) (centre along the ray, squared half length of
// the chord, sphere) into intervals; one whose two samples share a depth
// changes no state and is marked dead.  Whole warp.
__device__ __forceinline__ void make_intervals(uint4 *buf, int first, int nb, int lane) {
    __syncwarp();
    for (int i = first + lane; i < nb; i += 32) {
        const uint4 v = buf[i];
        const float c = __uint_as_float(v.x), t = __fsqrt_rn(__uint_as_float(v.y));
        const float e = __fsub_rn(c, t), x = __fadd_rn(c, t);
        buf[i] = e < x ? make_uint4(depth_key(e), depth_key(x), v.z + 1u, v.z + 1u) : make_uint4(kHigh, kHigh, kAll, kAll);
    }
    __syncwarp();
}

// Replaces the buffer's intervals by their components (whole warp); returns
// how many there are.  The first interval of a component becomes it, the
// others are marked dead (no key is above kHigh) and squeezed out.
__device__ __noinline__ int merge_buf(uint4 *buf, int nb, int lane) {
    unsigned from = 0;
    Comp c;
    while (next_comp(Ends<false>(buf, nb, lane), from, c)) {
        __syncwarp();
        int head = INT_MAX;
        for (int i = lane; i < nb; i += 32)
            if (buf[i].x == c.lo) head = min(head, i);
        head = __reduce_min_sync(kAll, head);
        for (int i = lane; i < nb; i += 32) {
            const unsigned e = buf[i].x;
            if (e < c.lo || e > c.hi || e == kHigh) continue;
            buf[i] = i == head ? make_uint4(c.lo, c.hi, c.lo_src, c.hi_src) : make_uint4(kHigh, kHigh, kAll, kAll);
        }
        __syncwarp();
        if (c.hi == kHigh) break;
        from = c.hi + 1u;
    }
    int n = 0;
    for (int i0 = 0; i0 < nb; i0 += 32) {
        const uint4 v = i0 + lane < nb ? buf[i0 + lane] : make_uint4(kHigh, kHigh, kAll, kAll);
        const unsigned live = __ballot_sync(kAll, v.x != kHigh);  // (also: every lane has read its slot)
        if (v.x != kHigh) buf[n + __popc(live & ((1u << lane) - 1u))] = v;
        n += __popc(live);
        __syncwarp();
    }
    return n;
}

// One sample of the result at `slot`: H's sample or the sphere's own.
__device__ __forceinline__ void put_result(const OffArgs &A, int b, long long hb, float pu, float pv, unsigned tag,
                                           long long slot, ldni_info_t *info) {
    if (slot >= pick(A.ocap, b)) {
        set_status(info, LDNI_ST_CAPACITY);
        return;
    }
    float d, nx, ny, nz;
    int id;
    if (!(tag & kSph)) {
        const long long k = hb + tag;
        d = pick(A.hd, b)[k];
        nx = pick(A.hx, b)[k];
        ny = pick(A.hy, b)[k];
        nz = pick(A.hz, b)[k];
        id = pick(A.ht, b)[k];
    } else {
        const unsigned sid = (tag & ~kSph) >> 1;
        float e, x, t, du, dv;
        sphere_hit(A.C[sid], b, pu, pv, A.r2, e, x, t, du, dv);
        const bool leaving = tag & 1u;
        const float n = __fdiv_rn(t, A.r);
        float nb = leaving ? n : -n, nu = __fdiv_rn(du, A.r), nv = __fdiv_rn(dv, A.r);
        if (A.inner) {  // the spheres are subtracted: inverted normals (Section 4.1)
            nb = -nb;
            nu = -nu;
            nv = -nv;
        }
        d = leaving ? x : e;
        nx = b == 0 ? nb : (b == 1 ? nv : nu);
        ny = b == 1 ? nb : (b == 2 ? nv : nu);
        nz = b == 2 ? nb : (b == 0 ? nv : nu);
        id = (int)(0x80000000u | sid);
    }
    pick(A.od, b)[slot] = d;
    pick(A.ox, b)[slot] = nx;
    pick(A.oy, b)[slot] = ny;
    pick(A.oz, b)[slot] = nz;
    pick(A.ot, b)[slot] = id;
}

// One pixel row of a tile of image b, a warp per ray.  The block
// walks the tile's list, kStage spheres at a time (the next ones' loads in
// flight), and stages those that reach its row (about a third), with their
// distance from the row, which all its rays share, in the list's order: the
// buffer's merges then fall on the same spheres in both passes, which agree
// on every ray.  (Slots handed out by one shared counter depended on the
// warps' timing, and a warp that was late to read that counter could find it
// cleared for the next round.)  Every warp then tests
// them against its ray; the ones that meet it become intervals, whose
// components are found by warp-wide minima and maxima, about a dozen sweeps
// over the five intervals a lane holds (150 a ray on the 128^2 flower by 2.5
// pixels).  Bound by issue: 50 M warp instructions at 58 % of the issue slots, 88 us.  Ordering
// the intervals' ends with a bitonic network and sweeping them with one lane,
// done in both passes, took 589 + 566 us (now 88, and 11 + 19 for the writes);
// half a tile per block, every list entry tested by every ray, 171 us.
// kDeep false: every ray's count, and the sources of its samples when there
// are at most kKept; kDeep true: writes the samples of the rays that have more.
template <bool kDeep>
__device__ __forceinline__ void ray_row(const OffArgs &A, int bx, int b, ldni_info_t *info) {
    __shared__ float4 sc[kStage];  // (centre along the ray, u, squared distance from the row, sphere)
    __shared__ uint4 sbuf[kOffWarps][kBuf];
    __shared__ int s_cnt[kStagePer * kOffWarps];  // staged spheres of each warp's 32, in list order
    __shared__ int s_deep;
    static_assert(kStagePer * kOffWarps <= 32, "a lane per count");
    if (threadIdx.x == 0) s_deep = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int tile = bx / kTile;
    const int i = tile % A.ntx * kTile + w, j = tile / A.ntx * kTile + bx % kTile;
    if (j >= A.res) return;  // the same for the whole block
    const bool mine = i < A.res;
    const long long p = (long long)j * A.res + i;
    const bool live = mine && (!kDeep || pick(A.cnt, b)[p] > kKept);
    const int bu = b == 2 ? 0 : b + 1, bv = b == 0 ? 2 : b - 1;
    const int l0 = pick(A.toff, b)[tile], nl = pick(A.toff, b)[tile + 1] - l0;
    const int *lst = pick(A.tlist, b) + l0;
    const float *HD = pick(A.hd, b);
    uint4 *buf = sbuf[w];
    long long hb = 0;
    int nh = 0, nb = 0;
    if (live) {
        const int *hoff = pick(A.hoff, b);
        long long he = hoff[p + 1];
        hb = hoff[p];
        if (hb < 0 || he < hb || he > pick(A.n, b)) {  // offsets that do not fit the stated sample count
            if (lane == 0) set_status(info, LDNI_ST_CAPACITY);
            hb = he = 0;
        }
        nh = (int)(he - hb);
        if ((nh & 1) && lane == 0 && !kDeep) {
            atomicAdd(&info->odd_rays, 1u);
            set_status(info, LDNI_ST_ODD);
        }
    }
    bool over = nh > kMaxHSamples, met = false;
    // H's solid intervals (outer) or its gaps (inner); an odd ray's last one has no end
    const int nhi = over || !live ? 0 : (A.inner ? nh / 2 + 1 : (nh + 1) / 2);
    for (int k0 = 0; k0 < nhi; k0 += 32) {
        const int k = 2 * (k0 + lane) - (A.inner ? 1 : 0);
        const bool in = k0 + lane < nhi;
        const unsigned lo = !in ? kHigh : (k < 0 ? kLow : depth_key(HD[hb + k]));
        const unsigned hi = !in ? kHigh : (k + 1 < nh ? depth_key(HD[hb + k + 1]) : kHigh);
        const bool some = lo < hi;
        const unsigned m = __ballot_sync(kAll, some);
        if (some) buf[nb + __popc(m & ((1u << lane) - 1u))] = make_uint4(lo, hi, 0u, 0u);
        nb += __popc(m);
    }
    int nfinal = nb;  // entries before this one are intervals, the others spheres that meet the ray
    const float pu = pix(i, A.o[bu], A.h), pv = pix(j, A.o[bv], A.h);
    int sid[kStagePer];
    float4 cc[kStagePer];
    auto fetch = [&](int base) {
#pragma unroll
        for (int k = 0; k < kStagePer; ++k) {
            const int idx = base + k * kOffWarps * 32 + (int)threadIdx.x;
            sid[k] = idx < nl ? lst[idx] : -1;
        }
#pragma unroll
        for (int k = 0; k < kStagePer; ++k) cc[k] = sid[k] >= 0 ? A.C[sid[k]] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    fetch(0);
    for (int base = 0; base < nl; base += kStage) {
        float dv2[kStagePer];
        unsigned in[kStagePer];
#pragma unroll
        for (int k = 0; k < kStagePer; ++k) {
            const float dv = __fsub_rn(pv, c4(cc[k], bv));
            dv2[k] = __fmul_rn(dv, dv);
            in[k] = __ballot_sync(kAll, sid[k] >= 0 && dv2[k] < A.r2);  // (du du + dv dv, rounded, is no smaller)
            if (lane == 0) s_cnt[k * kOffWarps + w] = __popc(in[k]);
        }
        __syncthreads();  // the counts are in; the previous round's spheres are read
        int upto = lane < kStagePer * kOffWarps ? s_cnt[lane] : 0;  // staged by the first lane + 1 of them
#pragma unroll
        for (int o = 1; o < kStagePer * kOffWarps; o <<= 1) {
            const int x = __shfl_up_sync(kAll, upto, o);
            if (lane >= o) upto += x;
        }
        const int ns = __shfl_sync(kAll, upto, kStagePer * kOffWarps - 1);
#pragma unroll
        for (int k = 0; k < kStagePer; ++k) {
            const int end = __shfl_sync(kAll, upto, k * kOffWarps + w);
            if ((in[k] >> lane) & 1u)
                sc[end - __popc(in[k] >> lane)] = make_float4(c4(cc[k], b), c4(cc[k], bu), dv2[k], __int_as_float(sid[k]));
        }
        fetch(base + kStage);
        __syncthreads();  // the spheres are staged; the counts are read
        for (int k0 = 0; k0 < ns && live && !over; k0 += 32) {
            float4 c;
            float q = INFINITY;
            if (k0 + lane < ns) {  // as sphere_hit
                c = sc[k0 + lane];
                const float du = __fsub_rn(pu, c.y);
                q = __fadd_rn(__fmul_rn(du, du), c.z);
            }
            const bool hit = q < A.r2;
            const unsigned m = __ballot_sync(kAll, hit);
            if (nb + __popc(m) > kBuf) {
                make_intervals(buf, nfinal, nb, lane);
                nb = nfinal = merge_buf(buf, nb, lane);
                over = nb > kMaxComp;
                if (over) break;
            }
            if (hit)
                buf[nb + __popc(m & ((1u << lane) - 1u))] =
                    make_uint4(__float_as_uint(c.x), __float_as_uint(__fsub_rn(A.r2, q)), __float_as_uint(c.w), 0u);
            nb += __popc(m);
            met = met || m != 0u;
        }
    }
    if (!live) return;
    if (over) {  // more than one warp holds: leave the ray empty and say so
        if (lane == 0) {
            set_status(info, LDNI_ST_EVENTS);
            if (!kDeep) pick(A.cnt, b)[p] = 0;
        }
        return;
    }
    make_intervals(buf, nfinal, nb, lane);
    // index on the ray of H's first sample with key k
    auto h_index = [&](unsigned k) {
        unsigned at = kAll;
        for (int h = lane; h < nh; h += 32)
            if (at == kAll && depth_key(HD[hb + h]) == k) at = (unsigned)h;
        return __reduce_min_sync(kAll, at);
    };
    const long long oslot = kDeep ? (long long)pick(A.ooff, b)[p] : 0;
    const int room = kDeep ? pick(A.cnt, b)[p] : 0;  // the ray's slots: what the count pass found
    unsigned tags[kKept] = {};
    int nout = 0;
    // one interval of the result, thinner than eps removed
    auto emit = [&](unsigned tag0, unsigned tag1) {
        if (kDeep) {
            if (lane < 2 && nout + lane < room) put_result(A, b, hb, pu, pv, lane ? tag1 : tag0, oslot + nout + lane, info);
        } else {
#pragma unroll
            for (int z = 0; z < kKept; z += 2)
                if (nout == z) {
                    tags[z] = tag0;
                    tags[z + 1] = tag1;
                }
        }
        nout += 2;
    };
    if (!met) {  // no sphere meets the ray: H stays as it is
        for (int k = 0; k + 1 < nh; k += 2) {
            if (!(__fsub_rn(HD[hb + k + 1], HD[hb + k]) < A.eps)) emit((unsigned)k, (unsigned)k + 1u);
        }
    } else {
        // A sphere met the ray: the step-by-step Booleans then also merge H's touching
        // intervals and drop its empty ones.
        auto sweep = [&](const auto &ends) {
            Comp c, prev{};
            bool first = true;
            unsigned from = 0;
            while (next_comp(ends, from, c)) {
                unsigned k0, k1, s0, s1;
                if (A.inner) {  // from the previous component's end to this one's beginning
                    k0 = prev.hi, s0 = prev.hi_src, k1 = c.lo, s1 = c.lo_src;
                } else {
                    k0 = c.lo, s0 = c.lo_src, k1 = c.hi, s1 = c.hi_src;
                }
                const bool whole = A.inner ? !first : c.hi != kHigh;
                if (whole && !(__fsub_rn(key_depth(k1), key_depth(k0)) < A.eps)) {
                    const unsigned side = A.inner ? 1u : 0u;  // where the result enters, the sphere leaves
                    emit(s0 ? (kSph | ((s0 - 1u) << 1) | side) : h_index(k0),
                         s1 ? (kSph | ((s1 - 1u) << 1) | (side ^ 1u)) : h_index(k1));
                }
                if (c.hi == kHigh) break;
                first = false;
                prev = c;
                from = c.hi + 1u;
            }
        };
        if (nb <= 32 * kRegs)
            sweep(Ends<true>(buf, nb, lane));
        else
            sweep(Ends<false>(buf, nb, lane));
    }
    if (!kDeep && lane == 0) {
        pick(A.cnt, b)[p] = nout;
        if (nout && nout <= kKept) {
            uint4 *kp = pick(A.kept, b) + 2 * p;
            kp[0] = make_uint4(tags[0], tags[1], tags[2], tags[3]);
            if (nout > 4) kp[1] = make_uint4(tags[4], tags[5], tags[6], tags[7]);
        }
        if (nout > kKept && atomicExch(&s_deep, 1) == 0) A.deep[1 + atomicAdd(A.deep, 1)] = b * (A.ntx * A.ntx * kTile) + bx;
    }
}

__global__ void __launch_bounds__(kOffWarps * 32) off_count(OffArgs A, ldni_info_t *info) {
    ray_row<false>(A, (int)blockIdx.x, A.img0 + (int)blockIdx.y, info);
}

// The rows that hold rays of more than kKept samples, from the list the count
// pass left (a launch over all rows spends 27 us finding none in most).
__global__ void __launch_bounds__(kOffWarps * 32) off_deep(OffArgs A, ldni_info_t *info) {
    const int rows = A.ntx * A.ntx * kTile, n = A.deep[0];
    for (int q = blockIdx.x; q < n; q += gridDim.x) {
        const int row = A.deep[1 + q];
        ray_row<true>(A, row % rows, row / rows, info);
        __syncthreads();  // the shared buffers are free again
    }
}

// The samples of the rays that have at most kKept, from the sources that the
// count pass left: a thread per ray of image img0 + blockIdx.y.
__global__ void __launch_bounds__(kThreads) off_write(OffArgs A, ldni_info_t *info) {
    const int b = A.img0 + blockIdx.y;
    const long long p = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (p >= (long long)A.res * A.res) return;
    const int n = pick(A.cnt, b)[p];
    if (n == 0 || n > kKept) return;
    const uint4 k = pick(A.kept, b)[2 * p], k2 = n > 4 ? pick(A.kept, b)[2 * p + 1] : k;
    const unsigned tag[kKept] = {k.x, k.y, k.z, k.w, k2.x, k2.y, k2.z, k2.w};
    const int bu = b == 2 ? 0 : b + 1, bv = b == 0 ? 2 : b - 1;
    const float pu = pix((int)p % A.res, A.o[bu], A.h), pv = pix((int)p / A.res, A.o[bv], A.h);
    const long long hb = max(pick(A.hoff, b)[p], 0), slot = pick(A.ooff, b)[p];
#pragma unroll
    for (int z = 0; z < kKept; ++z)
        if (z < n) put_result(A, b, hb, pu, pv, tag[z], slot + z, info);
}

struct OffWs {
    float4 *C;
    int *tcnt[3], *toff[3], *tlist[3], *cnt[3];
    uint4 *kept[3];
    int *deep;
    long long *partials;
    ldni_info_t *tinfo;
    size_t clear_bytes;  // tile counts and tinfo: one memset from tcnt[0]
};

long long tiles_per_sphere(double r_pixels) {
    const double span = std::ceil(2.0 * r_pixels) + 6.0;  // pixel centres a widened shadow can hold, and one more
    const long long per_side = (long long)std::ceil(span / kTile) + 1;
    return per_side * per_side;
}

bool carve_offset(Carver &c, long long S, int res, double r_pixels, OffWs &w) {
    const long long N = (long long)res * res;
    const long long ntx = (res + kTile - 1) / kTile, ntiles = ntx * ntx;
    const double pairs = (double)S * (double)tiles_per_sphere(r_pixels);
    if (pairs > (double)INT_MAX) return false;
    const long long tstride = (ntiles + 63) / 64 * 64;
    int *block = c.take<int>((size_t)(3 * tstride) + sizeof(ldni_info_t) / sizeof(int) + 16);
    for (int a = 0; a < 3; ++a) w.tcnt[a] = block ? block + a * tstride : nullptr;
    w.tinfo = block ? reinterpret_cast<ldni_info_t *>(block + 3 * tstride) : nullptr;
    w.clear_bytes = sizeof(int) * ((size_t)(3 * tstride) + sizeof(ldni_info_t) / sizeof(int) + 16);
    w.C = c.take<float4>((size_t)(S > 0 ? S : 1));
    for (int a = 0; a < 3; ++a) {
        w.toff[a] = c.take<int>((size_t)ntiles + 1);
        w.tlist[a] = c.take<int>((size_t)(pairs > 0 ? pairs : 1));
        w.cnt[a] = c.take<int>((size_t)N);
        w.kept[a] = a == 0 || N <= kKeptTogether ? c.take<uint4>(2 * (size_t)N) : w.kept[0];
    }
    w.deep = c.take<int>(1 + 3 * (size_t)ntiles * kTile);
    const size_t parts = std::max(csr_scan_partials(N), csr_scan_partials(ntiles));
    w.partials = c.take<long long>(parts * 3);
    return true;
}

}  // namespace
}  // namespace ldni

using namespace ldni;

extern "C" int ldni_offset_workspace_size(const int64_t *n, int32_t res, float r, float width, size_t *bytes) {
    if (!n || !bytes || res < 1 || res > 8192 || !(r > 0.0f) || !(width > 0.0f)) return LDNI_EINVAL;
    const long long S = (long long)n[0] + n[1] + n[2];
    if (n[0] < 0 || n[1] < 0 || n[2] < 0 || S >= (1ll << 29)) return LDNI_ETOOLARGE;
    Carver c(nullptr, 0);
    OffWs w{};
    const float h = width / (float)res;
    if (!carve_offset(c, S, res, (double)r / (double)h, w)) return LDNI_ETOOLARGE;
    *bytes = align_up(c.off);
    return LDNI_OK;
}

extern "C" int ldni_offset(const ldni_layers_t *H, const int64_t *n, const ldni_grid_t *grid, float r, int32_t inner,
                           float eps, ldni_layers_t *out, ldni_info_t *info, void *ws, size_t ws_bytes,
                           void *stream) {
    if (!H || !n || !grid_valid(grid) || !(r > 0.0f) || !(r < 3.0e38f) || (inner != 0 && inner != 1) || !out ||
        !info || !ws || !(eps >= 0.0f))
        return LDNI_EINVAL;
    const long long S = (long long)n[0] + n[1] + n[2];
    if (n[0] < 0 || n[1] < 0 || n[2] < 0 || S >= (1ll << 29)) return LDNI_ETOOLARGE;
    for (int a = 0; a < 3; ++a) {
        if (!H[a].offsets || (n[a] > 0 && (!H[a].depth || !H[a].nx || !H[a].ny || !H[a].nz || !H[a].tri_id)) ||
            H[a].capacity < n[a] || H[a].nrm8 || out[a].nrm8)  // FP32 normals only
            return LDNI_EINVAL;
        if (!out[a].offsets || out[a].capacity < 0 ||
            (out[a].capacity > 0 && (!out[a].depth || !out[a].nx || !out[a].ny || !out[a].nz || !out[a].tri_id)))
            return LDNI_EINVAL;
    }
    const int res = grid->res;
    const long long N = (long long)res * res;
    const float h = grid->width / (float)res;
    Carver c(ws, ws_bytes);
    OffWs w{};
    if (!carve_offset(c, S, res, (double)r / (double)h, w)) return LDNI_ETOOLARGE;
    if (!c.fits()) return LDNI_EWORKSPACE;
    OffArgs A{};
    long long acc = 0;
    for (int a = 0; a < 3; ++a) {
        A.hoff[a] = H[a].offsets;
        A.hd[a] = H[a].depth;
        A.hx[a] = H[a].nx;
        A.hy[a] = H[a].ny;
        A.hz[a] = H[a].nz;
        A.ht[a] = H[a].tri_id;
        A.base[a] = acc;
        A.n[a] = n[a];
        acc += n[a];
        A.tcnt[a] = w.tcnt[a];
        A.toff[a] = w.toff[a];
        A.tlist[a] = w.tlist[a];
        A.cnt[a] = w.cnt[a];
        A.kept[a] = w.kept[a];
        A.ooff[a] = out[a].offsets;
        A.od[a] = out[a].depth;
        A.ox[a] = out[a].nx;
        A.oy[a] = out[a].ny;
        A.oz[a] = out[a].nz;
        A.ot[a] = out[a].tri_id;
        A.ocap[a] = out[a].capacity;
        A.o[a] = grid->origin[a];
    }
    A.S = S;
    A.h = h;
    A.res = res;
    A.r = r;
    A.r2 = r * r;
    A.eps = eps;
    A.inner = inner;
    A.inv_h = 1.0f / h;
    for (int a = 0; a < 3; ++a)  // rounding of the bounds, and of the pixel centres o + (t + 1/2) h
        A.slack[a] = (float)std::min(1.0, 0.06 + std::ldexp(std::fabs((double)A.o[a]) + grid->width, -22) / h);
    A.C = w.C;
    A.deep = w.deep;
    A.ntx = (res + kTile - 1) / kTile;
    const long long ntiles = (long long)A.ntx * A.ntx;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (int rc_ = cuda_check(cudaMemsetAsync(w.tcnt[0], 0, w.clear_bytes, s))) return rc_;
    const unsigned rblocks = (unsigned)((N + kThreads - 1) / kThreads);
    const unsigned sblocks = (unsigned)((S + kThreads - 1) / kThreads);
    LDNI_LAUNCH(K_OFFSET, s, off_centres<<<dim3(rblocks, 3), kThreads, 0, s>>>(A));
    if (S > 0) LDNI_LAUNCH(K_OFFSET, s, off_bin<false><<<dim3(sblocks, 3), kThreads, 0, s>>>(A));
    int rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    {
        const int *cnts[3] = {w.tcnt[0], w.tcnt[1], w.tcnt[2]};
        int *offs[3] = {w.toff[0], w.toff[1], w.toff[2]};
        rc = csr_scan(cnts, offs, 3, ntiles, w.partials, w.tinfo, 0, s);
        if (rc != LDNI_OK) return rc;
    }
    // the counts become the fill cursors
    if (int rc_ = cuda_check(cudaMemsetAsync(w.tcnt[0], 0, w.clear_bytes, s))) return rc_;
    if (S > 0) LDNI_LAUNCH(K_OFFSET, s, off_bin<true><<<dim3(sblocks, 3), kThreads, 0, s>>>(A));
    const int together = N <= kKeptTogether ? 3 : 1;
    for (A.img0 = 0; A.img0 < 3; A.img0 += together) {
        if (int rc_ = cuda_check(cudaMemsetAsync(w.deep, 0, sizeof(int), s))) return rc_;
        LDNI_LAUNCH(K_OFFSET, s,
                    off_count<<<dim3((unsigned)(ntiles * kTile), together), kOffWarps * 32, 0, s>>>(A, info));
        rc = cuda_status();
        if (rc != LDNI_OK) return rc;
        const int *cnts[3] = {w.cnt[0], w.cnt[1], w.cnt[2]};
        int *offs[3] = {out[0].offsets, out[1].offsets, out[2].offsets};
        rc = csr_scan(cnts + A.img0, offs + A.img0, together, N, w.partials, info, A.img0, s);
        if (rc != LDNI_OK) return rc;
        LDNI_LAUNCH(K_OFFSET, s, off_write<<<dim3(rblocks, together), kThreads, 0, s>>>(A, info));
        LDNI_LAUNCH(K_OFFSET, s, off_deep<<<4 * num_sms(), kOffWarps * 32, 0, s>>>(A, info));
    }
    return cuda_status();
}
