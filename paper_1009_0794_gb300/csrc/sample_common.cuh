// Triangle traversal shared by the exact two-pass and the learned one-pass
// samplers: per-thread triangle setup, the exact crossing test and hit masks.
//
// A tile is kTilePix consecutive rays of one image in CSR order (rows
// p = j * res + i), so a tile's samples occupy one contiguous CSR range.
#pragma once

#include <climits>

#include "ldni_host.h"

namespace ldni {

constexpr int kTileBits = 12;
constexpr int kTilePix = 1 << kTileBits;  // rays per tile (= one scan chunk)
static_assert(kTilePix == kScanChunk, "a tile is one scan chunk");
constexpr int kBigPixels = 16;            // pixel-centre box of a thread-handled triangle (fits one mask)
constexpr int kHugePixels = 2048;         // boxes above this take whole blocks, smaller big ones a few threads
constexpr int kPairThreads = 4;             // at least so many
// Largest snapped extent (fixed-point units) of a triangle handled with
// 32-bit edge functions.  With every vertex and every visited pixel centre
// (plus one step beyond the box) within 32768 units of each other, each edge
// function |d_u (c_v - v) - d_v (c_u - u)| < 2 * 32767^2 < 2^31.
constexpr int kSmallExtent = 32000;

// Depth of a crossing, d = sum_k lambda_k a_k with lambda_k = E_k / A2 from
// the exact edge functions E_k (FP32 values of integers) and inv = 1 / A2:
// every operation is an explicit rounding, so every traversal (direct,
// binned, one-pass, batched) computes the same bits wherever it is inlined.
__device__ __forceinline__ float depth_of(float E0, float E1, float E2, float inv, float a0, float a1, float a2) {
    const float l0 = __fmul_rn(E0, inv), l1 = __fmul_rn(E1, inv), l2 = __fmul_rn(E2, inv);
    return __fmaf_rn(l2, a2, __fmaf_rn(l1, a1, __fmul_rn(l0, a0)));
}

// Per-thread view of one triangle: snapped lattice coordinates of its three
// vertices (all three world axes) and the world positions.
struct TriView {
    int q[3][3];  // [vertex][axis]
    float3 p[3];
};

// 0 = ok, else an LDNI_ST_* bit (bad index, unsnappable vertex)
__device__ __forceinline__ unsigned load_tri(const float *__restrict__ verts, const int *__restrict__ tris, int t,
                                             int nv, const GridDev &g, TriView &T) {
    const int id[3] = {__ldg(tris + 3 * (long long)t), __ldg(tris + 3 * (long long)t + 1),
                       __ldg(tris + 3 * (long long)t + 2)};
    if ((unsigned)id[0] >= (unsigned)nv || (unsigned)id[1] >= (unsigned)nv || (unsigned)id[2] >= (unsigned)nv)
        return LDNI_ST_INDEX;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float *v = verts + 3 * (long long)id[k];
        T.p[k] = make_float3(__ldg(v), __ldg(v + 1), __ldg(v + 2));
        ok &= snap(T.p[k].x, g.o[0], g.s, T.q[k][0]);
        ok &= snap(T.p[k].y, g.o[1], g.s, T.q[k][1]);
        ok &= snap(T.p[k].z, g.o[2], g.s, T.q[k][2]);
    }
    return ok ? 0u : LDNI_ST_RANGE;
}

__device__ __forceinline__ int owns_i(int du, int dv) { return (dv > 0 || (dv == 0 && du < 0)) ? 1 : 0; }

// Counter-clockwise projection of one triangle on one image, 32-bit form.
struct Setup32 {
    int u0, v0, u1, v1, u2, v2;
    float a0, a1, a2;
    int b0, b1, b2;
    float inv;  // 1 / area2
    int i0, j0, w, h;  // pixel-centre box: i0 .. i0+w-1, j0 .. j0+h-1
    int exiting;       // 1 if the face's projection was counter-clockwise (n_a > 0: the ray leaves the solid)

    // biased edge functions at pixel (i, j): inside iff all three are > 0
    __device__ __forceinline__ void edges(int i, int j, int &e0, int &e1, int &e2) const {
        const int cu = i * kSubpix + kHalfSubpix, cv = j * kSubpix + kHalfSubpix;
        e0 = (u1 - u0) * (cv - v0) - (v1 - v0) * (cu - u0) + b0;
        e1 = (u2 - u1) * (cv - v1) - (v2 - v1) * (cu - u1) + b1;
        e2 = (u0 - u2) * (cv - v2) - (v0 - v2) * (cu - u2) + b2;
    }
    // depth from the biased edge functions at a crossing: lambda_k from the
    // exact edge functions (bias removed); the edge opposite vertex k is k+1
    __device__ __forceinline__ float depth_from(int e0, int e1, int e2) const {
        return depth_of(__int2float_rn(e1 - b1), __int2float_rn(e2 - b2), __int2float_rn(e0 - b0), inv, a0, a1, a2);
    }
    __device__ __forceinline__ float depth(int i, int j) const {
        int e0, e1, e2;
        edges(i, j, e0, e1, e2);
        return depth_from(e0, e1, e2);
    }
    // visit every crossed pixel centre of the box: f(i, j, e0, e1, e2), with
    // the biased edge functions at that centre.  A box of at most 2 x 2
    // pixel centres (nearly every triangle of a mesh finer than the pixel
    // grid) is tested without a loop, so that the lanes of a warp, whose
    // boxes differ, run the same instructions; a larger box builds its hit
    // mask first and then visits the mask's bits.  Either way the crossings
    // come in row-major order.
    template <class F>
    __device__ __forceinline__ void for_each_hit(F &&f) const;
    // the box's crossings as bits x + w y (w * h <= kBigPixels)
    __device__ __forceinline__ unsigned hit_bits() const;
};

// 64-bit form for triangles too large for Setup32.
struct Setup64 {
    long long u0, v0, u1, v1, u2, v2;
    float a0, a1, a2;
    long long b0, b1, b2;
    float inv;
    int exiting;
    __device__ __forceinline__ void edges(int i, int j, long long &e0, long long &e1, long long &e2) const {
        const long long cu = (long long)i * kSubpix + kHalfSubpix, cv = (long long)j * kSubpix + kHalfSubpix;
        e0 = (u1 - u0) * (cv - v0) - (v1 - v0) * (cu - u0) + b0;
        e1 = (u2 - u1) * (cv - v1) - (v2 - v1) * (cu - u1) + b1;
        e2 = (u0 - u2) * (cv - v2) - (v0 - v2) * (cu - u2) + b2;
    }
    __device__ __forceinline__ bool inside(int i, int j) const {
        long long e0, e1, e2;
        edges(i, j, e0, e1, e2);
        return e0 > 0 && e1 > 0 && e2 > 0;
    }
    __device__ __forceinline__ float depth_from(long long e0, long long e1, long long e2) const {
        return depth_of(__ll2float_rn(e1 - b1), __ll2float_rn(e2 - b2), __ll2float_rn(e0 - b0), inv, a0, a1, a2);
    }
    __device__ __forceinline__ float depth_from(int e0, int e1, int e2) const {
        return depth_of(__int2float_rn(e1 - (int)b1), __int2float_rn(e2 - (int)b2), __int2float_rn(e0 - (int)b0), inv,
                        a0, a1, a2);
    }
    __device__ __forceinline__ float depth(int i, int j) const {
        long long e0, e1, e2;
        edges(i, j, e0, e1, e2);
        return depth_from(e0, e1, e2);
    }
    // its vertices lie within kSmallExtent of each other: edge functions at pixel centres of its box fit 32 bits
    __device__ __forceinline__ bool small() const {
        return max(u0, max(u1, u2)) - min(u0, min(u1, u2)) < kSmallExtent &&
               max(v0, max(v1, v2)) - min(v0, min(v1, v2)) < kSmallExtent;
    }
};

enum AxisKind { kNone = 0, kSmall = 1, kBig = 2 };

// Box test and (for small triangles) the 32-bit setup of image A; the
// reciprocal area for depths only when kDepth.
template <int A, bool kDepth = true>
__device__ __forceinline__ int setup_axis(const TriView &T, int res, Setup32 &S) {
    constexpr int U = (A + 1) % 3, V = (A + 2) % 3;
    int u0 = T.q[0][U], u1 = T.q[1][U], u2 = T.q[2][U];
    int v0 = T.q[0][V], v1 = T.q[1][V], v2 = T.q[2][V];
    const int umin = min(u0, min(u1, u2)), umax = max(u0, max(u1, u2));
    const int vmin = min(v0, min(v1, v2)), vmax = max(v0, max(v1, v2));
    // pixel centres 256 i + 128 inside [umin, umax] x [vmin, vmax]
    const int i0 = max((umin + 127) >> 8, 0), i1 = min((umax - 128) >> 8, res - 1);
    const int j0 = max((vmin + 127) >> 8, 0), j1 = min((vmax - 128) >> 8, res - 1);
    if (i0 > i1 || j0 > j1) return kNone;
    S.w = i1 - i0 + 1;
    S.h = j1 - j0 + 1;
    if (umax - umin >= kSmallExtent || vmax - vmin >= kSmallExtent || S.w * S.h > kBigPixels) return kBig;
    int A2 = (u1 - u0) * (v2 - v0) - (v1 - v0) * (u2 - u0);
    if (A2 == 0) return kNone;  // face parallel to the ray (Definition 1 note)
    float a0 = comp(T.p[0], A), a1 = comp(T.p[1], A), a2 = comp(T.p[2], A);
    S.exiting = A2 > 0 ? 1 : 0;
    if (A2 < 0) {  // turn counter-clockwise
        int x = u1; u1 = u2; u2 = x;
        x = v1; v1 = v2; v2 = x;
        const float y = a1; a1 = a2; a2 = y;
        A2 = -A2;
    }
    S.u0 = u0; S.v0 = v0; S.u1 = u1; S.v1 = v1; S.u2 = u2; S.v2 = v2;
    S.a0 = a0; S.a1 = a1; S.a2 = a2;
    S.b0 = owns_i(u1 - u0, v1 - v0);
    S.b1 = owns_i(u2 - u1, v2 - v1);
    S.b2 = owns_i(u0 - u2, v0 - v2);
    S.inv = kDepth ? __frcp_rn(__int2float_rn(A2)) : 0.0f;
    S.i0 = i0; S.j0 = j0; S.w = i1 - i0 + 1; S.h = j1 - j0 + 1;
    return kSmall;
}

// Crossings of the pixel box as a bit mask (bit b = pixel (i0 + b % w, j0 + b / w)).
__device__ __forceinline__ unsigned long long hit_mask(const Setup32 &S) {
    int r0, r1, r2;
    S.edges(S.i0, S.j0, r0, r1, r2);
    const int s0 = -(S.v1 - S.v0) * kSubpix, s1 = -(S.v2 - S.v1) * kSubpix, s2 = -(S.v0 - S.v2) * kSubpix;
    const int t0 = (S.u1 - S.u0) * kSubpix, t1 = (S.u2 - S.u1) * kSubpix, t2 = (S.u0 - S.u2) * kSubpix;
    unsigned long long m = 0;
    int bit = 0;
    for (int y = 0; y < S.h; ++y) {
        int e0 = r0, e1 = r1, e2 = r2;
        for (int x = 0; x < S.w; ++x, ++bit) {
            if ((e0 > 0) & (e1 > 0) & (e2 > 0)) m |= 1ull << bit;
            e0 += s0;
            e1 += s1;
            e2 += s2;
        }
        r0 += t0;
        r1 += t1;
        r2 += t2;
    }
    return m;
}

template <class F>
__device__ __forceinline__ void Setup32::for_each_hit(F &&f) const {
    if (w <= 2 && h <= 2) {
        // Edge functions one step beyond the box stay within int32: see kSmallExtent.
        int r0, r1, r2;
        edges(i0, j0, r0, r1, r2);
        const int s0 = -(v1 - v0) * kSubpix, s1 = -(v2 - v1) * kSubpix, s2 = -(v0 - v2) * kSubpix;
        const int t0 = (u1 - u0) * kSubpix, t1 = (u2 - u1) * kSubpix, t2 = (u0 - u2) * kSubpix;
        const unsigned w2 = w == 2, h2 = h == 2;
        const unsigned c00 = (r0 > 0) & (r1 > 0) & (r2 > 0);
        const unsigned c10 = w2 & (r0 + s0 > 0) & (r1 + s1 > 0) & (r2 + s2 > 0);
        const unsigned c01 = h2 & (r0 + t0 > 0) & (r1 + t1 > 0) & (r2 + t2 > 0);
        const unsigned c11 = w2 & h2 & (r0 + s0 + t0 > 0) & (r1 + s1 + t1 > 0) & (r2 + s2 + t2 > 0);
        unsigned m = c00 | (c10 << 1) | (c01 << 2) | (c11 << 3);  // bit x + 2 y
        while (m) {
            const int b = __ffs(m) - 1;
            m &= m - 1;
            const int x = b & 1, y = b >> 1;
            f(i0 + x, j0 + y, r0 + x * s0 + y * t0, r1 + x * s1 + y * t1, r2 + x * s2 + y * t2);
        }
        return;
    }
    const unsigned long long m = hit_mask(*this);
    const unsigned long long row_mask = w >= 64 ? ~0ull : ((1ull << w) - 1);
    for (int y = 0; y < h; ++y) {
        unsigned long long r = (m >> (y * w)) & row_mask;
        while (r) {
            const int x = __ffsll((long long)r) - 1;
            r &= r - 1;
            int e0, e1, e2;
            edges(i0 + x, j0 + y, e0, e1, e2);
            f(i0 + x, j0 + y, e0, e1, e2);
        }
    }
}

__device__ __forceinline__ unsigned Setup32::hit_bits() const {
    if (w <= 2 && h <= 2) {  // loop-free, as in for_each_hit
        int r0, r1, r2;
        edges(i0, j0, r0, r1, r2);
        const int s0 = -(v1 - v0) * kSubpix, s1 = -(v2 - v1) * kSubpix, s2 = -(v0 - v2) * kSubpix;
        const int t0 = (u1 - u0) * kSubpix, t1 = (u2 - u1) * kSubpix, t2 = (u0 - u2) * kSubpix;
        const unsigned w2 = w == 2, h2 = h == 2;
        const unsigned c00 = (r0 > 0) & (r1 > 0) & (r2 > 0);
        const unsigned c10 = w2 & (r0 + s0 > 0) & (r1 + s1 > 0) & (r2 + s2 > 0);
        const unsigned c01 = h2 & (r0 + t0 > 0) & (r1 + t1 > 0) & (r2 + t2 > 0);
        const unsigned c11 = w2 & h2 & (r0 + s0 + t0 > 0) & (r1 + s1 + t1 > 0) & (r2 + s2 + t2 > 0);
        return c00 | (c10 << 1) | (c01 << w) | (c11 << (w + 1));  // bit x + w y
    }
    return (unsigned)hit_mask(*this);
}

// 64-bit setup of image a for a queued big triangle; false when parallel.
__device__ __forceinline__ bool setup_big(const TriView &T, int a, int res, Setup64 &S, int &i0, int &i1, int &j0,
                                          int &j1) {
    const int U = (a + 1) % 3, V = (a + 2) % 3;
    const auto at = [&](int k, int c) { return (long long)(c == 0 ? T.q[k][0] : (c == 1 ? T.q[k][1] : T.q[k][2])); };
    long long u0 = at(0, U), u1 = at(1, U), u2 = at(2, U);
    long long v0 = at(0, V), v1 = at(1, V), v2 = at(2, V);
    long long A2 = (u1 - u0) * (v2 - v0) - (v1 - v0) * (u2 - u0);
    if (A2 == 0) return false;
    float a0 = comp(T.p[0], a), a1 = comp(T.p[1], a), a2 = comp(T.p[2], a);
    S.exiting = A2 > 0 ? 1 : 0;
    if (A2 < 0) {
        long long x = u1; u1 = u2; u2 = x;
        x = v1; v1 = v2; v2 = x;
        const float y = a1; a1 = a2; a2 = y;
        A2 = -A2;
    }
    S.u0 = u0; S.v0 = v0; S.u1 = u1; S.v1 = v1; S.u2 = u2; S.v2 = v2;
    S.a0 = a0; S.a1 = a1; S.a2 = a2;
    S.b0 = (v1 - v0 > 0 || (v1 == v0 && u1 - u0 < 0)) ? 1 : 0;
    S.b1 = (v2 - v1 > 0 || (v2 == v1 && u2 - u1 < 0)) ? 1 : 0;
    S.b2 = (v0 - v2 > 0 || (v0 == v2 && u0 - u2 < 0)) ? 1 : 0;
    S.inv = __frcp_rn(__ll2float_rn(A2));
    const long long umin = min(u0, min(u1, u2)), umax = max(u0, max(u1, u2));
    const long long vmin = min(v0, min(v1, v2)), vmax = max(v0, max(v1, v2));
    i0 = (int)max((umin + 127) >> 8, 0ll);
    i1 = (int)min((umax - 128) >> 8, (long long)res - 1);
    j0 = (int)max((vmin + 127) >> 8, 0ll);
    j1 = (int)min((vmax - 128) >> 8, (long long)res - 1);
    return i0 <= i1 && j0 <= j1;
}

// The crossed centres of a big pair's pixel box, swept by `step` threads of
// which this is number `first`, kBatch pixels at a time: hits(v, i, j, depth)
// for the batches with one, v[u] telling which of the kBatch pixels (i[u], j[u])
// are crossed and depth(u) the depth there.  The threads cover a patch 32, 16,
// ... pixels wide, as the box and their number allow, and the edge functions
// advance by additions, in 32 bits for nearly every triangle (Word unsigned:
// additions past the box may wrap, their results are not used), where a pixel
// of the flattened box took a 64-bit division and six 64-bit products.
template <int kBatch, class Word, class Int, class F>
__device__ __forceinline__ void sweep_patch(const Setup64 &S, int i0, int i1, int j0, int j1, int first, int step,
                                            F &&hits) {
    int lw = 0;  // the patch is 2^lw wide
    while (lw < 5 && (1 << lw) <= i1 - i0 && (2 << lw) <= step) ++lw;
    const int i = i0 + (first & ((1 << lw) - 1)), rows = step >> lw;
    int j = j0 + (first >> lw), x = i;
    if (j > j1 || x > i1) return;
    long long q0, q1, q2;
    S.edges(i, j, q0, q1, q2);
    Word r0 = (Word)q0, r1 = (Word)q1, r2 = (Word)q2, e0 = r0, e1 = r1, e2 = r2;
    const Word c0 = (Word)(S.v0 - S.v1) * kSubpix << lw, c1 = (Word)(S.v1 - S.v2) * kSubpix << lw,
               c2 = (Word)(S.v2 - S.v0) * kSubpix << lw;  // a patch to the right
    const Word t0 = (Word)(S.u1 - S.u0) * kSubpix * (Word)rows, t1 = (Word)(S.u2 - S.u1) * kSubpix * (Word)rows,
               t2 = (Word)(S.u0 - S.u2) * kSubpix * (Word)rows;  // the next patch row
    while (j <= j1) {
        bool v[kBatch], any = false;
        int px[kBatch], py[kBatch];
        Int f0[kBatch], f1[kBatch], f2[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            f0[u] = (Int)e0, f1[u] = (Int)e1, f2[u] = (Int)e2;
            px[u] = x, py[u] = j;
            v[u] = j <= j1 && f0[u] > 0 && f1[u] > 0 && f2[u] > 0;
            any |= v[u];
            x += 1 << lw;
            e0 += c0, e1 += c1, e2 += c2;
            if (x > i1) {
                x = i;
                j += rows;
                r0 += t0, r1 += t1, r2 += t2;
                e0 = r0, e1 = r1, e2 = r2;
            }
        }
        if (any) hits(v, px, py, [&](int u) { return S.depth_from(f0[u], f1[u], f2[u]); });
    }
}

template <int kBatch, class F>
__device__ __forceinline__ void sweep_box(const Setup64 &S, int i0, int i1, int j0, int j1, int first, int step,
                                          F &&hits) {
    if (S.small())
        sweep_patch<kBatch, unsigned, int>(S, i0, i1, j0, j1, first, step, hits);
    else
        sweep_patch<1, unsigned long long, long long>(S, i0, i1, j0, j1, first, step, hits);
}

// The fill pass's visit of the crossings among kN pixels of one face: all their
// cursors are in flight before any sample is stored.  off: the image's offsets,
// when a claimed slot has to be held against its ray's end (a fill that may see
// other crossings than its count did), else null.
constexpr int kFillBatch = 4;
template <int kN, class Depth>
__device__ __forceinline__ void fill_batch(const bool (&v)[kN], const int (&i)[kN], const int (&j)[kN], int res,
                                           int exiting, int t, int *cur, const int *off, float *D, int *Tr,
                                           long long cap, ldni_info_t *info, Depth depth) {
    unsigned c[kN], end[kN];
#pragma unroll
    for (int u = 0; u < kN; ++u) c[u] = v[u] ? (unsigned)cur[(long long)j[u] * res + i[u]] : 0u;
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        end[u] = 0xffffffffu;
        if (!v[u]) continue;
        const long long p = (long long)j[u] * res + i[u];
        if (c[u] & 0x80000000u) {
            c[u] = (c[u] & 0x7fffffffu) + (unsigned)exiting;
        } else {
            c[u] = (unsigned)atomicAdd(cur + p, 1);
            if (off) end[u] = (unsigned)off[p + 1];
        }
    }
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        if (!v[u]) continue;
        if (c[u] >= end[u] || (long long)c[u] >= cap) {
            set_status(info, LDNI_ST_CAPACITY);
            continue;
        }
        D[c[u]] = depth(u);
        Tr[c[u]] = t;
    }
}

// Queue of big (triangle, image) pairs: boxes up to kHugePixels from the
// front (a few threads each), larger ones from the back (blocks each); n[0],
// n[1] count the two ends.  The queue holds qcap entries.
template <class Code>
__device__ __forceinline__ void enqueue_big(Code *q, long long qcap, int *n, Code code, long long npx) {
    if (npx > kHugePixels)
        q[qcap - 1 - atomicAdd(n + 1, 1)] = code;
    else
        q[atomicAdd(n, 1)] = code;
}

// Visit every queued huge pair with body(code, first, step), which walks the
// pair's box with `step` threads.  Blocks blk of nblk: the pairs are shared out
// to groups of nblk / (huge pairs) blocks (at least one), each group sweeping
// its pairs with all its threads, so that a few faces of hundreds of thousands
// of pixels keep every SM busy and many huge faces run side by side.
template <class Code, class F>
__device__ __forceinline__ void for_each_huge(const Code *q, long long qcap, const int *n, int blk, int nblk, F &&body) {
    const int nh = n[1];
    if (nh <= 0) return;
    const int G = max(1, nblk / nh);  // blocks per huge pair
    const int groups = nblk / G, grp = blk / G, sub = blk - grp * G;
    if (grp >= groups) return;  // the blocks left over when nblk is no multiple of G
    for (int e = grp; e < nh; e += groups)
        body(q[qcap - 1 - e], sub * (int)blockDim.x + (int)threadIdx.x, G * (int)blockDim.x);
}

// Visit every queued pair in the same way: the medium pairs get a warp each, or
// fewer threads, down to kPairThreads, when there are more pairs than that
// leaves threads for (every thread of a pair repeats its loads and setup, and
// waits for its own crossings' slots: 306,000 pairs of a batch of 48 meshes take
// 56 us (count) and 203 us (fill) with 4 threads each, 190 and 604 with 32; the
// one-pass traversal's pairs of a 50,000-triangle sphere at 1280^2 164 and 549).
template <class Code, class F>
__device__ __forceinline__ void for_each_big(const Code *q, long long qcap, const int *n, int blk, int nblk, F &&body) {
    const int nmed = n[0];
    int pt = 32;
    while (pt > kPairThreads && (long long)nmed * pt > (long long)nblk * blockDim.x) pt >>= 1;
    const int gpb = blockDim.x / pt;
    for (int e = blk * gpb + (int)threadIdx.x / pt; e < nmed; e += nblk * gpb)
        body(q[e], (int)threadIdx.x & (pt - 1), pt);
    for_each_huge(q, qcap, n, blk, nblk, body);
}

__device__ __forceinline__ bool key_less(float d0, int t0, float d1, int t1) {
    return d0 < d1 || (d0 == d1 && t0 < t1);
}

// In-place insertion sort of one ray's samples (SoA arrays) by (depth, tri).
// Normals: FP32 in X, Y, Z, or packed 8-bit words in X with Y = Z = nullptr
// (moved as raw bits).
__device__ __forceinline__ void sort_ray_global(long long b, long long e, float *D, int *Tr, float *X, float *Y,
                                                float *Z) {
    const bool three = Y != nullptr;
    for (long long x = b + 1; x < e; ++x) {
        const float d = D[x];
        const int t = Tr[x];
        const float nx = X[x], ny = three ? Y[x] : 0.0f, nz = three ? Z[x] : 0.0f;
        long long y = x - 1;
        while (y >= b && key_less(d, t, D[y], Tr[y])) {
            D[y + 1] = D[y];
            Tr[y + 1] = Tr[y];
            X[y + 1] = X[y];
            if (three) {
                Y[y + 1] = Y[y];
                Z[y + 1] = Z[y];
            }
            --y;
        }
        D[y + 1] = d;
        Tr[y + 1] = t;
        X[y + 1] = nx;
        if (three) {
            Y[y + 1] = ny;
            Z[y + 1] = nz;
        }
    }
}


// ---- ordering by ranks ------------------------------------------------------------
// Sample i of a ray moves to position b + rank(i), the rank counting the
// samples with a smaller key (equal keys, which valid input never has, by
// index).  The key maps the depth's bits to an unsigned order in which -0 and
// +0 are equal, as under key_less, then the triangle index; every key is
// below ~0 because triangle indices are below INT_MAX.

__device__ __forceinline__ unsigned long long sort_key(float d, int t) {
    unsigned u = __float_as_uint(__fadd_rn(d, 0.0f));
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)u << 32) | (unsigned)(t ^ (int)0x80000000);
}

__device__ __forceinline__ int key_tri(unsigned long long k) { return (int)((unsigned)k ^ 0x80000000u); }

__device__ __forceinline__ int rank_step(unsigned long long kj, unsigned long long ki, int j, int i) {
    return (kj < ki) | ((kj == ki) & (j < i));
}

constexpr int kLanePer = 4;        // a lane orders rays of up to 4 samples by itself
constexpr int kLaneSort = 8;       // longest ray a lane sorts in registers
constexpr int kWarpSortMax = 128;  // longest ray a warp stages in shared memory
constexpr int kRankMax = 768;      // longest ray ordered by ranks in place

// one warp's staging area (3 KB): 128 samples, or 4 per lane, or 768 ranks
struct SortStage {
    unsigned long long key[kWarpSortMax];
    float d[kWarpSortMax], x[kWarpSortMax], y[kWarpSortMax], z[kWarpSortMax];
};
static_assert(sizeof(SortStage) >= kRankMax * sizeof(int), "ranks fit the stage");

struct RayOut {
    float *D;
    int *Tr;
    float *X, *Y, *Z;  // FP32 normals, or packed 8-bit normals in X with Y = Z = nullptr
};

// Unit normals of a mesh's triangles, w: packed 8-bit codes, or a table of the
// codes alone (codes).  An index outside the mesh (a slot that no crossing
// filled: the mesh changed between count and fill) reads as triangle 0.
struct NormalTable {
    const float4 *n;
    int nt;
    bool codes;
    __device__ __forceinline__ float4 operator()(int t) const {
        const int at = (unsigned)t < (unsigned)nt ? t : 0;
        return codes ? make_float4(0.0f, 0.0f, 0.0f, reinterpret_cast<const float *>(n)[at]) : n[at];
    }
};

__device__ __forceinline__ void put_normal(const RayOut &o, long long at, const float4 &q) {
    o.X[at] = o.Y ? q.x : q.w;
    if (o.Y) {
        o.Y[at] = q.y;
        o.Z[at] = q.z;
    }
}

// source of a ray's samples that sits where the ordered ray goes
struct InPlace {
    RayOut o;
    long long b;
    __device__ __forceinline__ void operator()(int i, float &d, int &t, float &x, float &y, float &z) const {
        d = o.D[b + i];
        t = o.Tr[b + i];
        x = o.X[b + i];
        y = o.Y ? o.Y[b + i] : 0.0f;
        z = o.Y ? o.Z[b + i] : 0.0f;
    }
};

__device__ __forceinline__ void stage_put(SortStage &st, int s, float d, int t, float x, float y, float z) {
    st.key[s] = sort_key(d, t);
    st.d[s] = d;
    st.x[s] = x;
    st.y[s] = y;
    st.z[s] = z;
}

__device__ __forceinline__ void stage_get(const SortStage &st, int s, const RayOut &o, long long dst) {
    o.D[dst] = st.d[s];
    o.Tr[dst] = key_tri(st.key[s]);
    o.X[dst] = st.x[s];
    if (o.Y) {
        o.Y[dst] = st.y[s];
        o.Z[dst] = st.z[s];
    }
}

// Stages samples [0, n) at slots base + i, then writes each to b + its rank
// among them; every sample is read before the first store.  kWarp: the 32
// lanes share the ray (lane l takes samples l, l + 32, ...); else one lane
// orders it alone.
template <bool kWarp, class Src>
__device__ __forceinline__ void rank_staged(long long b, int n, const Src &src, const RayOut &o, SortStage &st,
                                            int lane, int base) {
    const int first = kWarp ? lane : 0, step = kWarp ? 32 : 1;
    for (int i = first; i < n; i += step) {
        float d, x, y, z;
        int t;
        src(i, d, t, x, y, z);
        stage_put(st, base + i, d, t, x, y, z);
    }
    if (kWarp) __syncwarp();
    for (int i = first; i < n; i += step) {
        const unsigned long long ki = st.key[base + i];
        int r = 0;
        for (int j = 0; j < n; ++j) r += rank_step(st.key[base + j], ki, j, i);
        stage_get(st, base + i, o, b + r);
    }
    if (kWarp) __syncwarp();
}

// In-place ordering of a ray of kWarpSortMax < n <= kRankMax samples by the
// warp: ranks from the keys in global memory, then the permutation applied
// cycle by cycle by the first lane.
__device__ __forceinline__ void rank_long(long long b, int n, const RayOut &o, SortStage &st, int lane) {
    int *rank = reinterpret_cast<int *>(&st);
    for (int i = lane; i < n; i += 32) {
        const unsigned long long ki = sort_key(o.D[b + i], o.Tr[b + i]);
        int r = 0;
        for (int j = 0; j < n; ++j) r += rank_step(sort_key(o.D[b + j], o.Tr[b + j]), ki, j, i);
        rank[i] = r;
    }
    __syncwarp();
    if (lane == 0) {
        const InPlace at{o, b};
        for (int s0 = 0; s0 < n; ++s0) {
            int pos = rank[s0];
            if (pos < 0 || pos == s0) continue;
            rank[s0] = -1;
            float d, x, y, z;
            int t;
            at(s0, d, t, x, y, z);
            while (pos != s0) {  // carry the element to its place, pick up the one there
                const long long q = b + pos;
                float d2, x2, y2, z2;
                int t2;
                at(pos, d2, t2, x2, y2, z2);
                o.D[q] = d;
                o.Tr[q] = t;
                o.X[q] = x;
                if (o.Y) {
                    o.Y[q] = y;
                    o.Z[q] = z;
                }
                const int nxt = rank[pos];
                rank[pos] = -1;
                d = d2, t = t2, x = x2, y = y2, z = z2;
                pos = nxt;
            }
            o.D[b + s0] = d;
            o.Tr[b + s0] = t;
            o.X[b + s0] = x;
            if (o.Y) {
                o.Y[b + s0] = y;
                o.Z[b + s0] = z;
            }
        }
    }
    __syncwarp();
}

// Orders the rays of the 32 lanes of a warp; every lane calls it, with n = 0
// when it has nothing to order.  Rays of up to kLanePer samples are ordered
// by their own lane, up to kWarpSortMax by the warp from the staged samples,
// up to kRankMax by the warp in place (their samples must already sit at b),
// longer ones by their lane's insertion.  make(sb, b, o) gives the source of
// a ray whose samples are read from sb and go to b in o.  o is the same
// in every lane.
template <class Make>
__device__ __forceinline__ void order_warp_rays(long long b, int n, long long sb, const Make &make, const RayOut &o,
                                                SortStage &st, int lane) {
    if (n >= 2 && n <= kLanePer) rank_staged<false>(b, n, make(sb, b, o), o, st, lane, kLanePer * lane);
    if (n > kRankMax) sort_ray_global(b, b + n, o.D, o.Tr, o.X, o.Y, o.Z);
    __syncwarp();
    unsigned deep = __ballot_sync(0xffffffffu, n > kLanePer && n <= kRankMax);
    while (deep) {
        const int src = __ffs(deep) - 1;
        deep &= deep - 1;
        const long long bb = __shfl_sync(0xffffffffu, b, src);
        const long long sbb = __shfl_sync(0xffffffffu, sb, src);
        const int nn = __shfl_sync(0xffffffffu, n, src);
        if (nn <= kWarpSortMax)
            rank_staged<true>(bb, nn, make(sbb, bb, o), o, st, lane, 0);
        else
            rank_long(bb, nn, o, st, lane);
    }
}

// Rays of kLaneSort < n <= kFlatMax samples, ordered side by side: the samples
// of as many of the warp's rays as fit are staged one after another, whatever
// their lengths, and every lane ranks every 32nd of them within its own ray.
// (One ray at a time leaves most lanes of a warp idle on rays of ten or
// twenty samples, and moved every field through shared memory.)
constexpr int kFlatMax = 256;
struct FlatStage {
    unsigned long long key[kFlatMax];
    long long first[32];  // per lane: the ray's first slot
    int before[32];       // per lane: staged samples before the ray's
};
static_assert(sizeof(FlatStage) <= sizeof(SortStage), "shares the warp's staging area");

__device__ __forceinline__ void order_flat(long long b, int n, const RayOut &r, const NormalTable &nrm, SortStage &stage,
                                           int lane) {
    FlatStage &st = reinterpret_cast<FlatStage &>(stage);
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    for (int done = 0; done < total;) {
        const bool fits = incl - done <= kFlatMax;  // this round's rays, and those before
        const int m = __reduce_max_sync(0xffffffffu, fits ? incl : 0) - done;
        st.first[lane] = b;
        st.before[lane] = incl - n - done;
        __syncwarp();
        // (loads before stores throughout: the stores could be to anything for all the compiler knows)
        constexpr int kPer = kFlatMax / 32, kHalf = kPer / 2;
        float d[kPer];
        int at[kPer], t[kPer];  // the sample's ray (its lane), its triangle
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int s = 32 * q + lane;
            at[q] = 0;
            if (s >= m) continue;
            int lo = 0;  // the last lane that begins at or before s: the one ray that holds it
#pragma unroll
            for (int h = 16; h > 0; h >>= 1)
                if (st.before[lo + h] <= s) lo += h;
            at[q] = lo;
            const long long g = st.first[lo] + (s - st.before[lo]);
            d[q] = r.D[g];
            t[q] = r.Tr[g];
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q)
            if (32 * q + lane < m) st.key[32 * q + lane] = sort_key(d[q], t[q]);
        __syncwarp();
        const int upto = incl - done;  // lane: end of its ray
#pragma unroll
        for (int hq = 0; hq < kPer; hq += kHalf) {
            if (32 * hq >= m) break;  // the same for the whole warp
            long long g[kHalf];
            float4 nq[kHalf];
#pragma unroll
            for (int q = 0; q < kHalf; ++q) {
                const int s = 32 * (hq + q) + lane, L = at[hq + q];
                const int e = __shfl_sync(0xffffffffu, upto, L);
                if (s >= m) continue;
                const unsigned long long k = st.key[s];
                int rank = 0, j = st.before[L];
                for (; j + 4 <= e; j += 4) {  // four reads of shared memory in flight
                    unsigned long long o[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) o[h] = st.key[j + h];
#pragma unroll
                    for (int h = 0; h < 4; ++h) rank += rank_step(o[h], k, j + h, s);
                }
                for (; j < e; ++j) rank += rank_step(st.key[j], k, j, s);
                g[q] = st.first[L] + rank;
                nq[q] = nrm(t[hq + q]);
            }
#pragma unroll
            for (int q = 0; q < kHalf; ++q) {
                if (32 * (hq + q) + lane >= m) continue;
                r.D[g[q]] = d[hq + q];
                r.Tr[g[q]] = t[hq + q];
                put_normal(r, g[q], nq[q]);
            }
        }
        __syncwarp();
        done += m;
    }
}

// ---- ordering of samples that were filled without normals -----------------------------
//
// Two kernels order every ray and give its samples their normals: one for rays
// of few samples, nearly all of them, which lists the runs of 32 rays that hold
// others, and one for those.  Together in one kernel the long rays' registers
// spill in the short ones' path, and a block that meets many long rays makes the
// rest wait, which only images of few rays repay (kSmallSort).  Batch of 48 meshes,
// a quarter of them noisy tori with up to 92 layers: 85 + 141 us, 265 to 510 us in
// one; 1.31 M-triangle sphere at 2048^2: 73 + 6 us, 93 to 140 us in one.

// A lane's range of samples in one run of 32 rays p0 .. (whole warp); odd counts
// are reported if report.
__device__ __forceinline__ int ray_samples(const int *__restrict__ off, long long p0, long long N, long long cap,
                                           int lane, bool report, ldni_info_t *info, long long &b) {
    const long long p = p0 + lane;
    b = p < N ? off[p] : 0;
    long long e = __shfl_down_sync(0xffffffffu, b, 1);
    if (p >= N) return 0;
    if (lane == 31 || p + 1 == N) e = off[p + 1];
    if (report && ((e - b) & 1)) {
        atomicAdd(&info->odd_rays, 1u);
        set_status(info, LDNI_ST_ODD);
    }
    e = min(e, cap);
    return range_ok(b, max(b, e), cap, info) ? (int)max(e - b, 0ll) : 0;
}

// A ray of two samples from slot b on.  pairs8: the arrays are 8-byte aligned.
__device__ __forceinline__ void finish_pair(long long b, const RayOut &r, const NormalTable &nrm, bool pairs8) {
    const bool even = pairs8 && (b & 1) == 0;  // one 8-byte access per field
    float d0, d1;
    int t0, t1;
    if (even) {
        const float2 d = *reinterpret_cast<const float2 *>(r.D + b);
        const int2 t = *reinterpret_cast<const int2 *>(r.Tr + b);
        d0 = d.x, d1 = d.y, t0 = t.x, t1 = t.y;
    } else {
        d0 = r.D[b], d1 = r.D[b + 1], t0 = r.Tr[b], t1 = r.Tr[b + 1];
    }
    const bool swap = key_less(d1, t1, d0, t0);
    const float4 q0 = nrm(swap ? t1 : t0), q1 = nrm(swap ? t0 : t1);
    if (swap) {
        r.D[b] = d1, r.D[b + 1] = d0;
        r.Tr[b] = t1, r.Tr[b + 1] = t0;
    }
    if (even) {
        *reinterpret_cast<float2 *>(r.X + b) = r.Y ? make_float2(q0.x, q1.x) : make_float2(q0.w, q1.w);
        if (r.Y) {
            *reinterpret_cast<float2 *>(r.Y + b) = make_float2(q0.y, q1.y);
            *reinterpret_cast<float2 *>(r.Z + b) = make_float2(q0.z, q1.z);
        }
    } else {
        put_normal(r, b, q0);
        put_normal(r, b + 1, q1);
    }
}

// A ray of up to four samples from slot b on, ordered in registers.
__device__ __forceinline__ void finish_few(long long b, int n, const RayOut &r, const NormalTable &nrm) {
    float d[4];
    int t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        d[i] = i < n ? r.D[b + i] : INFINITY;
        t[i] = i < n ? r.Tr[b + i] : INT_MAX;
    }
    const auto order = [&](int i, int j) {
        if (key_less(d[j], t[j], d[i], t[i])) {
            const float x = d[i];
            d[i] = d[j];
            d[j] = x;
            const int y = t[i];
            t[i] = t[j];
            t[j] = y;
        }
    };
    order(0, 1);
    order(2, 3);
    order(0, 2);
    order(1, 3);
    order(1, 2);
#pragma unroll
    for (int h = 0; h < 4; h += 2) {  // two normals are read before either of their samples is stored
        if (h >= n) break;
        const float4 q0 = nrm(t[h]), q1 = nrm(h + 1 < n ? t[h + 1] : 0);
        r.D[b + h] = d[h];
        r.Tr[b + h] = t[h];
        put_normal(r, b + h, q0);
        if (h + 1 < n) {
            r.D[b + h + 1] = d[h + 1];
            r.Tr[b + h + 1] = t[h + 1];
            put_normal(r, b + h + 1, q1);
        }
    }
}

// A warp's rays (b, n) of other numbers of samples (n = 0: none in this lane).
__device__ __forceinline__ void finish_rest(long long b, int n, const RayOut &r, const NormalTable &nrm, SortStage &st,
                                         int lane) {
    if (n > 0 && n <= 4) {
        finish_few(b, n, r, nrm);
        n = 0;
    } else if (n > 4 && n <= kLaneSort) {
        // the lanes' rays side by side, each in its lane's registers (kLaneSort's network)
        unsigned long long key[kLaneSort];
        float d[kLaneSort];
#pragma unroll
        for (int i = 0; i < kLaneSort; ++i) {
            d[i] = i < n ? r.D[b + i] : 0.0f;
            key[i] = i < n ? sort_key(d[i], r.Tr[b + i]) : ~0ull;
        }
#pragma unroll
        for (int p = 1; p < kLaneSort; p <<= 1)  // Batcher's odd-even merge sort
#pragma unroll
            for (int k = p; k >= 1; k >>= 1)
#pragma unroll
                for (int j = k % p; j + k < kLaneSort; j += 2 * k)
#pragma unroll
                    for (int i = 0; i < k; ++i)
                        if (i + j + k < kLaneSort && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
                            const bool swap = key[i + j + k] < key[i + j];
                            const unsigned long long a = key[i + j], c = key[i + j + k];
                            const float x = d[i + j], y = d[i + j + k];
                            key[i + j] = swap ? c : a;
                            key[i + j + k] = swap ? a : c;
                            d[i + j] = swap ? y : x;
                            d[i + j + k] = swap ? x : y;
                        }
        // (a store could be to the table for all the compiler knows: four normals are read before the
        // first of their samples is stored, or each would wait for the one before)
#pragma unroll
        for (int h = 0; h < kLaneSort; h += 4) {
            if (h >= n) break;
            float4 q[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (h + i < n) q[i] = nrm(key_tri(key[h + i]));
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (h + i < n) {
                    r.D[b + h + i] = d[h + i];
                    r.Tr[b + h + i] = key_tri(key[h + i]);
                    put_normal(r, b + h + i, q[i]);
                }
        }
        n = 0;
    }
    const bool flat = n > 0 && n <= kFlatMax;
    if (__any_sync(0xffffffffu, flat)) order_flat(b, flat ? n : 0, r, nrm, st, lane);
    if (flat) n = 0;
    // longer rays are ordered in place, and get their normals first
    unsigned longer = __ballot_sync(0xffffffffu, n > 0);
    if (!longer) return;
    while (longer) {
        const int src = __ffs(longer) - 1;
        longer &= longer - 1;
        const long long bb = __shfl_sync(0xffffffffu, b, src);
        const int nn = __shfl_sync(0xffffffffu, n, src);
        for (int i = lane; i < nn; i += 32) put_normal(r, bb + i, nrm(r.Tr[bb + i]));
    }
    __syncwarp();
    order_warp_rays(b, n, b, [](long long, long long at, const RayOut &o) { return InPlace{o, at}; }, r, st, lane);
}

}  // namespace ldni
