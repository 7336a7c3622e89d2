// LDNI sampling of a closed triangle mesh, exact two-pass form (Section 3;
// Definitions 1-4).
//
// The paper renders the mesh n_max + 1 times through a stencil-routed
// OpenGL pipeline: pass 1 counts the depth complexity n_p of every pixel,
// passes 2..n_max each capture the n-th fragment, and the host post-sorts
// every pixel (Section 3, Appendix A).  Here the same count-then-fill
// structure runs as CUDA kernels with everything resident on the device:
//
//   count : one thread per triangle snaps its vertices once and, for each
//           requested image, counts every crossed pixel centre, and whether
//           the ray leaves the solid there (= the stencil pass);
//   scan  : counts -> CSR offsets (scan.cu), and every ray's count word becomes
//           its cursor;
//   fill  : the same traversal; every crossing takes a slot of its ray (a ray
//           of one entry and one exit: by that, else with an atomic) and
//           writes depth and triangle id there (= passes 2..n_max);
//   sort  : every ray orders its samples by (depth, tri_id) in place (= the
//           host post-sort) and takes their normals from a per-triangle table.
//
// The scattered 4-byte accesses of the fill are what bounds it, so it makes as
// few as the CSR form allows: for the 1.31 M-triangle sphere at 2048^2 146 us with
// 20 M stores and 10 M cursor loads, 454 us with 51 M stores, 10 M returned
// atomics and 10 M offset loads.  The normals, three fifths of a sample, are
// stored by the sort passes, ray after ray (79 us; 102 us when it had only the
// swaps to do).
//
// A fill may meet other crossings than its count did: the two are separate
// calls, and the cursors of a count serve one fill.  So no slot beyond its ray's
// end is written (a pair's slots are its own, other rays' claims are held
// against the next offset), and the crossings are counted once more: a fill
// that did not see as many as the count reports LDNI_ST_CAPACITY.
//
// Pairs of a triangle and an image whose pixel box is large are queued and swept
// by several threads, huge ones by whole blocks, with 64-bit edge functions where
// 32 bits do not hold them.
#include <algorithm>

#include "sample_common.cuh"

namespace ldni {
namespace {

constexpr int kThreads = 256;

struct Img {
    int *count[3];          // per-ray count words (count pass), cursors (fill pass)
    const int *offsets[3];  // CSR offsets
    float *depth[3];
    float *nx[3];
    float *ny[3];
    float *nz[3];
    int *tri[3];
    long long cap[3];
    float4 *nrm;            // per-triangle normals (x, y, z, packed codes)
    int nt;
    bool codes;             // ... of the codes alone
    bool pairs8;            // every sample array 8-byte aligned
    int *rest_n;            // listed runs of 32 rays left to sort_rest, and the list's length
    int rest_cap;
    unsigned *seen;         // [kSeen] crossings seen by fills since the count, in parts
};
constexpr int kSeen = 32;

// Adds a warp's crossings to the fill's (whole warp).
__device__ __forceinline__ void add_seen(const Img &o, unsigned seen) {
    seen = __reduce_add_sync(0xffffffffu, seen);
    if (seen && (threadIdx.x & 31) == 0) atomicAdd(o.seen + (blockIdx.x & (kSeen - 1)), seen);
}

__device__ __forceinline__ int *sel(int *const (&arr)[3], int a) { return a == 0 ? arr[0] : (a == 1 ? arr[1] : arr[2]); }

// The fill pass over a triangle's box, two crossings at a time: both cursors
// are in flight before either sample is stored.  m: the box's crossings, bit
// x + w y.
template <int A>
__device__ __forceinline__ void fill_hits(const Setup32 &S, unsigned m, int t, const Img &o, int res, ldni_info_t *info) {
    const int wdiv = (256 + S.w - 1) / S.w;  // y = (b * wdiv) >> 8 = b / w for b < 16, w <= 16
    int *cur = o.count[A];
    const int *off = o.offsets[A];
    const long long cap = o.cap[A];
    while (m) {
        int pr[2];
        unsigned c[2], end[2];
        float d[2];
        bool v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            v[u] = m != 0u;
            const int b = v[u] ? __ffs(m) - 1 : 0;
            m &= m - 1u;
            const int y = (b * wdiv) >> 8, x = b - y * S.w;
            pr[u] = (S.j0 + y) * res + S.i0 + x;
            c[u] = v[u] ? (unsigned)cur[pr[u]] : 0u;
            int e0, e1, e2;
            S.edges(S.i0 + x, S.j0 + y, e0, e1, e2);
            d[u] = S.depth_from(e0, e1, e2);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            end[u] = 0xffffffffu;
            if (!v[u]) continue;
            if (c[u] & 0x80000000u) {
                c[u] = (c[u] & 0x7fffffffu) + (unsigned)S.exiting;
            } else {
                c[u] = (unsigned)atomicAdd(cur + pr[u], 1);
                end[u] = (unsigned)off[pr[u] + 1];
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (!v[u]) continue;
            if (c[u] >= end[u] || (long long)c[u] >= cap) {
                set_status(info, LDNI_ST_CAPACITY);
                continue;
            }
            o.depth[A][c[u]] = d[u];
            o.tri[A][c[u]] = t;
        }
    }
}

// Returns the crossings filled.
template <bool kFill, int A>
__device__ __forceinline__ int tri_axis(const TriView &T, int t, const Img &o, int res, int *big_q, long long qcap,
                                        int *big_n, ldni_info_t *info) {
    Setup32 S;
    const int kind = setup_axis<A, kFill>(T, res, S);
    if (kind == kNone) return 0;
    if (kind == kBig) {
        if (!kFill) enqueue_big(big_q, qcap, big_n, t * 4 + A, (long long)S.w * S.h);  // the fill pass reuses it
        return 0;
    }
    if (!kFill) {
        const int word = count_word(S.exiting);
        S.for_each_hit([&](int i, int j, int, int, int) { atomicAdd(o.count[A] + (long long)j * res + i, word); });
        return 0;
    }
    const unsigned m = S.hit_bits();
    fill_hits<A>(S, m, t, o, res, info);
    return __popc(m);
}

// Entry t of the per-triangle table.
__device__ __forceinline__ void put_table(const TriView &T, int t, const Img &o) {
    float3 n;
    face_normal(T.p[0], T.p[1], T.p[2], n.x, n.y, n.z);
    const float code = __uint_as_float(encode_normal8(n.x, n.y, n.z));
    if (o.codes)
        reinterpret_cast<float *>(o.nrm)[t] = code;
    else
        o.nrm[t] = make_float4(n.x, n.y, n.z, code);
}

// Triangles of blocks blk of nblk, a thread each; big ones are queued (count
// pass).  A block takes its triangles on images ax_lo .. ax_hi.  Returns the
// thread's crossings (fill pass).
template <bool kFill>
__device__ __forceinline__ int tri_blocks(const float *__restrict__ verts, const int *__restrict__ tris, int nt, int nv,
                                          const GridDev &g, int ax_lo, int ax_hi, const Img &o, int *big_q,
                                          long long qcap, int *big_n, ldni_info_t *info, int blk, int nblk, bool table) {
    int seen = 0;
    for (int t = blk * blockDim.x + threadIdx.x; t < nt; t += nblk * blockDim.x) {
        TriView T;
        const unsigned bad = load_tri(verts, tris, t, nv, g, T);
        if (bad) {
            if (!kFill) set_status(info, bad);
            continue;
        }
        if (table) put_table(T, t, o);
        if (ax_lo <= 0 && 0 <= ax_hi) seen += tri_axis<kFill, 0>(T, t, o, g.res, big_q, qcap, big_n, info);
        if (ax_lo <= 1 && 1 <= ax_hi) seen += tri_axis<kFill, 1>(T, t, o, g.res, big_q, qcap, big_n, info);
        if (ax_lo <= 2 && 2 <= ax_hi) seen += tri_axis<kFill, 2>(T, t, o, g.res, big_q, qcap, big_n, info);
    }
    return seen;
}

// The queued big (triangle, image) pairs (for_each_big), each swept by its
// threads, on blocks blk of nblk.  Returns the thread's crossings (fill pass).
template <bool kFill>
__device__ __forceinline__ unsigned big_blocks(const float *__restrict__ verts, const int *__restrict__ tris, int nv,
                                               const GridDev &g, const Img &o, const int *big_q, long long qcap,
                                               const int *big_n, ldni_info_t *info, int blk, int nblk) {
    unsigned seen = 0;
    for_each_big(big_q, qcap, big_n, blk, nblk, [&](int code, int first, int step) {
        const int t = code >> 2, a = code & 3;
        TriView T;
        if (load_tri(verts, tris, t, nv, g, T)) return;
        Setup64 S;
        int i0, i1, j0, j1;
        if (!setup_big(T, a, g.res, S, i0, i1, j0, j1)) return;
        int *cnt = sel(o.count, a);
        if (!kFill) {
            const int word = count_word(S.exiting);
            sweep_box<1>(S, i0, i1, j0, j1, first, step, [&](auto &, auto &i, auto &j, auto) {
                atomicAdd(cnt + (long long)j[0] * g.res + i[0], word);
            });
            return;
        }
        float *D = a == 0 ? o.depth[0] : (a == 1 ? o.depth[1] : o.depth[2]);
        int *Tr = a == 0 ? o.tri[0] : (a == 1 ? o.tri[1] : o.tri[2]);
        const long long cap = a == 0 ? o.cap[0] : (a == 1 ? o.cap[1] : o.cap[2]);
        const int *off = a == 0 ? o.offsets[0] : (a == 1 ? o.offsets[1] : o.offsets[2]);
        sweep_box<kFillBatch>(S, i0, i1, j0, j1, first, step, [&](auto &v, auto &i, auto &j, auto depth) {
            for (bool hit : v) seen += hit;
            fill_batch(v, i, j, g.res, S.exiting, t, cnt, off, D, Tr, cap, info, depth);
        });
    });
    return seen;
}

// The count pass's triangles.  With gridDim.y > 1 a thread takes its triangle on
// one image, ax_lo + blockIdx.y, only (tri_grid).
__global__ void __launch_bounds__(kThreads) count_tri(const float *__restrict__ verts, const int *__restrict__ tris,
                                                      int nt, int nv, GridDev g, int ax_lo, int ax_hi, Img o, int *big_q,
                                                      long long qcap, int *big_n, ldni_info_t *info) {
    if (gridDim.y > 1) ax_lo = ax_hi = ax_lo + (int)blockIdx.y;
    tri_blocks<false>(verts, tris, nt, nv, g, ax_lo, ax_hi, o, big_q, qcap, big_n, info, (int)blockIdx.x,
                      (int)gridDim.x, false);
}

template <bool kFill>
__global__ void __launch_bounds__(kThreads) big_pass(const float *__restrict__ verts, const int *__restrict__ tris,
                                                     int nv, GridDev g, Img o, const int *big_q, long long qcap,
                                                     const int *big_n, ldni_info_t *info) {
    const unsigned seen = big_blocks<kFill>(verts, tris, nv, g, o, big_q, qcap, big_n, info, (int)blockIdx.x,
                                            (int)gridDim.x);
    if (kFill) add_seen(o, seen);
}

// The fill pass: the count has left the whole queue, so its pairs are filled
// beside the triangles, on the first `nbig` blocks.
__global__ void __launch_bounds__(kThreads, 4) fill_pass(const float *__restrict__ verts, const int *__restrict__ tris,
                                                         int nt, int nv, GridDev g, int ax_lo, int ax_hi, int nbig, Img o,
                                                         int *big_q, long long qcap, int *big_n, ldni_info_t *info) {
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *o.rest_n = 0;  // sort_rays fills it anew
    unsigned seen = 0;
    if ((int)blockIdx.x < nbig) {
        if (blockIdx.y != 0 || big_n[0] + big_n[1] == 0) return;
        seen = big_blocks<true>(verts, tris, nv, g, o, big_q, qcap, big_n, info, (int)blockIdx.x, nbig);
    } else {
        if (gridDim.y > 1) ax_lo = ax_hi = ax_lo + (int)blockIdx.y;
        seen = tri_blocks<true>(verts, tris, nt, nv, g, ax_lo, ax_hi, o, big_q, qcap, big_n, info,
                                (int)blockIdx.x - nbig, (int)gridDim.x - nbig, blockIdx.y == 0);
    }
    add_seen(o, seen);
}

struct Image {  // one image's arrays
    const int *off;
    RayOut r;
    long long cap;
};
__device__ __forceinline__ Image image_of(const Img &o, int a) {
    Image m;
    m.off = a == 0 ? o.offsets[0] : (a == 1 ? o.offsets[1] : o.offsets[2]);
    m.r.D = a == 0 ? o.depth[0] : (a == 1 ? o.depth[1] : o.depth[2]);
    m.r.Tr = a == 0 ? o.tri[0] : (a == 1 ? o.tri[1] : o.tri[2]);
    m.r.X = a == 0 ? o.nx[0] : (a == 1 ? o.nx[1] : o.nx[2]);
    m.r.Y = a == 0 ? o.ny[0] : (a == 1 ? o.ny[1] : o.ny[2]);
    m.r.Z = a == 0 ? o.nz[0] : (a == 1 ? o.nz[1] : o.nz[2]);
    m.cap = a == 0 ? o.cap[0] : (a == 1 ? o.cap[1] : o.cap[2]);
    return m;
}

// Per-ray ordering by (depth, tri_id) in place, and the samples' normals; also
// flags odd rays.  A warp takes 32 consecutive rays; the runs with rays of
// more than four samples are listed (image << 28 | run) for sort_rest.  (Rays of
// up to four here: torus of 1.2 M triangles at 1900^2 298 -> 283 us a call; spilled
// registers that cost the sphere, whose rays are all pairs, 5 us of 331.)
__global__ void __launch_bounds__(kThreads, 8) sort_rays(long long nrays, int ax_lo, Img o, int *rest,
                                                         ldni_info_t *info) {
    const int a = ax_lo + blockIdx.y;
    const Image m = image_of(o, a);
    const NormalTable nrm{o.nrm, o.nt, o.codes};
    const int lane = threadIdx.x & 31;
    for (long long base = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); base < nrays;
         base += (long long)gridDim.x * blockDim.x) {
        long long b;
        const int n = ray_samples(m.off, base, nrays, m.cap, lane, true, info, b);
        if (__any_sync(0xffffffffu, n > 4) && lane == 0) {
            const int at = atomicAdd(o.rest_n, 1);
            if (at < o.rest_cap) rest[at] = (a << 28) | (int)(base >> 5);
        }
        if (n == 2) finish_pair(b, m.r, nrm, o.pairs8);
        else if (n > 0 && n <= 4) finish_few(b, n, m.r, nrm);
    }
}

// As many crossings must have been met as the offsets have room for (a warp).
__device__ __forceinline__ void check_seen(long long nrays, int ax_lo, int ax_hi, const Img &o, ldni_info_t *info) {
    const int lane = threadIdx.x & 31;
    unsigned seen = __reduce_add_sync(0xffffffffu, o.seen[lane]);
    for (int a = ax_lo; a <= ax_hi; ++a) seen -= (unsigned)image_of(o, a).off[nrays];
    if (lane == 0 && seen != 0u) set_status(info, LDNI_ST_CAPACITY);
}

__global__ void __launch_bounds__(kThreads) sort_rest(long long nrays, int ax_lo, int ax_hi, Img o, const int *rest,
                                                      ldni_info_t *info) {
    __shared__ SortStage stage[kThreads / 32];
    const int lane = threadIdx.x & 31, warps = gridDim.x * (kThreads / 32), n_rest = min(*o.rest_n, o.rest_cap);
    if (blockIdx.x == 0 && threadIdx.x < 32) check_seen(nrays, ax_lo, ax_hi, o, info);
    for (int q = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); q < n_rest; q += warps) {
        const int code = rest[q];
        const Image m = image_of(o, code >> 28);
        long long b;
        const int n = ray_samples(m.off, (long long)(code & 0xfffffff) << 5, nrays, m.cap, lane, false, info, b);
        finish_rest(b, n <= 4 ? 0 : n, m.r, NormalTable{o.nrm, o.nt, o.codes}, stage[threadIdx.x >> 5], lane);
    }
}

// Both in one kernel, for images of few rays (kSmallSort).
__global__ void __launch_bounds__(kThreads, 4) sort_small(long long nrays, int ax_lo, Img o, ldni_info_t *info) {
    __shared__ SortStage stage[kThreads / 32];
    const int a = ax_lo + blockIdx.y;
    const Image m = image_of(o, a);
    const NormalTable nrm{o.nrm, o.nt, o.codes};
    const int lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 32)
        check_seen(nrays, ax_lo, ax_lo + (int)gridDim.y - 1, o, info);
    for (long long base = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); base < nrays;
         base += (long long)gridDim.x * blockDim.x) {
        long long b;
        const int n = ray_samples(m.off, base, nrays, m.cap, lane, true, info, b);
        if (n == 2) finish_pair(b, m.r, nrm, o.pairs8);
        if (__any_sync(0xffffffffu, n != 0 && n != 2))
            finish_rest(b, n == 2 ? 0 : n, m.r, nrm, stage[threadIdx.x >> 5], lane);
    }
}

// ---- tile binning (exact two-pass, binned) ------------------------------------
//
// The same crossings, counted and placed tile by tile instead of triangle by
// triangle: a counting sort bins every (triangle, image) pair to the 16 x 16
// pixel tiles its pixel box touches; one block per tile then stages the
// exact setup (snapped, oriented edge functions, depths, normal) of its
// triangles in shared memory, 128 at a time, and every thread - one pixel -
// tests them all.  A pixel counts its crossings in a register and, in the
// fill, writes them to its own front slots without any atomic; pairs whose
// box touches more than kMaxBinTiles tiles go to the big-triangle queue of
// the direct form, which takes the back slots.  The per-ray order comes from
// sort_rays, so the output equals the direct form's bit for bit.
constexpr int kBinTile = 16;      // pixels per tile side (one per thread)
constexpr int kMaxBinTiles = 16;  // tiles a binned pair may touch
static_assert(kBinTile * kBinTile == kThreads, "a tile is one pixel per thread");

struct BinImg {
    int *tile_cnt[3];   // pairs per tile (count), then the scatter's cursor
    int *tile_off[3];   // exclusive prefix of tile_cnt, tiles + 1 entries
    int *list[3];       // triangle indices, tile by tile
    int tiles_x;        // tiles per image side
};

// Pixel box of triangle T on image A, with its setup: 0 none, 1 small
// (Setup32 in S), 2 big (Setup64 in L); i0..i1, j0..j1 the pixel box.
template <int A>
__device__ __forceinline__ int classify(const TriView &T, int res, Setup32 &S, Setup64 &L, int &i0, int &i1,
                                        int &j0, int &j1, bool with_depth) {
    const int kind = with_depth ? setup_axis<A, true>(T, res, S) : setup_axis<A, false>(T, res, S);
    if (kind == kNone) return 0;
    if (kind == kSmall) {
        i0 = S.i0;
        j0 = S.j0;
        i1 = S.i0 + S.w - 1;
        j1 = S.j0 + S.h - 1;
        return 1;
    }
    return setup_big(T, A, res, L, i0, i1, j0, j1) ? 2 : 0;
}

__device__ __forceinline__ int tiles_touched(int i0, int i1, int j0, int j1) {
    return ((i1 / kBinTile) - (i0 / kBinTile) + 1) * ((j1 / kBinTile) - (j0 / kBinTile) + 1);
}

// kScatter false: count the pairs of every tile; true: write them into the
// tile lists, and queue the pairs that touch too many tiles.
template <bool kScatter, int A>
__device__ __forceinline__ void bin_axis(const TriView &T, int t, int res, const BinImg &b, int *big_q, long long qcap,
                                         int *big_n) {
    Setup32 S;
    Setup64 L;
    int i0, i1, j0, j1;
    const int kind = classify<A>(T, res, S, L, i0, i1, j0, j1, false);
    if (kind == 0) return;
    if (tiles_touched(i0, i1, j0, j1) > kMaxBinTiles) {
        if (kScatter) enqueue_big(big_q, qcap, big_n, t * 4 + A, (long long)(i1 - i0 + 1) * (j1 - j0 + 1));
        return;
    }
    for (int ty = j0 / kBinTile; ty <= j1 / kBinTile; ++ty)
        for (int tx = i0 / kBinTile; tx <= i1 / kBinTile; ++tx) {
            const int tile = ty * b.tiles_x + tx;
            if (!kScatter) {
                atomicAdd(b.tile_cnt[A] + tile, 1);
            } else {
                const int pos = atomicAdd(b.tile_cnt[A] + tile, 1);
                b.list[A][b.tile_off[A][tile] + pos] = t;
            }
        }
}

template <bool kScatter>
__global__ void __launch_bounds__(kThreads) bin_pass(const float *__restrict__ verts, const int *__restrict__ tris,
                                                     int nt, int nv, GridDev g, int ax_lo, int ax_hi, BinImg b, Img o,
                                                     int *big_q, long long qcap, int *big_n, ldni_info_t *info) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
        TriView T;
        const unsigned bad = load_tri(verts, tris, t, nv, g, T);
        if (bad) {
            if (!kScatter) set_status(info, bad);
            continue;
        }
        if (kScatter) put_table(T, t, o);
        if (ax_lo <= 0 && 0 <= ax_hi) bin_axis<kScatter, 0>(T, t, g.res, b, big_q, qcap, big_n);
        if (ax_lo <= 1 && 1 <= ax_hi) bin_axis<kScatter, 1>(T, t, g.res, b, big_q, qcap, big_n);
        if (ax_lo <= 2 && 2 <= ax_hi) bin_axis<kScatter, 2>(T, t, g.res, b, big_q, qcap, big_n);
    }
}

// One staged triangle of a tile: its setup (small: Setup32, big: Setup64),
// pixel box and id.
struct TileTri {
    Setup64 L;
    Setup32 S;
    int kind;  // 0 none, 1 small, 2 big
    int t;
    int i0, i1, j0, j1;
};

template <int A>
__device__ __forceinline__ void stage_tri(const float *__restrict__ verts, const int *__restrict__ tris, int nv,
                                          const GridDev &g, int t, bool fill, TileTri &R) {
    TriView T;
    R.kind = 0;
    R.t = t;
    if (load_tri(verts, tris, t, nv, g, T)) return;
    R.kind = classify<A>(T, g.res, R.S, R.L, R.i0, R.i1, R.j0, R.j1, fill);
}

// Block = tile (blockIdx.x) of image ax_lo + blockIdx.y; thread = pixel.
// Count pass: counts[p] = the count word of the pixel's binned crossings (before
// the big pairs add theirs).  Fill pass: the crossings take the ray's first
// slots, or a pair's by direction, and the cursor moves on for the big pairs.
constexpr int kTileStage = 128;  // triangles staged per round (26 KB of shared memory)

template <bool kFill>
__global__ void __launch_bounds__(kThreads) tile_pass(const float *__restrict__ verts, const int *__restrict__ tris,
                                                      int nv, GridDev g, int ax_lo, BinImg b, Img o,
                                                      ldni_info_t *info) {
    __shared__ TileTri st[kTileStage];
    const int a = ax_lo + blockIdx.y;
    const int tile = blockIdx.x;
    const int tx = tile % b.tiles_x, ty = tile / b.tiles_x;
    const int i = tx * kBinTile + (threadIdx.x % kBinTile), j = ty * kBinTile + (threadIdx.x / kBinTile);
    const bool mine = i < g.res && j < g.res;
    const int *lst = sel(b.list, a) + sel(b.tile_off, a)[tile];
    const int n = sel(b.tile_off, a)[tile + 1] - sel(b.tile_off, a)[tile];
    const long long p = (long long)j * g.res + i;
    int found = 0;          // count: the word so far; fill: the crossings so far
    unsigned cursor = 0;
    long long cap = 0;      // the slots end here
    if (kFill && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *o.rest_n = 0;  // sort_rays fills it anew
    if (kFill && mine) {
        cursor = (unsigned)sel(o.count, a)[p];
        cap = a == 0 ? o.cap[0] : (a == 1 ? o.cap[1] : o.cap[2]);
        const int *off = a == 0 ? o.offsets[0] : (a == 1 ? o.offsets[1] : o.offsets[2]);
        if (!(cursor >> 31)) cap = min(cap, (long long)off[p + 1]);  // (a pair's slots are its own)
    }
    for (int k0 = 0; k0 < n; k0 += kTileStage) {
        const int k = k0 + threadIdx.x;
        if (threadIdx.x < kTileStage && k < n) {
            if (a == 0) stage_tri<0>(verts, tris, nv, g, lst[k], kFill, st[threadIdx.x]);
            else if (a == 1) stage_tri<1>(verts, tris, nv, g, lst[k], kFill, st[threadIdx.x]);
            else stage_tri<2>(verts, tris, nv, g, lst[k], kFill, st[threadIdx.x]);
        }
        __syncthreads();
        const int m = min(kTileStage, n - k0);
        for (int r = 0; r < m && mine; ++r) {
            const TileTri &R = st[r];
            if (R.kind == 0 || i < R.i0 || i > R.i1 || j < R.j0 || j > R.j1) continue;
            float d = 0.0f;
            bool hit;
            if (R.kind == 1) {
                int e0, e1, e2;
                R.S.edges(i, j, e0, e1, e2);
                hit = (e0 > 0) & (e1 > 0) & (e2 > 0);
                if (kFill && hit) d = R.S.depth_from(e0, e1, e2);
            } else {
                hit = R.L.inside(i, j);
                if (kFill && hit) d = R.L.depth(i, j);
            }
            if (!hit) continue;
            const int exiting = R.kind == 1 ? R.S.exiting : R.L.exiting;
            if (kFill) {
                const long long at = (long long)(cursor & 0x7fffffffu) + (cursor >> 31 ? exiting : found);
                if (at >= cap) {
                    set_status(info, LDNI_ST_CAPACITY);
                } else {
                    (a == 0 ? o.depth[0] : (a == 1 ? o.depth[1] : o.depth[2]))[at] = d;
                    (a == 0 ? o.tri[0] : (a == 1 ? o.tri[1] : o.tri[2]))[at] = R.t;
                }
                ++found;
            } else {
                found = (int)((unsigned)found + (unsigned)count_word(exiting));
            }
        }
        __syncthreads();
    }
    if (kFill) add_seen(o, (unsigned)found);
    if (!mine) return;
    if (!kFill)
        sel(o.count, a)[p] = found;  // the big pairs add theirs afterwards
    else if (!(cursor >> 31))
        sel(o.count, a)[p] = (int)(cursor + (unsigned)found);  // the big pairs take the slots after these
}

struct SampleWs {
    int *count[3];
    int *big_n;          // two queue counts, rest's and the fill's right after the counts: one memset clears all
    int *rest;           // runs of 32 rays left to sort_rest
    long long rest_cap;
    long long qcap;
    size_t clear_bytes;
    long long *scan_words;
    int *big_q;
    float4 *nrm;
};

SampleWs carve_sample_ws(Carver &c, long long nt, int res, int naxes) {
    SampleWs w{};
    const long long N = (long long)res * res;
    const long long stride = (N + 63) / 64 * 64;  // every image's counts start 256-byte aligned
    int *block = c.take<int>((size_t)(stride * naxes + 3 + kSeen));
    for (int a = 0; a < naxes; ++a) w.count[a] = block ? block + (size_t)a * stride : nullptr;
    w.big_n = block ? block + (size_t)stride * naxes : nullptr;
    w.clear_bytes = sizeof(int) * (size_t)(stride * naxes + 3 + kSeen);
    w.rest_cap = (N + 31) / 32 * naxes;
    w.rest = c.take<int>((size_t)w.rest_cap);
    w.scan_words = c.take<long long>(csr_scan_partials(N) * naxes);
    w.qcap = nt * naxes > 0 ? nt * naxes : 1;
    w.big_q = c.take<int>((size_t)w.qcap);
    w.nrm = c.take<float4>((size_t)(nt > 0 ? nt : 1));
    return w;
}

struct Call {
    GridDev g;
    int ax_lo, ax_hi, naxes;
    long long nrays;
    Img o;
    SampleWs w;
    cudaStream_t s;
};

int prepare(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const ldni_grid_t *grid, int32_t axis,
            ldni_layers_t *out, ldni_info_t *info, void *ws, size_t ws_bytes, void *stream, bool need_samples,
            Call &C) {
    if (!grid_valid(grid) || !out || !info || !ws || axis < 0 || axis > LDNI_AXIS_ALL || nv <= 0 || nt < 0 ||
        (nt > 0 && (!verts || !tris)))
        return LDNI_EINVAL;
    if (nt > (INT_MAX / 4) || nv > INT_MAX) return LDNI_ETOOLARGE;
    C.ax_lo = axis == LDNI_AXIS_ALL ? 0 : axis;
    C.ax_hi = axis == LDNI_AXIS_ALL ? 2 : axis;
    C.naxes = C.ax_hi - C.ax_lo + 1;
    C.g = make_grid(grid);
    C.nrays = (long long)grid->res * grid->res;
    C.s = static_cast<cudaStream_t>(stream);
    Carver c(ws, ws_bytes);
    SampleWs w = carve_sample_ws(c, nt, grid->res, C.naxes);
    if (!c.fits()) return LDNI_EWORKSPACE;
    C.w = w;
    C.o = Img{};
    C.o.nrm = w.nrm;
    C.o.nt = (int)nt;
    C.o.rest_n = w.big_n + 2;
    C.o.rest_cap = (int)w.rest_cap;
    C.o.seen = reinterpret_cast<unsigned *>(w.big_n + 3);
    C.o.pairs8 = true;
    for (int k = 0; k < C.naxes; ++k) {
        const int a = C.ax_lo + k;
        const ldni_layers_t &L = out[k];
        if (!L.offsets) return LDNI_EINVAL;
        if (need_samples && !samples_ok(L)) return LDNI_EINVAL;
        if (L.capacity < 0) return LDNI_EINVAL;
        C.o.count[a] = w.count[k];
        C.o.offsets[a] = L.offsets;
        C.o.depth[a] = L.depth;
        normal_arrays(L, C.o.nx[a], C.o.ny[a], C.o.nz[a]);
        C.o.tri[a] = L.tri_id;
        C.o.cap[a] = L.capacity;
        for (const void *q : {(const void *)C.o.depth[a], (const void *)C.o.nx[a], (const void *)C.o.ny[a],
                              (const void *)C.o.nz[a], (const void *)C.o.tri[a]})
            C.o.pairs8 &= (reinterpret_cast<uintptr_t>(q) & 7) == 0;
    }
    return LDNI_OK;
}

int grid_blocks(long long work) {
    long long b = (work + kThreads - 1) / kThreads;
    const long long lim = (long long)num_sms() * current_tuning().tri_blocks_per_sm;
    if (b > lim) b = lim;
    return (int)(b > 0 ? b : 1);
}

// Blocks of a triangle pass.  A mesh that leaves threads of the chip idle is
// spread over its images too, which shortens each thread's chain of loads,
// setups and crossings to one image's: 1,280 triangles at 64^2 5.9 + 6.7 us (count and
// fill), one thread for all three images 9.3 + 14.9 us.
dim3 tri_grid(long long nt, int naxes) {
    const bool spread = naxes > 1 && nt * naxes <= (long long)num_sms() * 2048;
    return dim3((unsigned)grid_blocks(nt), spread ? (unsigned)naxes : 1u);
}

// Rays up to which the order is made in one kernel: below it the second launch
// costs more than the registers of the long rays' path, above it less.  us a
// call in one kernel and in two: 30,000-triangle torus 56 and 62 at 400^2 (three
// images), 87 and 91 at 700^2, 120 and 117 at 1000^2; 300,000-triangle sphere 57
// and 60, 87 and 87, 124 and 118.
constexpr long long kSmallSort = 2000000;

int run_count(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const Call &C, ldni_info_t *info) {
    if (int rc_ = cuda_check(cudaMemsetAsync(C.w.count[0], 0, C.w.clear_bytes, C.s))) return rc_;
    if (nt > 0) {
        LDNI_LAUNCH(K_COUNT_TRI, C.s,
                    count_tri<<<tri_grid(nt, C.naxes), kThreads, 0, C.s>>>(verts, tris, (int)nt, (int)nv, C.g, C.ax_lo,
                                                                          C.ax_hi, C.o, C.w.big_q, C.w.qcap,
                                                                          C.w.big_n, info));
        LDNI_LAUNCH(K_COUNT_BIG, C.s,
                    big_pass<false><<<5 * num_sms(), kThreads, 0, C.s>>>(verts, tris, (int)nv, C.g, C.o, C.w.big_q,
                                                                        C.w.qcap, C.w.big_n, info));
    }
    const int *cnt[3];
    int *off[3];
    for (int k = 0; k < C.naxes; ++k) {
        cnt[k] = C.w.count[k];
        off[k] = const_cast<int *>(C.o.offsets[C.ax_lo + k]);
    }
    int rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    return csr_scan(cnt, off, C.naxes, C.nrays, C.w.scan_words, info, C.ax_lo, C.s, nullptr, nullptr, kScanCursors);
}

void run_sort(const Call &C, ldni_info_t *info) {
    if (C.nrays * C.naxes <= kSmallSort) {
        LDNI_LAUNCH(K_SORT, C.s,
                    sort_small<<<dim3(grid_blocks(C.nrays), C.naxes), kThreads, 0, C.s>>>(C.nrays, C.ax_lo, C.o, info));
        return;
    }
    LDNI_LAUNCH(K_SORT, C.s,
                sort_rays<<<dim3(grid_blocks(C.nrays), C.naxes), kThreads, 0, C.s>>>(C.nrays, C.ax_lo, C.o, C.w.rest,
                                                                                    info));
    const long long runs = (C.nrays + 31) / 32 * C.naxes, blocks = (runs + kThreads / 32 - 1) / (kThreads / 32);
    LDNI_LAUNCH(K_SORT, C.s,
                sort_rest<<<(unsigned)std::min(blocks, 3ll * num_sms()), kThreads, 0, C.s>>>(
                    C.nrays, C.ax_lo, C.ax_hi, C.o, C.w.rest, info));
}

int run_fill(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, Call &C, ldni_info_t *info) {
    // images that all take packed normals need a table of the codes alone (16 -> 4 bytes a triangle)
    C.o.codes = true;
    for (int a = C.ax_lo; a <= C.ax_hi; ++a) C.o.codes &= C.o.ny[a] == nullptr;
    if (nt > 0) {
        // Beside the triangles, which saves a launch (4 to 6 us a call) and overlaps the two (300,000
        // triangles at 1900^2: 468 -> 412 us a call), except in large images of meshes whose mean face
        // covers a huge box: their pairs take whole blocks, and longer in this kernel's registers (1,000
        // triangles at 1900^2: 131 and 119 us).
        const bool beside = C.nrays <= (long long)kHugePixels * nt || C.nrays * C.naxes <= kSmallSort;
        const int nbig = beside ? 5 * num_sms() : 0;
        dim3 grid = tri_grid(nt, C.naxes);
        grid.x += (unsigned)nbig;
        LDNI_LAUNCH(K_FILL_TRI, C.s,
                    fill_pass<<<grid, kThreads, 0, C.s>>>(verts, tris, (int)nt, (int)nv, C.g, C.ax_lo, C.ax_hi, nbig,
                                                          C.o, C.w.big_q, C.w.qcap, C.w.big_n, info));
        if (!beside)
            LDNI_LAUNCH(K_FILL_BIG, C.s,
                        big_pass<true><<<5 * num_sms(), kThreads, 0, C.s>>>(verts, tris, (int)nv, C.g, C.o, C.w.big_q,
                                                                           C.w.qcap, C.w.big_n, info));
    }
    run_sort(C, info);
    return cuda_status();
}

// ---- binned form: workspace and launches --------------------------------------

struct BinWs {
    BinImg b;
    int *tile_cnt0;           // every image's tile counts (one clear)
    size_t tile_bytes;
    long long *tile_words;    // scan partials of the tile counts
    ldni_info_t *tile_info;   // the tile scan's report (not the caller's)
    int ntiles;
};

BinWs carve_bin_ws(Carver &c, long long nt, int res, int naxes) {
    BinWs w{};
    w.b.tiles_x = (res + kBinTile - 1) / kBinTile;
    w.ntiles = w.b.tiles_x * w.b.tiles_x;
    const long long stride = ((long long)w.ntiles + 1 + 63) / 64 * 64;
    int *cnt = c.take<int>((size_t)(stride * naxes));
    int *off = c.take<int>((size_t)(stride * naxes));
    const long long lcap = (long long)kMaxBinTiles * (nt > 0 ? nt : 1);
    int *lst = c.take<int>((size_t)(lcap * naxes));
    for (int a = 0; a < naxes; ++a) {
        w.b.tile_cnt[a] = cnt ? cnt + (size_t)a * stride : nullptr;
        w.b.tile_off[a] = off ? off + (size_t)a * stride : nullptr;
        w.b.list[a] = lst ? lst + (size_t)a * lcap : nullptr;
    }
    w.tile_cnt0 = cnt;
    w.tile_bytes = sizeof(int) * (size_t)(stride * naxes);
    w.tile_words = c.take<long long>(csr_scan_partials(w.ntiles) * naxes);
    w.tile_info = c.take<ldni_info_t>(1);
    return w;
}

// The binned image arrays indexed by image (a = ax_lo + k).
BinImg bin_view(const BinWs &w, const Call &C) {
    BinImg b{};
    b.tiles_x = w.b.tiles_x;
    for (int k = 0; k < C.naxes; ++k) {
        b.tile_cnt[C.ax_lo + k] = w.b.tile_cnt[k];
        b.tile_off[C.ax_lo + k] = w.b.tile_off[k];
        b.list[C.ax_lo + k] = w.b.list[k];
    }
    return b;
}

int run_binned_count(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const Call &C, const BinWs &w,
                     ldni_info_t *info) {
    if (int rc_ = cuda_check(cudaMemsetAsync(C.w.count[0], 0, C.w.clear_bytes, C.s))) return rc_;
    if (int rc_ = cuda_check(cudaMemsetAsync(w.tile_cnt0, 0, w.tile_bytes, C.s))) return rc_;
    const BinImg b = bin_view(w, C);
    if (nt > 0)
        LDNI_LAUNCH(K_BIN, C.s,
                    bin_pass<false><<<grid_blocks(nt), kThreads, 0, C.s>>>(verts, tris, (int)nt, (int)nv, C.g, C.ax_lo,
                                                                          C.ax_hi, b, C.o, C.w.big_q, C.w.qcap, C.w.big_n,
                                                                          info));
    const int *tc[3];
    int *to[3];
    for (int k = 0; k < C.naxes; ++k) {
        tc[k] = w.b.tile_cnt[k];
        to[k] = w.b.tile_off[k];
    }
    int rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    rc = csr_scan(tc, to, C.naxes, w.ntiles, w.tile_words, w.tile_info, 0, C.s);
    if (rc != LDNI_OK) return rc;
    if (int rc_ = cuda_check(cudaMemsetAsync(w.tile_cnt0, 0, w.tile_bytes, C.s))) return rc_;  // the scatter's cursors
    if (nt > 0)
        LDNI_LAUNCH(K_BIN, C.s,
                    bin_pass<true><<<grid_blocks(nt), kThreads, 0, C.s>>>(verts, tris, (int)nt, (int)nv, C.g, C.ax_lo,
                                                                         C.ax_hi, b, C.o, C.w.big_q, C.w.qcap, C.w.big_n,
                                                                         info));
    LDNI_LAUNCH(K_TILE, C.s,
                tile_pass<false><<<dim3(w.ntiles, C.naxes), kThreads, 0, C.s>>>(verts, tris, (int)nv, C.g, C.ax_lo, b,
                                                                               C.o, info));
    if (nt > 0)
        LDNI_LAUNCH(K_COUNT_BIG, C.s,
                    big_pass<false><<<5 * num_sms(), kThreads, 0, C.s>>>(verts, tris, (int)nv, C.g, C.o, C.w.big_q,
                                                                        C.w.qcap, C.w.big_n, info));
    const int *cnt[3];
    int *off[3];
    for (int k = 0; k < C.naxes; ++k) {
        cnt[k] = C.w.count[k];
        off[k] = const_cast<int *>(C.o.offsets[C.ax_lo + k]);
    }
    rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    return csr_scan(cnt, off, C.naxes, C.nrays, C.w.scan_words, info, C.ax_lo, C.s, nullptr, nullptr, kScanCursors);
}

int run_binned_fill(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const Call &C, const BinWs &w,
                    ldni_info_t *info) {
    const BinImg b = bin_view(w, C);
    LDNI_LAUNCH(K_TILE, C.s,
                tile_pass<true><<<dim3(w.ntiles, C.naxes), kThreads, 0, C.s>>>(verts, tris, (int)nv, C.g, C.ax_lo, b,
                                                                              C.o, info));
    if (nt > 0)
        LDNI_LAUNCH(K_FILL_BIG, C.s,
                    big_pass<true><<<5 * num_sms(), kThreads, 0, C.s>>>(verts, tris, (int)nv, C.g, C.o, C.w.big_q,
                                                                       C.w.qcap, C.w.big_n, info));
    run_sort(C, info);
    return cuda_status();
}

// prepare() plus the binned part of the workspace (after the direct form's).
int prepare_binned(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const ldni_grid_t *grid,
                   int32_t axis, ldni_layers_t *out, ldni_info_t *info, void *ws, size_t ws_bytes, void *stream,
                   bool need_samples, Call &C, BinWs &w) {
    int rc = prepare(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream, need_samples, C);
    if (rc != LDNI_OK) return rc;
    Carver c(ws, ws_bytes);
    carve_sample_ws(c, nt, grid->res, C.naxes);
    w = carve_bin_ws(c, nt, grid->res, C.naxes);
    return c.fits() ? LDNI_OK : LDNI_EWORKSPACE;
}

}  // namespace
}  // namespace ldni

using namespace ldni;

extern "C" int ldni_sample_workspace_size(int64_t nv, int64_t nt, int32_t res, int32_t axis, size_t *bytes) {
    if (!bytes || res < 1 || res > 8192 || nt < 0 || nv < 0 || axis < 0 || axis > LDNI_AXIS_ALL) return LDNI_EINVAL;
    Carver c(nullptr, 0);
    carve_sample_ws(c, nt, res, axis == LDNI_AXIS_ALL ? 3 : 1);
    *bytes = align_up(c.off);
    return LDNI_OK;
}

extern "C" int ldni_sample_count(const float *verts, int64_t nv, const int32_t *tris, int64_t nt,
                                 const ldni_grid_t *grid, int32_t axis, ldni_layers_t *out, ldni_info_t *info,
                                 void *ws, size_t ws_bytes, void *stream) {
    Call C;
    int rc = prepare(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream, false, C);
    if (rc != LDNI_OK) return rc;
    return run_count(verts, nv, tris, nt, C, info);
}

extern "C" int ldni_sample_fill(const float *verts, int64_t nv, const int32_t *tris, int64_t nt,
                                const ldni_grid_t *grid, int32_t axis, ldni_layers_t *out, ldni_info_t *info,
                                void *ws, size_t ws_bytes, void *stream) {
    Call C;
    int rc = prepare(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream, true, C);
    if (rc != LDNI_OK) return rc;
    return run_fill(verts, nv, tris, nt, C, info);
}

static int ldni_sample_exact2(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const ldni_grid_t *grid,
                       int32_t axis, ldni_layers_t *out, ldni_info_t *info, void *ws, size_t ws_bytes, void *stream) {
    Call C;
    int rc = prepare(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream, true, C);
    if (rc != LDNI_OK) return rc;
    rc = run_count(verts, nv, tris, nt, C, info);
    if (rc != LDNI_OK) return rc;
    return run_fill(verts, nv, tris, nt, C, info);
}

extern "C" int ldni_sample_binned_workspace_size(int64_t nv, int64_t nt, int32_t res, int32_t axis, size_t *bytes) {
    if (!bytes || res < 1 || res > 8192 || nt < 0 || nv < 0 || axis < 0 || axis > LDNI_AXIS_ALL) return LDNI_EINVAL;
    if (nt > (INT_MAX / (4 * kMaxBinTiles))) return LDNI_ETOOLARGE;
    Carver c(nullptr, 0);
    const int naxes = axis == LDNI_AXIS_ALL ? 3 : 1;
    carve_sample_ws(c, nt, res, naxes);
    carve_bin_ws(c, nt, res, naxes);
    *bytes = align_up(c.off);
    return LDNI_OK;
}

extern "C" int ldni_sample_binned_count(const float *verts, int64_t nv, const int32_t *tris, int64_t nt,
                                        const ldni_grid_t *grid, int32_t axis, ldni_layers_t *out, ldni_info_t *info,
                                        void *ws, size_t ws_bytes, void *stream) {
    if (nt > (INT_MAX / (4 * kMaxBinTiles))) return LDNI_ETOOLARGE;
    Call C;
    BinWs w;
    int rc = prepare_binned(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream, false, C, w);
    if (rc != LDNI_OK) return rc;
    return run_binned_count(verts, nv, tris, nt, C, w, info);
}

extern "C" int ldni_sample_binned_fill(const float *verts, int64_t nv, const int32_t *tris, int64_t nt,
                                       const ldni_grid_t *grid, int32_t axis, ldni_layers_t *out, ldni_info_t *info,
                                       void *ws, size_t ws_bytes, void *stream) {
    if (nt > (INT_MAX / (4 * kMaxBinTiles))) return LDNI_ETOOLARGE;
    Call C;
    BinWs w;
    int rc = prepare_binned(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream, true, C, w);
    if (rc != LDNI_OK) return rc;
    return run_binned_fill(verts, nv, tris, nt, C, w, info);
}

extern "C" int ldni_sample(const float *verts, int64_t nv, const int32_t *tris, int64_t nt, const ldni_grid_t *grid,
                           int32_t axis, int32_t mode, ldni_layers_t *out, ldni_info_t *info, void *ws,
                           size_t ws_bytes, void *stream) {
    if (mode == LDNI_MODE_EXACT2) return ldni_sample_exact2(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes,
                                                            stream);
    if (mode != LDNI_MODE_BINNED2) return LDNI_EINVAL;  // the learned one-pass form is ldni_sample_learned
    int rc = ldni_sample_binned_count(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream);
    if (rc != LDNI_OK) return rc;
    return ldni_sample_binned_fill(verts, nv, tris, nt, grid, axis, out, info, ws, ws_bytes, stream);
}
