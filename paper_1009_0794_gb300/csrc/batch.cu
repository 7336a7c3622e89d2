// Many meshes, of uneven size and resolution, sampled by ONE launch per stage
// (count, scan, fill, sort) for the whole batch - the exact two-pass form of
// sample.cu spread over every triangle, chunk and ray of the batch at once.
// Each block finds its mesh by a binary search over prefix tables that a setup
// kernel builds on the device from the caller's device array of item
// descriptors, so a batch call needs no host synchronisation and can be
// captured in a CUDA graph.  A block's triangles or rays are of one mesh: its
// descriptor's pointers are the same for all threads, and are read once (and
// its fixed-point scale is divided out once in the setup kernel: a division in
// FP64, at 1/64 of the FP32 rate, for every triangle and every thread of a big
// pair was most of the big passes' time: 308 -> 75 us for the counts of 48 meshes).
#include "lookback.cuh"
#include "sample_common.cuh"

namespace ldni {
namespace {

constexpr int kThreads = 256;

struct Tables {
    long long *tri_prefix;    // [count + 1]
    long long *tile_prefix;   // [count + 1]      tiles of kThreads triangles
    long long *chunk_prefix;  // [3 count + 1]  scan chunks
    long long *count_base;    // [3 count]      start of the image's counts
    float *scale;             // [count]        fixed-point units per world unit (an FP64 division)
    float4 *nrm;              // per-triangle normals of all items (x, y, z, packed codes)
    long long *big;           // queued big (item, triangle, image): item << 34 | tri << 2 | a
    long long qcap;
    int *big_n;               // counts of the queue's two ends, and of rest
    long long *rest;          // runs of 32 rays left to batch_rest
};

// k with prefix[k] <= x < prefix[k + 1], the same x in the whole warp: a search
// in 32 parts at a time (two dependent loads for up to a thousand entries, where
// halving took ten in every block's first microseconds).
__device__ __forceinline__ int find(const long long *prefix, int n, long long x) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int part = (hi - lo + 31) / 32, at = lo + (lane + 1) * part;
        const int k = __popc(__ballot_sync(0xffffffffu, at < hi && prefix[at] <= x));
        lo += k * part;
        hi = min(hi, lo + part);
    }
    return lo;
}

__device__ __forceinline__ GridDev grid_dev(const ldni_grid_t &g, float scale) {
    GridDev d;
    d.o[0] = g.origin[0];
    d.o[1] = g.origin[1];
    d.o[2] = g.origin[2];
    d.s = scale;
    d.res = g.res;
    return d;
}

// One block builds the prefix tables of the batch, kThreads items at a time:
// per item its triangles, and per image its rays, scan chunks and counts
// (padded to 64 ints); the images of an item have the same size.
__global__ void __launch_bounds__(kThreads) setup_kernel(const ldni_batch_item_t *items, int count, Tables T) {
    __shared__ long long sh[4][kThreads / 32 + 1];
    __shared__ long long carry[4];
    if (threadIdx.x < 4) carry[threadIdx.x] = 0;
    __syncthreads();
    for (int m0 = 0; m0 < count; m0 += kThreads) {
        const int m = m0 + threadIdx.x;
        long long v[4] = {0, 0, 0, 0};  // triangles, tiles; chunks, count ints of one image
        if (m < count) {
            const long long N = (long long)items[m].grid.res * items[m].grid.res;
            v[0] = items[m].nt;
            v[1] = (v[0] + kThreads - 1) / kThreads;
            v[2] = (N + kScanChunk - 1) / kScanChunk;
            v[3] = (N + 63) / 64 * 64;
        }
        long long ex[4], tot[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) ex[q] = block_exclusive_scan<kThreads>(q < 2 ? v[q] : 3 * v[q], sh[q], &tot[q]);
        if (m < count) {
            const ldni_grid_t &g = items[m].grid;
            T.scale[m] = (float)((double)g.res * (double)kSubpix / (double)g.width);  // as the host computes it
            T.tri_prefix[m] = carry[0] + ex[0];
            T.tile_prefix[m] = carry[1] + ex[1];
            for (int a = 0; a < 3; ++a) {
                T.chunk_prefix[3 * m + a] = carry[2] + ex[2] + a * v[2];
                T.count_base[3 * m + a] = carry[3] + ex[3] + a * v[3];
            }
        }
        __syncthreads();  // every thread has read the carries
        if (threadIdx.x < 4) carry[threadIdx.x] += tot[threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        T.tri_prefix[count] = carry[0];
        T.tile_prefix[count] = carry[1];
        T.chunk_prefix[3 * count] = carry[2];
    }
}

// The fill pass over a triangle's box, two crossings at a time: both cursors
// are in flight before either sample is stored (as the single-mesh fill).
// mk: the box's crossings, bit x + w y.
template <int A>
__device__ __forceinline__ void batch_fill_hits(const ldni_batch_item_t &it, const Setup32 &S, unsigned mk, int t,
                                                int *cur, int res, ldni_info_t *info) {
    const ldni_layers_t &L = it.out[A];
    float *D = L.depth;
    int *Tr = L.tri_id;
    const long long cap = L.capacity;
    const int wdiv = (256 + S.w - 1) / S.w;  // y = (b * wdiv) >> 8 = b / w for b < 16, w <= 16
    while (mk) {
        int pr[2];
        unsigned c[2];
        float d[2];
        bool v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            v[u] = mk != 0u;
            const int b = v[u] ? __ffs(mk) - 1 : 0;
            mk &= mk - 1u;
            const int y = (b * wdiv) >> 8, x = b - y * S.w;
            pr[u] = (S.j0 + y) * res + S.i0 + x;
            c[u] = v[u] ? (unsigned)cur[pr[u]] : 0u;
            int e0, e1, e2;
            S.edges(S.i0 + x, S.j0 + y, e0, e1, e2);
            d[u] = S.depth_from(e0, e1, e2);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (!v[u]) continue;
            c[u] = c[u] & 0x80000000u ? (c[u] & 0x7fffffffu) + (unsigned)S.exiting : (unsigned)atomicAdd(cur + pr[u], 1);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (!v[u]) continue;
            if ((long long)c[u] >= cap) {
                set_status(info, LDNI_ST_CAPACITY);
                continue;
            }
            D[c[u]] = d[u];
            Tr[c[u]] = t;
        }
    }
}

template <bool kFill, int A>
__device__ __forceinline__ void batch_axis(const ldni_batch_item_t &it, int m, const TriView &Tv, int t,
                                           int res, int *counts, const Tables &T, ldni_info_t *info) {
    Setup32 S;
    const int kind = setup_axis<A, kFill>(Tv, res, S);
    if (kind == kNone) return;
    if (kind == kBig) {
        if (!kFill)
            enqueue_big(T.big, T.qcap, T.big_n, ((long long)m << 34) | ((long long)t << 2) | A, (long long)S.w * S.h);
        return;
    }
    int *cnt = counts + T.count_base[3 * m + A];
    if (!kFill) {
        const int word = count_word(S.exiting);
        S.for_each_hit([&](int i, int j, int, int, int) { atomicAdd(cnt + (long long)j * res + i, word); });
        return;
    }
    batch_fill_hits<A>(it, S, S.hit_bits(), t, cnt, res, info);
}

template <bool kFill>
__global__ void __launch_bounds__(kThreads) batch_tri_pass(const ldni_batch_item_t *items, int count, Tables T,
                                                           int *counts, ldni_info_t *infos) {
    const long long tile = blockIdx.x;
    const int m = find(T.tile_prefix, count, tile);
    const ldni_batch_item_t &it = items[m];
    const long long t0 = (tile - T.tile_prefix[m]) * kThreads + threadIdx.x;
    if (t0 >= it.nt) return;
    const int t = (int)t0;
    const GridDev g = grid_dev(it.grid, T.scale[m]);
    TriView Tv;
    const unsigned bad = load_tri(it.verts, it.tris, t, (int)it.nv, g, Tv);
    if (bad) {
        if (!kFill) set_status(infos + m, bad);
        return;
    }
    if (kFill) {
        float3 n;
        face_normal(Tv.p[0], Tv.p[1], Tv.p[2], n.x, n.y, n.z);
        T.nrm[T.tri_prefix[m] + t] = make_float4(n.x, n.y, n.z, __uint_as_float(encode_normal8(n.x, n.y, n.z)));
    }
    batch_axis<kFill, 0>(it, m, Tv, t, g.res, counts, T, infos + m);
    batch_axis<kFill, 1>(it, m, Tv, t, g.res, counts, T, infos + m);
    batch_axis<kFill, 2>(it, m, Tv, t, g.res, counts, T, infos + m);
}

template <bool kFill>
__global__ void __launch_bounds__(kThreads, 4) batch_big(const ldni_batch_item_t *items, Tables T, int *counts,
                                                      ldni_info_t *infos) {
    for_each_big(T.big, T.qcap, T.big_n, (int)blockIdx.x, (int)gridDim.x,
                 [&](long long code, int first, int step) {
        const int m = (int)(code >> 34), t = (int)((code >> 2) & 0xFFFFFFFF), a = (int)(code & 3);
        const ldni_batch_item_t &it = items[m];
        const GridDev g = grid_dev(it.grid, T.scale[m]);
        TriView Tv;
        if (load_tri(it.verts, it.tris, t, (int)it.nv, g, Tv)) return;
        Setup64 S;
        int i0, i1, j0, j1;
        if (!setup_big(Tv, a, g.res, S, i0, i1, j0, j1)) return;
        int *cnt = counts + T.count_base[3 * m + a];
        if (!kFill) {
            const int word = count_word(S.exiting);
            sweep_box<1>(S, i0, i1, j0, j1, first, step, [&](auto &, auto &i, auto &j, auto) {
                atomicAdd(cnt + (long long)j[0] * g.res + i[0], word);
            });
            return;
        }
        const ldni_layers_t &L = it.out[a];
        float *D = L.depth;
        int *Tr = L.tri_id;
        const long long cap = L.capacity;
        sweep_box<kFillBatch>(S, i0, i1, j0, j1, first, step, [&](auto &v, auto &i, auto &j, auto depth) {
            fill_batch(v, i, j, g.res, S.exiting, t, cnt, nullptr, D, Tr, cap, infos + m, depth);
        });
    });
}

// Scan of every image's count words: chunks of all images in one launch; the
// look-back of a chunk stops at the first chunk of its own image.  Offsets go
// to the image, cursors over the words.  A thread's 16 words come as four
// 16-byte loads of whole lines per warp each: 45 us for the 12.5 M rays of 48
// meshes, 89 us with sixteen 4-byte loads 64 bytes apart.
__global__ void __launch_bounds__(kThreads) batch_scan(const ldni_batch_item_t *items, int count, Tables T,
                                                       int *counts, unsigned long long *words, ldni_info_t *infos,
                                                       int spin_limit) {
    constexpr int kSlices = kScanChunk / (4 * kThreads), kWarps = kThreads / 32;
    __shared__ long long tot[kSlices][kWarps];  // samples of each warp's words, per slice
    __shared__ long long s_chunk, s_base;
    const long long nchunks = T.chunk_prefix[3 * count];
    if (threadIdx.x == 0) s_chunk = (long long)atomicAdd(words + nchunks, 1ull);
    __syncthreads();
    const long long c = s_chunk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int img = find(T.chunk_prefix, 3 * count, c);
    const int m = img / 3, a = img % 3;
    const long long local = c - T.chunk_prefix[img];
    const long long N = (long long)items[m].grid.res * items[m].grid.res;
    int *cnt = counts + T.count_base[img];  // 256-byte aligned, padded to 64 words (zeros)
    int *out = items[m].out[a].offsets;
    const long long base = local * kScanChunk;
    int4 v[kSlices];
    long long xin[kSlices];  // samples before the thread's words within its warp
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
        const long long e = base + s * 4 * kThreads + threadIdx.x * 4;
        v[s] = e < N ? *reinterpret_cast<const int4 *>(cnt + e) : make_int4(0, 0, 0, 0);
    }
    long long wtot[kSlices];
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
        const long long mine = (long long)count_of(v[s].x) + count_of(v[s].y) + count_of(v[s].z) + count_of(v[s].w);
        long long x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        xin[s] = x - mine;
        wtot[s] = x;
    }
    if (lane == 31)
#pragma unroll
        for (int s = 0; s < kSlices; ++s) tot[s][warp] = wtot[s];
    __syncthreads();
    long long carry = 0;
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
        long long lead = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const long long t = tot[s][w];
            all += t;
            if (w < warp) lead += t;
        }
        xin[s] += carry + lead;
        carry += all;
    }
    if (threadIdx.x < 32) {
        // image-local status words: chunk 0 of the image starts at prefix 0
        const long long b = lookback_warp(words + T.chunk_prefix[img], (int)local, carry, infos + m, spin_limit);
        if (threadIdx.x == 0) s_base = b;
    }
    __syncthreads();
    const bool vec = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
#pragma unroll
    for (int s = 0; s < kSlices; ++s) {
        const long long e = base + s * 4 * kThreads + threadIdx.x * 4;
        if (e >= N) continue;
        const long long o0 = s_base + xin[s], o1 = o0 + count_of(v[s].x), o2 = o1 + count_of(v[s].y),
                        o3 = o2 + count_of(v[s].z);
        const auto clamp = [](long long x) { return (int)min(x, (long long)INT_MAX); };
        const int4 w = make_int4(clamp(o0), clamp(o1), clamp(o2), clamp(o3));
        *reinterpret_cast<int4 *>(cnt + e) = make_int4(make_cursor(w.x, v[s].x), make_cursor(w.y, v[s].y),
                                                       make_cursor(w.z, v[s].z), make_cursor(w.w, v[s].w));
        if (vec && e + 3 < N) {
            *reinterpret_cast<int4 *>(out + e) = w;
        } else {
            out[e] = w.x;
            if (e + 1 < N) out[e + 1] = w.y;
            if (e + 2 < N) out[e + 2] = w.z;
            if (e + 3 < N) out[e + 3] = w.w;
        }
    }
    if (local == T.chunk_prefix[img + 1] - T.chunk_prefix[img] - 1 && threadIdx.x == 0) {
        const long long n_img = s_base + carry;
        out[N] = (int)min(n_img, (long long)INT_MAX);
        infos[m].n[a] = n_img;
        if (n_img > INT_MAX) set_status(infos + m, LDNI_ST_TOOLARGE);
    }
}

// Ordering of every ray of the batch, and its samples' normals, as in the
// single-mesh sampling: kSortParts blocks per chunk, and the runs of 32 rays
// with others than two samples listed (image << 32 | run) for batch_rest.
constexpr int kSortParts = 4, kSortRays = kScanChunk / kSortParts;

struct ItemImage {
    const int *off;
    RayOut r;
    NormalTable nrm;
    long long cap, N;
    bool pairs8;
};
__device__ __forceinline__ ItemImage item_image(const ldni_batch_item_t *items, const Tables &T, int img) {
    const int m = img / 3, a = img % 3;
    const ldni_layers_t &L = items[m].out[a];
    ItemImage I;
    I.off = L.offsets;
    I.r = L.nrm8 ? RayOut{L.depth, L.tri_id, reinterpret_cast<float *>(L.nrm8), nullptr, nullptr}
                 : RayOut{L.depth, L.tri_id, L.nx, L.ny, L.nz};
    I.nrm = NormalTable{T.nrm + T.tri_prefix[m], (int)items[m].nt, false};
    I.cap = L.capacity;
    I.N = (long long)items[m].grid.res * items[m].grid.res;
    I.pairs8 = ((reinterpret_cast<uintptr_t>(I.r.D) | reinterpret_cast<uintptr_t>(I.r.Tr) |
                 reinterpret_cast<uintptr_t>(I.r.X) | reinterpret_cast<uintptr_t>(I.r.Y) |
                 reinterpret_cast<uintptr_t>(I.r.Z)) & 7) == 0;
    return I;
}

__global__ void __launch_bounds__(kThreads) batch_sort(const ldni_batch_item_t *items, int count, Tables T,
                                                       ldni_info_t *infos) {
    const int lane = threadIdx.x & 31;
    const long long c = blockIdx.x / kSortParts;
    const int img = find(T.chunk_prefix, 3 * count, c);
    const ItemImage I = item_image(items, T, img);
    const long long p0 = (c - T.chunk_prefix[img]) * kScanChunk + (blockIdx.x % kSortParts) * kSortRays;
    for (int q = threadIdx.x & ~31; q < kSortRays && p0 + q < I.N; q += kThreads) {
        long long b;
        const int n = ray_samples(I.off, p0 + q, I.N, I.cap, lane, true, infos + img / 3, b);
        if (__any_sync(0xffffffffu, n != 0 && n != 2) && lane == 0)
            T.rest[atomicAdd(T.big_n + 2, 1)] = ((long long)img << 32) | ((p0 + q) >> 5);
        if (n == 2) finish_pair(b, I.r, I.nrm, I.pairs8);
    }
}

__global__ void __launch_bounds__(kThreads) batch_rest(const ldni_batch_item_t *items, Tables T, ldni_info_t *infos) {
    __shared__ SortStage stage[kThreads / 32];
    const int lane = threadIdx.x & 31, warps = gridDim.x * (kThreads / 32);
    for (int q = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); q < T.big_n[2]; q += warps) {
        const long long code = T.rest[q];
        const int img = (int)(code >> 32);
        const ItemImage I = item_image(items, T, img);
        long long b;
        const int n = ray_samples(I.off, (code & 0xffffffffll) << 5, I.N, I.cap, lane, false, infos + img / 3, b);
        finish_rest(b, n == 2 ? 0 : n, I.r, I.nrm, stage[threadIdx.x >> 5], lane);
    }
}

struct BatchWs {
    Tables T;
    int *counts;
    size_t counts_bytes;  // counts and big_n are cleared by one memset
    unsigned long long *words;
    size_t words_bytes;
};

BatchWs carve_batch(Carver &c, const ldni_batch_item_t *items_host, int count) {
    BatchWs w{};
    long long cints = 0, chunks = 0, tris = 0;
    for (int m = 0; m < count; ++m) {
        const long long N = (long long)items_host[m].grid.res * items_host[m].grid.res;
        cints += 3 * ((N + 63) / 64 * 64);
        chunks += 3 * ((N + kScanChunk - 1) / kScanChunk);
        tris += items_host[m].nt;
    }
    w.counts = c.take<int>((size_t)cints + 64);
    w.T.big_n = w.counts ? w.counts + cints : nullptr;
    w.counts_bytes = sizeof(int) * ((size_t)cints + 64);
    w.words = c.take<unsigned long long>((size_t)chunks + 1);
    w.words_bytes = sizeof(unsigned long long) * ((size_t)chunks + 1);
    w.T.tri_prefix = c.take<long long>((size_t)count + 1);
    w.T.tile_prefix = c.take<long long>((size_t)count + 1);
    w.T.chunk_prefix = c.take<long long>(3 * (size_t)count + 1);
    w.T.count_base = c.take<long long>(3 * (size_t)count);
    w.T.scale = c.take<float>((size_t)count);
    w.T.nrm = c.take<float4>((size_t)(tris > 0 ? tris : 1));
    w.T.rest = c.take<long long>((size_t)chunks * (kScanChunk / 32));
    w.T.qcap = 3 * tris > 0 ? 3 * tris : 1;
    w.T.big = c.take<long long>((size_t)w.T.qcap);
    return w;
}

bool items_ok(const ldni_batch_item_t *items, int count) {
    for (int m = 0; m < count; ++m) {
        const ldni_batch_item_t &it = items[m];
        if (!grid_valid(&it.grid) || it.nv <= 0 || it.nt < 0 || (it.nt > 0 && (!it.verts || !it.tris)) ||
            it.nt > (1ll << 31) - 1 || it.nv > INT_MAX)
            return false;
        for (int a = 0; a < 3; ++a) {
            const ldni_layers_t &L = it.out[a];
            if (!L.offsets || L.capacity < 0 || !samples_ok(L))
                return false;
        }
    }
    return count < (1 << 29);
}

}  // namespace
}  // namespace ldni

using namespace ldni;

extern "C" int ldni_sample_batch_workspace_size(const ldni_batch_item_t *items_host, int32_t count, size_t *bytes) {
    if (!items_host || count < 1 || !bytes || !items_ok(items_host, count)) return LDNI_EINVAL;
    Carver c(nullptr, 0);
    carve_batch(c, items_host, count);
    *bytes = align_up(c.off);
    return LDNI_OK;
}

extern "C" int ldni_sample_batch(const ldni_batch_item_t *items_dev, const ldni_batch_item_t *items_host,
                                 int32_t count, ldni_info_t *infos, void *ws, size_t ws_bytes, void *stream) {
    if (!items_dev || !items_host || count < 1 || !infos || !ws || !items_ok(items_host, count)) return LDNI_EINVAL;
    Carver c(ws, ws_bytes);
    BatchWs w = carve_batch(c, items_host, count);
    if (!c.fits()) return LDNI_EWORKSPACE;
    long long tris = 0, tiles = 0, chunks = 0;
    for (int m = 0; m < count; ++m) {
        const long long N = (long long)items_host[m].grid.res * items_host[m].grid.res;
        tris += items_host[m].nt;
        tiles += (items_host[m].nt + kThreads - 1) / kThreads;
        chunks += 3 * ((N + kScanChunk - 1) / kScanChunk);
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (int rc_ = cuda_check(cudaMemsetAsync(w.counts, 0, w.counts_bytes, s))) return rc_;
    if (int rc_ = cuda_check(cudaMemsetAsync(w.words, 0, w.words_bytes, s))) return rc_;
    if (int rc_ = cuda_check(cudaMemsetAsync(infos, 0, sizeof(ldni_info_t) * (size_t)count, s))) return rc_;
    LDNI_LAUNCH(K_BATCH, s, setup_kernel<<<1, kThreads, 0, s>>>(items_dev, count, w.T));
    if (tris > 0) {
        LDNI_LAUNCH(K_BATCH, s, batch_tri_pass<false><<<(unsigned)tiles, kThreads, 0, s>>>(items_dev, count, w.T,
                                                                                             w.counts, infos));
        LDNI_LAUNCH(K_BATCH, s,
                    batch_big<false><<<5 * num_sms(), kThreads, 0, s>>>(items_dev, w.T, w.counts, infos));
    }
    LDNI_LAUNCH(K_BATCH, s,
                batch_scan<<<(unsigned)chunks, kThreads, 0, s>>>(items_dev, count, w.T, w.counts, w.words, infos,
                                                                  wait_limit()));
    if (tris > 0) {
        LDNI_LAUNCH(K_BATCH, s, batch_tri_pass<true><<<(unsigned)tiles, kThreads, 0, s>>>(items_dev, count, w.T,
                                                                                            w.counts, infos));
        LDNI_LAUNCH(K_BATCH, s,
                    batch_big<true><<<5 * num_sms(), kThreads, 0, s>>>(items_dev, w.T, w.counts, infos));
    }
    LDNI_LAUNCH(K_BATCH, s,
                batch_sort<<<(unsigned)(chunks * kSortParts), kThreads, 0, s>>>(items_dev, count, w.T, infos));
    LDNI_LAUNCH(K_BATCH, s, batch_rest<<<2 * num_sms(), kThreads, 0, s>>>(items_dev, w.T, infos));
    return cuda_status();
}
