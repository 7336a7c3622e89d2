// A chain of unions on one grid: out = P0 u P1 u ... u P(n-1), evaluated left
// to right with the Boolean of Section 4.1 at every step and the small-
// interval removal of Section 4.1.1 after every step - the repeated
// operation of offsetting and sweeps (Section 4.2: one union per sphere) and
// of any sequence of Booleans on one grid (Section 4.1.1 keeps such chains
// exact because every operand shares the grid).
//
// Every step treats each ray on its own, so the whole chain is a fold along
// each ray: a thread carries its ray's accumulated result from step to step
// and never waits for another ray or another step.  Two passes over the
// rays (count, then write, with the CSR scan between them) replace the n - 1
// Booleans of the step-by-step evaluation, whose intermediate images would
// each be written to and read back from memory.  Without small-interval
// removal the fold is a union of intervals (unite_pass); with it, or where that
// does not fit, it merges sample by sample (fold_pass).  The count pass leaves
// the sources of every interval it finds in a pool of records, from which the
// write pass copies them; a ray whose records find no room in the pool is
// folded again when it is written.
//
// The result equals the step-by-step chain bit for bit: each step is the
// same merge (merge.cuh) with the accumulated solid as the first operand, so
// at a shared depth the accumulated sample is kept, and a sample that first
// enters through part k >= 1 carries the second-operand mark (tri_id bit 31)
// from then on.
#include <algorithm>
#include <climits>

#include "ldni_host.h"
#include "merge.cuh"

namespace ldni {
namespace {

constexpr int kThreads = 128;
// Samples a ray's accumulated result may hold at any step.  A ray that needs
// more is left empty and reported (LDNI_ST_EVENTS).
constexpr int kChainMaxLayers = 64;

struct Entry {
    float d;
    int part;  // source part
    int idx;   // source sample in that part
};

// Sample range of ray p in part P.
__device__ __forceinline__ void part_range(const ldni_layers_t &P, long long p, int &b, int &e) {
    b = (int)min((long long)P.offsets[p], (long long)P.capacity);
    e = (int)min((long long)P.offsets[p + 1], (long long)P.capacity);
}

// Parts k0 .. k0 + 63 that have samples on ray p, as bits.  Most parts have
// none on most rays, and one part's offsets say nothing about where the next
// part's are, so the offsets of kAhead parts are loaded together: loaded part
// by part between the merges, 64 round trips to memory made up the fold.  odd
// counts the parts with an odd number of samples (Definition 4).
// (kN a time, down to one at the end of the parts: short chains would load
// their last part's offsets up to seven times over.)
template <int kN>
__device__ __forceinline__ unsigned long long present_step(const ldni_layers_t *__restrict__ parts, int &q0, long long p,
                                                           int &odd) {
    int b[kN], e[kN];
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        const int *off = parts[q0 + q].offsets;
        b[q] = __ldg(off + p);
        e[q] = __ldg(off + p + 1);
    }
    unsigned mask = 0;
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        odd += (e[q] - b[q]) & 1;
        mask |= e[q] != b[q] ? 1u << q : 0u;
    }
    q0 += kN;
    return (unsigned long long)mask << (q0 - kN);
}
__device__ __forceinline__ unsigned long long parts_present(const ldni_layers_t *__restrict__ parts, int count, int k0,
                                                            long long p, int &odd) {
    unsigned long long mask = 0;
    const int n = min(count - k0, 64);
    int q0 = 0;
    while (n - q0 >= 8) mask |= present_step<8>(parts + k0, q0, p, odd);
    if (n - q0 >= 4) mask |= present_step<4>(parts + k0, q0, p, odd);
    if (n - q0 >= 2) mask |= present_step<2>(parts + k0, q0, p, odd);
    if (n - q0 >= 1) mask |= present_step<1>(parts + k0, q0, p, odd);
    return mask;
}

// The fold of ray p: the accumulated samples in acc[cur] (returns their
// number), or -1 when a step needed more than kChainMaxLayers.  have(k0): the
// parts k0 .. k0 + 63 that may have samples on the ray.
template <class Have>
__device__ __forceinline__ int fold_ray(const ldni_layers_t *__restrict__ parts, int count, long long p, float eps,
                                        Entry (&acc)[2][kChainMaxLayers], int &cur, Have have) {
    cur = 0;
    int na = 0;
    for (int k0 = 0; k0 < count; k0 += 64) {
        unsigned long long todo = have(k0);
        if (k0 == 0) {
            if (todo & 1ull) {
                int b, e;
                part_range(parts[0], p, b, e);
                if (e - b > kChainMaxLayers) return -1;
                for (int x = b; x < e; ++x) acc[0][na++] = Entry{parts[0].depth[x], 0, x};
                // the first union merges touching intervals and removes thin ones even where it adds nothing
                if (count > 1) todo |= 2ull;
            }
            todo &= ~1ull;
        }
        // Uniting a merged result (strictly ascending, no interval that is empty or thinner than eps) with
        // nothing changes nothing: parts without samples are passed over.
        for (; todo; todo &= todo - 1ull) {
            const int k = k0 + __ffsll((long long)todo) - 1;
            const ldni_layers_t &P = parts[k];
            int b, e;
            part_range(P, p, b, e);
            if (e <= b && k > 1) continue;
            const Entry *A = acc[cur];
            Entry *O = acc[cur ^ 1];
            bool over = false;
            struct AccDepth {
                const Entry *a;
                __device__ __forceinline__ float operator[](int i) const { return a[i].d; }
            };
            const float *dB = P.depth + b;
            const int m = merge_core<int>(AccDepth{A}, 0, na, dB, 0, max(e - b, 0), LDNI_OP_UNION, eps,
                                          [&](bool pb, int pi, bool cb, int ci, int mm) {
                                              if (mm + 2 > kChainMaxLayers) {
                                                  over = true;
                                                  return;
                                              }
                                              O[mm] = pb ? Entry{dB[pi], k, b + pi} : A[pi];
                                              O[mm + 1] = cb ? Entry{dB[ci], k, b + ci} : A[ci];
                                          });
            if (over) return -1;
            na = m;
            cur ^= 1;
        }
    }
    return na;
}

// Without small-interval removal the chain's result on a ray is the union of
// all its parts' intervals, and where it changes state the chain keeps the
// sample of the first part whose own state changes there (every Boolean keeps
// the accumulated solid's sample at a shared depth).  So the union is kept as
// disjoint intervals, each new interval taking in the ones that it touches,
// and an end that it shares with one of them stays the earlier part's.
struct Span {
    float lo, hi;   // empty: lo > hi
    int2 slo, shi;  // (part, sample) of the ends
    __device__ __forceinline__ bool empty() const { return lo > hi; }
    // takes in s, if they touch (s: from earlier parts)
    __device__ __forceinline__ void take(Span &s) {
        if (!(s.lo <= hi && s.hi >= lo)) return;
        if (s.lo <= lo) {
            lo = s.lo;
            slo = s.slo;
        }
        if (s.hi >= hi) {
            hi = s.hi;
            shi = s.shi;
        }
        s.lo = INFINITY;
        s.hi = -INFINITY;
    }
};

// The intervals of a ray's parts in order, to add(span), which may say no; the
// samples of four parts are loaded together.  False where it said no, or a part
// has an odd count or repeated or unordered depths.
template <class Have, class Add>
__device__ __forceinline__ bool each_span(const ldni_layers_t *__restrict__ parts, int count, long long p, Have have,
                                          Add add) {
    for (int k0 = 0; k0 < count; k0 += 64) {
        unsigned long long todo = have(k0);
        while (todo) {
            constexpr int kTake = 4;
            int k[kTake], b[kTake], e[kTake];
            float d0[kTake], d1[kTake];
#pragma unroll
            for (int q = 0; q < kTake; ++q) {
                k[q] = todo ? k0 + __ffsll((long long)todo) - 1 : -1;
                todo &= todo - 1ull;  // (0 stays 0)
                b[q] = e[q] = 0;
                if (k[q] >= 0) part_range(parts[k[q]], p, b[q], e[q]);
            }
#pragma unroll
            for (int q = 0; q < kTake; ++q) {
                const bool some = e[q] - b[q] >= 2;
                d0[q] = some ? parts[k[q]].depth[b[q]] : 0.0f;
                d1[q] = some ? parts[k[q]].depth[b[q] + 1] : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kTake; ++q) {
                if (e[q] <= b[q]) continue;
                if ((e[q] - b[q]) & 1) return false;
                float l = d0[q], h = d1[q];
                for (int x = b[q];;) {
                    if (!(l < h) || !add(Span{l, h, {k[q], x}, {k[q], x + 1}})) return false;
                    x += 2;
                    if (x >= e[q]) break;
                    l = parts[k[q]].depth[x];
                    if (!(h < l)) return false;
                    h = parts[k[q]].depth[x + 1];
                }
            }
        }
    }
    return true;
}

// Adds a span to S (empty ones among them); false when there is no room.
template <int kN>
__device__ __forceinline__ bool add_span(Span (&S)[kN], Span s) {
    bool put = false;
#pragma unroll
    for (int i = 0; i < kN; ++i) s.take(S[i]);
#pragma unroll
    for (int i = 0; i < kN; ++i)
        if (!put && S[i].empty()) {
            S[i] = s;
            put = true;
        }
    return put;
}

// What the count pass leaves: every ray's count; a record per interval of its
// result; the rays left to fold_pass, from the front of one list, and those
// whose records found no room, from its back (a ray of the front that finds
// none stays in the list, the others of the front are marked -1).  Rays are
// numbered image N + ray.
struct Record {
    int ray, k;  // the interval's ray and its number there (-1: unused)
};
struct Rays {
    int *count[3];
    int4 *src;              // per record: (part, sample) of its ends; second part -1: a sample alone
    Record *rec;
    int *list;
    unsigned long long *n;  // front of the list, back of the list, records
    long long records, rays;
};

__device__ __forceinline__ void report_odd(int odd, ldni_info_t *info) {
    if (odd) {
        atomicAdd(&info->odd_rays, (unsigned)odd);
        set_status(info, LDNI_ST_ODD);
    }
}

// First record of each lane's `want` (whole warp), -1 where the pool has no
// room for all of them.
__device__ __forceinline__ long long claim_records(const Rays &rays, int want, int lane) {
    int upto = want;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += x;
    }
    const int all = __shfl_sync(0xffffffffu, upto, 31);
    if (all == 0) return 0;
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(rays.n + 2, (unsigned long long)all);
    const long long first = (long long)__shfl_sync(0xffffffffu, at, 0) + upto - want;
    if (first + want <= rays.records) return first;
    for (long long i = first; i < rays.records; ++i) rays.rec[i].k = -1;  // (at most one lane's)
    return -1;
}

__device__ __forceinline__ void put_record(const Rays &rays, long long at, long long ray, int k, int2 lo, int2 hi) {
    rays.src[at] = make_int4(lo.x, lo.y, hi.x, hi.y);
    rays.rec[at] = Record{(int)ray, k};
}

// Pass 1, when no thin intervals are removed: the rays whose results never have
// more than kSpans disjoint intervals; the others are listed.  Bound by the
// reads of the parts' offsets (201 MB for 64 parts at 512^2, three images) and
// the chain of loads of the rays that meet a part, a fifth of them: 95 us.
constexpr int kSpans = 4;

__global__ void __launch_bounds__(kThreads, 6) unite_pass(long long N, const ldni_layers_t *__restrict__ parts_all,
                                                          int count, Rays rays, ldni_info_t *info) {
    const int img = blockIdx.y, lane = threadIdx.x & 31;
    const ldni_layers_t *parts = parts_all + (size_t)img * count;
    // (whole warps: the rays' records are claimed together)
    for (long long base = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); base < N;
         base += (long long)gridDim.x * blockDim.x) {
        const long long p = base + lane;
        Span S[kSpans];
#pragma unroll
        for (int i = 0; i < kSpans; ++i) S[i] = Span{INFINITY, -INFINITY, {0, 0}, {0, 0}};
        bool left = false;
        if (p < N) {
            int odd = 0;
            const unsigned long long present = parts_present(parts, count, 0, p, odd);
            for (int k0 = 64; k0 < count; k0 += 64) parts_present(parts, count, k0, p, odd);
            report_odd(odd, info);
            if (present != 0 || count > 64)
                left = !each_span(parts, count, p,
                                  [&](int k0) { return k0 == 0 ? present : parts_present(parts, count, k0, p, odd); },
                                  [&](const Span &s) { return add_span<kSpans>(S, s); });
        }
        int m = 0;
        if (!left) {
            // ascending, the empty ones last
#pragma unroll
            for (int i = 0; i < kSpans - 1; ++i)
#pragma unroll
                for (int j = 0; j < kSpans - 1 - i; ++j)
                    if (S[j + 1].lo < S[j].lo) {
                        const Span t = S[j];
                        S[j] = S[j + 1];
                        S[j + 1] = t;
                    }
#pragma unroll
            for (int i = 0; i < kSpans; ++i) m += S[i].empty() ? 0 : 1;
        }
        const long long ray = N * img + p;
        const long long at = claim_records(rays, m, lane);
        if (at >= 0) {
#pragma unroll
            for (int i = 0; i < kSpans; ++i)
                if (i < m) put_record(rays, at + i, ray, i, S[i].slo, S[i].shi);
        } else if (m > 0) {
            rays.list[rays.rays - 1 - (long long)atomicAdd(rays.n + 1, 1ull)] = (int)ray;
        }
        if (left) rays.list[atomicAdd(rays.n, 1ull)] = (int)ray;
        if (p < N) rays.count[img][p] = 2 * m;
    }
}

// The samples src[0, n) (n <= kMax) to o from slot at on: all loads before the
// first store, which could otherwise be to the same memory.
template <int kMax>
__device__ __forceinline__ void put_samples(const ldni_layers_t *__restrict__ parts, const ldni_layers_t &o,
                                            const int2 (&src)[kMax], int n, long long at, ldni_info_t *info) {
    if (at + n > o.capacity) {
        set_status(info, LDNI_ST_CAPACITY);
        n = (int)max(0ll, (long long)o.capacity - at);
    }
    const bool packed = o.nrm8 != nullptr;
    float d[kMax], x[kMax], y[kMax], z[kMax];
    int t[kMax];
#pragma unroll
    for (int i = 0; i < kMax; ++i) {
        if (i >= n) continue;
        const ldni_layers_t &P = parts[src[i].x];
        d[i] = P.depth[src[i].y];
        x[i] = packed ? __uint_as_float(P.nrm8[src[i].y]) : P.nx[src[i].y];
        y[i] = packed ? 0.0f : P.ny[src[i].y];
        z[i] = packed ? 0.0f : P.nz[src[i].y];
        t[i] = P.tri_id[src[i].y];
        if (src[i].x != 0) t[i] |= (int)0x80000000u;
    }
#pragma unroll
    for (int i = 0; i < kMax; ++i) {
        if (i >= n) continue;
        o.depth[at + i] = d[i];
        if (packed) {
            o.nrm8[at + i] = __float_as_uint(x[i]);
        } else {
            o.nx[at + i] = x[i];
            o.ny[at + i] = y[i];
            o.nz[at + i] = z[i];
        }
        o.tri_id[at + i] = t[i];
    }
}

// The rays that unite_pass listed, or all of them (all: with thin intervals
// removed after every step, or one part alone): their counts and records.  On as
// many blocks as stay resident, whatever the list's length: three stacks of nine
// slabs at 512^2, where most rays are listed, 90 us, 212 on a block per SM.
__global__ void __launch_bounds__(kThreads) fold_pass(long long N, const ldni_layers_t *__restrict__ parts_all,
                                                      int count, int all, float eps, Rays rays, ldni_info_t *info) {
    Entry acc[2][kChainMaxLayers];
    const int lane = threadIdx.x & 31;
    const long long total = all ? rays.rays : (long long)rays.n[0];
    for (long long base = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); base < total;
         base += (long long)gridDim.x * blockDim.x) {
        const long long r = base + lane;
        const bool mine = r < total;
        const long long ray = !mine ? 0 : (all ? r : rays.list[r]);
        const int img = (int)(ray / N);
        const long long p = ray - img * N;
        int cur = 0, n = 0;
        if (mine) {
            const ldni_layers_t *parts = parts_all + (size_t)img * count;
            int odd = 0;
            const unsigned long long present = parts_present(parts, count, 0, p, odd);
            if (all) {
                for (int k0 = 64; k0 < count; k0 += 64) parts_present(parts, count, k0, p, odd);
                report_odd(odd, info);
            }
            n = fold_ray(parts, count, p, eps, acc, cur,
                         [&](int k0) { return k0 == 0 ? present : parts_present(parts, count, k0, p, odd); });
            if (n < 0) {
                set_status(info, LDNI_ST_EVENTS);
                n = 0;
            }
        }
        const int m = (n + 1) / 2;
        const long long at = claim_records(rays, m, lane);
        if (!mine) continue;
        if (at >= 0 || m == 0) {
            for (int i = 0; i < m; ++i) {
                const Entry lo = acc[cur][2 * i], hi = 2 * i + 1 < n ? acc[cur][2 * i + 1] : Entry{0.0f, -1, 0};
                put_record(rays, at + i, ray, i, make_int2(lo.part, lo.idx), make_int2(hi.part, hi.idx));
            }
            if (!all) rays.list[r] = -1;
        } else if (all) {
            rays.list[rays.rays - 1 - (long long)atomicAdd(rays.n + 1, 1ull)] = (int)ray;
        }
        rays.count[img][p] = n;
    }
}

// A ray without records: folded once more, and written.
__device__ __noinline__ void write_folded(const ldni_layers_t *__restrict__ parts, int count, long long p, float eps,
                                          const ldni_layers_t &o, ldni_info_t *info) {
    Entry acc[2][kChainMaxLayers];
    int cur, odd;
    const int n = fold_ray(parts, count, p, eps, acc, cur,
                           [&](int k0) { return parts_present(parts, count, k0, p, odd); });
    for (int x = 0; x < n; ++x) {
        const int2 one[1] = {{acc[cur][x].part, acc[cur][x].idx}};
        put_samples(parts, o, one, 1, (long long)o.offsets[p] + x, info);
    }
}

// The result's samples: a thread per record, then the rays without any.  A
// thread per ray with its kept sources spread a fifth of the threads' work over
// all of them: 41 us for 64 parts at 512^2, 22 now; folding deep rays again to
// write them took 330 us for the stacks of slabs, 68 now.
__global__ void __launch_bounds__(kThreads) chain_write(long long N, const ldni_layers_t *__restrict__ parts_all,
                                                        int count, int all, float eps, Rays rays, ldni_layers_t o0,
                                                        ldni_layers_t o1, ldni_layers_t o2, ldni_info_t *info) {
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    const long long claimed = (long long)rays.n[2], n = min(claimed, rays.records);
    for (long long i = first; i < n; i += step) {
        const Record R = rays.rec[i];
        const int4 v = rays.src[i];
        if (R.k < 0) continue;
        const int img = (unsigned)R.ray / (unsigned)N;
        const ldni_layers_t &o = img == 0 ? o0 : (img == 1 ? o1 : o2);
        const int2 from[2] = {{v.x, v.y}, {v.z, v.w}};
        put_samples(parts_all + (size_t)img * count, o, from, v.z < 0 ? 1 : 2,
                    (long long)o.offsets[R.ray - img * N] + 2 * R.k, info);
    }
    if (claimed <= rays.records) return;  // every ray has its records
    const long long front = all ? 0 : (long long)rays.n[0], back = (long long)rays.n[1];
    for (long long r = first; r < front + back; r += step) {
        const int ray = rays.list[r < front ? r : rays.rays - 1 - (r - front)];
        if (ray < 0) continue;
        const int img = (unsigned)ray / (unsigned)N;
        write_folded(parts_all + (size_t)img * count, count, ray - img * N, eps, img == 0 ? o0 : (img == 1 ? o1 : o2), info);
    }
}

struct ChainWs {
    Rays rays;
    long long *partials;
};

// Records: up to 32 a ray for small images, one for every three rays of large
// ones (a swept solid's rays are mostly empty): 16 bytes a ray in all, 0.8 GB for
// three images of 4096^2, where sources kept for every ray took 84.
ChainWs carve_chain_ws(Carver &c, int res, int nimg) {
    ChainWs w{};
    const long long N = (long long)res * res, rays = N * nimg;
    for (int j = 0; j < nimg; ++j) w.rays.count[j] = c.take<int>((size_t)N);
    w.rays.rays = rays;
    w.rays.records = std::min(rays * (kChainMaxLayers / 2), std::max(2ll << 20, rays / 3));
    w.rays.src = c.take<int4>((size_t)w.rays.records);
    w.rays.rec = c.take<Record>((size_t)w.rays.records);
    w.rays.list = c.take<int>((size_t)rays);
    w.rays.n = c.take<unsigned long long>(3);
    w.partials = c.take<long long>(csr_scan_partials(N) * nimg);
    return w;
}

int grid_for(long long N) {
    long long b = (N + kThreads - 1) / kThreads;
    const long long lim = (long long)num_sms() * 16;
    return (int)(b < 1 ? 1 : (b > lim ? lim : b));
}

}  // namespace
}  // namespace ldni

using namespace ldni;

extern "C" int ldni_union_chain_workspace_size(int32_t res, int32_t nimg, size_t *bytes) {
    if (!bytes || res < 1 || res > 8192 || nimg < 1 || nimg > 3) return LDNI_EINVAL;
    Carver c(nullptr, 0);
    carve_chain_ws(c, res, nimg);
    *bytes = align_up(c.off);
    return LDNI_OK;
}

extern "C" int ldni_union_chain(const ldni_layers_t *parts_dev, const ldni_layers_t *parts_host, int32_t count,
                                int32_t nimg, const ldni_grid_t *grid, float eps, ldni_layers_t *out,
                                ldni_info_t *info, void *ws, size_t ws_bytes, void *stream) {
    if (!parts_dev || !parts_host || count < 1 || nimg < 1 || nimg > 3 || !grid_valid(grid) || !out || !info ||
        !ws || !(eps >= 0.0f))
        return LDNI_EINVAL;
    for (int j = 0; j < nimg; ++j) {
        const ldni_layers_t &o = out[j];
        if (!o.offsets || o.capacity < 0 || !samples_ok(o)) return LDNI_EINVAL;
        const ldni_layers_t *fmt[2] = {&o, nullptr};
        bool packed = false, pk = false;
        if (!same_format(fmt, 1, &packed)) return LDNI_EINVAL;
        for (int k = 0; k < count; ++k) {
            const ldni_layers_t &P = parts_host[(size_t)j * count + k];
            fmt[1] = &P;
            if (!P.offsets || P.capacity < 0 || !samples_ok(P) || !same_format(fmt, 2, &pk)) return LDNI_EINVAL;
        }
    }
    Carver c(ws, ws_bytes);
    ChainWs w = carve_chain_ws(c, grid->res, nimg);
    if (!c.fits()) return LDNI_EWORKSPACE;
    const long long N = (long long)grid->res * grid->res;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    ldni_layers_t o[3] = {out[0], nimg > 1 ? out[1] : out[0], nimg > 2 ? out[2] : out[0]};
    const dim3 g((unsigned)grid_for(N), (unsigned)nimg);
    const unsigned blocks = (unsigned)grid_for(N * nimg);  // the lists' lengths are known on the device
    const int all = eps == 0.0f && count > 1 ? 0 : 1;
    if (int rc_ = cuda_check(cudaMemsetAsync(w.rays.n, 0, 3 * sizeof(unsigned long long), s))) return rc_;
    if (!all) LDNI_LAUNCH(K_CHAIN, s, unite_pass<<<g, kThreads, 0, s>>>(N, parts_dev, count, w.rays, info));
    LDNI_LAUNCH(K_CHAIN, s, fold_pass<<<blocks, kThreads, 0, s>>>(N, parts_dev, count, all, eps, w.rays, info));
    int rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    const int *cnt[3] = {w.rays.count[0], w.rays.count[1], w.rays.count[2]};
    int *off[3] = {out[0].offsets, nimg > 1 ? out[1].offsets : nullptr, nimg > 2 ? out[2].offsets : nullptr};
    rc = csr_scan(cnt, off, nimg, N, w.partials, info, 0, s);
    if (rc != LDNI_OK) return rc;
    LDNI_LAUNCH(K_CHAIN, s,
                chain_write<<<blocks, kThreads, 0, s>>>(N, parts_dev, count, all, eps, w.rays, o[0], o[1], o[2], info));
    return cuda_status();
}
