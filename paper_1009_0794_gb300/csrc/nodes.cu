// Grid-node classification from the three LDNIs (Section 5.1, Step 1): the
// rays of the x-, y- and z-LDNI meet at the res^3 nodes of the grid
// (Definition 3); a node is inside the solid when it lies in the solid
// volume of at least two of the three images, which settles the images'
// disagreements near the surface.
//
// Node (i, j, k) sits at (c_x(i), c_y(j), c_z(k)) with
// c_a(t) = fl32(o_a + fl32((t + 1/2) * h)), h = fl32(W / res): the pixel
// centres of the images.  Image a puts the node inside when an odd number of
// the samples of its ray through the node lie strictly below c_a (the
// odd-to-even ranges are inside, Section 2 after Proposition 1).
//
// A ray kernel turns each image into bit words along its rays, and a vote
// kernel takes 32 x 32 x 32 node cubes, turns the y and z words so that their
// bits run along x too, and writes the majority in the x-fastest output
// layout.  Nearly every cube lies wholly inside or outside, so the words of 32
// neighbouring rays are nearly always all ones or all zeros each: such a group
// is stored as one mask of 32 bits, which is already the turned word of all 32
// rows, and only a group that a surface crosses is stored word by word and
// turned bit by bit.  For 1024^3 nodes that leaves 25 MB of summaries where
// three whole bit volumes took 402 MB written and read again.
#include "ldni_host.h"

namespace ldni {
namespace {


__device__ __forceinline__ float node_c(int t, float o, float h) {
    return __fadd_rn(o, __fmul_rn((float)t + 0.5f, h));
}

// First node t in [0, res] with c(t) > d (c increases with t): a float
// estimate (inv_h: about 1 / h), then corrected with the exact node positions.
__device__ __forceinline__ int first_above(float d, int res, float o, float h, float inv_h) {
    const float est = (d - o) * inv_h - 0.5f;
    int t = !(est > 0.0f) ? 0 : (est >= (float)res ? res : (int)est);
    while (t > 0 && node_c(t - 1, o, h) > d) --t;
    while (t < res && !(node_c(t, o, h) > d)) ++t;
    return t;
}

// Node t of a ray is inside iff an odd number of the ray's depths lie below
// c(t), i.e. iff an odd number of the boundaries b_m = first_above(d_m) are
// <= t.  So the ray's bits are the XOR of one step per sample: the bits
// t >= b_m.  step_word gives the bits of word w (nodes 32 w .. 32 w + 31) of
// one step; bits of nodes t >= res are cleared by live_bits.
__device__ __forceinline__ unsigned step_word(int b, int w) {
    const int t0 = 32 * w;
    if (b <= t0) return 0xffffffffu;
    if (b >= t0 + 32) return 0u;
    return 0xffffffffu << (b - t0);
}

__device__ __forceinline__ void ray_range(const int *__restrict__ off, long long cap, long long p, long long &b,
                                          long long &e, ldni_info_t *info, bool report) {
    b = off[p];
    e = off[p + 1];
    if (((e - b) & 1) && report) {
        atomicAdd(&info->odd_rays, 1u);
        set_status(info, LDNI_ST_ODD);
    }
    if (e > cap) {
        if (report) set_status(info, LDNI_ST_CAPACITY);
        e = cap;
        b = min(b, e);
    }
}

// Transpose of the 32 x 32 bit matrix held by a warp, one row per lane (bit c
// of lane r = element (r, c)): afterwards lane r holds column r.  Five
// stages swap the off-diagonal blocks of width 16, 8, 4, 2, 1 between lanes
// r and r ^ j.
__device__ __forceinline__ unsigned warp_transpose32(unsigned x, int lane) {
    const unsigned lows[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int j = 16 >> s;
        const unsigned low = lows[s];
        const unsigned other = __shfl_xor_sync(0xffffffffu, x, j);
        x = (lane & j) ? ((x & ~low) | ((other & ~low) >> j)) : ((x & low) | ((other & low) << j));
    }
    return x;
}

// Bit words of the three images.  A group is 32 neighbouring rays (a lane
// each) of one node row, nb groups per row:
//   x-image ray p = k res + j: row k, column j (bits: nodes i)
//   y-image ray p = i res + k: row k, column i (bits: nodes j)
//   z-image ray p = j res + i: row j, column i (bits: nodes k)
// and has W words per ray.  sum[group W + w] = (the rays whose word w is all
// ones; 0 when every ray's word w is all ones or all zeros, else 1).  In the
// second case word[(group W + w) 32 + l] holds the words of an output row: of
// the x-image's ray l, and, the other two turned, of the row l of word w's 32
// nodes over the group's 32 columns.
struct NodeImg {
    const int *off[3];
    const float *depth[3];
    long long cap[3];
    float o[3];
    uint2 *sum[3];
    unsigned *word[3];
};

// Bits of nodes at or beyond res are left as they come: their lanes or words
// are never stored, or meet zeros in the vote.
// Bound by issue (76 % of the slots, 31 M warp instructions for the union of the
// noisy sphere and the knot at 1024^2): 38 us for the three images; the three
// launches that wrote every word took 37 us each.
constexpr int kRowsPerBlock = 8;  // a warp each (the y-image's offsets of 8 rows share their sectors)

__global__ void __launch_bounds__(32 * kRowsPerBlock) node_rays(NodeImg I, int res, int nb, int W, float h,
                                                                float inv_h, ldni_info_t *info) {
    const int a = blockIdx.z;
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.y * kRowsPerBlock + (threadIdx.x >> 5), col = blockIdx.x * 32 + lane;
    if (row >= res) return;  // the same for the whole warp
    const float o = I.o[a];
    const float *__restrict__ depth = I.depth[a];
    long long b = 0, e = 0;
    if (col < res)
        ray_range(I.off[a], I.cap[a], a == 1 ? (long long)col * res + row : (long long)row * res + col, b, e, info, true);
    const int n = (int)(e - b);
    int m = 0;
    int bm = n > 0 ? first_above(depth[b], res, o, h, inv_h) : res;
    unsigned after = 0;  // all ones once an odd number of boundaries lie before the current word
    const long long group = (long long)row * nb + blockIdx.x;
    uint2 *sum = I.sum[a] + group * W;
    unsigned *word = I.word[a] + group * W * 32;
    for (int w0 = 0; w0 < W; w0 += 32) {  // lane l holds the summary of word w0 + l
        uint2 mine = make_uint2(0u, 0u);
        const int w1 = min(w0 + 32, W);
        int w = w0;
        while (w < w1) {
            // words before the next boundary of any ray repeat the rays' states
            const int next = max(w, __reduce_min_sync(0xffffffffu, m < n ? bm >> 5 : W));
            const unsigned state = __ballot_sync(0xffffffffu, after != 0u);
            if (w0 + lane >= w && w0 + lane < next) mine = make_uint2(state, 0u);
            w = next;
            if (w >= w1) break;
            unsigned x = after;
            while (m < n && bm < 32 * w + 32) {  // boundaries that reach into this word
                x ^= step_word(bm, w);
                after = ~after;
                if (++m < n) bm = first_above(depth[b + m], res, o, h, inv_h);
            }
            const unsigned ones = __ballot_sync(0xffffffffu, x == 0xffffffffu);
            const unsigned mixed = __any_sync(0xffffffffu, x != 0u && x != 0xffffffffu);
            if (w0 + lane == w) mine = make_uint2(ones, mixed ? 1u : 0u);
            if (mixed) word[32LL * w + lane] = a == 0 ? x : warp_transpose32(x, lane);
            ++w;
        }
        if (w0 + lane < w1) sum[w0 + lane] = mine;
    }
}

// Majority words of the rows (k, j), j in 32-block jb, k among kVoteK of
// 32-block kb, for up to 32 words along i; a warp takes a row k at a time.
// Lane = (row within a store, word ib): a store covers 32 words of the output,
// several rows where a row is shorter, so that it is contiguous.  For word ib
// of row (k, j):
//   x: bit j of the mask of x-group (k, jb) at word ib, or that ray's word;
//   y: the mask of y-group (k, ib) at word jb, the same for every j;
//   z: the mask of z-group (j, ib) at word kb, the same for every k (shared
//      memory).
// The cubes that a surface crosses (a fifth of the words of a row of cubes that
// meets the solid) follow one by one, lane = row j.  Bound by the latency of
// the summaries and of those cubes' words (40 % issue, the 134 MB of output
// alone would take 20 us at 1024^3): 61 us; 173 us when every cube's words
// were read from bit volumes and turned, 76 us with summaries but a lane per
// row j, eight words each.
constexpr int kVoteWarps = 8, kVoteRows = 2, kVoteK = kVoteWarps * kVoteRows;
static_assert(kVoteRows == 2, "a warp's two rows are picked by selects");

__global__ void __launch_bounds__(32 * kVoteWarps) node_vote(NodeImg I, int res, int nb, int W, int log_words,
                                                             unsigned *out) {
    __shared__ unsigned zs[32][33];  // [j in block][word]: mask
    __shared__ unsigned zmix[32];    // [j in block]: the words whose group is mixed
    const int jb = blockIdx.y, kb = blockIdx.z / (32 / kVoteK), kpart = blockIdx.z % (32 / kVoteK);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ibl = lane & ((1 << log_words) - 1), ib = blockIdx.x * 32 + ibl, js = lane >> log_words;
    const bool live = ib < W;
    uint2 sx[kVoteRows], sy[kVoteRows], sz[32 / kVoteWarps];
#pragma unroll
    for (int r = 0; r < 32 / kVoteWarps; ++r) {
        const int j = jb * 32 + w + r * kVoteWarps;
        sz[r] = live && j < res ? I.sum[2][((long long)j * nb + ib) * W + kb] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int r = 0; r < kVoteRows; ++r) {
        const int k = kb * 32 + kpart * kVoteK + w + r * kVoteWarps;
        const bool in = live && k < res;
        sx[r] = in ? I.sum[0][((long long)k * nb + jb) * W + ib] : make_uint2(0u, 0u);
        sy[r] = in ? I.sum[1][((long long)k * nb + ib) * W + jb] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int r = 0; r < 32 / kVoteWarps; ++r) {
        const int jj = w + r * kVoteWarps;
        if (js == 0) zs[jj][ibl] = sz[r].x;
        const unsigned m = __ballot_sync(0xffffffffu, js == 0 && sz[r].y != 0u);
        if (lane == 0) zmix[jj] = m;
    }
    __syncthreads();
    unsigned zall = 0;  // words of cubes with a mixed z-group
#pragma unroll
    for (int jj = 0; jj < 32; ++jj) zall |= zmix[jj];
    const int per = 32 >> log_words;  // rows j per store
    const int jn = min(32, res - jb * 32);
#pragma unroll 1
    for (int r = 0; r < kVoteRows; ++r) {
        const int kk = kpart * kVoteK + w + r * kVoteWarps, k = kb * 32 + kk;
        if (k >= res) break;  // the same for the whole warp
        const unsigned xm = r == 0 ? sx[0].x : sx[1].x, y = r == 0 ? sy[0].x : sy[1].x;
        const bool xmix = (r == 0 ? sx[0].y : sx[1].y) != 0u, ymix = (r == 0 ? sy[0].y : sy[1].y) != 0u;
        const bool plain = live && !xmix && !ymix && !((zall >> ibl) & 1u);  // masks only
        unsigned *o = out + ((long long)k * res + jb * 32) * W + blockIdx.x * 32;
        {
            unsigned *oj = o + (long long)js * W + ibl;
            const long long step = (long long)per * W;
#pragma unroll 8
            for (int j = js; j < jn; j += per, oj += step) {
                const unsigned x = 0u - ((xm >> j) & 1u), z = zs[j][ibl];
                if (plain) *oj = (x & y) | (z & (x | y));  // at least two of three
            }
        }
        // the cubes that a surface crosses: lane = row j
        for (unsigned todo = __ballot_sync(0xffffffffu, live && !plain && js == 0); todo; todo &= todo - 1u) {
            const int c = __ffs(todo) - 1, ic = blockIdx.x * 32 + c;
            const unsigned xc = __shfl_sync(0xffffffffu, xm, c), yc = __shfl_sync(0xffffffffu, y, c);
            const bool xw = __shfl_sync(0xffffffffu, xmix, c), yw = __shfl_sync(0xffffffffu, ymix, c);
            const unsigned zm = (zmix[lane] >> c) & 1u;
            if (lane >= jn) continue;
            const unsigned x = xw ? I.word[0][(((long long)k * nb + jb) * W + ic) * 32 + lane] : 0u - ((xc >> lane) & 1u);
            const unsigned yy = yw ? I.word[1][(((long long)k * nb + ic) * W + jb) * 32 + lane] : yc;
            const unsigned z = zm ? I.word[2][(((long long)(jb * 32 + lane) * nb + ic) * W + kb) * 32 + kk] : zs[lane][c];
            o[(long long)lane * W + c] = (x & yy) | (z & (x | yy));
        }
    }
}

bool image_ok(const ldni_layers_t &L) {
    return L.offsets && L.capacity >= 0 && (L.capacity == 0 || L.depth);
}

}  // namespace
}  // namespace ldni

using namespace ldni;

extern "C" int ldni_classify_nodes_workspace_size(int32_t res, size_t *bytes) {
    if (!bytes || res < 1 || res > 4096) return LDNI_EINVAL;
    const size_t W = ((size_t)res + 31) / 32, groups = (size_t)res * W;  // as many groups in a row as words in a ray
    *bytes = 3 * (align_up(sizeof(uint2) * groups * W) + align_up(sizeof(unsigned) * groups * W * 32)) + kAlign;
    return LDNI_OK;
}

extern "C" int ldni_classify_nodes(const ldni_layers_t *L, const ldni_grid_t *grid, uint32_t *inside,
                                   ldni_info_t *info, void *ws, size_t ws_bytes, void *stream) {
    if (!L || !grid_valid(grid) || !inside || !info || !ws) return LDNI_EINVAL;
    for (int a = 0; a < 3; ++a)
        if (!image_ok(L[a])) return LDNI_EINVAL;
    const int res = grid->res;
    size_t need = 0;
    int rc = ldni_classify_nodes_workspace_size(res, &need);
    if (rc != LDNI_OK) return rc;
    if (ws_bytes < need) return LDNI_EWORKSPACE;
    const int W = (res + 31) / 32, nb = W;
    const size_t groups = (size_t)res * nb;
    Carver c(ws, ws_bytes);
    NodeImg I{};
    for (int a = 0; a < 3; ++a) {
        I.off[a] = L[a].offsets;
        I.depth[a] = L[a].depth;
        I.cap[a] = L[a].capacity;
        I.o[a] = grid->origin[a];
        I.sum[a] = c.take<uint2>(groups * W);
        I.word[a] = c.take<unsigned>(groups * W * 32);
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float hh = (float)grid->width / (float)res;  // FP32 division, as the node positions are defined
    LDNI_LAUNCH(K_NODES, s,
                node_rays<<<dim3(nb, (res + kRowsPerBlock - 1) / kRowsPerBlock, 3), 32 * kRowsPerBlock, 0, s>>>(
                    I, res, nb, W, hh, 1.0f / hh, info));
    int log_words = 0;  // lanes per row: the words of a row, at most 32
    while (log_words < 5 && (1 << log_words) < W) ++log_words;
    LDNI_LAUNCH(K_NODES, s,
                node_vote<<<dim3((W + 31) / 32, nb, nb * (32 / kVoteK)), 32 * kVoteWarps, 0, s>>>(I, res, nb, W,
                                                                                                  log_words, inside));
    return cuda_status();
}
