// Contouring, Steps 2 and 3 (Section 5.1): cell edges typed and regularised
// (Rules 1 and 2), the outside corners of every cell flooded through its
// empty edges into clusters, and one vertex per cluster at the minimum of
// the quadratic error function of its Hermite data (dual contouring).
//
// Grid nodes and their signs come from Step 1 (nodes.cu): node t of axis a
// at c_a(t) = fl32(o_a + fl32((t + 1/2) h)).  The edge (t, t + 1) along a
// lies on the ray of image a through its two other node indices and holds
// the ray's samples with c_a(t) <= d < c_a(t + 1), the samples that change
// Step 1's parity count between its end nodes.
//
// Readings the kernels follow (the paper leaves them open):
//  - Rule 1 keeps the first and last samples of a complex edge; Rule 2 keeps,
//    of an intersect edge's samples whose normal's a-component points from
//    the inside end to the outside end, the one nearest the midpoint (the
//    earlier on a tie; all samples compete when none points that way);
//  - a cluster takes the kept sample of each intersect edge at one of its
//    corners and, of a complex edge between outside corners, the sample
//    nearer each corner (a single one goes to the nearer corner); complex
//    edges between inside corners join no cluster;
//  - clusters are numbered by their lowest corner (di + 2 dj + 4 dk); every
//    cluster of a cell that meets an intersect, none-intersect or complex
//    edge yields a vertex;
//  - x = m + (A^T A)^+ (A^T b - A^T A m), m the points' mean, eigenvalues of
//    A^T A below 0.01 of the largest dropped (singular values below 0.1), its
//    sums in FP64 and solved to 1e-8 of its displacement from m (qef_solve); a
//    cluster with no Hermite data sits at the mean of its corners with no points.
//
// Stages: active-cell marks (edges with samples, from the samples; edges
// whose end signs differ, word-parallel from the node bits), their
// compaction, the active cells' records in a dense scratch, and the compaction
// of the cells that yield a vertex.
#include "ldni_host.h"

namespace ldni {
namespace {

constexpr int kThreads = 256;

struct CImg {
    const int *off[3];
    const float *d[3];
    const float *nx[3], *ny[3], *nz[3];
    long long cap[3];
};

__device__ __forceinline__ float node_c(int t, float o, float h) {
    return __fadd_rn(o, __fmul_rn((float)t + 0.5f, h));
}

// first node t in [0, res] with c(t) > d
__device__ __forceinline__ int first_above(float d, int res, float o, float h) {
    const float est = (d - o) / h - 0.5f;
    int t = !(est > 0.0f) ? 0 : (est >= (float)res ? res : (int)est);
    while (t > 0 && node_c(t - 1, o, h) > d) --t;
    while (t < res && !(node_c(t, o, h) > d)) ++t;
    return t;
}

template <class T>
__device__ __forceinline__ T pick(T const (&arr)[3], int a) {
    return a == 0 ? arr[0] : (a == 1 ? arr[1] : arr[2]);
}

__device__ __forceinline__ void mark(unsigned *act, int n, int Wc, int i, int j, int k) {
    if (i < 0 || j < 0 || k < 0 || i >= n || j >= n || k >= n) return;
    atomicOr(act + ((long long)k * n + j) * Wc + (i >> 5), 1u << (i & 31));
}

// Cells around every edge that holds a sample: a thread per ray of image
// blockIdx.y.
__global__ void __launch_bounds__(kThreads) mark_samples(CImg I, int res, float o0, float o1, float o2, float h,
                                                         unsigned *act, int Wc) {
    const int a = blockIdx.y;
    const long long p = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (p >= (long long)res * res) return;
    const int n = res - 1;
    const int *off = pick(I.off, a);
    const float *D = pick(I.d, a);
    const long long cap = pick(I.cap, a);
    const float oa = a == 0 ? o0 : (a == 1 ? o1 : o2);
    const int iu = (int)(p % res), iv = (int)(p / res);
    const long long e = min((long long)off[p + 1], cap);
    for (long long s = off[p]; s < e; ++s) {
        const int t = first_above(D[s], res, oa, h) - 1;  // c(t) <= d < c(t + 1)
        if (t < 0 || t >= n) continue;
        for (int du = 0; du < 2; ++du)
            for (int dv = 0; dv < 2; ++dv) {
                const int cu = iu - du, cv = iv - dv;
                if (a == 0) mark(act, n, Wc, t, cu, cv);
                else if (a == 1) mark(act, n, Wc, cv, t, cu);
                else mark(act, n, Wc, cu, cv, t);
            }
    }
}

// bits i of node row (j, k) where nodes i and i + 1 differ along x
__device__ __forceinline__ unsigned xdiff(const unsigned *node, int W, int res, int j, int k, int w) {
    const unsigned *row = node + ((long long)k * res + j) * W;
    const unsigned lo = row[w], hi = w + 1 < W ? row[w + 1] : 0u;
    return lo ^ ((lo >> 1) | (hi << 31));
}

__device__ __forceinline__ unsigned row_word(const unsigned *node, int W, int res, int j, int k, int w) {
    return (w < W) ? node[((long long)k * res + j) * W + w] : 0u;
}

// cell bit i from node-column bits i and i + 1
__device__ __forceinline__ unsigned spread(unsigned lo, unsigned hi) { return lo | (lo >> 1) | (hi << 31); }

// Cells around every edge whose end nodes differ: a thread per word of a
// cell row (j, k).  The cell and node bit volumes share the word width.
__global__ void __launch_bounds__(kThreads) mark_signs(const unsigned *node, int res, int W, unsigned *act, int Wc) {
    const int n = res - 1;
    const long long q = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (q >= (long long)n * n * Wc) return;
    const int w = (int)(q % Wc);
    const int j = (int)((q / Wc) % n), k = (int)(q / ((long long)Wc * n));
    // x-edges of the four node rows around cell row (j, k)
    unsigned m = xdiff(node, W, res, j, k, w) | xdiff(node, W, res, j + 1, k, w) | xdiff(node, W, res, j, k + 1, w) |
                 xdiff(node, W, res, j + 1, k + 1, w);
    // y-edges (node rows (j, k') and (j + 1, k'), k' = k, k + 1) and z-edges
    // (rows (j', k) and (j', k + 1), j' = j, j + 1), at node columns i, i + 1
    unsigned ylo = 0, yhi = 0, zlo = 0, zhi = 0;
    for (int dk = 0; dk < 2; ++dk) {
        ylo |= row_word(node, W, res, j, k + dk, w) ^ row_word(node, W, res, j + 1, k + dk, w);
        yhi |= row_word(node, W, res, j, k + dk, w + 1) ^ row_word(node, W, res, j + 1, k + dk, w + 1);
    }
    for (int dj = 0; dj < 2; ++dj) {
        zlo |= row_word(node, W, res, j + dj, k, w) ^ row_word(node, W, res, j + dj, k + 1, w);
        zhi |= row_word(node, W, res, j + dj, k, w + 1) ^ row_word(node, W, res, j + dj, k + 1, w + 1);
    }
    m |= spread(ylo, yhi) | spread(zlo, zhi);
    const int valid = n - 32 * w;  // cells i < n
    if (valid < 32) m &= (1u << valid) - 1u;
    if (m) atomicOr(act + ((long long)k * n + j) * Wc + w, m);
}

__global__ void __launch_bounds__(kThreads) count_words(const unsigned *act, long long nw, int *cnt) {
    const long long q = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (q < nw) cnt[q] = __popc(act[q]);
}

__global__ void __launch_bounds__(kThreads) list_cells(const unsigned *act, long long nw, const int *woff, int n,
                                                       int Wc, long long *cells, long long max_active,
                                                       ldni_info_t *info) {
    const long long q = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (q >= nw) return;
    unsigned m = act[q];
    long long at = woff[q];
    const long long row = q / Wc;  // k * n + j
    const int w = (int)(q % Wc);
    while (m) {
        const int b = __ffs(m) - 1;
        m &= m - 1;
        if (at >= max_active) {
            set_status(info, LDNI_ST_CAPACITY);
            return;
        }
        cells[at++] = row * n + 32 * w + b;  // i + n (j + n k)
    }
}

// ---- one cell --------------------------------------------------------------------

struct Edge {
    int a, q0, q1;  // axis, lower and upper corner
    int du, dv;     // ray node indices within the cell, along u and v
};

// Edge e = 4 a + x + 2 y of a cell.
__device__ __forceinline__ Edge cell_edge(int e) {
    const int x = e & 1, y = (e >> 1) & 1;
    if (e < 4) return Edge{0, 2 * x + 4 * y, 1 + 2 * x + 4 * y, x, y};  // x-edges at (j + x, k + y)
    if (e < 8) return Edge{1, x + 4 * y, x + 2 + 4 * y, y, x};          // y-edges at (i + x, k + y): (u, v) = (z, x)
    return Edge{2, x + 2 * y, x + 2 * y + 4, x, y};                     // z-edges at (i + x, j + y)
}

struct Sym3 {  // A^T A, A^T b, sum of points, count
    double xx, xy, xz, yy, yz, zz, bx, by, bz, px, py, pz;
    int n;
};

__device__ __forceinline__ void add_point(Sym3 &Q, const double (&P)[3], const double (&N)[3]) {
    Q.xx += N[0] * N[0];
    Q.xy += N[0] * N[1];
    Q.xz += N[0] * N[2];
    Q.yy += N[1] * N[1];
    Q.yz += N[1] * N[2];
    Q.zz += N[2] * N[2];
    const double nb = N[0] * P[0] + N[1] * P[1] + N[2] * P[2];
    Q.bx += N[0] * nb;
    Q.by += N[1] * nb;
    Q.bz += N[2] * nb;
    Q.px += P[0];
    Q.py += P[1];
    Q.pz += P[2];
    Q.n += 1;
}

// Cyclic Jacobi rotations on a symmetric 3 x 3 matrix: eigenvalues on the
// diagonal of S, eigenvectors in the columns of V.  The sweeps stop once the
// off-diagonal sum is below 1e-12 of the diagonal's: the eigenvalues are then
// exact to second order (about 1e-24 relative) and the eigenvectors to about
// 1e-12, while FP64 rounding keeps the off-diagonal near 1e-16 of the
// diagonal, so a stricter bound would only spend sweeps.
__device__ __forceinline__ void jacobi3(double S[3][3], double V[3][3]) {
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) V[r][c] = r == c ? 1.0 : 0.0;
    for (int sweep = 0; sweep < 32; ++sweep) {
        const double off = fabs(S[0][1]) + fabs(S[0][2]) + fabs(S[1][2]);
        const double dia = fabs(S[0][0]) + fabs(S[1][1]) + fabs(S[2][2]);
        if (!(off > 1e-300) || off <= 1e-12 * dia) break;
        for (int p = 0; p < 2; ++p)
            for (int q = p + 1; q < 3; ++q) {
                const double apq = S[p][q];
                if (fabs(apq) <= 1e-300) continue;
                const double theta = (S[q][q] - S[p][p]) / (2.0 * apq);
                const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                const double c = 1.0 / sqrt(t * t + 1.0), s = t * c;
                for (int r = 0; r < 3; ++r) {  // S <- J^T S J
                    const double srp = S[r][p], srq = S[r][q];
                    S[r][p] = c * srp - s * srq;
                    S[r][q] = s * srp + c * srq;
                }
                for (int r = 0; r < 3; ++r) {
                    const double spr = S[p][r], sqr = S[q][r];
                    S[p][r] = c * spr - s * sqr;
                    S[q][r] = s * spr + c * sqr;
                }
                S[p][q] = S[q][p] = 0.0;
                for (int r = 0; r < 3; ++r) {
                    const double vrp = V[r][p], vrq = V[r][q];
                    V[r][p] = c * vrp - s * vrq;
                    V[r][q] = s * vrp + c * vrq;
                }
            }
    }
}

// Any system, by the eigensolver: the general path of qef_solve.
__device__ __noinline__ void qef_solve_jacobi(const Sym3 &Q, double x[3]) {
    const double m[3] = {Q.px / Q.n, Q.py / Q.n, Q.pz / Q.n};
    double S[3][3] = {{Q.xx, Q.xy, Q.xz}, {Q.xy, Q.yy, Q.yz}, {Q.xz, Q.yz, Q.zz}};
    const double AtA[3][3] = {{Q.xx, Q.xy, Q.xz}, {Q.xy, Q.yy, Q.yz}, {Q.xz, Q.yz, Q.zz}};
    double r[3] = {Q.bx, Q.by, Q.bz};
    for (int a = 0; a < 3; ++a) r[a] -= AtA[a][0] * m[0] + AtA[a][1] * m[1] + AtA[a][2] * m[2];
    double V[3][3];
    jacobi3(S, V);
    const double lam[3] = {S[0][0], S[1][1], S[2][2]};
    const double top = fmax(lam[0], fmax(lam[1], lam[2]));
    double y[3];
    for (int c = 0; c < 3; ++c) {
        const double vr = V[0][c] * r[0] + V[1][c] * r[1] + V[2][c] * r[2];
        y[c] = (top > 0.0 && lam[c] >= 0.01 * top) ? vr / lam[c] : 0.0;
    }
    for (int a = 0; a < 3; ++a) x[a] = m[a] + V[a][0] * y[0] + V[a][1] * y[1] + V[a][2] * y[2];
}

// Cyclic Jacobi rotations in FP32 on the matrix (xx, xy, xz, yy, yz, zz): its
// eigenvectors, to FP32 accuracy, in the columns of V.
__device__ __forceinline__ void jacobi3f(float xx, float xy, float xz, float yy, float yz, float zz, float (&V)[3][3]) {
    float S[3][3] = {{xx, xy, xz}, {xy, yy, yz}, {xz, yz, zz}};
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) V[r][c] = r == c ? 1.0f : 0.0f;
#pragma unroll 1
    for (int sweep = 0; sweep < 8; ++sweep) {
        const float off = fabsf(S[0][1]) + fabsf(S[0][2]) + fabsf(S[1][2]);
        if (!(off > 1e-7f * (S[0][0] + S[1][1] + S[2][2]))) break;
#pragma unroll
        for (int z = 0; z < 3; ++z) {
            const int p = z == 2 ? 1 : 0, q = z == 0 ? 1 : 2, o = 3 - p - q;
            const float apq = S[p][q];
            if (fabsf(apq) < 1e-30f) continue;
            const float theta = 0.5f * (S[q][q] - S[p][p]) / apq;
            const float t = copysignf(1.0f, theta) / (fabsf(theta) + sqrtf(fmaf(theta, theta, 1.0f)));
            const float c = rsqrtf(fmaf(t, t, 1.0f)), s = t * c;
            S[p][p] -= t * apq;
            S[q][q] += t * apq;
            S[p][q] = S[q][p] = 0.0f;
            const float sop = S[o][p], soq = S[o][q];
            S[o][p] = S[p][o] = c * sop - s * soq;
            S[o][q] = S[q][o] = s * sop + c * soq;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const float vp = V[r][p], vq = V[r][q];
                V[r][p] = c * vp - s * vq;
                V[r][q] = s * vp + c * vq;
            }
        }
    }
}

__device__ __forceinline__ double dot3(const double (&a)[3], const double (&b)[3]) {
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// x = m + (A^T A)^+ (A^T b - A^T A m).  This GPU runs FP64 at 1/64 of its FP32
// rate, and the eigensolver took about 1,800 FP64 operations a cell (the whole
// call spent 400 of 529 us in it for the 255^3 cells of the united sphere and knot).
// Here FP32 rotations find the eigenvectors, about 100 FP64 operations make
// them orthonormal and give the matrix in their frame, S = V^T A V, whose
// off-diagonal entries e may be at most 4e-7 of the largest eigenvalue (the
// largest of 120,000 systems of unit normals at any spread: 2.7e-7):
//  - the eigenvalues differ from S's diagonal by at most 2 e, so the cut is
//    decided by the diagonal unless an entry lies within 1e-5 of it;
//  - turning the kept directions away from the dropped ones by
//    e / (gap of their eigenvalues) separates them to second order, below
//    1e-8 with the gaps of 0.004 asked for here;
//  - what is left is solved on the kept block with its off-diagonal entries, to
//    second order too, below 2e-9.
// A system that is not so clear (or not finite, or whose entries are too small
// for FP32 rotations, as of normals 1e-12 long) goes to the eigensolver.
__device__ __forceinline__ void qef_solve(const Sym3 &Q, double (&x)[3]) {
    const double inv_n = 1.0 / (double)Q.n;
    const double m[3] = {Q.px * inv_n, Q.py * inv_n, Q.pz * inv_n};
    const double r[3] = {Q.bx - (Q.xx * m[0] + Q.xy * m[1] + Q.xz * m[2]),
                         Q.by - (Q.xy * m[0] + Q.yy * m[1] + Q.yz * m[2]),
                         Q.bz - (Q.xz * m[0] + Q.yz * m[1] + Q.zz * m[2])};
    float F[3][3];
    jacobi3f((float)Q.xx, (float)Q.xy, (float)Q.xz, (float)Q.yy, (float)Q.yz, (float)Q.zz, F);
    double v[3][3];  // v[c]: direction c
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int a = 0; a < 3; ++a) v[c][a] = (double)F[a][c];
    double f = 1.5 - 0.5 * dot3(v[0], v[0]);  // one Newton step of 1 / |v|
#pragma unroll
    for (int a = 0; a < 3; ++a) v[0][a] *= f;
    f = dot3(v[0], v[1]);
#pragma unroll
    for (int a = 0; a < 3; ++a) v[1][a] -= f * v[0][a];
    f = 1.5 - 0.5 * dot3(v[1], v[1]);
#pragma unroll
    for (int a = 0; a < 3; ++a) v[1][a] *= f;
    v[2][0] = v[0][1] * v[1][2] - v[0][2] * v[1][1];
    v[2][1] = v[0][2] * v[1][0] - v[0][0] * v[1][2];
    v[2][2] = v[0][0] * v[1][1] - v[0][1] * v[1][0];
    double S[3][3], g[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double w[3] = {Q.xx * v[c][0] + Q.xy * v[c][1] + Q.xz * v[c][2],
                             Q.xy * v[c][0] + Q.yy * v[c][1] + Q.yz * v[c][2],
                             Q.xz * v[c][0] + Q.yz * v[c][1] + Q.zz * v[c][2]};
#pragma unroll
        for (int d = c; d < 3; ++d) S[c][d] = S[d][c] = dot3(v[d], w);
        g[c] = dot3(v[c], r);
    }
    // everything below that decides or corrects needs FP32 only; S and g keep their FP64 values
    const float l[3] = {(float)S[0][0], (float)S[1][1], (float)S[2][2]};
    const float top = fmaxf(l[0], fmaxf(l[1], l[2])), cut = 0.01f * top;
    bool clear = top > 1e-30f && top < 1e30f, keep[3];  // (the kept ones' FP32 reciprocals are finite)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        clear = clear && fabsf(l[c] - cut) > 1e-5f * top;
        keep[c] = l[c] >= cut;
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (d != c) clear = clear && fabsf((float)S[c][d]) <= 4e-7f * top;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (d != c && keep[c] && !keep[d]) clear = clear && l[c] - l[d] > 4e-3f * top;
    if (!clear) {
        qef_solve_jacobi(Q, x);
        return;
    }
    double u[3][3], h[3], inv[3], y[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // kept directions turned away from the dropped ones
        h[c] = g[c];
#pragma unroll
        for (int a = 0; a < 3; ++a) u[c][a] = v[c][a];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (d == c) continue;
            if (keep[c] && !keep[d]) {
                const double th = (double)((float)S[c][d] / (l[c] - l[d]));
                h[c] += th * g[d];
#pragma unroll
                for (int a = 0; a < 3; ++a) u[c][a] += th * v[d][a];
            }
        }
        const double i0 = (double)(keep[c] ? 1.0f / l[c] : 0.0f);
        inv[c] = i0 * (2.0 - S[c][c] * i0);  // 1 / S to FP64 accuracy, 0 for a dropped direction
        y[c] = h[c] * inv[c];
    }
    double z[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double t = h[c];
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (d != c && keep[d]) t -= S[c][d] * y[d];
        z[c] = t * inv[c];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = m[a] + u[0][a] * z[0] + u[1][a] * z[1] + u[2][a] * z[2];
}

constexpr int kCells = 128;        // cells per block
constexpr int kCellThreads = 128;  // threads per block

// The records of kCells active cells (of the first *nact of the list), and
// which of them yield a vertex.
//  1. a thread per cell finds the corner signs;
//  2. the kept samples of every (cell, edge) from its ray, the first with its
//     depth and normal;
//  3. a thread per cell: clusters as sets of corner bits, then one cluster at a
//     time, its points' sums in registers, and its vertex;
//  4. the records leave through shared memory in whole lines.
// Bound by FP64 in step 3 (1.5 M FP64 warp instructions, 74 us of that pipe):
// 124 us for the 255^3 cells of the united sphere and knot, 149 with twice the
// threads searching, 420 with the eigensolver for every cell.
__global__ void __launch_bounds__(kCellThreads) cell_kernel(CImg I, const unsigned *node, int res, int W, float o0,
                                                            float o1, float o2, float h, const long long *cells,
                                                            const int *nact, long long max_active, ldni_cell_t *rec,
                                                            int *flag) {
    __shared__ float4 pt[12][kCells];   // the edge's first kept sample: depth, normal
    __shared__ int second[12][kCells];  // its second kept sample, kOne: there is none, kNo: no sample at all
    __shared__ short ijk[3][kCells];
    __shared__ unsigned char corner[kCells];
    constexpr int kOne = -1, kNo = -2;
    const long long q0 = (long long)blockIdx.x * kCells;
    const long long total = min((long long)*nact, max_active);
    const int m = (int)max(0ll, min((long long)kCells, total - q0));  // cells of this block
    const int tid = threadIdx.x;
    if (tid < kCells && tid >= m && q0 + tid < max_active) flag[q0 + tid] = 0;
    if (m == 0) return;
    const int n = res - 1;
    long long ci = 0;
    if (tid < m) {
        ci = cells[q0 + tid];
        const int row = (int)(ci / n);
        const int i = (int)(ci - (long long)row * n), j = row % n, k = row / n;
        ijk[0][tid] = (short)i;
        ijk[1][tid] = (short)j;
        ijk[2][tid] = (short)k;
        unsigned sgn = 0;  // bit c: corner c inside
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const unsigned *nw = node + ((long long)(k + (r >> 1)) * res + j + (r & 1)) * W + (i >> 5);
            const unsigned b0 = nw[0] >> (i & 31);
            const unsigned b1 = (i & 31) == 31 ? nw[1] : b0 >> 1;
            sgn |= ((b0 & 1u) | ((b1 & 1u) << 1)) << (2 * r);
        }
        corner[tid] = (unsigned char)sgn;
    }
    __syncthreads();
    for (int task = tid; task < 12 * kCells; task += kCellThreads) {
        const int e = task / kCells, c = task % kCells;
        if (c >= m) continue;
        const Edge E = cell_edge(e);
        const int u = E.a == 2 ? 0 : E.a + 1, v = E.a == 0 ? 2 : E.a - 1;
        const long long p = (long long)(ijk[v][c] + E.dv) * res + ijk[u][c] + E.du;
        const int t = ijk[E.a][c];
        const int *off = pick(I.off, E.a);
        const float *D = pick(I.d, E.a);
        const int b0 = off[p], e0 = (int)min((long long)off[p + 1], pick(I.cap, E.a));
        const float oa = E.a == 0 ? o0 : (E.a == 1 ? o1 : o2);
        const float lo = node_c(t, oa, h), hi = node_c(t + 1, oa, h);
        const unsigned sgn = corner[c];
        const bool in0 = (sgn >> E.q0) & 1u, in1 = (sgn >> E.q1) & 1u;
        int first = -1, last = -1, s = b0;
        while (s < e0 && D[s] < lo) ++s;  // ascending depths
        for (; s < e0 && D[s] < hi; ++s) {
            if (first < 0) first = s;
            last = s;
        }
        int keep = first, more = first < 0 ? kNo : kOne;
        if (first >= 0 && last > first) {
            if (in0 != in1) {  // Rule 2
                const float *NA = E.a == 0 ? I.nx[0] : (E.a == 1 ? I.ny[1] : I.nz[2]);
                const float want = in0 ? 1.0f : -1.0f;
                const double mid = ((double)lo + (double)hi) / 2.0;
                bool fits = false;
                double bd = 0.0;
                for (int x = first; x <= last; ++x) {
                    const bool f = NA[x] * want > 0.0f;
                    const double dist = fabs((double)D[x] - mid);
                    if (x == first || (f && !fits) || (f == fits && dist < bd)) {
                        keep = x;
                        bd = dist;
                        fits = f;
                    }
                }
            } else {  // Rule 1
                more = last;
            }
        }
        if (first >= 0)
            pt[e][c] = make_float4(D[keep], pick(I.nx, E.a)[keep], pick(I.ny, E.a)[keep], pick(I.nz, E.a)[keep]);
        second[e][c] = more;
    }
    __syncthreads();
    ldni_cell_t R;
    R.cell = ci;
    R.nvert = 0;
    R.labels = 0xffffffffu;
    R.npts = 0;
    R.pad_ = 0;
#pragma unroll
    for (int x = 0; x < 12; ++x) R.v[x] = 0.0f;
    if (tid < m) {
        const int i = ijk[0][tid], j = ijk[1][tid], k = ijk[2][tid];
        const unsigned sgn = corner[tid], out = ~sgn & 0xffu;
        // per axis, bit c: the edge from corner c up along it is empty and both its ends are outside
        unsigned open[3] = {0, 0, 0}, held = 0;  // held: edges with samples
#pragma unroll
        for (int e = 0; e < 12; ++e) {
            const Edge E = cell_edge(e);
            if (second[e][tid] != kNo)
                held |= 1u << e;
            else
                open[E.a] |= (out >> E.q0) & (out >> E.q1) & 1u ? 1u << E.q0 : 0u;
        }
        // flood the outside corners through empty edges, clusters by lowest corner
        int ncl = 0;
        for (unsigned rest = out; rest; ++ncl) {
            unsigned c = rest & (0u - rest), was;
            do {
                was = c;
#pragma unroll
                for (int a = 0; a < 3; ++a) c |= ((c & open[a]) << (1 << a)) | ((c >> (1 << a)) & open[a]);
            } while (c != was);
            rest &= ~c;
            unsigned x = (c | (c << 12)) & 0x000f000fu;  // bit c to bit 4 c
            x = (x | (x << 6)) & 0x03030303u;
            x = (x | (x << 3)) & 0x11111111u;
            R.labels ^= x * (0xfu ^ (unsigned)ncl);
        }
        // edges that make a surface: ends of different sign, or samples between outside corners
        unsigned cross = 0, outer = 0;
#pragma unroll
        for (int e = 0; e < 12; ++e) {
            const Edge E = cell_edge(e);
            const unsigned b0 = (sgn >> E.q0) & 1u, b1 = (sgn >> E.q1) & 1u;
            cross |= (b0 ^ b1) << e;
            outer |= (1u ^ (b0 | b1)) << e;
        }
        if (ncl > 0 && (cross | (held & outer))) {
            R.nvert = min(ncl, 4);  // a record has room for four
            const auto label = [&](int q) { return (int)((R.labels >> (4 * q)) & 0xfu); };
            for (int g = 0; g < R.nvert; ++g) {
                Sym3 Q{0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
                for (unsigned todo = held & (cross | outer); todo; todo &= todo - 1u) {
                    const int e = __ffs(todo) - 1;
                    const Edge E = cell_edge(e);
                    const int s1 = second[e][tid];
                    const int l0 = label(E.q0), l1 = label(E.q1);
                    bool first = false, last = false;  // this cluster's samples of the edge
                    float4 f = pt[e][tid];
                    if ((cross >> e) & 1u) {
                        first = ((sgn >> E.q0) & 1u ? l1 : l0) == g;
                    } else if (s1 >= 0) {
                        first = l0 == g;
                        last = l1 == g;
                    } else {  // the nearer corner's
                        const int t = ijk[E.a][tid];
                        const float oa = E.a == 0 ? o0 : (E.a == 1 ? o1 : o2);
                        const double mid = ((double)node_c(t, oa, h) + (double)node_c(t + 1, oa, h)) / 2.0;
                        first = ((double)f.x < mid ? l0 : l1) == g;
                    }
                    if (!first && !last) continue;
                    const int iu = (E.a == 0 ? j : (E.a == 1 ? k : i)) + E.du, iv = (E.a == 0 ? k : (E.a == 1 ? i : j)) + E.dv;
                    const float ou = E.a == 0 ? o1 : (E.a == 1 ? o2 : o0), ov = E.a == 0 ? o2 : (E.a == 1 ? o0 : o1);
                    const float cu = node_c(iu, ou, h), cv = node_c(iv, ov, h);
                    for (int z = 0; z < 2; ++z) {
                        if (!(z ? last : first)) continue;
                        if (z) f = make_float4(pick(I.d, E.a)[s1], pick(I.nx, E.a)[s1], pick(I.ny, E.a)[s1], pick(I.nz, E.a)[s1]);
                        const double P[3] = {(double)(E.a == 0 ? f.x : (E.a == 1 ? cv : cu)),
                                             (double)(E.a == 1 ? f.x : (E.a == 2 ? cv : cu)),
                                             (double)(E.a == 2 ? f.x : (E.a == 0 ? cv : cu))};
                        const double N[3] = {(double)f.y, (double)f.z, (double)f.w};
                        add_point(Q, P, N);
                    }
                }
                double x[3];
                if (Q.n > 0) {
                    qef_solve(Q, x);
                } else {  // no Hermite data: the mean of the cluster's corners
                    int cs = 0;
                    x[0] = x[1] = x[2] = 0.0;
                    for (int c = 0; c < 8; ++c) {
                        if (label(c) != g) continue;
                        x[0] += (double)node_c(i + (c & 1), o0, h);
                        x[1] += (double)node_c(j + ((c >> 1) & 1), o1, h);
                        x[2] += (double)node_c(k + (c >> 2), o2, h);
                        ++cs;
                    }
                    for (int a = 0; a < 3; ++a) x[a] /= cs;
                }
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (v == g) {
                        R.v[3 * v] = (float)x[0];
                        R.v[3 * v + 1] = (float)x[1];
                        R.v[3 * v + 2] = (float)x[2];
                    }
                R.npts |= (unsigned)min(Q.n, 255) << (8 * g);
            }
        }
        flag[q0 + tid] = R.nvert > 0 ? 1 : 0;
    }
    __syncthreads();  // the points are read
    constexpr int kWords = (int)(sizeof(ldni_cell_t) / 4);
    static_assert(sizeof(pt) >= kCells * sizeof(ldni_cell_t), "the records fit where the points were");
    ldni_cell_t *out = reinterpret_cast<ldni_cell_t *>(&pt[0][0]);
    if (tid < m) out[tid] = R;
    __syncthreads();
    const int *from = reinterpret_cast<const int *>(out);
    int *to = reinterpret_cast<int *>(rec + q0);
    for (int x = tid; x < m * kWords; x += kCellThreads) to[x] = from[x];
}

// The cells with a vertex, in order: a warp copies 32 records, word by word.
__global__ void __launch_bounds__(kThreads) compact_cells(const ldni_cell_t *rec, const int *nact, long long n,
                                                          const int *flag, const int *at, ldni_cell_t *out,
                                                          long long cap, ldni_info_t *info) {
    const int lane = threadIdx.x & 31;
    const long long q0 = blockIdx.x * (long long)kThreads + (threadIdx.x & ~31), total = min((long long)*nact, n);
    if (q0 >= total) return;  // the same for the whole warp
    int slot = -1;
    if (q0 + lane < total && flag[q0 + lane]) {
        slot = at[q0 + lane];
        if (slot >= cap) {
            set_status(info, LDNI_ST_CAPACITY);
            slot = -1;
        }
    }
    constexpr int kWords = (int)(sizeof(ldni_cell_t) / 4);
    const int *from = reinterpret_cast<const int *>(rec + q0);
    int *to = reinterpret_cast<int *>(out);
    const int words = (int)min(32ll, total - q0) * kWords;
#pragma unroll 6
    for (int x = lane; x < 32 * kWords; x += 32) {
        const int c = x / kWords, s = __shfl_sync(0xffffffffu, slot, c);
        if (x < words && s >= 0) to[(long long)s * kWords + (x - c * kWords)] = from[x];
    }
}

struct ContourWs {
    unsigned *act;
    size_t act_bytes;
    int *wcnt, *woff;
    long long *cells;
    ldni_cell_t *rec;
    int *flag, *at;
    long long *partials;
    ldni_info_t *tinfo;
};

ContourWs carve_contour(Carver &c, int res, long long max_active) {
    ContourWs w{};
    const long long n = res - 1, Wc = (n + 31) / 32, nw = n * n * Wc;
    w.act = c.take<unsigned>((size_t)nw);
    w.act_bytes = sizeof(unsigned) * (size_t)nw;
    w.wcnt = c.take<int>((size_t)nw);
    w.woff = c.take<int>((size_t)nw + 1);
    w.cells = c.take<long long>((size_t)max_active);
    w.rec = c.take<ldni_cell_t>((size_t)max_active);
    w.flag = c.take<int>((size_t)max_active);
    w.at = c.take<int>((size_t)max_active + 1);
    w.partials = c.take<long long>(std::max(csr_scan_partials(nw), csr_scan_partials(max_active)));
    w.tinfo = c.take<ldni_info_t>(1);
    return w;
}

}  // namespace
}  // namespace ldni

using namespace ldni;

extern "C" int ldni_contour_workspace_size(int32_t res, int64_t max_active, size_t *bytes) {
    if (!bytes || res < 2 || res > 2048 || max_active < 1 || max_active > INT_MAX) return LDNI_EINVAL;
    Carver c(nullptr, 0);
    carve_contour(c, res, max_active);
    *bytes = align_up(c.off);
    return LDNI_OK;
}

extern "C" int ldni_contour_cells(const ldni_layers_t *L, const ldni_grid_t *grid, const uint32_t *inside,
                                  int64_t max_active, ldni_cell_t *cells, int64_t capacity, ldni_info_t *info,
                                  void *ws, size_t ws_bytes, void *stream) {
    if (!L || !grid_valid(grid) || !inside || !info || !ws || (capacity > 0 && !cells) || capacity < 0 ||
        max_active < 1 || max_active > INT_MAX)
        return LDNI_EINVAL;
    const int res = grid->res;
    if (res < 2 || res > 2048) return LDNI_EINVAL;
    CImg I{};
    for (int a = 0; a < 3; ++a) {
        if (!L[a].offsets || L[a].capacity < 0 || !samples_ok(L[a]) || L[a].nrm8) return LDNI_EINVAL;
        I.off[a] = L[a].offsets;
        I.d[a] = L[a].depth;
        I.nx[a] = L[a].nx;
        I.ny[a] = L[a].ny;
        I.nz[a] = L[a].nz;
        I.cap[a] = L[a].capacity;
    }
    Carver c(ws, ws_bytes);
    ContourWs w = carve_contour(c, res, max_active);
    if (!c.fits()) return LDNI_EWORKSPACE;
    const int n = res - 1, W = (res + 31) / 32, Wc = (n + 31) / 32;
    const long long nw = (long long)n * n * Wc;
    const float h = grid->width / (float)res;
    const float *o = grid->origin;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (int rc_ = cuda_check(cudaMemsetAsync(w.act, 0, w.act_bytes, s))) return rc_;
    if (int rc_ = cuda_check(cudaMemsetAsync(w.tinfo, 0, sizeof(ldni_info_t), s))) return rc_;
    const long long N = (long long)res * res;
    LDNI_LAUNCH(K_CONTOUR, s,
                mark_signs<<<(unsigned)((nw + kThreads - 1) / kThreads), kThreads, 0, s>>>(inside, res, W, w.act, Wc));
    LDNI_LAUNCH(K_CONTOUR, s,
                mark_samples<<<dim3((unsigned)((N + kThreads - 1) / kThreads), 3), kThreads, 0, s>>>(
                    I, res, o[0], o[1], o[2], h, w.act, Wc));
    LDNI_LAUNCH(K_CONTOUR, s,
                count_words<<<(unsigned)((nw + kThreads - 1) / kThreads), kThreads, 0, s>>>(w.act, nw, w.wcnt));
    int rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    {
        const int *cn[1] = {w.wcnt};
        int *of[1] = {w.woff};
        rc = csr_scan(cn, of, 1, nw, w.partials, w.tinfo, 0, s);
        if (rc != LDNI_OK) return rc;
    }
    // every later launch covers max_active cells and reads the active count
    // on the device, so the call needs no host synchronisation
    const int *nact = w.woff + nw;
    const unsigned ablocks = (unsigned)((max_active + kThreads - 1) / kThreads);
    LDNI_LAUNCH(K_CONTOUR, s,
                list_cells<<<(unsigned)((nw + kThreads - 1) / kThreads), kThreads, 0, s>>>(
                    w.act, nw, w.woff, n, Wc, w.cells, max_active, info));
    LDNI_LAUNCH(K_CONTOUR, s,
                cell_kernel<<<(unsigned)((max_active + kCells - 1) / kCells), kCellThreads, 0, s>>>(
                    I, inside, res, W, o[0], o[1], o[2], h, w.cells, nact, max_active, w.rec, w.flag));
    rc = cuda_status();
    if (rc != LDNI_OK) return rc;
    {
        const int *cn[1] = {w.flag};
        int *of[1] = {w.at};
        rc = csr_scan(cn, of, 1, max_active, w.partials, info, 0, s);
        if (rc != LDNI_OK) return rc;
    }
    LDNI_LAUNCH(K_CONTOUR, s,
                compact_cells<<<ablocks, kThreads, 0, s>>>(w.rec, nact, max_active, w.flag, w.at, cells, capacity,
                                                           info));
    return cuda_status();
}
