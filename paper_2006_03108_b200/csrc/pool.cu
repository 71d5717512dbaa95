// Distributed pooling layer on a feature-space partition with unbalanced halos (Section 4,
// "Sparse layers": pooling follows the convolution algorithms without weights; Section 3 and
// Appendix B: the halo widths of a strided kernel differ from worker to worker and some owned
// inputs may go unused).
//
// forward = halo exchange H (the library's in-place kernel), then the local sliding kernel over
// each worker's padded shard, starting at the first input the worker's block of the evenly split
// output needs; adjoint = local adjoint into every cell of the padded shard (ghosts included),
// then H*: as these two kernels, or (common windows, pool_adj_fused) as one that adds up the neighbours'
// outputs where H* would have brought their ghosts.  The local adjoint is evaluated in gather form -- a cell
// sums over the outputs whose window holds it, in ascending output order -- so overlapping windows need no atomics.
#include <algorithm>
#include <climits>
#include <cstring>
#include <vector>

#include "common.h"

namespace distdl {

constexpr int kPoolMaxWorkers = 32;
constexpr int kPoolThreadsX = 32, kPoolThreadsY = 8;

struct PoolShard {
    const float *in;       // forward: padded x;   adjoint: dy
    float *out;            // forward: y;          adjoint: padded dx
    int32_t *arg;          // position of the maximum inside the window (a * kw + b), or nullptr
    int32_t ph, pw;        // padded extents of the shard (rows, columns)
    int32_t oh, ow;        // this worker's block of the output
    int32_t i0, j0;        // padded-local index of the first input of output (0, 0)
    int32_t g0h, g0w;      // global index of padded-local index 0
    int32_t hlh, hlw;      // low ghost rows / columns
    int32_t bh, bw;        // bulk rows / columns
};

struct PoolParams {
    PoolShard s[kPoolMaxWorkers];
    int32_t planes, kh, kw, sh, sw, hg, wg, mode;
    int32_t wrows, wcols;  // rows and columns of workers
};

__host__ __device__ __forceinline__ int div_floor(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// One thread per output.  blockIdx.y = worker, blockIdx.x = (plane, row tile, column tile).
__global__ void __launch_bounds__(kPoolThreadsX *kPoolThreadsY)
pool_fwd_kernel(const __grid_constant__ PoolParams P, int tiles_x, int tiles_y) {
    stream_enter();
    const PoolShard &S = P.s[blockIdx.y];
    int rest = blockIdx.x;
    const int tx = rest % tiles_x;
    rest /= tiles_x;
    const int ty = rest % tiles_y;
    const int plane = rest / tiles_y;
    const int j = tx * kPoolThreadsX + threadIdx.x, i = ty * kPoolThreadsY + threadIdx.y;
    if (i >= S.oh || j >= S.ow || plane >= P.planes) return;
    const int r0 = S.i0 + i * P.sh, c0 = S.j0 + j * P.sw;
    const float *src = S.in + ((size_t)plane * S.ph + r0) * S.pw + c0;
    const size_t o = ((size_t)plane * S.oh + i) * S.ow + j;
    if (P.mode == DISTDL_POOL_AVG) {
        float acc = 0.f;
        for (int a = 0; a < P.kh; ++a)
            for (int b = 0; b < P.kw; ++b) acc = __fadd_rn(acc, src[a * S.pw + b]);
        S.out[o] = __fmul_rn(acc, 1.0f / (float)(P.kh * P.kw));
    } else {
        // largest value of the window clipped to the tensor; the first one in row-major order wins
        float best = 0.f;
        int where = -1;
        for (int a = 0; a < P.kh; ++a) {
            const int gi = S.g0h + r0 + a;
            if (gi < 0 || gi >= P.hg) continue;
            for (int b = 0; b < P.kw; ++b) {
                const int gj = S.g0w + c0 + b;
                if (gj < 0 || gj >= P.wg) continue;
                const float v = src[a * S.pw + b];
                if (where < 0 || v > best) {
                    best = v;
                    where = a * P.kw + b;
                }
            }
        }
        S.out[o] = best;
        if (S.arg) S.arg[o] = where < 0 ? 0 : where;
    }
}

// One thread per cell of the padded dx.  A cell (p, q) lies in the window of output (i, j) iff
// 0 <= p - i0 - i*sh < kh and likewise for the columns.
__global__ void __launch_bounds__(kPoolThreadsX *kPoolThreadsY)
pool_adj_kernel(const __grid_constant__ PoolParams P, int tiles_x, int tiles_y) {
    stream_enter();
    const PoolShard &S = P.s[blockIdx.y];
    int rest = blockIdx.x;
    const int tx = rest % tiles_x;
    rest /= tiles_x;
    const int ty = rest % tiles_y;
    const int plane = rest / tiles_y;
    const int q = tx * kPoolThreadsX + threadIdx.x, p = ty * kPoolThreadsY + threadIdx.y;
    if (p >= S.ph || q >= S.pw || plane >= P.planes) return;
    const int dp = p - S.i0, dq = q - S.j0;
    const int i_lo = max(0, div_floor(dp - P.kh + P.sh, P.sh)), i_hi = min(S.oh - 1, div_floor(dp, P.sh));
    const int j_lo = max(0, div_floor(dq - P.kw + P.sw, P.sw)), j_hi = min(S.ow - 1, div_floor(dq, P.sw));
    const float *dy = S.in + (size_t)plane * S.oh * S.ow;
    const int32_t *arg = S.arg ? S.arg + (size_t)plane * S.oh * S.ow : nullptr;
    float acc = 0.f;
    for (int i = i_lo; i <= i_hi; ++i)
        for (int j = j_lo; j <= j_hi; ++j) {
            if (P.mode == DISTDL_POOL_AVG) {
                acc = __fadd_rn(acc, dy[i * S.ow + j]);
            } else {
                const int a = dp - i * P.sh, b = dq - j * P.sw;
                if (arg[i * S.ow + j] == a * P.kw + b) acc = __fadd_rn(acc, dy[i * S.ow + j]);
            }
        }
    if (P.mode == DISTDL_POOL_AVG) acc = __fmul_rn(acc, 1.0f / (float)(P.kh * P.kw));
    S.out[((size_t)plane * S.ph + p) * S.pw + q] = acc;
}

// ---------------------------------------------------------------------------------------------
// Variants with the kernel and stride fixed at compile time (2 x 2 / 2, 3 x 3 / 2 and 3 x 3 / 1, the pooling layers of the
// usual networks).  A warp owns 64 columns (of outputs, adjoint: of groups of SH x SW cells) and marches down `rows` rows:
// what overlapping windows share stays in registers, the loads of the next step are issued before this step's arithmetic,
// and neighbouring lanes touch neighbouring addresses.  Same results as the general kernels above.
//
// What bounds them: device memory, instruction issue close behind.  Measured (B200, with H / H*, forward / adjoint, us; before: H* as a
// kernel of its own behind the local adjoint):
//   3 x 3 / 2 max, 16 x 16 x 1024 x 1024 on 4 x 4 workers    354 / 350   (354 / 417)
//   3 x 3 / 1 avg, 12 x 13 x 802 x 239 on 1 x 2               108 / 101   (108 / 127)
//   3 x 3 / 1 max, 2 x 7 x 752 x 84 on 3 x 4                  18.8 / 14.6  (18.8 / 15.7)
//   3 x 3 / 2 avg, 3 x 1 x 91 x 337 on 1 x 3                  3.9 / 3.1    (3.9 / 3.9)
// H in the forward kernel as well: ghosts copied by the warps that read them 349 of 357 us, but 3.9 -> 5.4 us for the last of these; read
// where they lie and written beside that 407 us: the forward's loop has no instructions to spare.  A maximum is taken per input row first
// (value, first position); a NaN counts as the scan in window order counts it: it wins only as the window's first cell.
// ---------------------------------------------------------------------------------------------
constexpr int kPoolCols = 2;           // columns per lane, 32 apart

template <int KW>
struct PoolRow {
    float x[KW];                       // AVG: the cells;  MAX: x[0] = first cell of the row inside the tensor
    float m;                           // MAX: largest cell that is a number, the first of equals
    int b;                             // and its column in the window
    __device__ __forceinline__ void set(const float (&v)[KW]) {
#pragma unroll
        for (int c = 0; c < KW; ++c) x[c] = v[c];
    }
    __device__ __forceinline__ void reduce() {
        float top = x[0];
#pragma unroll
        for (int c = 1; c < KW; ++c) top = fmaxf(top, x[c]);
        m = x[KW - 1];
        b = KW - 1;
#pragma unroll
        for (int c = KW - 2; c >= 0; --c)
            if (x[c] == top) {
                m = x[c];
                b = c;
            }
    }
    // the cells [lo, hi) of the row lie inside the tensor (at least one): the others take the value of the nearest of those,
    // which changes neither the maximum nor, once it is no smaller than lo, its first position
    __device__ __forceinline__ void reduce_clipped(int lo, int hi) {
#pragma unroll
        for (int c = KW - 2; c >= 0; --c)
            if (c < lo) x[c] = x[c + 1];
#pragma unroll
        for (int c = 1; c < KW; ++c)
            if (c >= hi) x[c] = x[c - 1];
        reduce();
        b = max(b, lo);
    }
};

template <int KH, int KW, int SH, int SW, int MODE>
__global__ void __launch_bounds__(kPoolThreadsX *kPoolThreadsY)
pool_fwd_fixed(const __grid_constant__ PoolParams P, int tiles_x, int tiles_y, int rows) {
    stream_enter();
    const PoolShard &S = P.s[blockIdx.y];
    int rest = blockIdx.x;
    const int tx = rest % tiles_x;
    rest /= tiles_x;
    const int ty = rest % tiles_y;
    const int plane = rest / tiles_y;
    const int lane = threadIdx.x, jb = tx * (32 * kPoolCols) + lane, i_begin = (ty * kPoolThreadsY + (int)threadIdx.y) * rows;
    const int i_end = min(i_begin + rows, S.oh);
    if (i_begin >= i_end || tx * (32 * kPoolCols) >= S.ow) return;
    bool on[kPoolCols], inside = true, some = true;         // all / at least one of the window's columns inside the tensor
    int lo[kPoolCols], hi[kPoolCols];                       // window columns inside the tensor
    const float *src[kPoolCols];
    const float *base = S.in + ((size_t)plane * S.ph + (S.i0 + i_begin * SH)) * S.pw + S.j0;
#pragma unroll
    for (int u = 0; u < kPoolCols; ++u) {
        const int j = min(jb + 32 * u, S.ow - 1);
        on[u] = jb + 32 * u < S.ow;
        src[u] = base + j * SW;
        const int gj = S.g0w + S.j0 + j * SW;
        lo[u] = max(0, -gj);
        hi[u] = min(KW, P.wg - gj);
        inside = inside && lo[u] == 0 && hi[u] == KW;
        some = some && lo[u] < hi[u];
    }
    inside = __all_sync(0xffffffffu, inside);
    some = __all_sync(0xffffffffu, some);
    float next[SH][kPoolCols][KW];
    PoolRow<KW> row[KH][kPoolCols];
    auto load = [&](float (&v)[kPoolCols][KW]) {            // one input row, and on to the next
#pragma unroll
        for (int u = 0; u < kPoolCols; ++u) {
#pragma unroll
            for (int c = 0; c < KW; ++c) v[u][c] = __ldg(src[u] + c);
            src[u] += S.pw;
        }
    };
    auto take = [&](int a, const float (&v)[kPoolCols][KW]) {
#pragma unroll
        for (int u = 0; u < kPoolCols; ++u) {
            row[a][u].set(v[u]);
            if (MODE == DISTDL_POOL_MAX) {
                if (inside) row[a][u].reduce();
                else row[a][u].reduce_clipped(lo[u], hi[u]);
            }
        }
    };
    // the rows that the first window shares with the one before it, then one step ahead
#pragma unroll
    for (int a = 0; a < KH - SH; ++a) {
        float v[kPoolCols][KW];
        load(v);
        take(a, v);
    }
#pragma unroll
    for (int a = 0; a < SH; ++a) load(next[a]);
    float *out = S.out + ((size_t)plane * S.oh + i_begin) * S.ow + jb;
    int32_t *arg = MODE == DISTDL_POOL_MAX && S.arg ? S.arg + ((size_t)plane * S.oh + i_begin) * S.ow + jb : nullptr;
    for (int i = i_begin; i < i_end; ++i) {
        float v[SH][kPoolCols][KW];
#pragma unroll
        for (int a = 0; a < SH; ++a)
#pragma unroll
            for (int u = 0; u < kPoolCols; ++u)
#pragma unroll
                for (int c = 0; c < KW; ++c) v[a][u][c] = next[a][u][c];
        if (i + 1 < i_end)
#pragma unroll
            for (int a = 0; a < SH; ++a) load(next[a]);
#pragma unroll
        for (int a = 0; a < SH; ++a) take(KH - SH + a, v[a]);
        const int gi = S.g0h + S.i0 + i * SH;               // tensor row of window row 0
        const bool full = some && gi >= 0 && gi + KH <= P.hg;   // no row of the window outside (3 x 3 / 1: 509 -> 465 us on 2 x 2 workers)
#pragma unroll
        for (int u = 0; u < kPoolCols; ++u) {
            float best = 0.f;
            int where = 0;
            if (MODE == DISTDL_POOL_AVG) {
#pragma unroll
                for (int a = 0; a < KH; ++a)
#pragma unroll
                    for (int c = 0; c < KW; ++c) best = __fadd_rn(best, row[a][u].x[c]);
                best = __fmul_rn(best, 1.0f / (float)(KH * KW));
            } else {
                if (full) {
                    const bool nan = row[0][u].x[0] != row[0][u].x[0];
                    best = nan ? row[0][u].x[0] : row[0][u].m;
                    where = nan ? lo[u] : row[0][u].b;
#pragma unroll
                    for (int a = 1; a < KH; ++a)
                        if (row[a][u].m > best) {
                            best = row[a][u].m;
                            where = a * KW + row[a][u].b;
                        }
                } else {
                    bool have = false;
#pragma unroll
                    for (int a = 0; a < KH; ++a) {
                        if (gi + a < 0 || gi + a >= P.hg || lo[u] >= hi[u]) continue;
                        const PoolRow<KW> &r = row[a][u];
                        if (!have) {
                            const bool nan = r.x[0] != r.x[0];
                            best = nan ? r.x[0] : r.m;
                            where = a * KW + (nan ? lo[u] : r.b);
                            have = true;
                        } else if (r.m > best) {
                            best = r.m;
                            where = a * KW + r.b;
                        }
                    }
                }
            }
            if (on[u]) {
                out[32 * u] = best;
                if (arg) arg[32 * u] = where;
            }
        }
        out += S.ow;
        if (arg) arg += S.ow;
#pragma unroll
        for (int a = 0; a < KH - SH; ++a)
#pragma unroll
            for (int u = 0; u < kPoolCols; ++u) row[a][u] = row[a + SH][u];
    }
}

// Cells of one row: lane l of a strip holds cells SW * (l + 32 u) + c.  Two to a lane are stored as 8-byte pairs; in rows that start off an
// 8-byte boundary (every other one at an odd pitch) a pair is a lane's second cell and the next lane's first (3 x 3 / 2 max, 16 x 16 x 1024 x
// 1024: 367 -> 359 us).
template <int SW, int NU>
__device__ __forceinline__ void pool_store_row(float *out, const float (&v)[NU][SW], int cols, int lane) {
    if (SW == 2 && cols == 64 * NU) {
        float *o = out + 2 * lane;
        if ((reinterpret_cast<uintptr_t>(out) & 7u) == 0) {
#pragma unroll
            for (int u = 0; u < NU; ++u) *reinterpret_cast<float2 *>(o + 64 * u) = make_float2(v[u][0], v[u][SW - 1]);
        } else {
            float next[NU];
#pragma unroll
            for (int u = 0; u < NU; ++u) next[u] = __shfl_sync(0xffffffffu, v[u][0], (lane + 1) & 31);
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                const float n = lane < 31 ? next[u] : next[u + 1 < NU ? u + 1 : u];
                if (u + 1 < NU || lane < 31) *reinterpret_cast<float2 *>(o + 64 * u + 1) = make_float2(v[u][SW - 1], n);
            }
            if (lane == 0) out[0] = v[0][0];
            if (lane == 31) o[64 * (NU - 1) + 1] = v[NU - 1][SW - 1];
        }
        return;
    }
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int c = 0; c < SW; ++c)
            if (SW * (lane + 32 * u) + c < cols) out[SW * (lane + 32 * u) + c] = v[u][c];
}

// Which columns of outputs the cells of a strip of the adjoint with H* in it meet: what the kernel computes with and what
// distdl_selftest_pool_adj_terms() replays.  A lane holds groups lane + 32 u of SW cells; the outputs that one meets are newest + 32 u - v.
template <int KW, int SW, int DW, int NU>
struct PoolStrip {
    static constexpr int EW = DW > 0 ? 1 : 0, NJ = (KW - 1 - DW) / SW + EW + 1;
    int newest;            // newest output column of the lane's first group
    int cols;              // cells of the strip
    bool left, right;      // the last column of the outputs on the left is met, the first column of those on the right
    __host__ __device__ __forceinline__ PoolStrip(const PoolShard &S, int wc, int wcols, int col0, int lane) {
        newest = col0 + lane + div_floor(S.hlw - S.j0, SW) + EW;
        cols = min(S.bw - col0 * SW, 32 * NU * SW);
        left = wc > 0 && col0 == 0 && newest - lane - (NJ - 1) < 0;
        // not in a shard's last strip only: where that is one column wide, the group at the end of the strip before it may lie under the output too
        right = wc + 1 < wcols && newest - lane + 32 * NU - 1 >= S.ow;
    }
    // window column under which output v of a group holds the group's cell c (outside 0 .. KW - 1: it does not)
    static constexpr __host__ __device__ __forceinline__ int window(int c, int v) { return c + DW + (v - EW) * SW; }
    // (x, at) in the place of the output on the left (right) of the shard's own.  The one on the left can be the newest of the first group
    // where windows do not overlap: a shard that begins with a whole window of its neighbour's.
    template <typename T>
    static __host__ __device__ __forceinline__ void put_left(T (&g)[NU][NJ], int (&code)[NU][NJ], T x, int at, int newest) {
#pragma unroll
        for (int v = KW > SW ? 1 : 0; v < NJ; ++v)
            if (newest - v == -1) {
                g[0][v] = x;
                code[0][v] = at;
            }
    }
    template <typename T>
    static __host__ __device__ __forceinline__ void put_right(T (&g)[NU][NJ], int (&code)[NU][NJ], T x, int at, int newest, int ow) {
#pragma unroll
        for (int u = 0; u < NU; ++u)
#pragma unroll
            for (int v = 0; v < NJ; ++v)
                if (newest + 32 * u - v == ow) {
                    g[u][v] = x;
                    code[u][v] = at;
                }
    }
};
// Row i of the outputs, counted from the own of worker w (shard S, in worker row wr): row il of the worker dr rows of workers below; false if there is none.
__host__ __device__ __forceinline__ bool pool_row_owner(const PoolParams &P, const PoolShard &S, int w, int wr, int i, int &dr, int &il) {
    dr = i < 0 ? -1 : i >= S.oh ? 1 : 0;
    if ((unsigned)(wr + dr) >= (unsigned)P.wrows) return false;
    const int oh = P.s[w + dr * P.wcols].oh;
    il = dr < 0 ? i + oh : dr ? i - S.oh : i;
    return (unsigned)il < (unsigned)oh;
}

// Adjoint with H* in it: every bulk cell sums over all outputs whose window holds it, the neighbours' among them, in ascending order, and
// the ghosts are cleared.  A lane owns groups of SH x SW bulk cells and marches down the rows of outputs; an output row is added to the KH
// rows of cells that its windows hold, whose sums move up by SH rows as the first of them are done.  The first column of a group is
// column DW of the windows that begin every SW columns, so the columns of a shard fill its strips whatever its ghosts (256 columns behind
// a ghost one: two strips of 64 groups, three when the groups begin with the windows).
// The outputs whose window holds cell column c of a group are J - v with window column b = c + DW + (v - EW) * SW < KW, known at compile
// time.  Rows of outputs above and below are read where they lie, the one column of outputs left and right of the shard that is met is
// fetched once by the lanes, a row each, and handed out by shuffles.
// NU columns of groups a lane: one where the shards are no wider than 32 groups (max 2 x 7 x 752 x 84 on 3 x 4 workers 20.2 -> 14.6 us), two
// otherwise (one for all: 350 -> 460 us at 16 x 16 x 1024 x 1024).  The next row is fetched before this one is added up, and four blocks fit a
// multiprocessor: with the fetch behind the sums 359 us, with three blocks 405, with five 375.
template <int KH, int KW, int SH, int SW, int MODE, int DW, int NU>
__device__ __forceinline__ void pool_adj_strip(const PoolParams &P, int w, int plane, int first_row, int rows, int col0, int lane) {
    using Strip = PoolStrip<KW, SW, DW, NU>;
    constexpr int NI = (KH + SH - 1) / SH, NJ = Strip::NJ;
    const PoolShard &S = P.s[w];
    const int wr = w / P.wcols, wc = w - wr * P.wcols;
    const int gi0 = div_floor(S.hlh - S.i0, SH) + first_row, bulk_end = S.hlh + S.bh;
    if (S.i0 + gi0 * SH >= bulk_end || col0 * SW >= S.bw) return;
    const int i_begin = gi0 - (NI - 1), i_end = min(gi0 + rows, div_floor(bulk_end - 1 - S.i0, SH) + 1);   // output rows
    const Strip strip(S, wc, P.wcols, col0, lane);
    const int j0 = strip.newest, cols = strip.cols;
    // outputs -1 and ow of row i_begin + lane
    const bool has_left = strip.left, has_right = strip.right;
    float sg[2] = {0.f, 0.f};
    int sc[2] = {-1, -1};
    if (has_left || has_right) {
        int dr, il;
        if (i_begin + lane < i_end && pool_row_owner(P, S, w, wr, i_begin + lane, dr, il)) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!(k ? has_right : has_left)) continue;
                const PoolShard &N = P.s[w + dr * P.wcols + 2 * k - 1];
                const size_t o = ((size_t)plane * N.oh + il) * N.ow + (k ? 0 : N.ow - 1);
                sg[k] = __ldg(N.in + o);
                if (MODE == DISTDL_POOL_MAX) sc[k] = __ldg(N.arg + o);
            }
        }
    }
    bool jok[NU][NJ], whole = true;
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int v = 0; v < NJ; ++v) {
            jok[u][v] = (unsigned)(j0 + 32 * u - v) < (unsigned)S.ow;
            whole = whole && jok[u][v];
        }
    whole = __all_sync(0xffffffffu, whole);
    const float *dy = S.in;
    const int32_t *arg = S.arg;
    bool row_ok = false;
    int at = i_begin, seek_at = i_begin;                   // output row to load next; row where the pointers move to another shard
    float gn[NU][NJ];
    int cn[NU][NJ];                                        // MAX: recorded position, -1 for an absent output
    auto load = [&]() {
        if (at == seek_at) {
            int dr, il = 0;
            row_ok = pool_row_owner(P, S, w, wr, at, dr, il);
            const PoolShard &N = P.s[row_ok ? w + dr * P.wcols : w];
            // above: down to row 0 (from a row above the shard above, which no window of this one's cells needs: to that shard)
            seek_at = dr < 0 ? (!row_ok && il < 0 ? at - il : 0) : dr == 0 ? S.oh : row_ok ? S.oh + N.oh : INT_MAX;
            const size_t o = ((size_t)plane * N.oh + il) * N.ow + j0;
            dy = N.in + o;
            if (MODE == DISTDL_POOL_MAX) arg = N.arg + o;
        }
        if (whole && row_ok) {
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int v = 0; v < NJ; ++v) {
                    gn[u][v] = __ldg(dy + (32 * u - v));
                    if (MODE == DISTDL_POOL_MAX) cn[u][v] = __ldg(arg + (32 * u - v));
                }
        } else {
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int v = 0; v < NJ; ++v) {
                    const bool on = row_ok && jok[u][v];
                    gn[u][v] = on ? __ldg(dy + (32 * u - v)) : 0.f;
                    if (MODE == DISTDL_POOL_MAX) cn[u][v] = on ? __ldg(arg + (32 * u - v)) : -1;
                }
        }
        dy += S.ow;
        if (MODE == DISTDL_POOL_MAX) arg += S.ow;
        ++at;
    };
    load();
    constexpr int SLOTS = KH > SH ? KH : SH;
    float acc[SLOTS][NU][SW];
#pragma unroll
    for (int a = 0; a < SLOTS; ++a)
#pragma unroll
        for (int u = 0; u < NU; ++u)
#pragma unroll
            for (int c = 0; c < SW; ++c) acc[a][u][c] = 0.f;
    // the ghost cell of every row that this lane clears: lanes 0 on left of the strip, lanes 16 on right of it
    const bool left = col0 == 0 && S.hlw > 0, right = col0 * SW + cols == S.bw && S.hlw + S.bw < S.pw;
    const bool clears = lane < 16 ? left && lane < S.hlw : right && lane - 16 < S.pw - S.hlw - S.bw;
    const int clear_at = lane < 16 ? lane - S.hlw : cols + lane - 16;
    float *shard = S.out + (size_t)plane * S.ph * S.pw;
    float *out = shard + (size_t)(S.i0 + gi0 * SH) * S.pw + (S.hlw + col0 * SW);       // first cell of the strip
#pragma unroll 1
    for (int i = i_begin; i < i_end; ++i) {
        float g[NU][NJ];
        int code[NU][NJ];
#pragma unroll
        for (int u = 0; u < NU; ++u)
#pragma unroll
            for (int v = 0; v < NJ; ++v) {
                g[u][v] = gn[u][v];
                code[u][v] = cn[u][v];
            }
        if (i + 1 < i_end) load();
        if (has_left) {
            const float x = __shfl_sync(0xffffffffu, sg[0], i - i_begin);
            const int c = MODE == DISTDL_POOL_MAX ? __shfl_sync(0xffffffffu, sc[0], i - i_begin) : 0;
            Strip::put_left(g, code, x, c, j0);
        }
        if (has_right) {
            const float x = __shfl_sync(0xffffffffu, sg[1], i - i_begin);
            const int c = MODE == DISTDL_POOL_MAX ? __shfl_sync(0xffffffffu, sc[1], i - i_begin) : 0;
            Strip::put_right(g, code, x, c, j0, S.ow);
        }
#pragma unroll
        for (int a = 0; a < KH; ++a)
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int c = 0; c < SW; ++c)
#pragma unroll
                    for (int v = NJ - 1; v >= 0; --v) {
                        const int b = Strip::window(c, v);
                        if (b < 0 || b >= KW) continue;                                // compile-time
                        if (MODE == DISTDL_POOL_AVG || code[u][v] == a * KW + b) acc[a][u][c] = __fadd_rn(acc[a][u][c], g[u][v]);
                    }
        if (i >= gi0) {
#pragma unroll
            for (int r = 0; r < SH; ++r) {
                const int p = S.i0 + i * SH + r;
                if (p >= S.hlh && p < bulk_end) {
                    if (MODE == DISTDL_POOL_AVG)
#pragma unroll
                        for (int u = 0; u < NU; ++u)
#pragma unroll
                            for (int c = 0; c < SW; ++c) acc[r][u][c] = __fmul_rn(acc[r][u][c], 1.0f / (float)(KH * KW));
                    pool_store_row<SW, NU>(out, acc[r], cols, lane);
                    if (clears) out[clear_at] = 0.f;
                }
                out += S.pw;
            }
        }
#pragma unroll
        for (int a = 0; a < SLOTS; ++a)
#pragma unroll
            for (int u = 0; u < NU; ++u)
#pragma unroll
                for (int c = 0; c < SW; ++c) acc[a][u][c] = a + SH < SLOTS ? acc[a + SH < SLOTS ? a + SH : a][u][c] : 0.f;
    }
    // ghost rows above and below this strip
    const int qa = left ? 0 : S.hlw + col0 * SW, qb = right ? S.pw : S.hlw + col0 * SW + cols;
    if (first_row == 0)
        for (int p = 0; p < S.hlh; ++p)
            for (int q = qa + lane; q < qb; q += 32) shard[(size_t)p * S.pw + q] = 0.f;
    if (S.i0 + (gi0 + rows) * SH >= bulk_end)
        for (int p = bulk_end; p < S.ph; ++p)
            for (int q = qa + lane; q < qb; q += 32) shard[(size_t)p * S.pw + q] = 0.f;
}

template <int KH, int KW, int SH, int SW, int MODE, int NU>
__global__ void __launch_bounds__(kPoolThreadsX *kPoolThreadsY, 4)
pool_adj_fused(const __grid_constant__ PoolParams P, int tiles_x, int tiles_y, int rows) {
    stream_enter();
    const PoolShard &S = P.s[blockIdx.y];
    int rest = blockIdx.x;
    const int tx = rest % tiles_x;
    rest /= tiles_x;
    const int ty = rest % tiles_y;
    const int plane = rest / tiles_y;
    const int first_row = (ty * kPoolThreadsY + (int)threadIdx.y) * rows, col0 = tx * (32 * NU);
    const int shift = S.hlw - S.j0 - SW * div_floor(S.hlw - S.j0, SW);
    if (SW == 1 || shift == 0) pool_adj_strip<KH, KW, SH, SW, MODE, 0, NU>(P, blockIdx.y, plane, first_row, rows, col0, threadIdx.x);
    else pool_adj_strip<KH, KW, SH, SW, MODE, SW - 1, NU>(P, blockIdx.y, plane, first_row, rows, col0, threadIdx.x);
}

// Adjoint of the local layer alone (H* follows), where a shard meets more than a column of a neighbour's outputs or the images are small and many: a
// lane owns the SH x SW cells {i0 + SH * gi + r, j0 + SW * gj + c} of a group and marches down gi.  The outputs whose window holds cell (r, c) of the
// group are (gi - t, gj - v) with window positions a = r + t * SH < KH, b = c + v * SW < KW, all known at compile time; the outputs (gi - t, .) of the
// rows above stay in registers, and every cell picks its terms (ascending output order = descending t, v).
template <int KH, int KW, int SH, int SW, int MODE>
__global__ void __launch_bounds__(kPoolThreadsX *kPoolThreadsY)
pool_adj_fixed(const __grid_constant__ PoolParams P, int tiles_x, int tiles_y, int rows) {
    stream_enter();
    const PoolShard &S = P.s[blockIdx.y];
    int rest = blockIdx.x;
    const int tx = rest % tiles_x;
    rest /= tiles_x;
    const int ty = rest % tiles_y;
    const int plane = rest / tiles_y;
    constexpr int NI = (KH + SH - 1) / SH, NJ = (KW + SW - 1) / SW;
    // the first group holds padded row / column 0
    const int gi0 = div_floor(-S.i0, SH) + (ty * kPoolThreadsY + (int)threadIdx.y) * rows;
    const int gj0 = div_floor(-S.j0, SW) + tx * (32 * kPoolCols) + (int)threadIdx.x;
    if (S.i0 + gi0 * SH >= S.ph) return;
    const float *dy = S.in + (size_t)plane * S.oh * S.ow;
    const int32_t *arg = MODE == DISTDL_POOL_MAX ? S.arg + (size_t)plane * S.oh * S.ow : nullptr;
    float *out = S.out + ((size_t)plane * S.ph + (S.i0 + gi0 * SH)) * S.pw + (S.j0 + gj0 * SW);
    bool jok[kPoolCols][NJ], cok[kPoolCols][SW];
#pragma unroll
    for (int u = 0; u < kPoolCols; ++u) {
        const int gj = gj0 + 32 * u;
#pragma unroll
        for (int v = 0; v < NJ; ++v) jok[u][v] = (unsigned)(gj - v) < (unsigned)S.ow;
#pragma unroll
        for (int c = 0; c < SW; ++c) cok[u][c] = (unsigned)(S.j0 + gj * SW + c) < (unsigned)S.pw;
    }
    // MAX: recorded position, -1 for an absent output;  AVG: 0 present, -1 absent
    float g[NI][kPoolCols][NJ], gn[kPoolCols][NJ];
    int code[NI][kPoolCols][NJ], cn[kPoolCols][NJ];
    auto load = [&](int i, float (&gv)[kPoolCols][NJ], int (&cv)[kPoolCols][NJ]) {
        const bool ok = (unsigned)i < (unsigned)S.oh;
        const int o = i * S.ow + gj0;
#pragma unroll
        for (int u = 0; u < kPoolCols; ++u)
#pragma unroll
            for (int v = 0; v < NJ; ++v) {
                gv[u][v] = 0.f;
                cv[u][v] = -1;
                if (ok && jok[u][v]) {
                    gv[u][v] = __ldg(dy + o + (32 * u - v));
                    cv[u][v] = MODE == DISTDL_POOL_MAX ? __ldg(arg + o + (32 * u - v)) : 0;
                }
            }
    };
#pragma unroll
    for (int t = 1; t < NI; ++t) load(gi0 - t, g[t], code[t]);
    load(gi0, gn, cn);
    for (int gi = gi0; gi < gi0 + rows; ++gi) {
        const int p0 = S.i0 + gi * SH;
        if (p0 >= S.ph) break;
#pragma unroll
        for (int u = 0; u < kPoolCols; ++u)
#pragma unroll
            for (int v = 0; v < NJ; ++v) {
                g[0][u][v] = gn[u][v];
                code[0][u][v] = cn[u][v];
            }
        if (gi + 1 < gi0 + rows) load(gi + 1, gn, cn);
#pragma unroll
        for (int r = 0; r < SH; ++r) {
            if ((unsigned)(p0 + r) < (unsigned)S.ph) {
#pragma unroll
                for (int u = 0; u < kPoolCols; ++u)
#pragma unroll
                    for (int c = 0; c < SW; ++c) {
                        float acc = 0.f;
#pragma unroll
                        for (int t = NI - 1; t >= 0; --t)
#pragma unroll
                            for (int v = NJ - 1; v >= 0; --v) {
                                if (r + t * SH >= KH || c + v * SW >= KW) continue;      // compile-time
                                const bool take = code[t][u][v] == (MODE == DISTDL_POOL_AVG ? 0 : (r + t * SH) * KW + (c + v * SW));
                                if (take) acc = __fadd_rn(acc, g[t][u][v]);
                            }
                        if (MODE == DISTDL_POOL_AVG) acc = __fmul_rn(acc, 1.0f / (float)(KH * KW));
                        if (cok[u][c]) out[32 * SW * u + c] = acc;
                    }
            }
            out += S.pw;
        }
#pragma unroll
        for (int t = NI - 1; t > 0; --t)
#pragma unroll
            for (int u = 0; u < kPoolCols; ++u)
#pragma unroll
                for (int v = 0; v < NJ; ++v) {
                    g[t][u][v] = g[t - 1][u][v];
                    code[t][u][v] = code[t - 1][u][v];
                }
    }
}

template <int KH, int KW, int SH, int SW>
static void launch_pool_fixed(const PoolParams &P, dim3 grid, dim3 block, int tiles_x, int tiles_y, int rows, bool adjoint, bool fused, int nu, cudaStream_t s) {
    const auto run = [&](auto kernel) { launch_in_stream(kernel, grid, block, 0, s, P, tiles_x, tiles_y, rows); };
    constexpr int AVG = DISTDL_POOL_AVG, MAX = DISTDL_POOL_MAX;
    const bool avg = P.mode == AVG;
    if (!adjoint) avg ? run(pool_fwd_fixed<KH, KW, SH, SW, AVG>) : run(pool_fwd_fixed<KH, KW, SH, SW, MAX>);
    else if (fused && nu == 1) avg ? run(pool_adj_fused<KH, KW, SH, SW, AVG, 1>) : run(pool_adj_fused<KH, KW, SH, SW, MAX, 1>);
    else if (fused) avg ? run(pool_adj_fused<KH, KW, SH, SW, AVG, 2>) : run(pool_adj_fused<KH, KW, SH, SW, MAX, 2>);
    else avg ? run(pool_adj_fixed<KH, KW, SH, SW, AVG>) : run(pool_adj_fixed<KH, KW, SH, SW, MAX>);
}

struct PoolDim {
    std::vector<int64_t> out_start, out_size;
    std::vector<int32_t> hlo, hhi;
};

static distdl_status_t pool_dim(int64_t n, int32_t p, int32_t k, int32_t s, int32_t pad_lo, int32_t pad_hi, PoolDim &d,
                                const char *what) {
    d.hlo.resize(p);
    d.hhi.resize(p);
    const distdl_status_t st = distdl_halo_widths_1d(n, p, k, s, 1, pad_lo, pad_hi, d.hlo.data(), d.hhi.data(), nullptr, nullptr);
    if (st != DISTDL_OK) return st;
    const int64_t m = (n + pad_lo + pad_hi - k) / s + 1;
    const int64_t q = m / p, r = m % p;
    d.out_start.resize(p);
    d.out_size.resize(p);
    int64_t at = 0;
    for (int32_t c = 0; c < p; ++c) {
        d.out_size[c] = q + (c < r ? 1 : 0);
        d.out_start[c] = at;
        at += d.out_size[c];
    }
    (void)what;
    return DISTDL_OK;
}

// A layer's geometry and kernel; the shards' addresses are filled in by the call.
struct PoolPlan {
    PoolParams P;
    int fixed;                       // which of the compile-time variants, 0: the general kernels
    bool fusable;                    // the adjoint's kernel can have H* in it
    int64_t max_rows, max_cols;      // of the largest shard: outputs, of the adjoint padded cells
};

static distdl_status_t pool_plan(const distdl_partition *p, int32_t kh, int32_t kw, int32_t sh, int32_t sw, int32_t plh, int32_t phh,
                                 int32_t plw, int32_t phw, int32_t mode, bool adjoint, const char *what, PoolPlan &plan) {
    if (p->rank != 4 || p->dtype != DISTDL_F32) return fail(DISTDL_ERR_SHAPE, "%s: needs a rank-4 F32 partition", what);
    if (p->any_periodic()) return fail(DISTDL_ERR_UNSUPPORTED, "%s: periodic partitions are not supported by the fused layers", what);
    if (p->pshape[0] != 1 || p->pshape[1] != 1)
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: only the feature-space dimensions may be partitioned", what);
    if (p->num_workers > kPoolMaxWorkers) return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d workers", what, kPoolMaxWorkers);
    if (mode != DISTDL_POOL_AVG && mode != DISTDL_POOL_MAX) return fail(DISTDL_ERR_INVALID_ARG, "%s: bad mode", what);
    if (kh < 1 || kw < 1 || sh < 1 || sw < 1 || plh < 0 || phh < 0 || plw < 0 || phw < 0)
        return fail(DISTDL_ERR_INVALID_ARG, "%s: bad kernel, stride or padding", what);
    if (kh > 16 || kw > 16) return fail(DISTDL_ERR_UNSUPPORTED, "%s: kernels beyond 16 x 16", what);
    PoolDim dh, dw;
    distdl_status_t st = pool_dim(p->global_shape[2], p->pshape[2], kh, sh, plh, phh, dh, what);
    if (st != DISTDL_OK) return st;
    st = pool_dim(p->global_shape[3], p->pshape[3], kw, sw, plw, phw, dw, what);
    if (st != DISTDL_OK) return st;
    for (int32_t c = 0; c < p->pshape[2]; ++c)
        if (p->hlo[2][c] != dh.hlo[c] || p->hhi[2][c] != dh.hhi[c])
            return fail(DISTDL_ERR_SHAPE, "%s: ghost rows of worker row %d are (%d, %d), this kernel needs (%d, %d)", what, c,
                        p->hlo[2][c], p->hhi[2][c], dh.hlo[c], dh.hhi[c]);
    for (int32_t c = 0; c < p->pshape[3]; ++c)
        if (p->hlo[3][c] != dw.hlo[c] || p->hhi[3][c] != dw.hhi[c])
            return fail(DISTDL_ERR_SHAPE, "%s: ghost columns of worker column %d are (%d, %d), this kernel needs (%d, %d)", what,
                        c, p->hlo[3][c], p->hhi[3][c], dw.hlo[c], dw.hhi[c]);
    for (int k = 0; k < 2; ++k)
        if (p->hlo[k][0] != 0 || p->hhi[k][0] != 0) return fail(DISTDL_ERR_SHAPE, "%s: ghosts along batch or channels", what);

    PoolParams &P = plan.P;
    memset(&P, 0, sizeof(P));
    P.planes = (int32_t)(p->global_shape[0] * p->global_shape[1]);
    P.kh = kh;
    P.kw = kw;
    P.sh = sh;
    P.sw = sw;
    P.hg = (int32_t)p->global_shape[2];
    P.wg = (int32_t)p->global_shape[3];
    P.mode = mode;
    P.wrows = p->pshape[2];
    P.wcols = p->pshape[3];
    int64_t &max_rows = plan.max_rows, &max_cols = plan.max_cols;
    max_rows = max_cols = 0;
    // the compile-time variants
    const int fixed = plan.fixed = (kh == 2 && kw == 2 && sh == 2 && sw == 2) ? 1 : (kh == 3 && kw == 3 && sh == 2 && sw == 2) ? 2
                                 : (kh == 3 && kw == 3 && sh == 1 && sw == 1) ? 3 : 0;
    // the adjoint with H* in it: where there is an H* (a ghost anywhere)
    bool fused = fixed && adjoint && !p->adj_host.tiles.empty();
    for (int32_t w = 0; w < p->num_workers; ++w) {
        const int32_t r = w / p->pshape[3], c = w % p->pshape[3];
        PoolShard &S = P.s[w];
        S.ph = (int32_t)p->padded_extent(2, r);
        S.pw = (int32_t)p->padded_extent(3, c);
        S.oh = (int32_t)dh.out_size[r];
        S.ow = (int32_t)dw.out_size[c];
        S.g0h = (int32_t)(p->start[2][r] - p->hlo[2][r]);
        S.g0w = (int32_t)(p->start[3][c] - p->hlo[3][c]);
        S.hlh = p->hlo[2][r];
        S.hlw = p->hlo[3][c];
        S.bh = (int32_t)p->size[2][r];
        S.bw = (int32_t)p->size[3][c];
        S.i0 = (int32_t)(dh.out_start[r] * sh - plh - S.g0h);
        S.j0 = (int32_t)(dw.out_start[c] * sw - plw - S.g0w);
        if (S.oh > 0 && (S.i0 < 0 || S.i0 + (int64_t)(S.oh - 1) * sh + kh > S.ph))
            return fail(DISTDL_ERR_SHAPE, "%s: worker row %d does not hold the inputs of its outputs", what, r);
        if (S.ow > 0 && (S.j0 < 0 || S.j0 + (int64_t)(S.ow - 1) * sw + kw > S.pw))
            return fail(DISTDL_ERR_SHAPE, "%s: worker column %d does not hold the inputs of its outputs", what, c);
        max_rows = std::max<int64_t>(max_rows, adjoint ? S.ph : S.oh);
        max_cols = std::max<int64_t>(max_cols, adjoint ? S.pw : S.ow);
        // it hands one column of the neighbours' outputs on either side from lane to lane, and a lane clears one ghost cell a row
        fused = fused && S.oh >= 1 && S.ow >= kw && S.hlw <= 16 && S.pw - S.hlw - S.bw <= 16 &&
                (c == 0 || div_floor(S.hlw - S.j0 - kw + sw, sw) >= -1) && (c + 1 == p->pshape[3] || div_floor(S.hlw + S.bw - 1 - S.j0, sw) <= S.ow);
    }
    plan.fusable = fused;
    return DISTDL_OK;
}

// Rows and columns of what the threads walk, and the launch over them.
struct PoolLaunch {
    int64_t max_rows, max_cols;      // threads' cells or outputs (general), lanes' (fixed), groups (adjoint, fixed)
    int nu;                          // columns (adjoint: of groups) per lane
    int rows, tiles_x, tiles_y;      // rows per warp (fixed) or thread; tiles per plane
};

static PoolLaunch pool_launch(const PoolPlan &plan, int32_t workers, bool adjoint, bool fused, int sms) {
    const PoolParams &P = plan.P;
    const int fixed = plan.fixed;
    PoolLaunch L;
    int64_t &max_rows = L.max_rows, &max_cols = L.max_cols;
    max_rows = plan.max_rows;
    max_cols = plan.max_cols;
    if (fixed && adjoint && !fused) {
        // groups of sh x sw cells; the group lattice starts up to one group before cell 0
        max_rows = max_rows / P.sh + 2;
        max_cols = max_cols / P.sw + 2;
    } else if (fixed && adjoint) {
        // groups of sh x sw bulk cells, the first row of groups may begin above the bulk
        max_rows = max_cols = 0;
        for (int32_t w = 0; w < workers; ++w) {
            const PoolShard &S = P.s[w];
            max_rows = std::max<int64_t>(max_rows, div_floor(S.hlh + S.bh - 1 - S.i0, P.sh) - div_floor(S.hlh - S.i0, P.sh) + 1);
            max_cols = std::max<int64_t>(max_cols, (S.bw + P.sw - 1) / P.sw);
        }
    }
    // the compile-time variants: 64 (or 32) columns and up to 16 rows (20 of the fused adjoint) per warp, fewer where eight warps would leave some without a row
    // or an SM would have fewer than 16 warps
    L.nu = fused && max_cols <= 32 ? 1 : kPoolCols;
    const int cols = fixed ? 32 * L.nu : kPoolThreadsX;
    L.tiles_x = (int)((max_cols + cols - 1) / cols);
    L.rows = 1;
    if (fixed) {
        const int64_t all = (int64_t)workers * P.planes * L.tiles_x * max_rows;      // rows of 64 columns
        L.rows = (int)std::min<int64_t>(fused ? 20 : 16, std::max<int64_t>(2, std::min((max_rows + kPoolThreadsY - 1) / kPoolThreadsY, all / (16 * sms))));
    }
    L.tiles_y = (int)((max_rows + kPoolThreadsY * L.rows - 1) / (kPoolThreadsY * L.rows));
    if (fixed) L.rows = (int)((max_rows + kPoolThreadsY * L.tiles_y - 1) / (kPoolThreadsY * L.tiles_y));      // equal shares
    return L;
}

// Whether the adjoint with H* in it is the faster one.  It saves H*'s launch (3 us) and passes over cells and ghosts, but a warp takes about 0.3 ns of
// the device longer to begin: where it finds its neighbours' outputs, the column beside the shard, the ghosts to clear.  So small images in large
// batches, whose warps have two or three rows each, are for the two kernels.  Fitted to 830 layers (both ways timed, calls back to back, 0.1 to 24 M cells, 8 to 8192 planes
// of 10 to 1024 rows and columns on up to 4 x 4 workers): within 0.6 % of the better way on average, where fusing
// nearly all of them was 8 % behind.
//   2 x 2 / 2 avg, 1024 x 16 x 14 x 14 on 1 x 2 workers fused 59.6, two kernels 27.5 us;   4096 x 62 x 62 on 2 x 2 81 / 52;   64 x 258 x 258 on 4 x 4 10.5 / 12.1
//   2 x 2 / 2 max, 1024 x 62 x 62 on 2 x 2 25.2 / 17.6;   192 x 362 x 358 on 2 x 3 36.1 / 39.5
//   3 x 3 / 2 max, 4096 x 62 x 62 on 2 x 2 105 / 77;   192 x 362 x 358 on 2 x 3 38.2 / 47.6
//   3 x 3 / 1 avg, 4096 x 30 x 30 on 2 x 2 91.7 / 86.9;   512 x 126 x 126 on 2 x 2 33.7 / 68.3
static bool pool_fused_pays(const PoolPlan &plan, int32_t workers, const PoolLaunch &L, int sms) {
    const PoolParams &P = plan.P;
    const int64_t warps = (int64_t)workers * P.planes * L.tiles_x * ((L.max_rows + L.rows - 1) / L.rows);
    const int64_t cells = (int64_t)P.planes * P.hg * P.wg, beside = (int64_t)P.planes * (P.wcols - 1) * P.hg;      // rows that meet a shard end
    int64_t limit = (int64_t)sms * 74;
    if (plan.fixed == 3) limit = (int64_t)sms * 100 + cells / 160 + beside / 4;
    else if (plan.fixed == 2) limit += cells / 600 + beside / 40;
    else if (P.mode == DISTDL_POOL_AVG) limit += cells / 1600;
    return warps < limit;
}

// terms[k * q + b]: output column (counted from the shard's own) that the adjoint with H* in it adds to bulk column q as window column b.
template <int KW, int SW, int DW, int NU>
static void pool_column_terms(const PoolShard &S, int wc, int wcols, int32_t *terms) {
    using Strip = PoolStrip<KW, SW, DW, NU>;
    constexpr int kNone = INT_MIN;
    for (int col0 = 0; col0 * SW < S.bw; col0 += 32 * NU) {
        for (int lane = 0; lane < 32; ++lane) {
            const Strip strip(S, wc, wcols, col0, lane);
            const int newest = strip.newest;
            int g[NU][Strip::NJ], code[NU][Strip::NJ];
            for (int u = 0; u < NU; ++u)
                for (int v = 0; v < Strip::NJ; ++v) g[u][v] = (unsigned)(newest + 32 * u - v) < (unsigned)S.ow ? newest + 32 * u - v : kNone;
            if (strip.left) Strip::put_left(g, code, -1, 0, newest);
            if (strip.right) Strip::put_right(g, code, S.ow, 0, newest, S.ow);
            for (int u = 0; u < NU; ++u)
                for (int c = 0; c < SW; ++c)
                    for (int v = 0; v < Strip::NJ; ++v) {
                        const int cell = SW * (lane + 32 * u) + c, b = Strip::window(c, v);
                        if (cell < strip.cols && b >= 0 && b < KW) terms[KW * (SW * col0 + cell) + b] = g[u][v];
                    }
        }
    }
}
template <int KW, int SW>
static void pool_column_terms(const PoolShard &S, int wc, int wcols, int nu, int32_t *terms) {
    if (SW == 1 || (S.hlw - S.j0 - SW * div_floor(S.hlw - S.j0, SW)) == 0)
        nu == 1 ? pool_column_terms<KW, SW, 0, 1>(S, wc, wcols, terms) : pool_column_terms<KW, SW, 0, 2>(S, wc, wcols, terms);
    else
        nu == 1 ? pool_column_terms<KW, SW, SW - 1, 1>(S, wc, wcols, terms) : pool_column_terms<KW, SW, SW - 1, 2>(S, wc, wcols, terms);
}

static distdl_status_t pool_impl(const distdl_partition *p, const void *const *in, void *const *out, void *const *arg,
                                 int32_t kh, int32_t kw, int32_t sh, int32_t sw, int32_t plh, int32_t phh, int32_t plw,
                                 int32_t phw, int32_t mode, void *stream, bool adjoint, const char *what) {
    clear_error();
    if (!p || !in || !out) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL argument", what);
    PoolPlan plan;
    distdl_status_t st = pool_plan(p, kh, kw, sh, sw, plh, phh, plw, phw, mode, adjoint, what, plan);
    if (st != DISTDL_OK) return st;
    if (mode == DISTDL_POOL_MAX && adjoint && !arg) return fail(DISTDL_ERR_INVALID_ARG, "%s: max pooling needs argmax", what);
    PoolParams &P = plan.P;
    for (int32_t w = 0; w < p->num_workers; ++w) {
        PoolShard &S = P.s[w];
        if (!in[w] || !out[w]) return fail(DISTDL_ERR_INVALID_ARG, "%s: shard pointer %d is NULL", what, w);
        S.in = (const float *)in[w];
        S.out = (float *)out[w];
        S.arg = arg ? (int32_t *)arg[w] : nullptr;
        if (mode == DISTDL_POOL_MAX && adjoint && !S.arg) return fail(DISTDL_ERR_INVALID_ARG, "%s: argmax[%d] is NULL", what, w);
    }
    // H and H* work on the padded shards: what they ask of them holds for the layer as well
    st = halo_check_shards(p, adjoint ? out : const_cast<void *const *>(reinterpret_cast<const void *const *>(in)), what);
    if (st != DISTDL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int fixed = plan.fixed;
    int sms = 0;
    if (fixed) {
        int dev = 0;
        DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
        DISTDL_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    }
    bool fused = plan.fusable;
    PoolLaunch L = pool_launch(plan, p->num_workers, adjoint, fused, sms);
    if (fused && !pool_fused_pays(plan, p->num_workers, L, sms)) {
        fused = false;
        L = pool_launch(plan, p->num_workers, adjoint, fused, sms);
    }
    const int rows = L.rows, tiles_x = L.tiles_x, tiles_y = L.tiles_y, nu = L.nu;
    const int64_t blocks = (int64_t)tiles_x * tiles_y * P.planes;
    if (blocks >= ((int64_t)1 << 31)) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles", what);
    const dim3 grid((unsigned)blocks, (unsigned)p->num_workers), block(kPoolThreadsX, kPoolThreadsY);
    if (!adjoint) {
        // H in place on the padded input, then the local layer
        st = distdl_halo_fwd(p, const_cast<void *const *>(reinterpret_cast<const void *const *>(in)), stream);
        if (st != DISTDL_OK) return st;
    }
    if (blocks > 0) {
        if (fixed == 1) launch_pool_fixed<2, 2, 2, 2>(P, grid, block, tiles_x, tiles_y, rows, adjoint, fused, nu, s);
        else if (fixed == 2) launch_pool_fixed<3, 3, 2, 2>(P, grid, block, tiles_x, tiles_y, rows, adjoint, fused, nu, s);
        else if (fixed == 3) launch_pool_fixed<3, 3, 1, 1>(P, grid, block, tiles_x, tiles_y, rows, adjoint, fused, nu, s);
        else if (!adjoint) launch_in_stream(pool_fwd_kernel, grid, block, 0, s, P, tiles_x, tiles_y);
        else launch_in_stream(pool_adj_kernel, grid, block, 0, s, P, tiles_x, tiles_y);
    }
    DISTDL_CUDA_CHECK(cudaGetLastError());
    if (!adjoint || fused) return DISTDL_OK;
    return distdl_halo_adj(p, out, stream);
}

}  // namespace distdl

extern "C" distdl_status_t distdl_pool_fwd(const distdl_partition_t *p, void *const *x, int32_t kh, int32_t kw, int32_t sh,
                                           int32_t sw, int32_t pad_h_lo, int32_t pad_h_hi, int32_t pad_w_lo,
                                           int32_t pad_w_hi, int32_t mode, void *const *y, void *const *argmax,
                                           void *stream) {
    return distdl::pool_impl(p, reinterpret_cast<const void *const *>(x), y, argmax, kh, kw, sh, sw, pad_h_lo, pad_h_hi,
                             pad_w_lo, pad_w_hi, mode, stream, false, "pool_fwd");
}

extern "C" distdl_status_t distdl_pool_adj(const distdl_partition_t *p, const void *const *dy, const void *const *argmax,
                                           int32_t kh, int32_t kw, int32_t sh, int32_t sw, int32_t pad_h_lo,
                                           int32_t pad_h_hi, int32_t pad_w_lo, int32_t pad_w_hi, int32_t mode,
                                           void *const *dx, void *stream) {
    // the positions are only read here; pool_impl shares one pointer type with the forward call
    return distdl::pool_impl(p, dy, dx, (void *const *)argmax, kh, kw, sh, sw, pad_h_lo, pad_h_hi, pad_w_lo, pad_w_hi, mode,
                             stream, true, "pool_adj");
}

// Which outputs the adjoint with H* in it adds to the rows (dim 0) or columns (dim 1) of a worker's bulk, by the rules of the kernel.
extern "C" distdl_status_t distdl_selftest_pool_adj_terms(const distdl_partition_t *p, int32_t k, int32_t stride, int32_t pad_lo, int32_t pad_hi,
                                                          int32_t mode, int32_t worker, int32_t dim, int32_t *fused, int32_t *terms, int32_t num_terms) {
    using namespace distdl;
    clear_error();
    const char *what = "selftest_pool_adj_terms";
    if (!p || !fused || !terms || worker < 0 || worker >= p->num_workers || dim < 0 || dim > 1) return fail(DISTDL_ERR_INVALID_ARG, "%s: bad argument", what);
    PoolPlan plan;
    const distdl_status_t st = pool_plan(p, k, k, stride, stride, pad_lo, pad_hi, pad_lo, pad_hi, mode, true, what, plan);
    if (st != DISTDL_OK) return st;
    *fused = 0;
    if (!plan.fusable) return DISTDL_OK;
    const int sms = 148;                                        // a B200's
    const PoolLaunch launch = pool_launch(plan, p->num_workers, true, true, sms);
    const int nu = launch.nu;
    *fused = pool_fused_pays(plan, p->num_workers, launch, sms) ? 2 : 1;
    const PoolParams &P = plan.P;
    const PoolShard &S = P.s[worker];
    const int wr = worker / P.wcols, wc = worker % P.wcols, cells = dim ? S.bw : S.bh;
    if (num_terms < k * cells) return fail(DISTDL_ERR_INVALID_ARG, "%s: need %d terms", what, k * cells);
    for (int i = 0; i < k * cells; ++i) terms[i] = -1;
    std::vector<int32_t> own(dim ? k * cells : 0, INT_MIN);
    if (dim) {
        if (plan.fixed == 1) pool_column_terms<2, 2>(S, wc, P.wcols, nu, own.data());
        else if (plan.fixed == 2) pool_column_terms<3, 2>(S, wc, P.wcols, nu, own.data());
        else pool_column_terms<3, 1>(S, wc, P.wcols, nu, own.data());
    }
    std::vector<int32_t> first(dim ? P.wcols : P.wrows, 0);          // outputs of the workers before each
    for (size_t w = 1; w < first.size(); ++w) first[w] = first[w - 1] + (dim ? P.s[w - 1].ow : P.s[(w - 1) * P.wcols].oh);
    if (dim) {
        for (int i = 0; i < k * cells; ++i)
            if (own[i] != INT_MIN) terms[i] = first[wc] + own[i];
    } else {
        // cell row p is a = p - i0 - i * stride rows into the windows of output row i
        for (int q = 0; q < cells; ++q)
            for (int a = (S.hlh + q - S.i0) - stride * div_floor(S.hlh + q - S.i0, stride); a < k; a += stride) {
                int dr, il;
                if (pool_row_owner(P, S, worker, wr, div_floor(S.hlh + q - S.i0 - a, stride), dr, il)) terms[k * q + a] = first[wr + dr] + il;
            }
    }
    return DISTDL_OK;
}
