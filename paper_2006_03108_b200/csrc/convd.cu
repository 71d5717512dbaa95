// Distributed depthwise convolution layer on a feature-space partition (Section 4, "Sparse
// layers"): forward = halo exchange H followed by the local sliding-kernel layer, adjoint =
// local adjoint followed by H*.  Both are fused: the rows a warp works on are staged in shared
// memory straight from the bulk of whichever shard owns them (or zeros outside the tensor), so ghost
// data never makes a round trip through device memory.  The adjoint is evaluated in gather form (a
// correlation of dy with the kernel rotated by 180 degrees), which equals "scatter locally, then add
// the ghosts into the neighbours' bulk" without any atomics, and it leaves the ghosts of dx zero as
// H* does.  The parameter gradients (adjoint convolution algorithm) use the same staging:
//   dw^_k[c,a,b] = sum_{n,i,j} dy_k[n,c,i,j] * (H x)_k[n,c,i+a,j+b],   db^_k[c] = sum dy_k[n,c,i,j],
//   dw = R_k dw^_k,  db = R_k db^_k      (every worker holds a copy of the kernel).
//
// Every warp works alone: it owns a strip of 32 * NC columns and a segment of rows of one plane of one
// shard and marches down the rows.  Rows arrive in a ring of its own, by one bulk copy per row, a group
// of rows ahead; a block never meets at a barrier.  A bulk copy wants both addresses on 16-byte
// boundaries and no more: a row starts in the ring at the same offset from such a boundary as in device
// memory, so any row pitch is as good as another.  Lane l reads columns l, l + 32, ... (no bank conflicts at
// any offset), a pair of columns 32 apart is one packed operand, and every input row is read once and added
// to the K output rows it belongs to (their sums rotate through registers).
//
// What bounds it: device memory (8 bytes per cell) for 3 x 3 and 5 x 5, instruction issue close behind; 5 x 5: 20 shared
// reads and 50 packed FMAs per row and four columns of a lane, about 45 other instructions, half of them done once per
// group of rows.  Measured (B200, forward / adjoint / gradients, ms; before: tiles of 32 x 128 staged by a block, bulk tensor
// copies where every row pitch allowed them):
//   3 x 3, 4 x 12 x 515 x 509 on 3 x 2 workers (odd pitches)     0.018 / 0.018 / 0.025   (0.067 / 0.069 / 0.087)
//   5 x 5, 16 x 16 x 1024 x 1024 on 4 x 4                        0.381 / 0.473 / 0.562   (0.435 / 0.503 / 0.556)
//   3 x 3,  8 x 16 x 1024 x 1024 on 4 x 4                        0.197 / 0.203 / 0.190   (0.365 / 0.199 / 0.510)
//   7 x 7,  8 x 16 x 1024 x 1024 on 4 x 4                        0.365 / 0.388 / 0.476   (0.583 / 0.453 / 1.047)
// dy read straight into registers, two rows ahead, instead of through the ring: 0.610 (5 x 5 gradients).
#include <algorithm>
#include <cstring>

#include "common.h"
#include "conv_common.h"
#include "tma.h"

namespace distdl {

constexpr int kDwWarps = 4;
constexpr int kDwThreads = 32 * kDwWarps;
// Warps of a block, forward and adjoint.  The warps work alone: blocks of one even out the multiprocessors, and no warp's place
// stays empty until its neighbours are done (5 x 5 forward / adjoint: 16 x 16 x 1024 x 1024 on 4 x 4 workers 407 / 492 -> 381 / 478 us, 4 x 16 x
// 512 x 512 on 2 x 2 36.3 / 38.4 -> 34.3 / 36.6; 7 x 7, 8 x 16 x 1024 x 1024 on 4 x 4 384 / 408 -> 370 / 389).  3 x 3, bound by memory alone, is
// faster with blocks of four (8 x 16 x 1024 x 1024 195 / 202 us, one 205 / 212; 4 x 12 x 515 x 509 on 3 x 2 17.7 / 17.8, one 20.0 / 20.5).
__host__ __device__ constexpr int dw_row_warps(int K) { return K == 3 ? kDwWarps : 1; }
constexpr uint64_t kConvWaitLimitNs = 2000000000ull;

__device__ int g_conv_status = 0;

struct DwParams {
    const float *in[kConvMaxWorkers];
    float *out[kConvMaxWorkers];            // forward / adjoint
    const float *dy[kConvMaxWorkers];       // parameter gradients
    int32_t bh[kConvMaxWorkers];            // bulk rows per worker-row coordinate
    int32_t bw[kConvMaxWorkers];            // bulk columns per worker-column coordinate
    const float *w;                         // [C, K, K]
    const float *bias;                      // [C] or nullptr
    float *partial;                         // parameter gradients: [C][slices][kGradRow]
    int32_t ph, pw, channels, planes;
    int32_t seg_rows;                       // rows of a segment
    int32_t items;                          // forward / adjoint: all; parameter gradients: of one channel
    int32_t slices;                         // parameter gradients: blocks per channel
    uint32_t zero;                          // 0, see fresh()
    FastDiv strips, pw_div, segs, ph_div, chan_div, slice_div;
};

template <int K, int NC, bool GRAD>
struct DwCfg {
    static constexpr int PH = K / 2;
    static constexpr int W = 32 * NC;                                   // columns of a strip
    // rows of a group (whole turns of the K running sums): what is done once per group is done by a lane per row; as many
    // as leave room for four blocks on an SM (7 x 7, whose weights or sums take more registers: three)
    static constexpr int G = GRAD ? (K == 3 ? 6 : K) : (K == 3 ? 12 : K == 5 ? 10 : 7);
    static constexpr int D = 2;                                         // groups in the ring
    static constexpr int PITCH = (W + 2 * PH + 3 + 3) / 4 * 4;          // a row starts up to three floats in
    static constexpr int PITCHY = (W + 3 + 3) / 4 * 4;
    static constexpr int RING = D * G * PITCH, RINGY = D * G * PITCHY, SIDE = D * G * 2 * PH;
    // per warp, in floats: rows (x, then dy), where each lane reads (three pointers), barriers, cells from the shards beside,
    // offset of every row
    static constexpr int WARP_FLOATS = (RING + (GRAD ? RINGY : 0) + 3 * 64 + 2 * D + SIDE + D * G * (GRAD ? 2 : 1) + 3) / 4 * 4;
};

__device__ __forceinline__ void dw_bulk_copy(uint32_t dst, const float *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// (w, w) pairs of one channel, in floats, whole 16-byte units
__host__ __device__ constexpr int dw_weight_floats(int K) { return (2 * K * K + 3) / 4 * 4; }

// Rows of arrays without ghosts travel in whole 16-byte blocks.  Whether the last block of a row may reach past the end of the
// array: of a plane's last row, and of any whose rows are shorter than the three cells that a block takes in beyond one (beyond a
// bulk row of a padded array lie more than three ghost cells).
__host__ __device__ inline bool dw_may_pass_end(int i, int bh, int bw) { return i == bh - 1 || bw < 3; }
// Whether the block of cells [first, first + n) does.
__host__ __device__ inline bool dw_past_end(const float *first, int n, const float *end) {
    return first + ((n + 3 + (int)((reinterpret_cast<uintptr_t>(first) >> 2) & 3)) & ~3) - (int)((reinterpret_cast<uintptr_t>(first) >> 2) & 3) > end;
}
// Cells of such a row that its whole blocks hold; the up to three behind them are copied one by one.
__host__ __device__ inline int dw_whole(const float *first, int n) {
    const int tail = (n + (int)((reinterpret_cast<uintptr_t>(first) >> 2) & 3)) & 3;
    return n > tail ? n - tail : 0;
}

// One warp's work: plane, shard (r, c), first row and column, rows and columns of the segment.
struct DwItem {
    int plane, r, c, i0, j0, rows, cols;
    bool valid;
};

// strip fastest, then worker column, segment, worker row, plane: warps that run together work on neighbouring columns and
// rows, so the halo cells of one sit in lines that another has just brought into L2
__device__ __forceinline__ DwItem dw_item(const DwParams &P, uint32_t id, int W) {
    DwItem t;
    t.j0 = (int)fast_rem(P.strips, id) * W;
    t.c = (int)fast_rem(P.pw_div, id);
    t.i0 = (int)fast_rem(P.segs, id) * P.seg_rows;
    t.r = (int)fast_rem(P.ph_div, id);
    t.plane = (int)id;
    const int bh = P.bh[t.r], bw = P.bw[t.c];
    t.valid = t.i0 < bh && t.j0 < bw;
    t.rows = min(P.seg_rows, bh - t.i0);
    t.cols = min(W, bw - t.j0);
    return t;
}

// Ring of rows of one warp.  Group g holds input rows g * G ... of the item (row t = bulk row i0 - PH + t) and, for the
// parameter gradients, dy rows g * G ... (bulk row i0 + t).
// IO: ghost width of the input layout.
template <int K, int NC, int IO, bool GRAD>
struct DwRing {
    using C = DwCfg<K, NC, GRAD>;
    float *x, *y, *side;
    // of this lane: first cell of row (i0 - PH + lane) (lanes 16 on, gradients: dy row i0 + lane - 16), and of that column left /
    // right of the shard that issue_side() gives it, as if the rows went on above and below the shard; in shared memory
    const float **from;
    int *off, *offy;                        // float offset of tile column 0 inside the row's slot, -1: a row of zeros
    uint32_t bars;
    uint32_t phases;

    __device__ __forceinline__ void init(float *mem, int lane) {
        x = mem;
        y = x + C::RING;
        from = reinterpret_cast<const float **>(y + (GRAD ? C::RINGY : 0));
        bars = smem_u32(from + 96);
        side = reinterpret_cast<float *>(from + 96 + C::D);
        off = reinterpret_cast<int *>(side + C::SIDE);
        offy = off + C::D * C::G;
        phases = 0;
        if (lane == 0) {
            for (int d = 0; d < C::D; ++d) mbar_init(bars + 8 * d, GRAD ? 2 * C::G : C::G);
            fence_barrier_init();
        }
        __syncwarp();
    }

    __device__ __forceinline__ const float *cell(const DwParams &P, const DwItem &t, int r, int c, int i, int j) {
        const int pitch = P.bw[c] + 2 * IO;
        return P.in[r * P.pw + c] + (size_t)t.plane * (uint32_t)((P.bh[r] + 2 * IO) * pitch) + ((i + IO) * pitch + IO + j);
    }
    // Pointers of an item's first group.
    __device__ __forceinline__ void begin(const DwParams &P, const DwItem &t, int lane) {
        const float *f = cell(P, t, t.r, t.c, t.i0 - C::PH + lane, max(t.j0 - C::PH, 0));
        if (GRAD && lane >= 16)
            f = P.dy[t.r * P.pw + t.c] + (size_t)t.plane * (uint32_t)(P.bh[t.r] * P.bw[t.c]) + ((t.i0 + lane - 16) * P.bw[t.c] + t.j0);
        from[lane] = f;
        const int l = lane / C::PH, q = lane - l * C::PH;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            int cc, jj;
            const bool ok = conv_owner(P.bw, P.pw, t.c, s ? t.j0 + t.cols + q : t.j0 - C::PH + q, cc, jj);
            from[32 * (1 + s) + lane] = ok && cc != t.c ? cell(P, t, t.r, cc, t.i0 - C::PH + l, jj) : nullptr;
        }
    }

    // One lane, one row: copies the cells [first, first + n) (the 16-byte blocks that hold them) so that `first` lands at
    // column `col` of slot `slot`.  Returns the offset of column 0 in the slot.
    __device__ __forceinline__ int row_copy(const float *first, int n, int col, float *slot, uint32_t bar) {
        const int m = (int)((reinterpret_cast<uintptr_t>(first) >> 2) & 3);
        const int o = (m - col) & 3;
        const uint32_t bytes = (uint32_t)((m + n + 3) & ~3) * 4u;
        mbar_expect_tx(bar, bytes);
        dw_bulk_copy(smem_u32(slot + o + col - m), first - m, bytes, bar);
        return o;
    }
    // The columns beside the shard, lane -> (row, column) of group g; s: 0 left, 1 right.
    __device__ __forceinline__ void issue_side(const DwParams &P, const DwItem &t, int g, int lane, int s) {
        const int d = g % C::D;
        const int l = lane / C::PH, q = lane - l * C::PH;
        if (lane >= C::G * C::PH) return;
        const float *f = from[32 * (1 + s) + lane];
        float *dst = side + ((d * 2 + s) * C::G + l) * C::PH + q;
        const int i = t.i0 - C::PH + g * C::G + l;
        if (f && (unsigned)i < (unsigned)P.bh[t.r]) {
            cp_async4_to(smem_u32(dst), f + g * C::G * (P.bw[t.c + 2 * s - 1] + 2 * IO));
        } else {
            // above or below the shard, outside the tensor, or (a last strip narrower than the halo of the one before it) not
            // a column beside the shard at all: then nobody asks for the zero
            int cc, jj, rr, ii;
            if (f && l + g * C::G < t.rows + K - 1 && conv_owner(P.bh, P.ph, t.r, i, rr, ii) &&
                conv_owner(P.bw, P.pw, t.c, s ? t.j0 + t.cols + q : t.j0 - C::PH + q, cc, jj))
                cp_async4_to(smem_u32(dst), cell(P, t, rr, cc, ii, jj));
            else
                *dst = 0.f;
        }
    }
    __device__ __forceinline__ void complete_side(const DwParams &P, const DwItem &t, int g, int lane, int s) {
        const int d = g % C::D;
        const int l = lane / C::PH, q = lane - l * C::PH;
        if (lane >= C::G * C::PH) return;
        const int j = s ? t.j0 + t.cols + q : t.j0 - C::PH + q;
        if (j >= 0 && j < P.bw[t.c]) return;
        const int o = off[d * C::G + l];
        if (o >= 0) x[(d * C::G + l) * C::PITCH + o + (s ? C::PH + t.cols + q : q)] = side[((d * 2 + s) * C::G + l) * C::PH + q];
    }

    __device__ __forceinline__ void issue(const DwParams &P, const DwItem &t, int g, int lane) {
        const int d = g % C::D;
        const int bw = P.bw[t.c];
        const uint32_t bar = bars + 8 * d;
        const int ja = max(t.j0 - C::PH, 0), n = min(t.j0 + t.cols + C::PH, bw) - ja, col = ja - (t.j0 - C::PH);
        fence_proxy_async();
        // Parameter gradients, a group of rows of this shard only, none of them a plane's last: one copy a lane, x and dy alike (5 x 5, 16 x 16 x
        // 1024 x 1024 577 -> 571 us, 3 x 3, 8 x 16 x 1024 x 1024 235 -> 223; nothing to gain where all rows are x: forward 381 -> 383).
        if (GRAD && t.i0 + g * C::G >= C::PH && (g + 1) * C::G <= t.rows && t.i0 + (g + 1) * C::G < P.bh[t.r] && bw >= 3) {
            const bool dy = lane >= 16;
            const int l = lane & 15;
            if (l < C::G) {
                const float *f = from[lane] + g * C::G * (dy ? bw : bw + 2 * IO);
                float *slot = dy ? y + (d * C::G + l) * C::PITCHY : x + (d * C::G + l) * C::PITCH;
                (dy ? offy : off)[d * C::G + l] = row_copy(f, dy ? t.cols : n, dy ? 0 : col, slot, bar);
            }
        } else {
            if (lane < C::G) {
                const int i = t.i0 - C::PH + g * C::G + lane;
                const float *f = from[lane] + g * C::G * (bw + 2 * IO);
                float *slot = x + (d * C::G + lane) * C::PITCH;
                int rr = t.r, ii = i;
                bool ok = true;
                if ((unsigned)i >= (unsigned)P.bh[t.r]) {
                    ok = g * C::G + lane < t.rows + K - 1 && conv_owner(P.bh, P.ph, t.r, i, rr, ii);
                    if (ok) f = cell(P, t, rr, t.c, ii, ja);
                }
                int o = -1;
                if (!ok) {
                    mbar_expect_tx(bar, 0);
                } else if (IO == 0 && dw_may_pass_end(ii, P.bh[rr], bw) &&
                           dw_past_end(f, n, P.in[rr * P.pw + t.c] + (size_t)P.planes * (uint32_t)(P.bh[rr] * bw))) {
                    // the last row of a shard (or the last few): its whole blocks at once, then up to three cells.  Cell by cell, one load
                    // after another, the lane kept a small layer waiting (3 x 3, 9 x 2 x 43 x 101 on 4 x 1 workers, adjoint / gradients 9.1 / 14.1
                    // -> 7.1 / 12.2 us).
                    const int whole = dw_whole(f, n);
                    if (whole) {
                        o = row_copy(f, whole, col, slot, bar);
                    } else {
                        mbar_expect_tx(bar, 0);
                        o = 0;
                    }
                    for (int e = whole; e < n; ++e) cp_async4_to(smem_u32(slot + o + col + e), f + e);
                } else {
                    o = row_copy(f, n, col, slot, bar);
                }
                off[d * C::G + lane] = o;
            }
            if (GRAD && lane >= 16 && lane < 16 + C::G) {
                int o = 0;
                const int l = lane - 16, i = t.i0 + g * C::G + l;
                const float *f = from[lane] + g * C::G * bw;
                float *slot = y + (d * C::G + l) * C::PITCHY;
                if (i >= t.i0 + t.rows) {
                    mbar_expect_tx(bar, 0);
                } else if (dw_may_pass_end(i, P.bh[t.r], bw) &&
                           dw_past_end(f, t.cols, P.dy[t.r * P.pw + t.c] + (size_t)P.planes * (uint32_t)(P.bh[t.r] * bw))) {
                    const int whole = dw_whole(f, t.cols);
                    if (whole) o = row_copy(f, whole, 0, slot, bar);
                    else mbar_expect_tx(bar, 0);
                    for (int e = whole; e < t.cols; ++e) cp_async4_to(smem_u32(slot + o + e), f + e);
                } else {
                    o = row_copy(f, t.cols, 0, slot, bar);
                }
                offy[d * C::G + l] = o;
            }
        }
        // cells of the shards beside this one (zeros outside the tensor)
        if (t.j0 == 0) issue_side(P, t, g, lane, 0);
        if (t.j0 + t.cols + C::PH > bw) issue_side(P, t, g, lane, 1);
    }

    // Waits for group g and completes its rows.  False (for the whole warp) if the bulk copies never arrived.
    __device__ __forceinline__ bool arrive(const DwParams &P, const DwItem &t, int g, int lane) {
        const int d = g % C::D;
        const uint32_t bar = bars + 8 * d, parity = (phases >> d) & 1u;
        bool ok = mbar_try_wait(bar, parity);
        if (!ok) {
            const uint64_t t0 = global_timer();
            while (!(ok = mbar_try_wait(bar, parity)) && global_timer() - t0 < kConvWaitLimitNs) {}
        }
        phases ^= 1u << d;
        cp_async_wait_group<C::D - 1>();
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) atomicExch(&g_conv_status, (int)DISTDL_ERR_TIMEOUT);
            const uint64_t t0 = global_timer();
            while (global_timer() - t0 < 1000000ull) {}      // copies still in flight may land
            return false;
        }
        if (t.j0 == 0) complete_side(P, t, g, lane, 0);
        if (t.j0 + t.cols + C::PH > P.bw[t.c]) complete_side(P, t, g, lane, 1);
        // rows above the first and below the last of the tensor (the first or last groups of an item)
        if ((g == 0 && t.i0 == 0) || (g + 1) * C::G > t.rows + K - 1 - C::PH) {
#pragma unroll 1
            for (int l = 0; l < C::G; ++l)
                if (off[d * C::G + l] < 0)
                    for (int e = lane; e < C::PITCH; e += 32) x[(d * C::G + l) * C::PITCH + e] = 0.f;
            __syncwarp();
            if (lane < C::G && off[d * C::G + lane] < 0) off[d * C::G + lane] = 0;
        }
        if (GRAD) {
            // dy rows and columns beyond the segment are zeros, and so is what they meet in x
            if (t.cols < C::W) {
                const int gap = C::W - t.cols;
                for (int e0 = 0; e0 < C::G * gap; e0 += 32) {
                    const int l = (e0 + lane) / gap, e = e0 + lane - l * gap;
                    if (l < C::G) {
                        y[(d * C::G + l) * C::PITCHY + offy[d * C::G + l] + t.cols + e] = 0.f;
                        x[(d * C::G + l) * C::PITCH + max(off[d * C::G + l], 0) + t.cols + 2 * C::PH + e] = 0.f;
                    }
                }
            }
            if ((g + 1) * C::G > t.rows) {
#pragma unroll 1
                for (int l = 0; l < C::G; ++l)
                    if (g * C::G + l >= t.rows)
                        for (int e = lane; e < C::PITCHY; e += 32) y[(d * C::G + l) * C::PITCHY + e] = 0.f;
            }
        }
        __syncwarp();
        return true;
    }
};

// Offset (modulo four) of tile column 0, i.e. of bulk column j0 - PH, from a 16-byte boundary when every row starts on one.
__host__ __device__ constexpr int dw_offset(int K, int io) { return (4 + io - K / 2) & 3; }

// The inputs of four neighbouring columns of a row, and of the K - 1 columns beside them, in 16-byte units; O: offset of the
// first of them in the first unit (-1: not used).  pair(e): inputs e, e + 1.
template <int K, int O>
struct DwWindow {
    static constexpr int NU = (O + 4 + K - 1 + 3) / 4;
    uint64_t P[2 * NU], Q[2 * NU - 1];          // (x[2i], x[2i+1]) as they lie, (x[2i+1], x[2i+2]) put together
    __device__ __forceinline__ void load(const float *x, uint32_t zero) {
#pragma unroll
        for (int v = 0; v < NU; ++v) {
            const ulonglong2 f = *reinterpret_cast<const ulonglong2 *>(x + 4 * v);
            P[2 * v] = f.x;
            P[2 * v + 1] = f.y;
        }
#pragma unroll
        for (int v = 0; v < 2 * NU - 1; ++v) {
            float a0, a1, b0, b1;
            unpack2(P[v], a0, a1);
            unpack2(P[v + 1], b0, b1);
            Q[v] = pack2(fresh(a1, zero), fresh(b0, zero));
        }
    }
    __device__ __forceinline__ uint64_t pair(int e) const { return ((O + e) & 1) ? Q[(O + e) / 2] : P[(O + e) / 2]; }
};
template <int K>
struct DwWindow<K, -1> {
    __device__ __forceinline__ void load(const float *, uint32_t) {}
    __device__ __forceinline__ uint64_t pair(int) const { return 0ull; }
};

// K: kernel extent (odd).  ADJ: false = forward (padded x -> bulk-shaped y), true = adjoint
// (bulk-shaped dy -> padded dx, rotated kernel, ghosts of dx cleared).
//
// VEC (NC = 4): every row of every input shard starts on a 16-byte boundary.  Then the offset of a row in the ring is the same for
// all of them, a lane owns four neighbouring columns, reads 16 bytes at a time and makes the pairs that start at an odd
// offset itself: 5 x 5 forward, two reads and six exclusive-ors instead of twenty reads per row.
template <int K, bool ADJ, int NC, bool VEC>
__global__ void __launch_bounds__(32 * dw_row_warps(K), (K == 7 ? 12 : 16) / dw_row_warps(K))
conv_rows_kernel(const __grid_constant__ DwParams P) {
    stream_enter();
    using C = DwCfg<K, NC, false>;
    constexpr int OO = ADJ ? C::PH : 0;                     // ghost width of the output layout
    extern __shared__ __align__(16) float smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t id = blockIdx.x * dw_row_warps(K) + warp;
    if (id >= (uint32_t)P.items) return;
    const DwItem t = dw_item(P, id, C::W);
    if (!t.valid) return;

    DwRing<K, NC, ADJ ? 0 : C::PH, false> ring;
    ring.init(smem + warp * (C::WARP_FLOATS + dw_weight_floats(K)), lane);
    // (w, w) pairs of this channel, [column b][row a]
    uint64_t *wp = reinterpret_cast<uint64_t *>(smem + warp * (C::WARP_FLOATS + dw_weight_floats(K)) + C::WARP_FLOATS);
    uint32_t ch = (uint32_t)t.plane;
    ch = fast_rem(P.chan_div, ch);
    const int nr = t.rows + K - 1, ng = (nr + C::G - 1) / C::G;
    ring.begin(P, t, lane);
#pragma unroll
    for (int g = 0; g < C::D - 1; ++g) {
        if (g < ng) ring.issue(P, t, g, lane);
        cp_async_commit();
    }
    for (int e = lane; e < K * K; e += 32) {
        const int a = e / K, b = e - a * K;
        const float w = __ldg(P.w + (size_t)ch * K * K + (ADJ ? K * K - 1 - e : e));      // adjoint: rotated
        wp[b * K + a] = pack2(w, w);
    }
    const float bias = !ADJ && P.bias ? __ldg(P.bias + ch) : 0.f;
    const uint64_t bias2 = pack2(bias, bias);
    __syncwarp();
    uint64_t w[K][K];
#pragma unroll
    for (int b = 0; b < K; ++b)
#pragma unroll
        for (int a = 0; a < K; ++a) w[b][a] = wp[b * K + a];

    const int bh = P.bh[t.r], bw = P.bw[t.c];
    const int pitch = bw + 2 * OO;
    float *plane = P.out[t.r * P.pw + t.c] + (size_t)t.plane * (bh + 2 * OO) * pitch;
    float *out = plane + (size_t)(t.i0 + OO) * pitch + (OO + t.j0 + (VEC ? 4 : 1) * lane);
    const bool first_col = ADJ && t.j0 == 0, last_col = ADJ && t.j0 + t.cols == bw;

    bool in[NC];
#pragma unroll
    for (int p = 0; p < NC; ++p) in[p] = (VEC ? 4 * lane + p : lane + 32 * p) < t.cols;
    const uint32_t zero = P.zero;
    uint64_t acc[K][NC / 2];                                // sums of output row o: slot o % K
#pragma unroll
    for (int s = 0; s < K; ++s)
#pragma unroll
        for (int p = 0; p < NC / 2; ++p) acc[s][p] = bias2;
    for (int g = 0; g < ng; ++g) {
        __syncwarp();                                       // the slot about to be refilled has been read
        if (g + C::D - 1 < ng) ring.issue(P, t, g + C::D - 1, lane);
        cp_async_commit();
        if (!ring.arrive(P, t, g, lane)) break;
        const int slot = (g % C::D) * C::G;
        const float *xg = ring.x + slot * C::PITCH + (VEC ? 4 : 1) * lane;
#pragma unroll
        for (int l = 0; l < C::G; ++l) {
            constexpr int last = K - 1;
            const int ph = l % K, done = (l + 1) % K;       // input row g * G + l; the output row that it completes
            const float *xr = xg + l * C::PITCH + (VEC ? 0 : ring.off[slot + l]);
            DwWindow<K, VEC ? dw_offset(K, ADJ ? 0 : C::PH) : -1> win;
            win.load(xr, zero);
#pragma unroll
            for (int b = 0; b < K; ++b) {
                uint64_t X[NC / 2];
#pragma unroll
                for (int p = 0; p < NC / 2; ++p) X[p] = VEC ? win.pair(2 * p + b) : pack2(xr[b + 64 * p], xr[b + 64 * p + 32]);
                // this input row is kernel row a of the output row a rows above; a = 0 begins a new sum
#pragma unroll
                for (int a = 0; a < K; ++a)
#pragma unroll
                    for (int p = 0; p < NC / 2; ++p)
                        acc[(ph - a + K) % K][p] = fma2(X[p], w[b][a], a == 0 && b == 0 ? bias2 : acc[(ph - a + K) % K][p]);
            }
            // rows beyond the segment (of its first and last groups) make sums that are never written
            if ((unsigned)(g * C::G + l - last) < (unsigned)t.rows) {
                float v[NC];
#pragma unroll
                for (int p = 0; p < NC / 2; ++p) unpack2(acc[done][p], v[2 * p], v[2 * p + 1]);
                if (VEC) {
                    const uint32_t align = (uint32_t)reinterpret_cast<uintptr_t>(out);
                    if (in[3] && (align & 15u) == 0) {
                        *reinterpret_cast<float4 *>(out) = make_float4(v[0], v[1], v[2], v[NC - 1]);
                    } else if (in[3] && (align & 7u) == 0) {
                        *reinterpret_cast<float2 *>(out) = make_float2(v[0], v[1]);
                        *reinterpret_cast<float2 *>(out + 2) = make_float2(v[NC - 2], v[NC - 1]);
                    } else {
#pragma unroll
                        for (int p = 0; p < NC; ++p)
                            if (in[p]) out[p] = v[p];
                    }
                } else {
#pragma unroll
                    for (int p = 0; p < NC; ++p)
                        if (in[p]) out[32 * p] = v[p];
                }
                // adjoint: the ghost columns beside the row
                if (first_col && lane < C::PH) out[-C::PH - (VEC ? 3 : 0) * lane] = 0.f;
                if (last_col && lane < C::PH) out[t.cols - (VEC ? 3 : 0) * lane] = 0.f;
                out += pitch;
            }
        }
    }
    cp_async_wait_group<0>();
    if (ADJ) {
        // ghost rows above and below this strip
        const int p0 = first_col ? 0 : OO + t.j0, p1 = last_col ? pitch : OO + t.j0 + t.cols;
        for (int r = 0; r < C::PH; ++r) {
            if (t.i0 == 0)
                for (int q = p0 + lane; q < p1; q += 32) plane[(size_t)r * pitch + q] = 0.f;
            if (t.i0 + t.rows == bh)
                for (int q = p0 + lane; q < p1; q += 32) plane[(size_t)(bh + OO + r) * pitch + q] = 0.f;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Parameter gradients.  A block is one (channel, slice): its warps take the items slice * 4 + warp,
// + 4 * slices, ... of that channel's planes, so the K * K + 1 running sums stay in registers from item to
// item; the last K rows of dy do as well, and every row of x meets all of them.  At the end the sums are
// folded (pair halves, lanes by shuffles, warps in order) into one row of the scratch table; a second
// small kernel adds the rows of a channel in order.  The assignment of items to sums is static, so the
// result does not change from run to run.
// ---------------------------------------------------------------------------------------------
constexpr int kGradRow = 64;   // floats per (channel, slice) row of the scratch table (K * K + 1 <= 50 used)

template <int K, int NC, bool VEC>
__global__ void __launch_bounds__(kDwThreads, K == 7 ? 3 : 4)
conv_grad_rows_kernel(const __grid_constant__ DwParams P) {
    stream_enter();
    using C = DwCfg<K, NC, true>;
    extern __shared__ __align__(16) float smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t rest = blockIdx.x;
    const int sl = (int)fast_rem(P.slice_div, rest), ch = (int)rest;
    DwRing<K, NC, C::PH, true> ring;
    ring.init(smem + warp * C::WARP_FLOATS, lane);
    uint64_t acc[K][K], accb[NC / 2];
    const uint64_t ones = pack2(1.f, 1.f);
    const uint32_t zero = P.zero;
#pragma unroll
    for (int a = 0; a < K; ++a)
#pragma unroll
        for (int b = 0; b < K; ++b) acc[a][b] = 0ull;
#pragma unroll
    for (int p = 0; p < NC / 2; ++p) accb[p] = 0ull;

    bool ok = true;
#pragma unroll 1
    for (int id = sl * kDwWarps + warp; id < P.items && ok; id += kDwWarps * P.slices) {
        DwItem t = dw_item(P, (uint32_t)id, C::W);
        if (!t.valid) continue;
        t.plane = t.plane * P.channels + ch;
        const int nr = t.rows + K - 1, ng = (nr + C::G - 1) / C::G;
        __syncwarp();
        ring.begin(P, t, lane);
#pragma unroll
        for (int g = 0; g < C::D - 1; ++g) {
            if (g < ng) ring.issue(P, t, g, lane);
            cp_async_commit();
        }
        uint64_t dyh[K][NC / 2];                            // dy row o: slot o % K
#pragma unroll
        for (int s = 0; s < K; ++s)
#pragma unroll
            for (int p = 0; p < NC / 2; ++p) dyh[s][p] = 0ull;
        for (int g = 0; g < ng; ++g) {
            __syncwarp();
            if (g + C::D - 1 < ng) ring.issue(P, t, g + C::D - 1, lane);
            cp_async_commit();
            ok = ring.arrive(P, t, g, lane);
            if (!ok) break;
            const int slot = (g % C::D) * C::G;
            const float *xg = ring.x + slot * C::PITCH + (VEC ? 4 : 1) * lane, *yg = ring.y + slot * C::PITCHY + (VEC ? 4 : 1) * lane;
            // Row l of the group: kernel row a meets dy row g * G + l - a.  At both ends of an item (not `whole`) some of those are no rows of
            // it.  Their products are left out: zeros in their place make NaN of an infinite cell that the tap does not reach.  (The 7 x 7
            // kernels and the 5 x 5 ones off 16-byte rows have no registers for it and take the zeros: 500 -> 680 us, 72 -> 87.)
            constexpr bool SKIP = K == 3 || VEC;
            const bool whole = g > 0 && (g + 1) * C::G <= t.rows;
            auto row = [&](int l, bool all) {
                const int ph = l % K;
                const float *xr = xg + l * C::PITCH + (VEC ? 0 : ring.off[slot + l]);
                const float *yr = yg + l * C::PITCHY + (VEC ? 0 : ring.offy[slot + l]);
                if (VEC) {
                    const ulonglong2 f = *reinterpret_cast<const ulonglong2 *>(yr);
                    dyh[ph][0] = f.x;
                    dyh[ph][NC / 2 - 1] = f.y;
                } else {
#pragma unroll
                    for (int p = 0; p < NC / 2; ++p) dyh[ph][p] = pack2(yr[64 * p], yr[64 * p + 32]);
                }
#pragma unroll
                for (int p = 0; p < NC / 2; ++p) accb[p] = fma2(dyh[ph][p], ones, accb[p]);
                DwWindow<K, VEC ? dw_offset(K, C::PH) : -1> win;
                win.load(xr, zero);
                auto X = [&](int b, int p) { return VEC ? win.pair(2 * p + b) : pack2(xr[b + 64 * p], xr[b + 64 * p + 32]); };
                if (SKIP) {
                    uint64_t x[K][NC / 2];
#pragma unroll
                    for (int b = 0; b < K; ++b)
#pragma unroll
                        for (int p = 0; p < NC / 2; ++p) x[b][p] = X(b, p);
#pragma unroll
                    for (int a = 0; a < K; ++a)
                        if (all || (unsigned)(g * C::G + l - a) < (unsigned)t.rows) {
#pragma unroll
                            for (int b = 0; b < K; ++b)
#pragma unroll
                                for (int p = 0; p < NC / 2; ++p) acc[a][b] = fma2(x[b][p], dyh[(ph - a + K) % K][p], acc[a][b]);
                        }
                } else {
#pragma unroll
                    for (int b = 0; b < K; ++b)
#pragma unroll
                        for (int p = 0; p < NC / 2; ++p) {
                            const uint64_t x = X(b, p);
#pragma unroll
                            for (int a = 0; a < K; ++a) acc[a][b] = fma2(x, dyh[(ph - a + K) % K][p], acc[a][b]);
                        }
                }
            };
            if (K == 3 && whole) {                          // a copy of its own: 8 x 16 x 1024 x 1024 225 -> 196 us
#pragma unroll
                for (int l = 0; l < C::G; ++l) row(l, true);
            } else {
#pragma unroll
                for (int l = 0; l < C::G; ++l)
                    if (g * C::G + l < nr) row(l, whole);
            }
        }
    }
    cp_async_wait_group<0>();
    __syncthreads();                                        // the rings are free
    float *red = smem;                                      // [warp][K * K + 1]
#pragma unroll
    for (int q = 0; q <= K * K; ++q) {
        float lo, hi, v;
        if (q < K * K) {
            unpack2(acc[q / K][q % K], lo, hi);
            v = lo + hi;
        } else {
            v = 0.f;
#pragma unroll
            for (int p = 0; p < NC / 2; ++p) {
                unpack2(accb[p], lo, hi);
                v += lo + hi;
            }
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
        if (lane == 0) red[warp * (K * K + 1) + q] = v;
    }
    __syncthreads();
    for (int q = threadIdx.x; q <= K * K; q += kDwThreads) {
        float v = red[q];
#pragma unroll
        for (int w = 1; w < kDwWarps; ++w) v += red[w * (K * K + 1) + q];
        P.partial[((size_t)ch * P.slices + sl) * kGradRow + q] = v;
    }
}

// dw[c, :, :] and db[c] = the slices' rows of channel c: thread group h adds rows h, h + H, ..., the groups are added in order
constexpr int kDwFoldGroups = 16;
__global__ void __launch_bounds__(64 * kDwFoldGroups)
conv_grad_finish_kernel(const float *partial, int slices, int taps, float *dw, float *db) {
    stream_enter();
    __shared__ float part[kDwFoldGroups][64];
    const int ch = blockIdx.x, t = threadIdx.x & 63, h = threadIdx.x >> 6;
    float v = 0.f;
    if (t <= taps) {
        const float *row = partial + (size_t)ch * slices * kGradRow + t;
#pragma unroll 4
        for (int s = h; s < slices; s += kDwFoldGroups) v += row[(size_t)s * kGradRow];
    }
    part[h][t] = v;
    __syncthreads();
    if (h > 0 || t > taps) return;
    v = part[0][t];
#pragma unroll
    for (int k = 1; k < kDwFoldGroups; ++k) v += part[k][t];
    if (t < taps) dw[(size_t)ch * taps + t] = v;
    else if (db) db[ch] = v;
}

int conv_take_status() {
    int st = 0;
    if (cudaMemcpyFromSymbol(&st, g_conv_status, sizeof(int)) != cudaSuccess) return -1;
    if (st != 0) {
        const int zero = 0;
        cudaMemcpyToSymbol(g_conv_status, &zero, sizeof(int));
    }
    return st;
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
template <int K, int NC>
static constexpr int dw_smem_bytes(bool grad) {
    return (grad ? kDwWarps * DwCfg<K, NC, true>::WARP_FLOATS : dw_row_warps(K) * (DwCfg<K, NC, false>::WARP_FLOATS + dw_weight_floats(K))) * 4;
}

// Resident blocks of a kernel on the current device; sets the kernel's shared-memory limit on the first call.
template <typename Kernel>
static distdl_status_t dw_resident(Kernel kernel, int threads, int smem, int (&blocks_on)[kMaxDevicesPerProcess], int *blocks) {
    int dev = 0;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevicesPerProcess)
        return fail(DISTDL_ERR_UNSUPPORTED, "device index %d: at most %d devices per process", dev, kMaxDevicesPerProcess);
    std::lock_guard<std::mutex> setup_lock(setup_mutex());      // first calls from several threads set up once
    if (blocks_on[dev] == 0) {
        int sms = 0, per_sm = 0;
        DISTDL_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        DISTDL_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        DISTDL_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
        blocks_on[dev] = sms * std::max(per_sm, 1);
    }
    *blocks = blocks_on[dev];
    return DISTDL_OK;
}

// Checks shared by all entry points; fills the geometry.
static distdl_status_t dw_geometry(const distdl_partition *p, int32_t kh, int32_t kw, const char *what, DwParams *P, int64_t *max_bh, int64_t *max_bw) {
    if (!p) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL partition", what);
    if (p->rank != 4 || p->dtype != DISTDL_F32) return fail(DISTDL_ERR_SHAPE, "%s: needs a rank-4 F32 partition", what);
    if (p->any_periodic()) return fail(DISTDL_ERR_UNSUPPORTED, "%s: periodic partitions are not supported by the fused layers", what);
    if (p->pshape[0] != 1 || p->pshape[1] != 1)
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: only the feature-space dimensions may be partitioned", what);
    if (kh != kw || (kh != 3 && kh != 5 && kh != 7))
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: kernel %d x %d (supported: 3x3, 5x5, 7x7)", what, kh, kw);
    if (p->num_workers > kConvMaxWorkers) return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d workers", what, kConvMaxWorkers);
    const int h = kh / 2;
    for (int k = 0; k < 4; ++k)
        for (int32_t c = 0; c < p->pshape[k]; ++c) {
            const int want = k < 2 ? 0 : h;
            if (p->hlo[k][c] != want || p->hhi[k][c] != want)
                return fail(DISTDL_ERR_SHAPE, "%s: halo widths must be 0,0,%d,%d on every side", what, h, h);
        }
    *max_bh = *max_bw = 0;
    for (int32_t r = 0; r < p->pshape[2]; ++r) *max_bh = std::max<int64_t>(*max_bh, P->bh[r] = (int32_t)p->size[2][r]);
    for (int32_t c = 0; c < p->pshape[3]; ++c) *max_bw = std::max<int64_t>(*max_bw, P->bw[c] = (int32_t)p->size[3][c]);
    P->ph = p->pshape[2];
    P->pw = p->pshape[3];
    P->channels = (int32_t)p->global_shape[1];
    P->planes = (int32_t)(p->global_shape[0] * p->global_shape[1]);
    return DISTDL_OK;
}

// Strips of 64 columns instead of 128 where they leave fewer lanes without a column (a narrow strip pays about a sixth more
// per column for what is done once per row).
// Nor where wide strips, in segments of eight rows, leave a scheduler of the device with one warp at most: it goes at the pace of one warp's
// instructions, and half the columns are half of them (forward, adjoint and gradients, 7 x 7, 1 x 10 x 375 x 111: 33.7 -> 26.1 us; 5 x 5, 1 x 3
// x 33 x 169 on 1 x 2 workers 26.0 -> 22.0, 2 x 1 x 217 x 753 on 4 x 3 24.7 -> 22.1).
static int64_t dw_schedulers() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        sms = 148;                          // no device: a B200's
    }
    return 4 * (int64_t)sms;
}
static bool dw_narrow(const DwParams &P, int64_t max_bh, int64_t max_bw) {
    if (2 * ((max_bw + 63) / 64) * 7 < 4 * ((max_bw + 127) / 128) * 6) return true;
    return ((max_bw + 127) / 128) * ((max_bh + 7) / 8) * P.ph * P.pw * P.planes <= dw_schedulers();
}

// Rows per segment: the smallest estimated time, turns of the resident warps times rows an item reads (its halo, whole
// groups and about a dozen rows' worth of start-up included), and of equal ones the longest segments.  For a number of turns the most segments that
// fit into them are the best, as long as whole groups of rows allow, and more turns than the fewest by two dozen do not pay: the same
// rows as by trying all numbers of segments in 99 % of sizes, within 3 % in the others, in under half a microsecond of host time whatever the rows (67
// us for shards of 65536).
static int dw_segment(int K, int group, int64_t max_bh, int64_t strips_and_planes, int64_t warps) {
    int64_t best = max_bh;
    double best_cost = 0;
    const int64_t most = std::max<int64_t>(1, (max_bh - 1) / 7);                    // segments of eight rows
    const int64_t fewest = (strips_and_planes + warps - 1) / warps;
    for (int64_t t = fewest; t < fewest + 24; ++t) {
        const int64_t n = std::min(most, std::max<int64_t>(1, t * warps / strips_and_planes));
        const int64_t read = ((max_bh + n - 1) / n + K - 1 + group - 1) / group * group;          // whole groups
        const int64_t fit = (max_bh + read - K) / (read - K + 1), rows = (max_bh + fit - 1) / fit;   // the fewest segments that read as much
        const int64_t turns = (strips_and_planes * ((max_bh + rows - 1) / rows) + warps - 1) / warps;
        const double cost = (double)turns * ((rows + K - 1 + group - 1) / group * group + 12);
        if (best_cost == 0 || cost < best_cost) {
            best = rows;
            best_cost = cost;
        }
        if (n == most) break;
    }
    return (int)best;
}

static distdl_status_t dw_items(DwParams *P, int K, int64_t max_bh, int64_t max_bw, int strip, int group, int64_t planes, int64_t warps,
                                const char *what) {
    const int64_t strips = (max_bw + strip - 1) / strip;
    P->seg_rows = dw_segment(K, group, max_bh, strips * P->pw * P->ph * planes, warps);
    const int64_t segs = (max_bh + P->seg_rows - 1) / P->seg_rows, items = strips * P->pw * segs * P->ph * planes;
    if (items >= ((int64_t)1 << 31) - 1024) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles", what);
    P->items = (int32_t)items;
    P->strips = make_fast_div((uint32_t)strips);
    P->pw_div = make_fast_div((uint32_t)P->pw);
    P->segs = make_fast_div((uint32_t)segs);
    P->ph_div = make_fast_div((uint32_t)P->ph);
    P->chan_div = make_fast_div((uint32_t)P->channels);
    return DISTDL_OK;
}

// Whether every row of a layout with ghosts of width io starts on a 16-byte boundary.
static bool dw_aligned_rows(const DwParams &P, int io) {
    for (int32_t c = 0; c < P.pw; ++c)
        if ((P.bw[c] + 2 * io) % 4) return false;
    return true;
}

template <int K, bool ADJ, int NC, bool VEC>
static distdl_status_t launch_conv_rows(DwParams &P, int64_t max_bh, int64_t max_bw, cudaStream_t s, const char *what) {
    constexpr int smem = dw_smem_bytes<K, NC>(false), warps = dw_row_warps(K);
    static int blocks_on[kMaxDevicesPerProcess] = {0};
    int blocks = 0;
    distdl_status_t st = dw_resident(conv_rows_kernel<K, ADJ, NC, VEC>, 32 * warps, smem, blocks_on, &blocks);
    if (st != DISTDL_OK) return st;
    st = dw_items(&P, K, max_bh, max_bw, 32 * NC, DwCfg<K, NC, false>::G, P.planes, (int64_t)blocks * warps, what);
    if (st != DISTDL_OK) return st;
    launch_in_stream(conv_rows_kernel<K, ADJ, NC, VEC>, (unsigned)((P.items + warps - 1) / warps), 32 * warps, smem, s, P);
    DISTDL_CUDA_CHECK(cudaGetLastError());
    return DISTDL_OK;
}

template <int K, bool ADJ>
static distdl_status_t launch_conv(DwParams &P, int64_t max_bh, int64_t max_bw, cudaStream_t s, const char *what) {
    if (dw_narrow(P, max_bh, max_bw)) return launch_conv_rows<K, ADJ, 2, false>(P, max_bh, max_bw, s, what);
    return dw_aligned_rows(P, ADJ ? 0 : K / 2) ? launch_conv_rows<K, ADJ, 4, true>(P, max_bh, max_bw, s, what)
                                               : launch_conv_rows<K, ADJ, 4, false>(P, max_bh, max_bw, s, what);
}

static distdl_status_t conv_impl(const distdl_partition *p, const void *const *in, const void *w, const void *bias,
                                 int32_t kh, int32_t kw, void *const *out, void *stream, bool adj, const char *what) {
    clear_error();
    if (!p || !in || !w || !out) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL argument", what);
    DwParams P;
    memset(&P, 0, sizeof(P));
    int64_t max_bh = 0, max_bw = 0;
    const distdl_status_t st = dw_geometry(p, kh, kw, what, &P, &max_bh, &max_bw);
    if (st != DISTDL_OK) return st;
    if (!aligned16(w) || (bias && !aligned16(bias))) return fail(DISTDL_ERR_ALIGNMENT, "%s: w / bias not 16-byte aligned", what);
    for (int32_t wk = 0; wk < p->num_workers; ++wk) {
        if (!in[wk] || !out[wk]) return fail(DISTDL_ERR_INVALID_ARG, "%s: shard pointer %d is NULL", what, wk);
        if (!aligned16(in[wk]) || !aligned16(out[wk])) return fail(DISTDL_ERR_ALIGNMENT, "%s: shard %d is not 16-byte aligned", what, wk);
        P.in[wk] = (const float *)in[wk];
        P.out[wk] = (float *)out[wk];
    }
    P.w = (const float *)w;
    P.bias = (const float *)bias;
    cudaStream_t s = (cudaStream_t)stream;
    if (!adj)
        return kh == 3 ? launch_conv<3, false>(P, max_bh, max_bw, s, what) : kh == 5 ? launch_conv<5, false>(P, max_bh, max_bw, s, what)
                                                                                     : launch_conv<7, false>(P, max_bh, max_bw, s, what);
    return kh == 3 ? launch_conv<3, true>(P, max_bh, max_bw, s, what) : kh == 5 ? launch_conv<5, true>(P, max_bh, max_bw, s, what)
                                                                                : launch_conv<7, true>(P, max_bh, max_bw, s, what);
}

// Geometry and slices of the parameter gradients: shared by the workspace query and the launch.
template <int K, int NC, bool VEC>
static distdl_status_t grad_plan_rows(DwParams *P, int64_t max_bh, int64_t max_bw, int64_t batch, const char *what) {
    static int blocks_on[kMaxDevicesPerProcess] = {0};
    int blocks = 0;
    distdl_status_t st = dw_resident(conv_grad_rows_kernel<K, NC, VEC>, kDwThreads, dw_smem_bytes<K, NC>(true), blocks_on, &blocks);
    if (st != DISTDL_OK) return st;
    // as many slices per channel as give every block an SM slot of its own (one wave), never more than warps' items
    const int64_t slices = std::max<int64_t>(1, blocks / P->channels);
    st = dw_items(P, K, max_bh, max_bw, 32 * NC, DwCfg<K, NC, true>::G, batch, slices * kDwWarps, what);
    if (st != DISTDL_OK) return st;
    P->slices = (int32_t)std::min<int64_t>(slices, (P->items + kDwWarps - 1) / kDwWarps);
    P->slice_div = make_fast_div((uint32_t)P->slices);
    if ((int64_t)P->slices * P->channels >= ((int64_t)1 << 31)) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles", what);
    return DISTDL_OK;
}

// Which kernel: narrow strips, wide ones, or wide ones with 16-byte reads (rows of x and of dy on 16-byte boundaries: both
// are for 5 x 5, whose ghosts are four columns together, when the bulk is a multiple of four columns wide).
enum DwGradKind { kDwNarrow, kDwWide, kDwVector };

static distdl_status_t grad_plan(const distdl_partition *p, int32_t kh, int32_t kw, const char *what, DwParams *P, DwGradKind *kind) {
    int64_t max_bh = 0, max_bw = 0;
    const distdl_status_t st = dw_geometry(p, kh, kw, what, P, &max_bh, &max_bw);
    if (st != DISTDL_OK) return st;
    const int64_t n = p->global_shape[0];
    *kind = dw_narrow(*P, max_bh, max_bw) ? kDwNarrow : kh == 5 && dw_aligned_rows(*P, 0) ? kDwVector : kDwWide;
    if (*kind == kDwNarrow)
        return kh == 3 ? grad_plan_rows<3, 2, false>(P, max_bh, max_bw, n, what) : kh == 5 ? grad_plan_rows<5, 2, false>(P, max_bh, max_bw, n, what)
                                                                                           : grad_plan_rows<7, 2, false>(P, max_bh, max_bw, n, what);
    if (*kind == kDwVector) return grad_plan_rows<5, 4, true>(P, max_bh, max_bw, n, what);
    return kh == 3 ? grad_plan_rows<3, 4, false>(P, max_bh, max_bw, n, what) : kh == 5 ? grad_plan_rows<5, 4, false>(P, max_bh, max_bw, n, what)
                                                                                       : grad_plan_rows<7, 4, false>(P, max_bh, max_bw, n, what);
}

template <int K>
static distdl_status_t launch_grad(const DwParams &P, DwGradKind kind, float *dw, float *db, cudaStream_t s) {
    const unsigned grid = (unsigned)(P.slices * P.channels);
    if (kind == kDwNarrow) launch_in_stream(conv_grad_rows_kernel<K, 2, false>, grid, kDwThreads, dw_smem_bytes<K, 2>(true), s, P);
    else if (kind == kDwVector && K == 5) launch_in_stream(conv_grad_rows_kernel<5, 4, true>, grid, kDwThreads, dw_smem_bytes<5, 4>(true), s, P);
    else launch_in_stream(conv_grad_rows_kernel<K, 4, false>, grid, kDwThreads, dw_smem_bytes<K, 4>(true), s, P);
    DISTDL_CUDA_CHECK(cudaGetLastError());
    launch_in_stream(conv_grad_finish_kernel, P.channels, 64 * kDwFoldGroups, 0, s, P.partial, P.slices, K * K, dw, db);
    DISTDL_CUDA_CHECK(cudaGetLastError());
    return DISTDL_OK;
}

}  // namespace distdl

extern "C" distdl_status_t distdl_conv_adj_params_workspace(const distdl_partition_t *p, int32_t kh, int32_t kw,
                                                            int64_t *bytes) {
    using namespace distdl;
    clear_error();
    if (!bytes) return fail(DISTDL_ERR_INVALID_ARG, "conv_adj_params_workspace: NULL argument");
    DwParams P;
    memset(&P, 0, sizeof(P));
    DwGradKind kind = kDwWide;
    const distdl_status_t st = grad_plan(p, kh, kw, "conv_adj_params_workspace", &P, &kind);
    if (st != DISTDL_OK) return st;
    *bytes = (int64_t)P.channels * P.slices * kGradRow * (int64_t)sizeof(float);
    return DISTDL_OK;
}

extern "C" distdl_status_t distdl_conv_adj_params(const distdl_partition_t *p, const void *const *x,
                                                  const void *const *dy, int32_t kh, int32_t kw, void *dw, void *db,
                                                  void *workspace, int64_t workspace_bytes, void *stream) {
    using namespace distdl;
    clear_error();
    const char *what = "conv_adj_params";
    if (!p || !x || !dy || !dw || !workspace) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL argument", what);
    DwParams P;
    memset(&P, 0, sizeof(P));
    DwGradKind kind = kDwWide;
    const distdl_status_t st = grad_plan(p, kh, kw, what, &P, &kind);
    if (st != DISTDL_OK) return st;
    const int64_t need = (int64_t)P.channels * P.slices * kGradRow * (int64_t)sizeof(float);
    if (workspace_bytes < need) return fail(DISTDL_ERR_INVALID_ARG, "%s: workspace of %lld bytes, %lld needed", what,
                                            (long long)workspace_bytes, (long long)need);
    if (!aligned16(dw) || !aligned16(workspace) || (db && !aligned16(db)))
        return fail(DISTDL_ERR_ALIGNMENT, "%s: dw / db / workspace not 16-byte aligned", what);
    for (int32_t wk = 0; wk < p->num_workers; ++wk) {
        if (!x[wk] || !dy[wk]) return fail(DISTDL_ERR_INVALID_ARG, "%s: shard pointer %d is NULL", what, wk);
        if (!aligned16(x[wk]) || !aligned16(dy[wk])) return fail(DISTDL_ERR_ALIGNMENT, "%s: shard %d is not 16-byte aligned", what, wk);
        P.in[wk] = (const float *)x[wk];
        P.dy[wk] = (const float *)dy[wk];
    }
    P.partial = (float *)workspace;
    cudaStream_t s = (cudaStream_t)stream;
    if (kh == 3) return launch_grad<3>(P, kind, (float *)dw, (float *)db, s);
    if (kh == 5) return launch_grad<5>(P, kind, (float *)dw, (float *)db, s);
    return launch_grad<7>(P, kind, (float *)dw, (float *)db, s);
}

extern "C" distdl_status_t distdl_conv_fwd(const distdl_partition_t *p, const void *const *x, const void *w,
                                           const void *bias, int32_t kh, int32_t kw, void *const *y, void *stream) {
    return distdl::conv_impl(p, x, w, bias, kh, kw, y, stream, false, "conv_fwd");
}
extern "C" distdl_status_t distdl_conv_adj(const distdl_partition_t *p, const void *const *dy, const void *w,
                                           int32_t kh, int32_t kw, void *const *dx, void *stream) {
    return distdl::conv_impl(p, dy, w, nullptr, kh, kw, dx, stream, true, "conv_adj");
}

// Every row that the adjoint (gradients: the parameter gradients) copies out of arrays without ghosts, by the rules of the kernels.
extern "C" distdl_status_t distdl_selftest_conv_row_reads(const distdl_partition_t *p, int32_t k, int32_t gradients, int64_t *floats_past_end,
                                                          int64_t *rows_cut) {
    using namespace distdl;
    clear_error();
    if (!floats_past_end || !rows_cut) return fail(DISTDL_ERR_INVALID_ARG, "selftest_conv_row_reads: NULL argument");
    DwParams P;
    memset(&P, 0, sizeof(P));
    int64_t max_bh = 0, max_bw = 0;
    const distdl_status_t st = dw_geometry(p, k, k, "selftest_conv_row_reads", &P, &max_bh, &max_bw);
    if (st != DISTDL_OK) return st;
    *floats_past_end = *rows_cut = 0;
    const int strip = dw_narrow(P, max_bh, max_bw) ? 64 : 128;
    const uintptr_t base = 256;                                 // never read: addresses only
    for (int32_t w = 0; w < p->num_workers; ++w) {
        const int bh = P.bh[w / P.pw], bw = P.bw[w % P.pw];
        const int64_t cells = (int64_t)P.planes * bh * bw;
        const float *end = reinterpret_cast<const float *>(base + 4 * (uintptr_t)cells);
        for (int64_t row = 0; row < (int64_t)P.planes * bh; ++row)
            for (int j0 = 0; j0 < bw; j0 += strip) {
                const int cols = std::min(strip, bw - j0);
                const int halo = gradients ? 0 : k / 2, ja = std::max(j0 - halo, 0), n = std::min(j0 + cols + halo, bw) - ja;
                const uintptr_t first = base + 4 * (uintptr_t)(row * bw + ja);
                const float *f = reinterpret_cast<const float *>(first);
                const bool cut = dw_may_pass_end((int)(row % bh), bh, bw) && dw_past_end(f, n, end);
                const int lead = (int)((first >> 2) & 3), in_blocks = cut ? dw_whole(f, n) : n;
                *rows_cut += cut;
                if (in_blocks) *floats_past_end = std::max<int64_t>(*floats_past_end, row * bw + ja - lead + ((lead + in_blocks + 3) & ~3) - cells);
            }
    }
    return DISTDL_OK;
}
