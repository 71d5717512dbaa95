// Generalized convolution layer: channels partitioned as well (Section 4, "Sparse layers": forward /
// adjoint convolution algorithms with x on 1 x P_ci x P_0 x P_1, y on 1 x P_co x P_0 x P_1, weights on
// P_co x P_ci and the work partition 1 x P_co x P_ci x P_0 x P_1).
//   forward:  x <- H x;  x^ <- B x (to the P_co copies);  y^_{ijs} <- Conv(w_{ij}, b_i on j = 0; x^_{js});
//             y_{is} <- R over j, in order.
//   adjoint:  dy^ <- B dy (to the P_ci copies);  dx^_{ijs} <- [dConv]*(dy^_{ijs});  dx_{js} <- R over i, in
//             order;  dx <- H* dx  (gather form: a correlation of dy with the rotated kernels).
// With every shard in one memory the broadcasts are implicit and the sum-reduce is the running sum of
// the block that owns an output tile: it walks through the blocks of the reduced channel partition in
// worker order and through the channels of a block in channel order, so the order of the sum is fixed.
// H / H* are fused: a tile is staged with its ghost rows and columns straight from the bulk of the
// neighbouring shards (zeros outside the tensor), and the adjoint writes the zeros that H* leaves in the
// ghosts of dx together with the tile beside them.
#include <algorithm>
#include <cstring>
#include <vector>

#include "common.h"
#include "conv_common.h"

namespace distdl {

constexpr int kCgThreads = 128;
constexpr int kCgMaxPairs = 4;          // output-channel pairs per thread
constexpr int kMaxChanBlocks = 8;       // P_co, P_ci
constexpr int kMaxGroups = 128;         // groups of up to 2 * kCgMaxPairs output channels

// Shape of the tiles of one launch.  A tile is tn images x th rows x px * seg columns of one shard and one group of
// output channels; thread -> (image, row, segment of px columns).
struct CgShape {
    int32_t px;                         // consecutive pixels of a row per thread: 8 or 4
    int32_t tn, th, seg;
    int32_t rows, cols, pitch;          // staged rows and columns of one image, floats from row to row
    int32_t tile_floats;                // one staged channel
    int32_t entries;                    // staged cells: tn * rows * cols
    int32_t smem_bytes;
};

struct ConvGParams {
    const float *in[kConvMaxWorkers];       // shards of the input tensor, channel block after channel block
    float *out[kConvMaxWorkers];
    int32_t bh[kConvMaxWorkers], bw[kConvMaxWorkers];   // bulk rows / columns per worker row / column
    const float *w[kMaxChanBlocks * kMaxChanBlocks];    // weight blocks, worker order i * P_ci + j
    const float *bias[kMaxChanBlocks];      // forward only; per block of output channels, may be null
    int32_t cnt_out[kMaxChanBlocks], cnt_in[kMaxChanBlocks];   // channels per block of the output / input partition
    int32_t ph, pw, p_in, pci, batch;
    uint8_t grp_block[kMaxGroups], grp_count[kMaxGroups];
    uint16_t grp_first[kMaxGroups];
    CgShape t;
    FastDiv groups, tiles_x, pw_div, tiles_y, ph_div, cols, rows, tn, seg, half_th;
};

// Blocks per SM that the registers allow: 168 a thread for eight pixels (a whole row of taps read ahead), 128 for four.
constexpr int cg_blocks(int px) { return px == 8 ? 3 : 4; }

// What bounds it: the fp32 pipe.  A thread owns PX pixels of a row and up to eight output channels; the accumulators
// are pairs of channels, so a weight pair is two neighbouring floats of the staged table (one 16-byte broadcast read
// feeds two pairs) and an input value is duplicated once and used by every tap and channel: 5 x 5, eight channels, eight
// pixels, 800 packed FMAs per input channel and thread beside about 125 other instructions.  With pairs of pixels instead
// (two channels per thread, as many packed FMAs as now for a quarter of the outputs) every input channel was staged four
// times as often.  The rows of taps are unrolled, so that the next row's reads overlap the FMAs of this one; that takes
// 168 registers with eight pixels, and three blocks an SM are faster with it than four without (1.14 -> 1.10 ms below).
// Blocks of one or two warps instead, one image each: 54 us instead of 40, the weights are staged for fewer outputs.
//
// Measured (forward / adjoint, B200): 16 -> 16 channels, 5 x 5, 4 x 1024 x 1024 on 2 x 2 workers 1.10 / 1.12 ms = 49 TFLOP/s
// (1.48 / 1.59 ms with two channels a block; packed FMAs alone, as an outer product in registers, reach 59 TFLOP/s);
// 6 -> 16 channels, 256 images of 28 x 28 on 2 x 2 workers 0.040 / 0.044 ms (0.82 / 0.79 ms).
//
// Small images are packed: a tile may span several images, so 14 x 14 shards fill the threads (32 x 128 tiles left 95 %
// of them idle).  Cells are staged one by one (4-byte asynchronous copies), which takes any row pitch and any mixture of
// neighbours; where each cell comes from is worked out once per tile and kept in a table, a channel then costs one table
// read, one pointer read and one copy per cell.  Two buffers, one barrier per input channel.
template <int K, bool ADJ, int CP, int PX>
__global__ void __launch_bounds__(kCgThreads, cg_blocks(PX))
convg_kernel(const __grid_constant__ ConvGParams G) {
    constexpr int PH = K / 2, CT = 2 * CP;
    constexpr int NF = ((PX + K - 1 + 3) / 4) * 4;         // floats of a thread's window per row
    constexpr int WF = ((K * K * CT + 3) / 4) * 4;
    constexpr int io = ADJ ? 0 : PH, oo = ADJ ? PH : 0;    // ghost width of the input / output layout
    extern __shared__ __align__(16) float smem[];
    const CgShape &T = G.t;
    float *tiles = smem;
    float *wbuf = tiles + 2 * T.tile_floats;
    uint2 *table = reinterpret_cast<uint2 *>(wbuf + 2 * WF);
    const float **ptrs = reinterpret_cast<const float **>(table + T.entries);     // [2][9 * tn]
    const int tid = threadIdx.x;

    uint32_t id = blockIdx.x;
    const int g = (int)fast_rem(G.groups, id);             // groups fastest: they read the same input tile
    const int tx = (int)fast_rem(G.tiles_x, id);
    const int c = (int)fast_rem(G.pw_div, id);
    const int ty = (int)fast_rem(G.tiles_y, id);
    const int r = (int)fast_rem(G.ph_div, id);
    const int n0 = (int)id * T.tn;
    const int bh = G.bh[r], bw = G.bw[c];
    const int i0 = ty * T.th, j0 = tx * PX * T.seg;
    const bool live = i0 < bh && j0 < bw;                  // shards smaller than the largest
    const int ob = G.grp_block[g], o0 = G.grp_first[g], oc = G.grp_count[g];
    const int spatial = G.ph * G.pw;

    // where every staged cell comes from (each thread reads back its own entries only): while the kernel before this one ends
    for (int e = tid; live && e < T.entries; e += kCgThreads) {
        uint32_t q = (uint32_t)e;
        const int s = (int)fast_rem(G.cols, q);
        const int ry = (int)fast_rem(G.rows, q);
        const int tn = (int)q;
        const int dst = (tn * T.rows + ry) * T.pitch + s;
        int i = i0 - PH + ry, j = j0 - PH + s, dr = 1, dc = 1;
        bool ok = n0 + tn < G.batch;
        if (i < 0) {
            dr = 0;
            ok = ok && r > 0;
            if (ok) i += G.bh[r - 1];
            ok = ok && i >= 0;
        } else if (i >= bh) {
            dr = 2;
            i -= bh;
            ok = ok && r + 1 < G.ph;
            if (ok) ok = i < G.bh[r + 1];
        }
        int w = bw;
        if (j < 0) {
            dc = 0;
            ok = ok && c > 0;
            if (ok) w = G.bw[c - 1];
            j += w;
            ok = ok && j >= 0;
        } else if (j >= bw) {
            dc = 2;
            j -= bw;
            ok = ok && c + 1 < G.pw;
            if (ok) w = G.bw[c + 1];
            ok = ok && j < w;
        }
        if (ok) {
            table[e] = make_uint2((uint32_t)(i * (w + 2 * io) + j), (uint32_t)dst | ((uint32_t)((3 * dr + dc) * T.tn + tn) << 16));
        } else {
            table[e] = make_uint2(0xffffffffu, 0u);
            tiles[dst] = 0.f;
            tiles[T.tile_floats + dst] = 0.f;
        }
    }
    if (oc < CT)
        for (int idx = tid; idx < 2 * WF; idx += kCgThreads) wbuf[idx] = 0.f;
    stream_enter();
    if (!live) return;

    // First cell (bulk row 0, column 0) of the channel's plane in every neighbour, per image.  Channels come one after another: with four
    // pixels a thread its pointer and its weights' offsets are worked out at the first channel of a block and moved on from there (1 x 14
    // x 61 x 68, 3 x 3, forward / adjoint / gradients 33.6 -> 30.4 us, 29.0 with the table above ahead of the wait as well); with eight there is
    // no register for it (16 -> 16 channels at 1024 x 1024: 1.10 -> 1.12 ms).
    constexpr bool KEEP = PX == 4;
    const float *plane_p = nullptr;
    uint32_t plane_step = 0;
    auto set_pointers = [&](int ib, int cl, int b) {
        for (int t = tid; t < 9 * T.tn; t += kCgThreads) {
            if (KEEP && cl > 0 && t == tid) {
                plane_p += plane_step;
                ptrs[b * 9 * T.tn + t] = plane_p;
                continue;
            }
            uint32_t q = (uint32_t)t;
            const int tn = (int)fast_rem(G.tn, q);
            const int rr = r + (int)q / 3 - 1, cc = c + (int)q % 3 - 1;
            const float *p = nullptr;
            if (rr >= 0 && rr < G.ph && cc >= 0 && cc < G.pw) {
                const uint32_t pitch = (uint32_t)(G.bw[cc] + 2 * io);
                const uint32_t step = (uint32_t)(G.bh[rr] + 2 * io) * pitch;
                p = G.in[ib * spatial + rr * G.pw + cc] + (size_t)((n0 + tn) * G.cnt_in[ib] + cl) * step + (io * pitch + io);
                if (KEEP && t == tid) plane_step = step;
            }
            if (KEEP && t == tid) plane_p = p;
            ptrs[b * 9 * T.tn + t] = p;
        }
    };
    // this thread's weights of a channel: their offsets in the block, and the channel's first
    constexpr int NW = (K * K * CT + kCgThreads - 1) / kCgThreads;
    int w_off[NW], w_step = 0;
    const float *w_p = nullptr;
    const uint32_t tiles_s = (uint32_t)__cvta_generic_to_shared(tiles), wbuf_s = (uint32_t)__cvta_generic_to_shared(wbuf);
    auto stage = [&](int ib, int cl, int b) {
        const uint32_t dst0 = tiles_s + (uint32_t)(b * T.tile_floats) * 4u;
        const float *const *pt = ptrs + b * 9 * T.tn;
        for (int e = tid; e < T.entries; e += kCgThreads) {
            const uint2 t = table[e];
            if (t.x != 0xffffffffu) cp_async4_to(dst0 + (t.y & 0xffffu) * 4u, pt[t.y >> 16] + t.x);
        }
        const int s_out = ADJ ? K * K : G.cnt_in[ib] * K * K, s_in = ADJ ? G.cnt_out[ob] * K * K : K * K;
        const float *first = (ADJ ? G.w[ib * G.pci + ob] : G.w[ob * G.pci + ib]) + (size_t)o0 * s_out;
        if constexpr (KEEP) {
            if (cl == 0) {
                w_p = first;
                w_step = s_in;
#pragma unroll
                for (int k = 0; k < NW; ++k) {
                    const int idx = tid + k * kCgThreads, tap = idx / CT, o = idx - tap * CT;
                    w_off[k] = idx < K * K * CT && o < oc ? o * s_out + (ADJ ? K * K - 1 - tap : tap) : -1;      // adjoint: rotated
                }
            }
#pragma unroll
            for (int k = 0; k < NW; ++k)
                if (w_off[k] >= 0) cp_async4_to(wbuf_s + (uint32_t)(b * WF + tid + k * kCgThreads) * 4u, w_p + w_off[k]);
            w_p += w_step;
        } else {
            const float *wsrc = first + (size_t)cl * s_in;
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const int idx = tid + k * kCgThreads, tap = idx / CT, o = idx - tap * CT;
                if (idx < K * K * CT && o < oc)
                    cp_async4_to(wbuf_s + (uint32_t)(b * WF + idx) * 4u, wsrc + (size_t)o * s_out + (ADJ ? K * K - 1 - tap : tap));
            }
        }
    };
    auto advance = [&](int &ib, int &cl) {
        if (++cl == G.cnt_in[ib]) {
            cl = 0;
            ++ib;
        }
    };

    // this thread's item: neighbouring threads take the two rows of a pair, so that (with a row pitch of an odd number of
    // float4s) the 16-byte reads of eight consecutive lanes fall into eight different bank groups
    uint32_t rest = (uint32_t)tid >> 1;
    const int seg = (int)fast_rem(G.seg, rest);
    const int row = 2 * (int)fast_rem(G.half_th, rest) + (tid & 1);
    const int img = (int)rest;
    const bool active = img < T.tn && n0 + img < G.batch && i0 + row < bh && j0 + PX * seg < bw;
    const int xoff = (img * T.rows + row) * T.pitch + PX * seg;

    uint64_t acc[PX][CP];
#pragma unroll
    for (int q = 0; q < CP; ++q) {
        float b0 = 0.f, b1 = 0.f;
        if (!ADJ && G.bias[ob]) {
            if (2 * q < oc) b0 = __ldg(G.bias[ob] + o0 + 2 * q);
            if (2 * q + 1 < oc) b1 = __ldg(G.bias[ob] + o0 + 2 * q + 1);
        }
#pragma unroll
        for (int p = 0; p < PX; ++p) acc[p][q] = pack2(b0, b1);
    }

    int sib = 0, scl = 0;                   // channel to stage next
    int pib = 0, pcl = 0;                   // channel whose pointers are set next
    set_pointers(pib, pcl, 0);
    advance(pib, pcl);
    __syncthreads();
    stage(sib, scl, 0);
    advance(sib, scl);
    cp_async_commit();
    if (pib < G.p_in) {
        set_pointers(pib, pcl, 1);
        advance(pib, pcl);
    }
    int buf = 0;
    bool more = true;
    while (more) {
        cp_async_wait_group<0>();
        __syncthreads();        // this channel has arrived; the other buffer has been read; the next pointers are set
        more = sib < G.p_in;
        if (more) {
            stage(sib, scl, buf ^ 1);
            advance(sib, scl);
            cp_async_commit();
            if (pib < G.p_in) {
                set_pointers(pib, pcl, buf);
                advance(pib, pcl);
            }
        }
        if (active) {
            const float *xb = tiles + buf * T.tile_floats + xoff;
            const float *wb = wbuf + buf * WF;
#pragma unroll
            for (int a = 0; a < K; ++a) {
                float x[NF];
#pragma unroll
                for (int v = 0; v < NF / 4; ++v) {
                    const float4 f = *reinterpret_cast<const float4 *>(xb + 4 * v);
                    x[4 * v] = f.x;
                    x[4 * v + 1] = f.y;
                    x[4 * v + 2] = f.z;
                    x[4 * v + 3] = f.w;
                }
                uint64_t xx[PX + K - 1];
#pragma unroll
                for (int v = 0; v < PX + K - 1; ++v) xx[v] = pack2(x[v], x[v]);
#pragma unroll
                for (int b = 0; b < K; ++b) {
                    uint64_t w[CP];
                    if (CP % 2 == 0) {
#pragma unroll
                        for (int q = 0; q < CP; q += 2) {
                            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(wb + b * CT + 2 * q);
                            w[q] = v.x;
                            w[q + 1] = v.y;
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < CP; ++q) w[q] = *reinterpret_cast<const uint64_t *>(wb + b * CT + 2 * q);
                    }
#pragma unroll
                    for (int p = 0; p < PX; ++p)
#pragma unroll
                        for (int q = 0; q < CP; ++q) acc[p][q] = fma2(xx[p + b], w[q], acc[p][q]);
                }
                xb += T.pitch;
                wb += K * CT;
            }
        }
        buf ^= 1;
    }

    // Store: two channels at a time through shared memory, so that a warp writes consecutive cells whatever the row pitch.
    // The rectangle written is the tile, in the adjoint extended through the ghost layers wherever it touches a face.
    const int th = min(T.th, bh - i0), tw = min(PX * T.seg, bw - j0), imgs = min(T.tn, G.batch - n0);
    const int top = ADJ && i0 == 0 ? oo : 0, bottom = ADJ && i0 + th == bh ? oo : 0;
    const int left = ADJ && j0 == 0 ? oo : 0, right = ADJ && j0 + tw == bw ? oo : 0;
    const int er = th + top + bottom, ew = tw + left + right;
    const uint32_t pitch_o = (uint32_t)(bw + 2 * oo), plane_o = (uint32_t)(bh + 2 * oo) * pitch_o;
    const int chan = G.cnt_out[ob];
    float *obase = G.out[ob * spatial + r * G.pw + c] + ((size_t)n0 * chan + o0) * plane_o;
    const int spitch = PX * T.seg;
    __syncthreads();                        // the tiles and the cell table are free
    for (int idx = tid; idx < imgs * er; idx += kCgThreads) {
        const int im = idx / er, y = idx - im * er;
        const bool ghost = y < top || y >= top + th;
        table[idx] = make_uint2((uint32_t)im * (uint32_t)chan * plane_o + (uint32_t)(i0 + oo - top + y) * pitch_o + (uint32_t)(j0 + oo - left),
                                ghost ? 0xffffffffu : (uint32_t)((im * T.th + (y - top)) * spitch));
    }
    const int per_ch = T.tn * T.th * spitch;                                    // floats of one channel
    const int vw = ADJ ? 0 : ((bw & 3) == 0 ? tw / 4 : 0);                      // whole rows of aligned float4s
    const int cw = vw ? vw : ew;
    const int step_row = kCgThreads / cw, step_col = kCgThreads - step_row * cw;
#pragma unroll
    for (int q = 0; q < CP; ++q) {
        if (2 * q >= oc) break;
        if (q > 0) __syncthreads();
        if (active) {
            float lo[PX], hi[PX];
#pragma unroll
            for (int p = 0; p < PX; ++p) unpack2(acc[p][q], lo[p], hi[p]);
            float *d = tiles + (img * T.th + row) * spitch + PX * seg;
#pragma unroll
            for (int p = 0; p < PX; p += 4) {
                *reinterpret_cast<float4 *>(d + p) = make_float4(lo[p], lo[p + 1], lo[p + 2], lo[p + 3]);
                *reinterpret_cast<float4 *>(d + per_ch + p) = make_float4(hi[p], hi[p + 1], hi[p + 2], hi[p + 3]);
            }
        }
        __syncthreads();
        float *o_lo = obase + (size_t)(2 * q) * plane_o;
        const bool two = 2 * q + 1 < oc;
        int y = tid / cw, x = tid - y * cw;
        while (y < imgs * er) {
            const uint2 t = table[y];
            if (vw) {
                const float *s = tiles + t.y + 4 * x;
                *reinterpret_cast<float4 *>(o_lo + t.x + 4 * x) = *reinterpret_cast<const float4 *>(s);
                if (two) *reinterpret_cast<float4 *>(o_lo + plane_o + t.x + 4 * x) = *reinterpret_cast<const float4 *>(s + per_ch);
            } else {
                const bool in = t.y != 0xffffffffu && (unsigned)(x - left) < (unsigned)tw;
                const float *s = tiles + (in ? t.y + (uint32_t)(x - left) : 0u);
                o_lo[t.x + x] = in ? s[0] : 0.f;
                if (two) o_lo[plane_o + t.x + x] = in ? s[per_ch] : 0.f;
            }
            y += step_row;
            x += step_col;
            if (x >= cw) {
                x -= cw;
                ++y;
            }
        }
    }
}

static CgShape cg_shape(int K, int px, int tn, int th, int seg, int cp) {
    CgShape t;
    memset(&t, 0, sizeof(t));
    const int nf = ((px + K - 1 + 3) / 4) * 4;
    t.px = px;
    t.tn = tn;
    t.th = th;
    t.seg = seg;
    t.rows = th + K - 1;
    t.cols = px * seg + K - 1;
    t.pitch = (std::max(t.cols, px * (seg - 1) + nf) + 3) / 4 * 4;
    if ((t.pitch / 4) % 2 == 0) t.pitch += 4;
    t.tile_floats = tn * t.rows * t.pitch;
    t.entries = tn * t.rows * t.cols;
    t.smem_bytes = 2 * t.tile_floats * 4 + 2 * ((K * K * 2 * cp + 3) / 4 * 4) * 4 + t.entries * 8 + 2 * 9 * tn * 8;
    return t;
}

// Tile shape: the one with the smallest estimated time, tiles per SM times the cost of a tile in thread-cycles: the
// packed FMAs of 128 threads (2.5 cycles each, as measured for a register outer product) plus the staging of its cells
// (about eight instructions each); the last wave of an SM takes 0.45 of a full one, whatever is in it, and 0.55 in proportion.
// Up to 56 KB of shared memory keep four blocks on an SM.  Sizes are tried from the largest down in steps of a fifth, shards cut
// into that many equal tiles, and what cannot win by its FMAs alone is passed over: 1 to 2 us of host time.  Four pixels a thread spend a tenth more on the same outputs (weights are read for
// half as many FMAs), but make twice the warps: 16 images of 28 x 28, 6 -> 16 channels, forward 12.6 us with eight pixels,
// 9.8 with four; 256 images 46.8 and 39.6; 1024 images 148 and 146, their adjoint 138 and 153.
static CgShape cg_choose(int K, int cp, int max_bh, int max_bw, int batch, int workers, int groups, int sms) {
    CgShape best;
    memset(&best, 0, sizeof(best));
    double best_cost = 0;
    const double per_tile = 1.0 / sms;
    for (int px = 8; px >= 4; px -= 4) {
        const double fma = kCgThreads * (double)(K * K) * px * cp * (px == 4 ? 2.75 : 2.5);
        const int res = cg_blocks(px);
        int nx_before = 0;
        for (int try_seg = kCgThreads / px; try_seg >= 1; try_seg -= std::max(1, try_seg / 5)) {
            const int nx = (max_bw + px * try_seg - 1) / (px * try_seg);
            if (nx == nx_before) continue;
            nx_before = nx;
            const int seg = (max_bw + px * nx - 1) / (px * nx);
            int ny_before = 0;
            for (int try_th = kCgThreads / seg / 2 * 2; try_th >= 2; try_th -= std::max(2, try_th / 10 * 2)) {
                const int ny = (max_bh + try_th - 1) / try_th;
                if (ny == ny_before) continue;
                ny_before = ny;
                const int th = ((max_bh + ny - 1) / ny + 1) & ~1;
                const int room = kCgThreads / (th * seg);
                for (int tn = std::min(room, batch); tn >= 1; tn /= 2) {
                    const int64_t tiles = (int64_t)(nx * ny) * ((int64_t)(workers * groups) * (tn == 1 ? batch : (batch + tn - 1) / tn));
                    const int per_sm = (int)(int64_t)((double)(tiles + sms - 1) * per_tile), last = per_sm % res;
                    const double waves = per_sm - last + (last ? 0.45 * res + 0.55 * last : 0.0);
                    if (best.tn != 0 && waves * fma >= best_cost) continue;
                    const CgShape t = cg_shape(K, px, tn, th, seg, cp);
                    if (t.smem_bytes > 56 * 1024 || t.tile_floats > 32767) continue;
                    const double cost = waves * (fma + 8.0 * t.entries);
                    if (best.tn == 0 || cost < best_cost) {
                        best = t;
                        best_cost = cost;
                    }
                }
            }
        }
    }
    return best;
}

template <int K, bool ADJ, int CP, int PX>
static distdl_status_t launch_convg(const ConvGParams &G, int64_t blocks, cudaStream_t s) {
    static bool configured_on[kMaxDevicesPerProcess] = {false};
    int dev = 0;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevicesPerProcess)
        return fail(DISTDL_ERR_UNSUPPORTED, "device index %d: at most %d devices per process", dev, kMaxDevicesPerProcess);
    {
        std::lock_guard<std::mutex> setup_lock(setup_mutex());
        if (!configured_on[dev]) {
            DISTDL_CUDA_CHECK(cudaFuncSetAttribute(convg_kernel<K, ADJ, CP, PX>, cudaFuncAttributeMaxDynamicSharedMemorySize, 56 * 1024));
            configured_on[dev] = true;
        }
    }
    launch_in_stream(convg_kernel<K, ADJ, CP, PX>, (unsigned)blocks, kCgThreads, G.t.smem_bytes, s, G);
    DISTDL_CUDA_CHECK(cudaGetLastError());
    return DISTDL_OK;
}

template <int K, bool ADJ>
static distdl_status_t launch_convg_pairs(const ConvGParams &G, int cp, int64_t blocks, cudaStream_t s) {
    switch (cp) {
        case 1: return G.t.px == 8 ? launch_convg<K, ADJ, 1, 8>(G, blocks, s) : launch_convg<K, ADJ, 1, 4>(G, blocks, s);
        case 2: return G.t.px == 8 ? launch_convg<K, ADJ, 2, 8>(G, blocks, s) : launch_convg<K, ADJ, 2, 4>(G, blocks, s);
        case 3: return G.t.px == 8 ? launch_convg<K, ADJ, 3, 8>(G, blocks, s) : launch_convg<K, ADJ, 3, 4>(G, blocks, s);
        default: return G.t.px == 8 ? launch_convg<K, ADJ, 4, 8>(G, blocks, s) : launch_convg<K, ADJ, 4, 4>(G, blocks, s);
    }
}

// px: partition of the tensor with n_ci channels (x, dx); the other tensor (y, dy) has n_co channels on pco
// blocks and the same spatial partition.  Forward: in = x (padded), out = y (bulk-shaped); adjoint: in = dy
// (bulk-shaped), out = dx (padded, ghosts cleared).
static distdl_status_t convg_impl(const distdl_partition *px, int64_t nco, int32_t pco, const void *const *in,
                                  const void *const *w, const void *const *bias, int32_t kh, int32_t kw,
                                  void *const *out, void *stream, bool adj, const char *what) {
    clear_error();
    if (!px || !in || !w || !out) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL argument", what);
    if (px->rank != 4 || px->dtype != DISTDL_F32) return fail(DISTDL_ERR_SHAPE, "%s: needs a rank-4 F32 partition", what);
    if (px->any_periodic()) return fail(DISTDL_ERR_UNSUPPORTED, "%s: periodic partitions are not supported by the fused layers", what);
    if (px->pshape[0] != 1) return fail(DISTDL_ERR_UNSUPPORTED, "%s: the batch dimension may not be partitioned", what);
    if (kh != kw || (kh != 3 && kh != 5 && kh != 7))
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: kernel %d x %d (supported: 3x3, 5x5, 7x7)", what, kh, kw);
    const int32_t pci = px->pshape[1], ph = px->pshape[2], pw = px->pshape[3];
    if (pco < 1 || nco < pco) return fail(DISTDL_ERR_SHAPE, "%s: %lld output channels on %d blocks", what, (long long)nco, pco);
    if (pci > kMaxChanBlocks || pco > kMaxChanBlocks)
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d blocks of a channel partition", what, kMaxChanBlocks);
    if ((int64_t)std::max(pci, pco) * ph * pw > kConvMaxWorkers)
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d shards of one tensor", what, kConvMaxWorkers);
    const int h = kh / 2;
    for (int k = 0; k < 4; ++k)
        for (int32_t c = 0; c < px->pshape[k]; ++c) {
            const int want = k < 2 ? 0 : h;
            if (px->hlo[k][c] != want || px->hhi[k][c] != want)
                return fail(DISTDL_ERR_SHAPE, "%s: halo widths must be 0,0,%d,%d on every side", what, h, h);
        }
    ConvGParams G;
    memset(&G, 0, sizeof(G));
    int64_t max_bh = 0, max_bw = 0;
    for (int32_t r = 0; r < ph; ++r) max_bh = std::max<int64_t>(max_bh, G.bh[r] = (int32_t)px->size[2][r]);
    for (int32_t c = 0; c < pw; ++c) max_bw = std::max<int64_t>(max_bw, G.bw[c] = (int32_t)px->size[3][c]);
    G.ph = ph;
    G.pw = pw;
    G.batch = (int32_t)px->global_shape[0];
    // channel blocks: the evenly split n_ci (from the partition) and n_co
    std::vector<int64_t> co_start, co_size;
    split_evenly(nco, pco, co_start, co_size);
    const int32_t p_out = adj ? pci : pco, p_in = adj ? pco : pci;
    for (int32_t b = 0; b < pci; ++b) (adj ? G.cnt_out : G.cnt_in)[b] = (int32_t)px->size[1][b];
    for (int32_t b = 0; b < pco; ++b) (adj ? G.cnt_in : G.cnt_out)[b] = (int32_t)co_size[b];
    G.p_in = p_in;
    G.pci = pci;
    // groups: as few as hold every channel of a block at up to eight per thread, of equal size
    int groups = 0, cp = 1;
    for (int32_t b = 0; b < p_out; ++b) {
        const int64_t cnt = G.cnt_out[b], parts = (cnt + 2 * kCgMaxPairs - 1) / (2 * kCgMaxPairs);
        if (groups + parts > kMaxGroups) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many output channels", what);
        for (int64_t q = 0, first = 0; q < parts; ++q) {
            const int64_t size = cnt / parts + (q < cnt % parts ? 1 : 0);
            G.grp_block[groups] = (uint8_t)b;
            G.grp_first[groups] = (uint16_t)first;
            G.grp_count[groups] = (uint8_t)size;
            cp = std::max(cp, (int)(size + 1) / 2);
            first += size;
            ++groups;
        }
    }
    const int spatial = ph * pw;
    for (int32_t k = 0; k < p_in * spatial; ++k) {
        if (!in[k]) return fail(DISTDL_ERR_INVALID_ARG, "%s: input shard %d is NULL", what, k);
        if (!aligned16(in[k])) return fail(DISTDL_ERR_ALIGNMENT, "%s: input shard %d is not 16-byte aligned", what, k);
        G.in[k] = (const float *)in[k];
    }
    for (int32_t k = 0; k < p_out * spatial; ++k) {
        if (!out[k]) return fail(DISTDL_ERR_INVALID_ARG, "%s: output shard %d is NULL", what, k);
        if (!aligned16(out[k])) return fail(DISTDL_ERR_ALIGNMENT, "%s: output shard %d is not 16-byte aligned", what, k);
        G.out[k] = (float *)out[k];
    }
    for (int32_t k = 0; k < pco * pci; ++k) {
        if (!w[k]) return fail(DISTDL_ERR_INVALID_ARG, "%s: weight block %d is NULL", what, k);
        G.w[k] = (const float *)w[k];
    }
    if (!adj && bias)
        for (int32_t b = 0; b < pco; ++b) G.bias[b] = (const float *)bias[b];
    int dev = 0, sms = 148;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    DISTDL_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    G.t = cg_choose(kh, cp, (int)max_bh, (int)max_bw, G.batch, ph * pw, groups, sms);
    const int64_t tiles_x = (max_bw + G.t.px * G.t.seg - 1) / (G.t.px * G.t.seg), tiles_y = (max_bh + G.t.th - 1) / G.t.th;
    const int64_t total = tiles_x * tiles_y * ph * pw * ((G.batch + G.t.tn - 1) / G.t.tn) * groups;
    if (total >= ((int64_t)1 << 31)) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles", what);
    G.groups = make_fast_div((uint32_t)groups);
    G.tiles_x = make_fast_div((uint32_t)tiles_x);
    G.pw_div = make_fast_div((uint32_t)pw);
    G.tiles_y = make_fast_div((uint32_t)tiles_y);
    G.ph_div = make_fast_div((uint32_t)ph);
    G.cols = make_fast_div((uint32_t)G.t.cols);
    G.rows = make_fast_div((uint32_t)G.t.rows);
    G.tn = make_fast_div((uint32_t)G.t.tn);
    G.seg = make_fast_div((uint32_t)G.t.seg);
    G.half_th = make_fast_div((uint32_t)(G.t.th / 2));
    cudaStream_t s = (cudaStream_t)stream;
    if (!adj)
        return kh == 3 ? launch_convg_pairs<3, false>(G, cp, total, s) : kh == 5 ? launch_convg_pairs<5, false>(G, cp, total, s)
                                                                                 : launch_convg_pairs<7, false>(G, cp, total, s);
    return kh == 3 ? launch_convg_pairs<3, true>(G, cp, total, s) : kh == 5 ? launch_convg_pairs<5, true>(G, cp, total, s)
                                                                            : launch_convg_pairs<7, true>(G, cp, total, s);
}

// ---------------------------------------------------------------------------------------------
// Parameter gradients (adjoint convolution algorithm):
//   dw^_{ijs}[o,c,a,b] = sum_{n,i,j} dy_{is}[n,o,i,j] * (H x)_{js}[n,c,i+a,j+b],   db^_{is}[o] = sum dy_{is}[n,o,i,j],
//   dw_{ij} = R_s dw^_{ijs},  db_i = R_s db^_{is}      (s: feature-space workers).
// A work item is (group of output channels, group of input channels, slice): the tiles slice, slice + S, ... of all images
// and workers, so the running sums stay in registers from tile to tile.  At the end of an item the block adds up its
// splits in order and writes one row of K * K + 1 values per channel pair to the scratch table; a second small kernel adds
// the rows of a pair in order.  The assignment of tiles to sums is static, so the result does not change from run to run.
// The error of an fp32 sum grows with its length, so a running sum takes at most kGgSumTerms terms (one tile at least): longer
// shares of tiles are several launches, each adding its sums onto the rows (0.6 to 1.3 % of the time, 8 us a launch; as a loop
// inside the kernel the accumulators' second life costs the inner loop a tenth).
//
// What bounds it: the fp32 pipe.  A thread owns one input channel c, one kernel row a and all OC output channels of the
// group, and walks along the rows of the tile four pixels at a time: K * OC sums as pairs (even pixels, odd pixels), one new
// 16-byte unit of x and OC broadcast units of dy per step, 2 K OC packed FMAs (80 for 5 x 5, eight channels, beside about
// 20 other instructions).  The (c, a) combinations of a block share the staged dy, the rows of the tile are split over what
// is left of the threads, and one more combination reads ones instead of x: its sums are db.  Lanes that own pixels
// instead (all K * K sums of one or two channel pairs per lane) spend as many instructions on putting x pairs together and
// on folding lanes as on FMAs.
// Measured (B200): 16 -> 16 channels, 5 x 5, 4 x 1024 x 1024 on 2 x 2 workers 1.41 ms = 38 TFLOP/s (1.94 ms with one channel
// pair per block, both its tiles staged again for every pair); 6 -> 16 channels, 256 images of 28 x 28 0.063 ms (1.61 ms).
// Two steps per turn instead of moving the window: 1.63 ms (spills); 192 threads with 168 registers: 1.67 ms.
// ---------------------------------------------------------------------------------------------
constexpr int kGradRow = 64;            // floats per row of the scratch table (K * K + 1 <= 50 used)
constexpr int kGgThreads = 256;
constexpr int kGgSmem = 112 * 1024;     // two blocks per SM
constexpr int kGgSumTerms = 2560;
// output channels of a group: more would need more than the 128 registers of two blocks per SM
constexpr int gg_max_oc(int k) { return k == 7 ? 4 : 8; }

struct GgShape {
    int32_t tn, th, seg;                // tile: tn images x th rows x 4 * seg columns
    int32_t rows, units, pitch;         // staged x rows of one image, 16-byte units and floats per row
    int32_t x_floats;                   // one staged input channel
    int32_t px;                         // pixels of a tile = floats of one staged dy channel
    int32_t buf_floats;                 // x of all input channels, then dy: per four pixels the units of all output channels
    int32_t smem_bytes;
};

struct ConvGGradParams {
    const float *x[kConvMaxWorkers], *dy[kConvMaxWorkers];
    int32_t bh[kConvMaxWorkers], bw[kConvMaxWorkers];
    int32_t x_start[8], x_cnt[8], y_start[8], y_cnt[8];     // channels of every block
    int32_t cgrp[9], ogrp[9];           // first group of every block; [blocks]: all groups
    int32_t x_blocks, y_blocks, ph, pw, batch, n_x;
    int32_t slices;                     // slices per pair of groups
    int32_t xc, splits;                 // input channels per block; splits of a tile's rows
    int32_t tiles;                      // tiles of one channel: workers, images, rows, columns
    int32_t run;                        // tiles of a launch: a whole number of turns of the slices
    int32_t first, last;                // those of this launch
    uint32_t zero;                      // 0, see fresh()
    float *partial;                     // [pairs][slices][kGradRow]
    GgShape t;
    FastDiv slice_div, cgrp_div, tiles_x, pw_div, tiles_y, ph_div, units, rows, seg, th;
};

// FIRST, MORE: whether this may be the launch of an item's first tiles, and one of those after it.  Compiled apart for 5 x 5 and 7 x 7 (5 x 5,
// 2 -> 6 channels, 501 x 508: 18.7 us, as one kernel 19.3); 3 x 3 is faster as one (8 -> 6, 8 x 509 x 513: 119.7 us, apart 122).
template <int K, int OC, bool FIRST, bool MORE>
__global__ void __launch_bounds__(kGgThreads, 2)
convg_grad_kernel(const __grid_constant__ ConvGGradParams G) {
    stream_enter();
    constexpr int PH = K / 2;
    constexpr int NU = (4 + K - 1 + 3) / 4;                 // 16-byte units of x that four pixels of a kernel row need
    extern __shared__ __align__(16) float smem[];           // two buffers, then a row of ones
    const GgShape &T = G.t;
    const int tid = threadIdx.x;
    const int spatial = G.ph * G.pw;

    uint32_t rest = blockIdx.x;
    const int sl = (int)fast_rem(G.slice_div, rest);
    const int cg = (int)fast_rem(G.cgrp_div, rest);
    const int og = (int)rest;
    int jb = 0, ib = 0;
    while (cg >= G.cgrp[jb + 1]) ++jb;
    while (og >= G.ogrp[ib + 1]) ++ib;
    // groups of a block: equal sizes, the first ones one channel larger
    const int cparts = G.cgrp[jb + 1] - G.cgrp[jb], cq = cg - G.cgrp[jb];
    const int oparts = G.ogrp[ib + 1] - G.ogrp[ib], oq = og - G.ogrp[ib];
    const int xcnt = G.x_cnt[jb], ycnt = G.y_cnt[ib];
    const int cbase = xcnt / cparts, crem = xcnt - cbase * cparts, obase = ycnt / oparts, orem = ycnt - obase * oparts;
    const int xc = cbase + (cq < crem ? 1 : 0), c0 = cq * cbase + min(cq, crem);
    const int oc = obase + (oq < orem ? 1 : 0), o0 = oq * obase + min(oq, orem);

    const int combos = G.xc * K + 1;
    const int split = tid / combos, combo = tid - split * combos;
    const bool is_ones = combo == combos - 1;
    const int my_c = combo / K, my_a = combo - my_c * K;
    const bool active = split < G.splits && (is_ones || my_c < xc);
    const int x_pitch = is_ones ? 0 : T.pitch;
    const uint32_t zero = G.zero;

    uint64_t acc[OC][K];
#pragma unroll
    for (int k = 0; k < OC; ++k)
#pragma unroll
        for (int b = 0; b < K; ++b) acc[k][b] = 0ull;
    for (int i = tid; i < T.pitch; i += kGgThreads) smem[2 * T.buf_floats + i] = 1.f;
    for (int b = 0; b < 2; ++b)         // output channels that no copy ever writes
        for (int i = tid; i < OC * T.px; i += kGgThreads)
            if ((i >> 2) % OC >= oc) smem[b * T.buf_floats + G.xc * T.x_floats + i] = 0.f;

    const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(smem);
    // Cells are staged in units of four: one 16-byte copy where the unit lies inside one shard and its rows start on
    // 16-byte boundaries, element by element otherwise.  Where a unit comes from is worked out once for all channels.
    auto stage = [&](uint32_t L, int buf) {
        const int tx = (int)fast_rem(G.tiles_x, L);
        const int c = (int)fast_rem(G.pw_div, L);
        const int ty = (int)fast_rem(G.tiles_y, L);
        const int r = (int)fast_rem(G.ph_div, L);
        const int n0 = (int)L * T.tn;
        const int bh = G.bh[r], bw = G.bw[c];
        const int i0 = ty * T.th, j0 = tx * 4 * T.seg;
        if (i0 >= bh || j0 >= bw) return false;
        const int th = min(T.th, bh - i0), tw = min(4 * T.seg, bw - j0);
        const int need_rows = th + K - 1, need_cols = tw + K - 1;
        const bool x_wide = ((bw + 2 * PH) & 3) == 0, y_wide = (bw & 3) == 0;
        float *xs = smem + buf * T.buf_floats, *ds = xs + G.xc * T.x_floats;
        const uint32_t xs_s = smem_s + (uint32_t)(buf * T.buf_floats) * 4u, ds_s = xs_s + (uint32_t)(G.xc * T.x_floats) * 4u;
        for (int e = tid; e < T.tn * T.rows * T.units; e += kGgThreads) {
            uint32_t q = (uint32_t)e;
            const int s = 4 * (int)fast_rem(G.units, q);
            const int line = (int)q;                        // row of all images
            const int ry = (int)fast_rem(G.rows, q);
            const int tn = (int)q;
            const uint32_t dst = (uint32_t)(line * T.pitch + s);
            int rr, i;
            const bool row_ok = conv_owner(G.bh, G.ph, r, i0 - PH + ry, rr, i) && n0 + tn < G.batch && ry < need_rows;
            const int j = j0 - PH + s;
            if (row_ok && x_wide && j >= 0 && j + 4 <= bw && s + 4 <= need_cols) {
                const uint32_t pitch = (uint32_t)(bw + 2 * PH), plane = (uint32_t)(G.bh[rr] + 2 * PH) * pitch;
                const float *p = G.x[jb * spatial + rr * G.pw + c] + (size_t)((n0 + tn) * xcnt + c0) * plane +
                                 ((uint32_t)(i + PH) * pitch + (uint32_t)(PH + j));
                uint32_t d = xs_s + dst * 4u;
#pragma unroll 1
                for (int k = 0; k < xc; ++k, p += plane, d += (uint32_t)T.x_floats * 4u) cp_async16_to(d, p);
            } else {
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    int cc, jj;
                    // cells that no pixel of the tile reads are zero: they meet the zeros of the dy tile
                    const bool ok = row_ok && s + f < need_cols && conv_owner(G.bw, G.pw, c, j + f, cc, jj);
                    if (ok) {
                        const uint32_t pitch = (uint32_t)(G.bw[cc] + 2 * PH), plane = (uint32_t)(G.bh[rr] + 2 * PH) * pitch;
                        const float *p = G.x[jb * spatial + rr * G.pw + cc] + (size_t)((n0 + tn) * xcnt + c0) * plane +
                                         ((uint32_t)(i + PH) * pitch + (uint32_t)(PH + jj));
                        uint32_t d = xs_s + (dst + (uint32_t)f) * 4u;
#pragma unroll 1
                        for (int k = 0; k < xc; ++k, p += plane, d += (uint32_t)T.x_floats * 4u) cp_async4_to(d, p);
                    } else {
#pragma unroll 1
                        for (int k = 0; k < xc; ++k) xs[k * T.x_floats + dst + f] = 0.f;
                    }
                }
            }
        }
        const uint32_t plane_y = (uint32_t)bh * (uint32_t)bw;
        const float *dysh = G.dy[ib * spatial + r * G.pw + c];
        for (int e = tid; e < T.tn * T.th * T.seg; e += kGgThreads) {
            uint32_t q = (uint32_t)e;
            const int col = 4 * (int)fast_rem(G.seg, q);
            const int row = (int)fast_rem(G.th, q);
            const int tn = (int)q;
            const bool row_ok = n0 + tn < G.batch && row < th;
            const float *p = dysh + (size_t)((n0 + tn) * ycnt + o0) * plane_y + ((uint32_t)(i0 + row) * (uint32_t)bw + (uint32_t)(j0 + col));
            if (row_ok && y_wide && col + 4 <= tw) {
                uint32_t d = ds_s + (uint32_t)(e * OC) * 16u;
#pragma unroll 1
                for (int k = 0; k < oc; ++k, p += plane_y, d += 16u) cp_async16_to(d, p);
            } else {
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    if (row_ok && col + f < tw) {
                        const float *pf = p + f;
                        uint32_t d = ds_s + (uint32_t)(4 * e * OC + f) * 4u;
#pragma unroll 1
                        for (int k = 0; k < oc; ++k, pf += plane_y, d += 16u) cp_async4_to(d, pf);
                    } else {
#pragma unroll 1
                        for (int k = 0; k < oc; ++k) ds[4 * (e * OC + k) + f] = 0.f;
                    }
                }
            }
        }
        return true;
    };

    int L = (MORE ? G.first : 0) + sl, buf = 0;
    bool cur = L < G.last && stage((uint32_t)L, 0);
    cp_async_commit();
    while (L < G.last) {
        cp_async_wait_group<0>();
        __syncthreads();                // this tile has arrived, the other buffer has been read
        const int next = L + G.slices;
        const bool nxt = next < G.last && stage((uint32_t)next, buf ^ 1);
        cp_async_commit();
        if (cur && active) {
            const float *xt = is_ones ? smem + 2 * T.buf_floats : smem + buf * T.buf_floats + my_c * T.x_floats + my_a * T.pitch;
            const float *dt = smem + buf * T.buf_floats + G.xc * T.x_floats;
#pragma unroll 1
            for (int line = split; line < T.tn * T.th; line += G.splits) {
                const int img = (int)fast_quot(G.th, (uint32_t)line);
                const float *xp = xt + (line + img * (K - 1)) * x_pitch;        // an image has th + K - 1 staged rows
                const float *dp = dt + line * (4 * OC * T.seg);
                uint64_t U[NU][2];
#pragma unroll
                for (int v = 0; v + 1 < NU; ++v) {
                    const ulonglong2 f = *reinterpret_cast<const ulonglong2 *>(xp + 4 * v);
                    U[v][0] = f.x;
                    U[v][1] = f.y;
                }
                xp += 4 * (NU - 1);
#pragma unroll 1
                for (int q = 0; q < T.seg; ++q) {
                    const ulonglong2 f = *reinterpret_cast<const ulonglong2 *>(xp);
                    U[NU - 1][0] = f.x;
                    U[NU - 1][1] = f.y;
                    uint64_t Q[2 * NU - 1];                 // U holds (x[2i], x[2i+1]), Q (x[2i+1], x[2i+2])
#pragma unroll
                    for (int v = 0; v < 2 * NU - 1; ++v) {
                        float a0, a1, b0, b1;
                        unpack2(U[v / 2][v % 2], a0, a1);
                        unpack2(U[(v + 1) / 2][(v + 1) % 2], b0, b1);
                        Q[v] = pack2(fresh(a1, zero), fresh(b0, zero));
                    }
#pragma unroll
                    for (int k = 0; k < OC; ++k) {
                        const ulonglong2 d = *reinterpret_cast<const ulonglong2 *>(dp + 4 * k);
#pragma unroll
                        for (int b = 0; b < K; ++b) acc[k][b] = fma2((b & 1) ? Q[b / 2] : U[b / 4][b / 2 % 2], d.x, acc[k][b]);
#pragma unroll
                        for (int b = 0; b < K; ++b)
                            acc[k][b] = fma2((b & 1) ? Q[b / 2 + 1] : U[(b / 2 + 1) / 2][(b / 2 + 1) % 2], d.y, acc[k][b]);
                    }
                    // the window moves on by one unit (moves: two steps per turn instead need registers that are not there)
#pragma unroll
                    for (int v = 0; v + 1 < NU; ++v) {
                        U[v][0] = U[v + 1][0];
                        U[v][1] = U[v + 1][1];
                    }
                    xp += 4;
                    dp += 4 * OC;
                }
            }
        }
        cur = nxt;
        L = next;
        buf ^= 1;
    }
    // add up: the two halves of a pair, then the splits in order, onto the launches before; one row per channel pair
    __syncthreads();
    if (active)
#pragma unroll
        for (int k = 0; k < OC; ++k)
#pragma unroll
            for (int b = 0; b < K; ++b) {
                float lo, hi;
                unpack2(acc[k][b], lo, hi);
                smem[(k * K + b) * (G.splits * combos) + tid] = lo + hi;
            }
    __syncthreads();
    for (int idx = tid; idx < oc * K * combos; idx += kGgThreads) {
        const int kb = idx / combos, cb = idx - kb * combos;
        const int k = kb / K, b = kb - k * K;
        const bool ones = cb == combos - 1;
        const int ch = ones ? 0 : cb / K;
        if (ones ? b > 0 : ch >= xc) continue;              // the sums against ones are the same for every b
        const float *src = smem + kb * (G.splits * combos) + cb;
        float v = src[0];
        for (int s = 1; s < G.splits; ++s) v += src[s * combos];
        const size_t pair = (size_t)(G.y_start[ib] + o0 + k) * G.n_x + (G.x_start[jb] + c0 + ch);
        float *sum = G.partial + (pair * G.slices + sl) * kGradRow + (ones ? K * K : (cb - ch * K) * K + b);
        *sum = MORE && (!FIRST || G.first) ? *sum + v : v;
    }
}

// One block per channel pair: the rows of its slices added in a fixed order -- thread group h takes rows h, h + H, ..., the
// groups' sums are added in order -- into tap t of dw block (i, j) at [o_local][c_local]; the last entry of the c = 0
// pairs goes to db_i[o_local].
constexpr int kGradFoldGroups = 8;
struct ConvGGradOut {
    float *dw[64];
    float *db[8];
};
__global__ void __launch_bounds__(64 * kGradFoldGroups)
convg_grad_finish_kernel(const __grid_constant__ ConvGGradParams G, const __grid_constant__ ConvGGradOut O, int taps) {
    stream_enter();
    __shared__ float part[kGradFoldGroups][64];
    const int q = blockIdx.x, t = threadIdx.x & 63, h = threadIdx.x >> 6;
    const int o = q / G.n_x, c = q - o * G.n_x;
    float v = 0.f;
    if (t < taps || (t == taps && c == 0)) {
        const float *row = G.partial + (size_t)q * G.slices * kGradRow + t;
#pragma unroll 8
        for (int s = h; s < G.slices; s += kGradFoldGroups) v += row[(size_t)s * kGradRow];
    }
    part[h][t] = v;
    __syncthreads();
    if (h > 0 || t > taps) return;
    v = part[0][t];
#pragma unroll
    for (int k = 1; k < kGradFoldGroups; ++k) v += part[k][t];
    int ib = 0, jb = 0;
    while (ib + 1 < G.y_blocks && o >= G.y_start[ib + 1]) ++ib;
    while (jb + 1 < G.x_blocks && c >= G.x_start[jb + 1]) ++jb;
    if (t < taps) O.dw[ib * G.x_blocks + jb][((size_t)(o - G.y_start[ib]) * G.x_cnt[jb] + (c - G.x_start[jb])) * taps + t] = v;
    else if (O.db[ib] && c == 0) O.db[ib][o - G.y_start[ib]] = v;
}

static GgShape gg_shape(int K, int tn, int th, int seg, int xc, int oc) {
    GgShape t;
    memset(&t, 0, sizeof(t));
    const int nu = (4 + K - 1 + 3) / 4;
    t.tn = tn;
    t.th = th;
    t.seg = seg;
    t.rows = th + K - 1;
    t.units = (4 * seg + K - 1 + 3) / 4;
    // eight lanes are eight consecutive (channel, kernel row) combinations: an odd number of units per row and, from channel
    // to channel, K rows' worth of units modulo eight put their 16-byte reads into eight different bank groups
    int pu = std::max(t.units, seg - 1 + nu);
    pu += 1 - pu % 2;
    int xu = tn * t.rows * pu;
    while ((xu - K * pu) % 8 != 0) ++xu;
    t.pitch = 4 * pu;
    t.x_floats = 4 * xu;
    t.px = tn * th * 4 * seg;
    t.buf_floats = xc * t.x_floats + oc * t.px;
    const int fold = oc * K * kGgThreads * 4;               // the sums of all threads, at the end
    t.smem_bytes = std::max((2 * t.buf_floats + t.pitch) * 4, fold);
    return t;
}

// Tile shape with the smallest estimated time of a launch: tiles per block times warp instructions per tile (a packed FMA
// counts 2.5: the rate of a register outer product), staging 40 per unit and 2 or 12 more per channel.  Sizes are tried from
// the largest down in steps of a fifth, shards cut into that many equal tiles, and what cannot win by its FMAs alone is passed
// over: 3 to 7 us of host time (7 to 27 us with every size in turn).
static GgShape gg_choose(int K, int xc, int splits, int oc, int max_bh, int max_bw, int batch, int workers, int slots, double *tile_cost) {
    GgShape best;
    memset(&best, 0, sizeof(best));
    double best_cost = 0;
    const bool x_wide = (max_bw + K - 1) % 4 == 0, y_wide = max_bw % 4 == 0;
    int nx_before = 0;
    for (int try_seg = 32; try_seg >= 1; try_seg -= std::max(1, try_seg / 5)) {
        const int nx = (max_bw + 4 * try_seg - 1) / (4 * try_seg);
        if (nx == nx_before) continue;
        nx_before = nx;
        const int seg = (max_bw + 4 * nx - 1) / (4 * nx);
        int ny_before = 0;
        for (int try_th = 128; try_th >= 1; try_th -= std::max(1, try_th / 5)) {
            const int ny = (max_bh + try_th - 1) / try_th;
            if (ny == ny_before) continue;
            ny_before = ny;
            const int th = (max_bh + ny - 1) / ny;
            // the sums of all threads and one image's dy alone bound the images of a tile
            const int room = std::min(64, kGgSmem / (2 * 4 * (oc * th * 4 * seg + xc * (th + K - 1) * 4 * seg)));
            for (int tn = std::min(room, batch); tn >= 1; tn -= std::max(1, tn / 5)) {
                const int64_t tiles = (int64_t)(nx * ny) * ((int64_t)workers * (tn == 1 ? batch : (batch + tn - 1) / tn));
                const double turns = (double)((tiles + slots - 1) / slots);
                const double compute = 8.0 * ((tn * th + splits - 1) / splits) * (seg * (2.0 * K * oc * 2.5 + oc + 10) + 20);
                if (best.tn != 0 && turns * (compute + 1200) >= best_cost) continue;
                const GgShape t = gg_shape(K, tn, th, seg, xc, oc);
                if (t.smem_bytes > kGgSmem) continue;
                const double staging = (tn * t.rows * t.units * (40.0 + xc * (x_wide ? 2 : 12)) + tn * th * seg * (20.0 + oc * (y_wide ? 2 : 12))) / 32;
                const double cost = turns * (compute + staging + 1200);
                if (best.tn == 0 || cost < best_cost) {
                    best = t;
                    best_cost = cost;
                    *tile_cost = cost / turns;
                }
            }
        }
    }
    return best;
}

static int64_t gg_tiles(const GgShape &t, int64_t max_bh, int64_t max_bw, int64_t batch, int64_t workers) {
    return (max_bw + 4 * t.seg - 1) / (4 * t.seg) * ((max_bh + t.th - 1) / t.th) * workers * ((batch + t.tn - 1) / t.tn);
}

// Geometry, groups and slices: shared by the workspace query and the launch.
static distdl_status_t convg_grad_plan(const distdl_partition *px, int64_t nco, int32_t pco, int32_t kh, int32_t kw,
                                       const char *what, ConvGGradParams *G, int *oc_out, int *grid) {
    if (!px) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL partition", what);
    if (px->rank != 4 || px->dtype != DISTDL_F32) return fail(DISTDL_ERR_SHAPE, "%s: needs a rank-4 F32 partition", what);
    if (px->any_periodic()) return fail(DISTDL_ERR_UNSUPPORTED, "%s: periodic partitions are not supported by the fused layers", what);
    if (px->pshape[0] != 1) return fail(DISTDL_ERR_UNSUPPORTED, "%s: the batch dimension may not be partitioned", what);
    if (kh != kw || (kh != 3 && kh != 5 && kh != 7))
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: kernel %d x %d (supported: 3x3, 5x5, 7x7)", what, kh, kw);
    const int32_t pci = px->pshape[1], ph = px->pshape[2], pw = px->pshape[3];
    if (pco < 1 || nco < pco) return fail(DISTDL_ERR_SHAPE, "%s: %lld output channels on %d blocks", what, (long long)nco, pco);
    if (pci > 8 || pco > 8) return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than 8 blocks of a channel partition", what);
    if ((int64_t)std::max(pci, pco) * ph * pw > kConvMaxWorkers)
        return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d shards of one tensor", what, kConvMaxWorkers);
    const int h = kh / 2;
    for (int k = 0; k < 4; ++k)
        for (int32_t c = 0; c < px->pshape[k]; ++c) {
            const int want = k < 2 ? 0 : h;
            if (px->hlo[k][c] != want || px->hhi[k][c] != want)
                return fail(DISTDL_ERR_SHAPE, "%s: halo widths must be 0,0,%d,%d on every side", what, h, h);
        }
    int64_t max_bh = 0, max_bw = 0;
    for (int32_t r = 0; r < ph; ++r) max_bh = std::max<int64_t>(max_bh, G->bh[r] = (int32_t)px->size[2][r]);
    for (int32_t c = 0; c < pw; ++c) max_bw = std::max<int64_t>(max_bw, G->bw[c] = (int32_t)px->size[3][c]);
    const int64_t pairs = nco * px->global_shape[1];
    if (pairs > 65536) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles or channel pairs", what);
    G->ph = ph;
    G->pw = pw;
    G->batch = (int32_t)px->global_shape[0];
    G->n_x = (int32_t)px->global_shape[1];
    G->x_blocks = pci;
    G->y_blocks = pco;
    std::vector<int64_t> co_start, co_size;
    split_evenly(nco, pco, co_start, co_size);
    // output channels: as few groups as hold a block, of equal size
    int max_x = 0, oc = 2;
    G->cgrp[0] = G->ogrp[0] = 0;
    for (int32_t b = 0; b < pco; ++b) {
        G->y_start[b] = (int32_t)co_start[b];
        const int cnt = G->y_cnt[b] = (int32_t)co_size[b];
        const int parts = (cnt + gg_max_oc(kh) - 1) / gg_max_oc(kh);
        oc = std::max(oc, ((cnt + parts - 1) / parts + 1) / 2 * 2);
        G->ogrp[b + 1] = G->ogrp[b] + parts;
    }
    // input channels per block: threads that own no combination against staging dy for every group of them
    for (int32_t b = 0; b < pci; ++b) max_x = std::max(max_x, (int)px->size[1][b]);
    int xc = 1;
    double best = -1;
    for (int a = 1; a <= 8 && a <= max_x; ++a) {
        const int g = (max_x + a - 1) / a, splits = kGgThreads / (a * kh + 1);
        const double cost = g * (8.0 * kh * oc * 1.4 / splits + (1.4 * a + oc) * 0.06);
        if (best < 0 || cost < best) {
            best = cost;
            xc = a;
        }
    }
    for (int32_t b = 0; b < pci; ++b) {
        G->x_start[b] = (int32_t)px->start[1][b];
        G->x_cnt[b] = (int32_t)px->size[1][b];
        G->cgrp[b + 1] = G->cgrp[b] + (G->x_cnt[b] + xc - 1) / xc;
    }
    G->xc = xc;
    G->splits = kGgThreads / (xc * kh + 1);
    int dev = 0, sms = 148;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    DISTDL_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // Slices: as many as fill the resident blocks once -- or, where many groups leave that far from full or past it, the number
    // (16 at most: it is the size of the scratch table) whose turns of the resident blocks take the least time; 15000: what a block
    // spends besides its tiles.  5 x 5, 128 x 128: 80 -> 80 channels, four images, 943 us with the two slices that fit, now 687; 136 ->
    // 144, two images (more groups than blocks), 1403 and 987.
    const int64_t group_pairs = (int64_t)G->cgrp[pci] * G->ogrp[pco], resident = 2 * (int64_t)sms;
    int64_t slots = std::max<int64_t>(1, resident / group_pairs);
    double tile_cost = 0;
    const auto choose = [&]() {
        G->t = gg_choose(kh, xc, G->splits, oc, (int)max_bh, (int)max_bw, G->batch, ph * pw, (int)slots, &tile_cost);
        return gg_tiles(G->t, max_bh, max_bw, G->batch, ph * pw);
    };
    int64_t tiles = choose();
    if (slots < 16) {
        const auto time = [&](int64_t n) {
            return (double)((n * group_pairs + resident - 1) / resident) * ((double)((tiles + n - 1) / n) * tile_cost + 15000);
        };
        int64_t best_slots = slots;
        for (int64_t n = 1; n <= std::min<int64_t>(16, tiles); ++n)
            if (time(n) < 0.97 * time(best_slots)) best_slots = n;
        if (best_slots != slots) {
            slots = best_slots;
            tiles = choose();
        }
    }
    if (tiles >= ((int64_t)1 << 31)) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles or channel pairs", what);
    const int64_t tiles_x = (max_bw + 4 * G->t.seg - 1) / (4 * G->t.seg), tiles_y = (max_bh + G->t.th - 1) / G->t.th;
    G->tiles = (int32_t)tiles;
    const int64_t slices = std::min<int64_t>(slots, tiles);
    G->slices = (int32_t)slices;
    // launches with equal shares of a slice's tiles, none with more terms to a sum than the limit
    const int64_t terms = (int64_t)((G->t.tn * G->t.th + G->splits - 1) / G->splits) * 2 * G->t.seg, share = (tiles + slices - 1) / slices;
    const int64_t most = std::max<int64_t>(1, kGgSumTerms / terms), launches = (share + most - 1) / most;
    G->run = (int32_t)std::min<int64_t>(tiles, (share + launches - 1) / launches * slices);
    G->slice_div = make_fast_div((uint32_t)slices);
    G->cgrp_div = make_fast_div((uint32_t)G->cgrp[pci]);
    G->tiles_x = make_fast_div((uint32_t)tiles_x);
    G->pw_div = make_fast_div((uint32_t)pw);
    G->tiles_y = make_fast_div((uint32_t)tiles_y);
    G->ph_div = make_fast_div((uint32_t)ph);
    G->units = make_fast_div((uint32_t)G->t.units);
    G->rows = make_fast_div((uint32_t)G->t.rows);
    G->seg = make_fast_div((uint32_t)G->t.seg);
    G->th = make_fast_div((uint32_t)G->t.th);
    *oc_out = oc;
    *grid = (int)(slices * group_pairs);
    return DISTDL_OK;
}

template <int K, int OC>
static distdl_status_t launch_convg_grad(ConvGGradParams &G, const ConvGGradOut &O, int grid, int pairs, cudaStream_t s) {
    static bool configured_on[kMaxDevicesPerProcess] = {false};
    int dev = 0;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevicesPerProcess)
        return fail(DISTDL_ERR_UNSUPPORTED, "device index %d: at most %d devices per process", dev, kMaxDevicesPerProcess);
    {
        std::lock_guard<std::mutex> setup_lock(setup_mutex());
        if (!configured_on[dev]) {
            DISTDL_CUDA_CHECK(cudaFuncSetAttribute(convg_grad_kernel<K, OC, true, K == 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGgSmem));
            DISTDL_CUDA_CHECK(cudaFuncSetAttribute(convg_grad_kernel<K, OC, K == 3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGgSmem));
            configured_on[dev] = true;
        }
    }
    for (int64_t at = 0; at < G.tiles; at += G.run) {
        G.first = (int32_t)at;
        G.last = (int32_t)std::min<int64_t>(G.tiles, at + G.run);
        if (at == 0) launch_in_stream(convg_grad_kernel<K, OC, true, K == 3>, grid, kGgThreads, G.t.smem_bytes, s, G);
        else launch_in_stream(convg_grad_kernel<K, OC, K == 3, true>, grid, kGgThreads, G.t.smem_bytes, s, G);
        DISTDL_CUDA_CHECK(cudaGetLastError());
    }
    launch_in_stream(convg_grad_finish_kernel, pairs, 64 * kGradFoldGroups, 0, s, G, O, K * K);
    DISTDL_CUDA_CHECK(cudaGetLastError());
    return DISTDL_OK;
}

template <int K>
static distdl_status_t launch_convg_grad_channels(ConvGGradParams &G, const ConvGGradOut &O, int oc, int grid, int pairs, cudaStream_t s) {
    constexpr int most = gg_max_oc(K);
    if (oc == 2) return launch_convg_grad<K, 2>(G, O, grid, pairs, s);
    if (oc == 4) return launch_convg_grad<K, 4>(G, O, grid, pairs, s);
    if (oc == 6) return launch_convg_grad<K, most < 6 ? most : 6>(G, O, grid, pairs, s);
    return launch_convg_grad<K, most>(G, O, grid, pairs, s);
}

}  // namespace distdl

extern "C" distdl_status_t distdl_convg_fwd(const distdl_partition_t *px, int64_t nco, int32_t pco, const void *const *x,
                                            const void *const *w, const void *const *bias, int32_t kh, int32_t kw,
                                            void *const *y, void *stream) {
    return distdl::convg_impl(px, nco, pco, x, w, bias, kh, kw, y, stream, false, "convg_fwd");
}
extern "C" distdl_status_t distdl_convg_adj(const distdl_partition_t *px, int64_t nco, int32_t pco, const void *const *dy,
                                            const void *const *w, int32_t kh, int32_t kw, void *const *dx, void *stream) {
    return distdl::convg_impl(px, nco, pco, dy, w, nullptr, kh, kw, dx, stream, true, "convg_adj");
}

extern "C" distdl_status_t distdl_convg_adj_params_workspace(const distdl_partition_t *px, int64_t nco, int32_t pco,
                                                             int32_t kh, int32_t kw, int64_t *bytes) {
    using namespace distdl;
    clear_error();
    if (!bytes) return fail(DISTDL_ERR_INVALID_ARG, "convg_adj_params_workspace: NULL argument");
    ConvGGradParams G;
    memset(&G, 0, sizeof(G));
    int oc = 2, grid = 0;
    const distdl_status_t st = convg_grad_plan(px, nco, pco, kh, kw, "convg_adj_params_workspace", &G, &oc, &grid);
    if (st != DISTDL_OK) return st;
    *bytes = nco * G.n_x * G.slices * kGradRow * (int64_t)sizeof(float);
    return DISTDL_OK;
}

extern "C" distdl_status_t distdl_convg_adj_params(const distdl_partition_t *px, int64_t nco, int32_t pco,
                                                   const void *const *x, const void *const *dy, int32_t kh, int32_t kw,
                                                   void *const *dw, void *const *db, void *workspace,
                                                   int64_t workspace_bytes, void *stream) {
    using namespace distdl;
    clear_error();
    const char *what = "convg_adj_params";
    if (!px || !x || !dy || !dw || !workspace) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL argument", what);
    ConvGGradParams G;
    memset(&G, 0, sizeof(G));
    int oc = 2, grid = 0;
    const distdl_status_t st = convg_grad_plan(px, nco, pco, kh, kw, what, &G, &oc, &grid);
    if (st != DISTDL_OK) return st;
    const int64_t need = nco * G.n_x * G.slices * kGradRow * (int64_t)sizeof(float);
    if (workspace_bytes < need) return fail(DISTDL_ERR_INVALID_ARG, "%s: workspace of %lld bytes, %lld needed", what,
                                            (long long)workspace_bytes, (long long)need);
    if (!aligned16(workspace)) return fail(DISTDL_ERR_ALIGNMENT, "%s: workspace not 16-byte aligned", what);
    for (int32_t k = 0; k < G.x_blocks * G.ph * G.pw; ++k) {
        if (!x[k]) return fail(DISTDL_ERR_INVALID_ARG, "%s: x shard %d is NULL", what, k);
        if (!aligned16(x[k])) return fail(DISTDL_ERR_ALIGNMENT, "%s: x shard %d is not 16-byte aligned", what, k);
        G.x[k] = (const float *)x[k];
    }
    for (int32_t k = 0; k < G.y_blocks * G.ph * G.pw; ++k) {
        if (!dy[k]) return fail(DISTDL_ERR_INVALID_ARG, "%s: dy shard %d is NULL", what, k);
        if (!aligned16(dy[k])) return fail(DISTDL_ERR_ALIGNMENT, "%s: dy shard %d is not 16-byte aligned", what, k);
        G.dy[k] = (const float *)dy[k];
    }
    ConvGGradOut O;
    memset(&O, 0, sizeof(O));
    for (int32_t k = 0; k < G.x_blocks * G.y_blocks; ++k) {
        if (!dw[k]) return fail(DISTDL_ERR_INVALID_ARG, "%s: dw block %d is NULL", what, k);
        O.dw[k] = (float *)dw[k];
    }
    if (db)
        for (int32_t b = 0; b < G.y_blocks; ++b) O.db[b] = (float *)db[b];
    G.partial = (float *)workspace;
    cudaStream_t s = (cudaStream_t)stream;
    const int pairs = (int)nco * G.n_x;
    if (kh == 3) return launch_convg_grad_channels<3>(G, O, oc, grid, pairs, s);
    if (kh == 5) return launch_convg_grad_channels<5>(G, O, oc, grid, pairs, s);
    return launch_convg_grad_channels<7>(G, O, oc, grid, pairs, s);
}
