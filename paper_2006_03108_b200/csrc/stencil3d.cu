// Distributed star-stencil layer on a rank-3 tensor (Section 4, "Sparse layers": a sliding-kernel
// layer on a feature-space partition is the halo exchange H followed by the local kernel; its
// adjoint is the local adjoint followed by H*).  The kernel is a star: one 1-D kernel of radius R
// per dimension,
//   y[i] = sum_d sum_{k=-R..R} w[d][k+R] * x[i + k e_d],     x = 0 outside the tensor,
// which is the shape of the finite-difference operators of the volumetric problems the paper
// names as its target.  Both directions are fused with their exchange: a thread block reads the
// planes, rows and columns it needs straight from the bulk of whichever shard owns them, so no
// ghost cell is ever written to or read from device memory by the forward pass.  The adjoint is
// the same star with every 1-D kernel reversed, evaluated in gather form on the bulk-shaped dy,
// written into the bulk of the padded dx shards whose ghosts are cleared as H* leaves them.
//
// Blocking: a block (four warps) owns 16 rows x 64 columns (or 8 x 128) of one shard and marches through a chunk
// of planes.  A thread owns 4 consecutive columns of two consecutive rows and keeps the running sums of the
// 2R+1 outputs around the current plane in registers: a cell of plane p is tap 2R - i of output p - R + i, and the
// sum moves from slot i + 1 to slot i as the destination of that very FMA (a queue of the 2R+1 input planes instead costs
// 2R+1 register moves per cell).  The current plane with R extra rows above / below and R extra columns left / right
// lies in shared memory (y and x neighbours, added to the output in the middle; a star needs no corners); the two rows of a
// thread share their y neighbours, 2R + 2 plane rows, two of them its own.  Planes arrive by asynchronous copies
// straight into a ring of five, four planes ahead: a plane's cells are needed at once when it becomes the current one, so
// one plane of registers does not cover the latency of device memory.  One barrier per plane.  Rows that do not start on
// 16-byte boundaries (R < 4 on the padded side) are copied four bytes a lane, a warp's cells next to one another.
// Issue bounds it, not memory: 116 of ~300 instructions a plane are the warp's FMA (25 taps on eight cells, pairs
// packed but for the odd column shifts), and a fourth block per multiprocessor makes it 301 us from 233.  At 512^3, R = 4,
// forward 308 -> 233 us, adjoint 365 -> 264 us, where reading and writing the bulk once takes 164 us and 170 us (those with tiles of 8 x 128; 16 x 64
// forward and adjoint 565 -> 540 us together, shards that 128 columns do not fit: 296 x 226 x 96 on 1 x 1 x 2 workers 102 -> 43, 201 x 238 x 44 on
// 1 x 2 x 4 195 -> 103, 151 x 307 x 238 on 3 x 3 x 4, R = 2, 140 -> 85).  The rest
// of the radii and sizes gain by the rule for the chunks as well (200^3, R = 2: 61 -> 32 and 78 -> 31 us; 64^3, R = 4: 40 -> 6.4 us).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "common.h"
#include "conv_common.h"

namespace distdl {

constexpr int kStMaxWorkers = 64;
constexpr int kStMaxPerDim = 8;
constexpr int kStMaxR = 4;
constexpr int kStRpt = 2;             // consecutive rows per thread
constexpr int kStThreads = 128;
// Tile of LANES threads a row: 16 rows x 64 columns or 8 x 128
__host__ __device__ constexpr int st_rows(int lanes) { return kStRpt * (kStThreads / lanes); }
__host__ __device__ constexpr int st_cols(int lanes) { return 4 * lanes; }
constexpr int kStLead = 4;            // shared-memory column of the tile's first column (keeps rows 16-byte aligned)
__host__ __device__ constexpr int st_pitch(int lanes) { return kStLead + st_cols(lanes) + 4; }
constexpr int kStDepth = 5;           // planes in the ring (4 and 6 measure the same within 2 %)
// Blocks per multiprocessor.  With 16-byte copies a fourth block of the wide stars costs more in registers (128 instead of 168: moves and
// spills) than it hides; scalar copies have latency left for it (22 x 126 x 103 shards, R = 4, 576 blocks: 56 -> 48 and 74 -> 58 us; a
// single 240 x 155 x 201 shard: 35 -> 39 us).
template <int R, bool VEC>
constexpr int kStBlocks = VEC && R >= 3 ? 3 : 4;

struct StencilParams {
    const float *in[kStMaxWorkers];
    float *out[kStMaxWorkers];
    int32_t bz[kStMaxPerDim], by[kStMaxPerDim], bx[kStMaxPerDim];   // bulk extents per worker coordinate
    int32_t pz, py, px;
    int32_t in_off, out_off;          // ghost width of the input / output layout (R or 0)
    int32_t tiles_y, tiles_x, chunks_z;
    int32_t chunk;                    // planes a block marches through
    int32_t clear_ghosts;             // adjoint: the ghosts of the output shards are set to zero
    int32_t vec_out;                  // rows of the output start on 16-byte boundaries and hold whole vectors
    // taps [d][k + R], already reversed for the adjoint; the three centre taps meet the same cell and are added up in [0][R]
    float w[3][2 * kStMaxR + 1];
    uint64_t w2[3][2 * kStMaxR + 1];  // the same as (w, w) pairs
};

// Owner of coordinate c along one dimension, seen from worker coordinate s: the worker itself, or the
// one below / above (a ghost is never wider than the neighbour's bulk).  Returns false outside the tensor.
__device__ __forceinline__ bool st_owner(const int32_t *b, int p, int s, int c, int &so, int &co) {
    so = s;
    co = c;
    if (c < 0) {
        so = s - 1;
        if (so < 0) return false;
        co = c + b[so];
        return co >= 0;
    }
    if (c >= b[s]) {
        so = s + 1;
        if (so >= p) return false;
        co = c - b[s];
        return co < b[so];
    }
    return true;
}

// Copy of 16 / 4 bytes, or that many zeros (bytes = 0: nothing is read); nothing at all where `on` is false.
__device__ __forceinline__ void st_copy16(uint32_t dst, const float *src, uint32_t bytes, bool on) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n@p cp.async.cg.shared.global [%0], [%1], 16, %2;\n}"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void st_copy4(uint32_t dst, const float *src, uint32_t bytes, bool on) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n@p cp.async.ca.shared.global [%0], [%1], 4, %2;\n}"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"((uint32_t)on) : "memory");
}

template <int R, int LANES>
constexpr int st_smem_bytes() { return kStDepth * (st_rows(LANES) + 2 * R) * st_pitch(LANES) * 4; }

// Ghost shell of an output shard but for the row ends, which the threads that write the rows clear: the ghost planes below and
// above, and the ghost rows of each bulk plane, which lie next to those of the plane before it in memory.  All of them are
// contiguous runs and every block of the shard takes an equal share (block j of n).
template <bool VEC>
__device__ __forceinline__ void st_clear(float *out, int bz, int opy, int opx, int oo, int j, int n) {
    auto zero = [&](size_t at, size_t end) {
        if (VEC)
            for (at += 4 * threadIdx.x; at < end; at += 4 * kStThreads) *reinterpret_cast<float4 *>(out + at) = make_float4(0.f, 0.f, 0.f, 0.f);
        else
            for (at += threadIdx.x; at < end; at += kStThreads) out[at] = 0.f;
    };
    const size_t plane = (size_t)opy * opx, rows = (size_t)oo * opx, ghosts = oo * plane;
    for (int i = j; i <= bz; i += n) zero((i + oo) * plane - (i > 0 ? rows : 0), (i + oo) * plane + (i < bz ? rows : 0));
    const size_t piece = (ghosts + 4 * (size_t)n - 1) / (4 * (size_t)n) * 4, lo = min(j * piece, ghosts), hi = min(lo + piece, ghosts);
    zero(lo, hi);
    zero((bz + oo) * plane + lo, (bz + oo) * plane + hi);
}

template <int R, bool VEC, int LANES>
__global__ void __launch_bounds__(kStThreads, kStBlocks<R, VEC>)
stencil3d_kernel(const __grid_constant__ StencilParams P) {
    stream_enter();
    constexpr int kStRows = st_rows(LANES), kStCols = st_cols(LANES), kStPitch = st_pitch(LANES);
    extern __shared__ __align__(16) float ring[];          // planes of kStRows + 2 R rows
    constexpr int kPlane = (kStRows + 2 * R) * kStPitch;
    constexpr int N = 2 * R + 1;
    // Copies: 16 bytes a thread, the LANES threads of a row together, or (4 bytes a thread) 32 columns of a row at a time, a warp together
    constexpr int CL = VEC ? LANES : 32, CE = VEC ? 1 : kStCols / 32;      // threads that copy a row, copies of each
    constexpr int CG = kStThreads / CL, CR = kStRows / CG;                // groups of such threads, rows of a tile that each copies
    constexpr int HR = (2 * R + CG - 1) / CG;                              // extra rows that each copies per plane
    const int group = threadIdx.x / LANES, lane = threadIdx.x % LANES;
    const int cgroup = threadIdx.x / CL, clane = threadIdx.x % CL;
    // block -> (shard, plane chunk, row tile, column tile), column tile fastest
    int rest = blockIdx.x;
    const int tx = rest % P.tiles_x;
    rest /= P.tiles_x;
    const int ty = rest % P.tiles_y;
    rest /= P.tiles_y;
    const int cz = rest % P.chunks_z;
    const int shard = rest / P.chunks_z;
    const int sx = shard % P.px, sy = (shard / P.px) % P.py, sz = shard / (P.px * P.py);
    const int bz = P.bz[sz], by = P.by[sy], bx = P.bx[sx];
    const int oo = P.out_off;
    const int opy = by + 2 * oo, opx = bx + 2 * oo;
    const int x0 = tx * kStCols, y0 = ty * kStRows, z0 = cz * P.chunk;
    if (x0 >= bx || y0 >= by || z0 >= bz) return;
    const int z1 = min(z0 + P.chunk, bz);
    const int th = min(kStRows, by - y0), tw = min(kStCols, bx - x0);
    const int io = P.in_off;
    const int ipx = bx + 2 * io;                       // input row pitch of every shard in this worker column

    const int rw = kStRpt * group;                     // first of this thread's rows inside the tile
    const int x = x0 + 4 * lane;
    const bool col_ok = x < bx;
    bool row_ok[kStRpt];
#pragma unroll
    for (int r = 0; r < kStRpt; ++r) row_ok[r] = y0 + rw + r < by;

    // Everything that does not change from plane to plane is resolved once: for each kind of copy a pointer that walks from plane to
    // plane, the step (the plane stride of the owning shard, in elements: a shard holds fewer than 2^31 of them) and the bytes
    // to read (0: zeros, and the pointer stands still)
    // the columns that this thread copies of a row: its own four, or where rows are not aligned every 32nd
    const int xc = VEC ? x : x0 + clane, rc = CR == kStRpt ? rw : CR * cgroup;        // and the first of the rows
    // which of them lie inside the shard: flags where the store's can serve for the rows, counts otherwise (registers)
    const int cols_in = bx - xc, rows_in = by - y0 - rc;
    bool col_flag[CE];
#pragma unroll
    for (int e = 0; e < CE; ++e) col_flag[e] = VEC ? col_ok : xc + 32 * e < bx;
    auto row_in = [&](int r) { return CR == kStRpt ? row_ok[r < kStRpt ? r : 0] : r < rows_in; };
    auto col_in = [&](int e) { return CR == kStRpt ? col_flag[e] : 32 * e < cols_in; };
    auto copy4 = [&](uint32_t dst, const float *src, uint32_t bytes, bool on) {
        if (VEC) {
            st_copy16(dst, src, bytes, on && col_ok);
        } else {
#pragma unroll
            for (int e = 0; e < CE; ++e) st_copy4(dst + 128 * e, src + 32 * e, bytes, on && col_in(e));
        }
    };
    constexpr uint32_t kBytes = VEC ? 16 : 4;
    const uint32_t copy_dst = (uint32_t)((kStLead + (VEC ? 4 : 1) * clane) * 4);
    const uint32_t ipy = (uint32_t)(by + 2 * io);
    const uint32_t own_off = (uint32_t)(y0 + rc + io) * (uint32_t)ipx + (uint32_t)(xc + io);   // first row it copies
    const uint32_t own_stride = ipy * (uint32_t)ipx;                   // the same in the shards below and above
    const float *own_p = P.in[shard];
    uint32_t own_bytes = 0;
    // this thread's cell of plane zp (any plane within R of the chunk)
    auto own_at = [&](int zp) {
        int s3 = shard, n = bz;
        if (zp < 0) {
            s3 = sz > 0 ? shard - P.py * P.px : -1;
            n = sz > 0 ? P.bz[sz - 1] : 0;
            zp += n;
        } else if (zp >= bz) {
            s3 = sz + 1 < P.pz ? shard + P.py * P.px : -1;
            n = sz + 1 < P.pz ? P.bz[sz + 1] : 0;
            zp -= bz;
        }
        own_bytes = s3 >= 0 && col_in(0) && (unsigned)zp < (unsigned)n ? kBytes : 0u;
        own_p = own_bytes ? P.in[s3] + ((uint32_t)(zp + io) * own_stride + own_off) : P.in[shard];
    };
    // extra rows of the current plane: row h of the 2R (R above the tile, R below) goes to group h % CG
    const float *hrow_p[HR];
    uint32_t hrow_step[HR], hrow_bytes[HR], hrow_dst[HR];
#pragma unroll
    for (int i = 0; i < HR; ++i) {
        const int h = cgroup + CG * i;
        hrow_p[i] = P.in[shard];
        hrow_step[i] = hrow_bytes[i] = 0;
        // its row in the shared-memory plane: the rows below follow the tile's last one
        hrow_dst[i] = (uint32_t)(((h < R ? h : th + h) * kStPitch) * 4) + copy_dst;
        const int hy = h < R ? y0 - R + h : y0 + th + (h - R);
        int so, yo;
        if (h < 2 * R && col_in(0) && st_owner(P.by, P.py, sy, hy, so, yo)) {
            hrow_bytes[i] = kBytes;
            hrow_step[i] = (uint32_t)(P.by[so] + 2 * io) * (uint32_t)ipx;
            hrow_p[i] = P.in[(sz * P.py + so) * P.px + sx] + (uint32_t)(z0 + io) * hrow_step[i] +
                        ((uint32_t)(yo + io) * (uint32_t)ipx + (uint32_t)(xc + io));
        }
    }
    // threads 0 .. kStRows * 2R - 1: one cell of an extra column
    const int hc_row = threadIdx.x / (2 * R), hc_c = threadIdx.x % (2 * R);
    const bool hc_active = (int)threadIdx.x < kStRows * 2 * R && y0 + hc_row < by;
    const int hc_x = hc_c < R ? x0 - R + hc_c : x0 + tw + (hc_c - R);
    const uint32_t hcol_dst = (uint32_t)(((R + hc_row) * kStPitch + kStLead + (hc_x - x0)) * 4);
    const float *hcol_p = P.in[shard];
    uint32_t hcol_step = 0, hcol_bytes = 0;
    {
        int so, xo;
        if (hc_active && st_owner(P.bx, P.px, sx, hc_x, so, xo)) {
            const uint32_t pitch = (uint32_t)(P.bx[so] + 2 * io);
            hcol_bytes = 4u;
            hcol_step = ipy * pitch;
            hcol_p = P.in[(sz * P.py + sy) * P.px + so] + (uint32_t)(z0 + io) * hcol_step + ((uint32_t)(y0 + hc_row + io) * pitch + (uint32_t)(xo + io));
        }
    }
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    const uint32_t own_dst = ring_s + (uint32_t)((R + rc) * kStPitch * 4) + copy_dst;
    own_at(z0 - R);
    // plane zp into the slot `at` bytes into the ring: own cells, and if it is to be the current one a vector of each extra row and
    // one extra-column cell; cells beyond the bulk are written by the extra-row / extra-column threads only
    auto issue = [&](int zp, uint32_t at) {
#pragma unroll
        for (int r = 0; r < CR; ++r) copy4(own_dst + at + (uint32_t)(r * kStPitch * 4), own_p + r * ipx, own_bytes, row_in(r));
        if (zp + 1 == 0 || zp + 1 == bz) own_at(zp + 1);
        else own_p += own_bytes ? own_stride : 0u;
        if (zp >= z0 && zp < z1) {
#pragma unroll
            for (int i = 0; i < HR; ++i) {
                copy4(ring_s + at + hrow_dst[i], hrow_p[i], hrow_bytes[i], (2 * R) % CG == 0 || cgroup + CG * i < 2 * R);
                hrow_p[i] += hrow_step[i];
            }
            st_copy4(ring_s + at + hcol_dst, hcol_p, hcol_bytes, hc_active);
            hcol_p += hcol_step;
        }
    };

    // sums of the outputs p - R .. p + R around plane p
    uint64_t acc[N][kStRpt][2];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int r = 0; r < kStRpt; ++r) acc[i][r][0] = acc[i][r][1] = 0ull;
    // a plane's cells as z neighbours (the middle tap: the three centre taps together); the sums move on by one slot
    auto z_taps = [&](const float4 (&v)[kStRpt]) {
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int r = 0; r < kStRpt; ++r) {
                acc[i][r][0] = fma2(P.w2[0][2 * R - i], pack2(v[r].x, v[r].y), i + 1 < N ? acc[i + 1 < N ? i + 1 : i][r][0] : 0ull);
                acc[i][r][1] = fma2(P.w2[0][2 * R - i], pack2(v[r].z, v[r].w), i + 1 < N ? acc[i + 1 < N ? i + 1 : i][r][1] : 0ull);
            }
    };

    float *optr = P.out[shard] + ((size_t)(z0 + oo) * opy + (size_t)(y0 + rw + oo)) * opx + (x + oo);
    const size_t oplane = (size_t)opy * opx;
    const bool clear_x = P.clear_ghosts && oo > 0 && (x == 0 || x + 4 >= bx);   // threads at the row ends

    // output plane z - R is complete
    auto store = [&]() {
        if (col_ok && row_ok[0]) {
#pragma unroll
            for (int r = 0; r < kStRpt; ++r) {
                if (!row_ok[r]) continue;
                float o[4];
                unpack2(acc[0][r][0], o[0], o[1]);
                unpack2(acc[0][r][1], o[2], o[3]);
                float *op = optr + (size_t)r * opx;
                if (R == 4 ? VEC : P.vec_out) {
                    *reinterpret_cast<float4 *>(op) = make_float4(o[0], o[1], o[2], o[3]);
                } else {
                    op[0] = o[0];
                    if (x + 1 < bx) op[1] = o[1];
                    if (x + 2 < bx) op[2] = o[2];
                    if (x + 3 < bx) op[3] = o[3];
                }
                // adjoint: the ghost columns beside this row are cleared by the threads that write the row's
                // ends, so that they land in the same lines of memory as the row itself
                if (clear_x) {
                    if (x == 0) {
                        if (VEC && R == 4) *reinterpret_cast<float4 *>(op - 4) = make_float4(0.f, 0.f, 0.f, 0.f);
                        else
                            for (int c = 1; c <= oo; ++c) op[-c] = 0.f;
                    }
                    if (x + 4 >= bx) {
                        if (VEC && R == 4) *reinterpret_cast<float4 *>(op + 4) = make_float4(0.f, 0.f, 0.f, 0.f);
                        else
                            for (int c = 0; c < oo; ++c) op[bx - x + c] = 0.f;
                    }
                }
            }
        }
        optr += oplane;
    };
#pragma unroll 1
    for (int i = 0; i < kStDepth - 1; ++i) {
        if (z0 - R + i < z1 + R) issue(z0 - R + i, i * kPlane * 4);
        cp_async_commit();
    }
    // in the shadow of the first planes' arrival (ahead of their copies it costs 12 us of 233 at 512^3, clearing or not)
    if (P.clear_ghosts && oo > 0) {
        const int ny = (by + kStRows - 1) / kStRows, nx = (bx + kStCols - 1) / kStCols;   // this shard's blocks
        st_clear<VEC && R == 4>(P.out[shard], bz, opy, opx, oo, (cz * ny + ty) * nx + tx, (bz + P.chunk - 1) / P.chunk * ny * nx);
    }
    uint32_t at = 0;                                       // slot of this plane, in bytes; the one before it is free
#pragma unroll 1
    for (int z = z0 - R; z < z1 + R; ++z) {
        const bool centre = z >= z0 && z < z1;             // the planes around the chunk are only z neighbours
        cp_async_wait_group<kStDepth - 2>();
        __syncthreads();                                   // this plane has arrived; the one before it has been read
        if (z + kStDepth - 1 < z1 + R) issue(z + kStDepth - 1, at == 0 ? (kStDepth - 1) * kPlane * 4 : at - kPlane * 4);
        cp_async_commit();
        const float *pl = reinterpret_cast<const float *>(reinterpret_cast<const char *>(ring) + at);
        at = at == (kStDepth - 1) * kPlane * 4 ? 0u : at + kPlane * 4;
        float4 cur[kStRpt];
#pragma unroll
        for (int r = 0; r < kStRpt; ++r) {
            const float *c = pl + (R + rw + r) * kStPitch + kStLead + 4 * lane;
            cur[r] = *reinterpret_cast<const float4 *>(c);
        }
        z_taps(cur);
        if (centre && col_ok && row_ok[0]) {
            // x neighbours: the vectors left and right of the own one; shifts by an even number of columns as pairs
#pragma unroll
            for (int r = 0; r < kStRpt; ++r) {
                float xs[12], o[4];
                const float4 l = *reinterpret_cast<const float4 *>(pl + (R + rw + r) * kStPitch + 4 * lane);
                const float4 rt = *reinterpret_cast<const float4 *>(pl + (R + rw + r) * kStPitch + 4 * lane + 8);
                xs[0] = l.x; xs[1] = l.y; xs[2] = l.z; xs[3] = l.w;
                const float4 c = cur[r];
                xs[4] = c.x; xs[5] = c.y; xs[6] = c.z; xs[7] = c.w;
                xs[8] = rt.x; xs[9] = rt.y; xs[10] = rt.z; xs[11] = rt.w;
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    if (k == R || ((k - R) & 1)) continue;
#pragma unroll
                    for (int p = 0; p < 2; ++p)
                        acc[R][r][p] = fma2(P.w2[2][k], pack2(xs[4 + 2 * p + k - R], xs[5 + 2 * p + k - R]), acc[R][r][p]);
                }
                unpack2(acc[R][r][0], o[0], o[1]);
                unpack2(acc[R][r][1], o[2], o[3]);
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    if (!((k - R) & 1)) continue;
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[e] = fmaf(P.w[2][k], xs[4 + e + k - R], o[e]);
                }
                acc[R][r][0] = pack2(o[0], o[1]);
                acc[R][r][1] = pack2(o[2], o[3]);
            }
            // y neighbours: the rows rw .. rw + 2R + RPT - 1 of the plane, each read once and used by every
            // row of the thread it is a neighbour of (tap k of row r is plane row rw + r + k)
            auto y_taps = [&](int j, const float4 &v) {
#pragma unroll
                for (int r = 0; r < kStRpt; ++r) {
                    const int k = j - r;
                    if (k < 0 || k >= N || k == R) continue;
                    acc[R][r][0] = fma2(P.w2[1][k], pack2(v.x, v.y), acc[R][r][0]);
                    acc[R][r][1] = fma2(P.w2[1][k], pack2(v.z, v.w), acc[R][r][1]);
                }
            };
            // its own rows are in registers already (in a ragged last tile such a row may be an extra row of the plane)
#pragma unroll
            for (int r = 0; r < kStRpt; ++r) y_taps(R + r, cur[r]);
#pragma unroll
            for (int j = 0; j < N + kStRpt - 1; ++j)
                if (j < R || j >= R + kStRpt) y_taps(j, *reinterpret_cast<const float4 *>(pl + (rw + j) * kStPitch + kStLead + 4 * lane));
        }
        if (z >= z0 + R) store();
    }
}

template <int R, int LANES>
static distdl_status_t launch_stencil(const StencilParams &P, unsigned grid, bool vec, cudaStream_t s) {
    constexpr int smem = st_smem_bytes<R, LANES>();
    static bool configured_on[kMaxDevicesPerProcess] = {false};
    int dev = 0;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevicesPerProcess)
        return fail(DISTDL_ERR_UNSUPPORTED, "device index %d: at most %d devices per process", dev, kMaxDevicesPerProcess);
    {
        std::lock_guard<std::mutex> setup_lock(setup_mutex());
        if (!configured_on[dev]) {
            DISTDL_CUDA_CHECK(cudaFuncSetAttribute(stencil3d_kernel<R, true, LANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            DISTDL_CUDA_CHECK(cudaFuncSetAttribute(stencil3d_kernel<R, false, LANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            configured_on[dev] = true;
        }
    }
    if (vec) launch_in_stream(stencil3d_kernel<R, true, LANES>, grid, kStThreads, smem, s, P);
    else launch_in_stream(stencil3d_kernel<R, false, LANES>, grid, kStThreads, smem, s, P);
    DISTDL_CUDA_CHECK(cudaGetLastError());
    return DISTDL_OK;
}

// Planes per block.  A block's time goes with its planes and the 2R around them, and with how many blocks share its
// multiprocessor: 0.62 / 0.79 / 0.96 us a plane for one, two, three of them.  Small chunks fill the device and even out its last
// wave, long ones read fewer planes twice: of the chunks in steps of a quarter the one with the least time by this count.
static int32_t st_chunk(int64_t planes, int64_t tiles, int radius, bool vec, int sms) {
    const int64_t resident = !vec ? kStBlocks<4, false> : radius <= 2 ? kStBlocks<2, true> : kStBlocks<4, true>;
    int64_t best = planes, best_cost = INT64_MAX;
    for (int64_t c = 4;; c += std::max<int64_t>(1, c / 4)) {
        const int64_t chunks = (planes + c - 1) / c, chunk = (planes + chunks - 1) / chunks;
        const int64_t n = (tiles * chunks + sms - 1) / sms, last = n % resident;
        const int64_t cost = (n / resident * (45 + 17 * resident) + (last ? 45 + 17 * last : 0)) * (chunk + 2 * radius);
        if (cost < best_cost) {
            best_cost = cost;
            best = chunk;
        }
        if (c >= planes) return (int32_t)best;
    }
}

static distdl_status_t stencil_impl(const distdl_partition *p, const void *const *in, const float *w, int32_t radius,
                                    void *const *out, void *stream, bool adj, const char *what) {
    clear_error();
    if (!p || !in || !w || !out) return fail(DISTDL_ERR_INVALID_ARG, "%s: NULL argument", what);
    if (p->rank != 3 || p->dtype != DISTDL_F32) return fail(DISTDL_ERR_SHAPE, "%s: needs a rank-3 F32 partition", what);
    if (p->any_periodic()) return fail(DISTDL_ERR_UNSUPPORTED, "%s: periodic partitions are not supported by the fused layers", what);
    if (radius < 1 || radius > kStMaxR) return fail(DISTDL_ERR_UNSUPPORTED, "%s: radius %d (supported: 1..%d)", what, radius, kStMaxR);
    if (p->num_workers > kStMaxWorkers) return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d workers", what, kStMaxWorkers);
    for (int k = 0; k < 3; ++k) {
        if (p->pshape[k] > kStMaxPerDim)
            return fail(DISTDL_ERR_UNSUPPORTED, "%s: more than %d workers along a dimension", what, kStMaxPerDim);
        for (int32_t c = 0; c < p->pshape[k]; ++c)
            if (p->hlo[k][c] != radius || p->hhi[k][c] != radius)
                return fail(DISTDL_ERR_SHAPE, "%s: halo widths must equal the radius %d on every side", what, radius);
    }
    StencilParams P;
    memset(&P, 0, sizeof(P));
    int64_t mz = 0, my = 0, mx = 0;
    for (int32_t c = 0; c < p->pshape[0]; ++c) mz = std::max<int64_t>(mz, P.bz[c] = (int32_t)p->size[0][c]);
    for (int32_t c = 0; c < p->pshape[1]; ++c) my = std::max<int64_t>(my, P.by[c] = (int32_t)p->size[1][c]);
    for (int32_t c = 0; c < p->pshape[2]; ++c) mx = std::max<int64_t>(mx, P.bx[c] = (int32_t)p->size[2][c]);
    P.pz = p->pshape[0];
    P.py = p->pshape[1];
    P.px = p->pshape[2];
    P.in_off = adj ? 0 : radius;
    P.out_off = adj ? radius : 0;
    P.clear_ghosts = adj ? 1 : 0;
    // 16-byte accesses: every row of the layout starts on a 16-byte boundary and holds whole vectors
    bool whole = true;
    for (int32_t c = 0; c < p->pshape[2]; ++c) whole = whole && (P.bx[c] % 4) == 0;
    const bool vec = whole && P.in_off % 4 == 0;
    P.vec_out = whole && P.out_off % 4 == 0;
    // 16 rows x 64 columns where that makes fewer tiles, or as many with 16-byte copies: fewer rows and vectors around a tile (512^3, R = 4, pair 565 ->
    // 540 us); with 4-byte copies and as many tiles the longer rows win (66 x 305 x 202 on 3 x 4 x 1 workers, R = 1: 33.3 against 31.9 us).
    const auto tiles = [&](int lanes) { return ((mx + st_cols(lanes) - 1) / st_cols(lanes)) * ((my + st_rows(lanes) - 1) / st_rows(lanes)); };
    const int lanes = tiles(16) < tiles(32) || (tiles(16) == tiles(32) && vec) ? 16 : 32;
    P.tiles_x = (int32_t)((mx + st_cols(lanes) - 1) / st_cols(lanes));
    P.tiles_y = (int32_t)((my + st_rows(lanes) - 1) / st_rows(lanes));
    for (int d = 0; d < 3; ++d)
        for (int k = 0; k <= 2 * radius; ++k) P.w[d][k] = adj ? w[d * (2 * radius + 1) + (2 * radius - k)] : w[d * (2 * radius + 1) + k];
    P.w[0][radius] = (float)((double)P.w[0][radius] + (double)P.w[1][radius] + (double)P.w[2][radius]);
    for (int d = 0; d < 3; ++d)
        for (int k = 0; k <= 2 * radius; ++k) {
            uint32_t bits;
            memcpy(&bits, &P.w[d][k], 4);
            P.w2[d][k] = (uint64_t)bits << 32 | bits;
        }
    for (int32_t wk = 0; wk < p->num_workers; ++wk) {
        if (!in[wk] || !out[wk]) return fail(DISTDL_ERR_INVALID_ARG, "%s: shard pointer %d is NULL", what, wk);
        if (!aligned16(in[wk]) || !aligned16(out[wk])) return fail(DISTDL_ERR_ALIGNMENT, "%s: shard %d is not 16-byte aligned", what, wk);
        if (p->shard_elems(wk) >= ((int64_t)1 << 31)) return fail(DISTDL_ERR_UNSUPPORTED, "%s: shard %d too large", what, wk);
        P.in[wk] = (const float *)in[wk];
        P.out[wk] = (float *)out[wk];
    }
    int dev = 0, sms = 0;
    DISTDL_CUDA_CHECK(cudaGetDevice(&dev));
    DISTDL_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    P.chunk = st_chunk(mz, (int64_t)p->num_workers * P.tiles_y * P.tiles_x, radius, vec, sms);
    P.chunks_z = (int32_t)((mz + P.chunk - 1) / P.chunk);
    const int64_t blocks = (int64_t)p->num_workers * P.chunks_z * P.tiles_y * P.tiles_x;
    if (blocks >= ((int64_t)1 << 31)) return fail(DISTDL_ERR_UNSUPPORTED, "%s: too many tiles", what);
    cudaStream_t s = (cudaStream_t)stream;
    const auto run = [&](auto r) {
        constexpr int R = decltype(r)::value;
        return lanes == 16 ? launch_stencil<R, 16>(P, (unsigned)blocks, vec, s) : launch_stencil<R, 32>(P, (unsigned)blocks, vec, s);
    };
    switch (radius) {
        case 1: return run(std::integral_constant<int, 1>{});
        case 2: return run(std::integral_constant<int, 2>{});
        case 3: return run(std::integral_constant<int, 3>{});
        default: return run(std::integral_constant<int, 4>{});
    }
}

}  // namespace distdl

extern "C" distdl_status_t distdl_stencil3d_fwd(const distdl_partition_t *p, const void *const *x, const float *w,
                                                int32_t radius, void *const *y, void *stream) {
    return distdl::stencil_impl(p, x, w, radius, y, stream, false, "stencil3d_fwd");
}
extern "C" distdl_status_t distdl_stencil3d_adj(const distdl_partition_t *p, const void *const *dy, const float *w,
                                                int32_t radius, void *const *dx, void *stream) {
    return distdl::stencil_impl(p, dy, w, radius, dx, stream, true, "stencil3d_adj");
}
