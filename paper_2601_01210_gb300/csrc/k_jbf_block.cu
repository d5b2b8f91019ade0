// The block form of the second filter stage (jbf_block.cuh): its persistent tile loop and its
// instantiations. Tiles, flags, tile counter, copies one tile ahead and bounded waits as in
// jbf_tma.cuh.
#include <type_traits>

#include "jbf_block.cuh"
#include "ray.cuh"
#include "tile_queue.cuh"
#include "tma_info.h"

namespace dz {

namespace {

// A frame's outputs, copied into shared memory once per CTA.
struct BlockOut {
    float *depth;
    uint8_t *valid;
    int32_t gw, gh;
};

// What a frame's points take besides (POINTS).
struct BlockPoints {
    float4 *points;
    int64_t cap;
    const uint32_t *row, *seg;   // valid pixels in the rows before, and before a segment of its row
    float c2w[12];
    float ifx, ify, cx, cy;
};

__device__ __forceinline__ void copy_word(uint32_t *dst, const uint32_t *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// POINTS: the valid pixels' coloured points are written here as well, each at its place in row-major
// order: row_pre and seg_pre (bp_rows_kernel) give the place of a warp's first pixel of a row, ballots
// the rest. The depth, the colour and the validity are at hand, so that the compaction's own pass over
// the three maps (and its count of the validity map) falls away: on eight 1080p frames (cold caches)
// this kernel takes 120 us instead of 96 and the row prefixes 7, the compaction kernels took 69; one
// frame: 28.5 instead of 25, 6, and 15.5.
template <int R, int NW, bool POINTS>
__global__ void __launch_bounds__(NW * 32, 16 / NW) jbf_block_kernel(const BatchDev *__restrict__ B, const StageArgs a) {
    using G = BlockGeom<R, NW>;
    constexpr int TW = G::TW, TH = G::TH;
    extern __shared__ __align__(128) uint8_t smem[];
    auto rawA = [&](int b) { return smem + b * (G::RAW_A + G::RAW_B); };
    auto rawB = [&](int b) { return smem + b * (G::RAW_A + G::RAW_B) + G::RAW_A; };
    uint32_t *const sc = reinterpret_cast<uint32_t *>(smem + G::OFF_STAGED);
    uint64_t *const bar = reinterpret_cast<uint64_t *>(smem + G::OFF_BAR);
    __shared__ TileQueueMem s_queue;
    __shared__ BlockOut s_out[kMaxBatch];
    __shared__ BlockPoints s_pts[POINTS ? kMaxBatch : 1];
    __shared__ uint32_t s_place[6 * NW][2];
    const int nf = B->n_frames;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto copies = [&](int fi, int x0, int y0, int buf) {
        const FrameDev &F = B->f[fi];
        mbar_expect_tx(&bar[buf], G::TX_BYTES);
        tma_load_2d(rawA(buf), &F.tm[TM_RGB], (3 * x0 - G::RGB_LEAD) / 4, y0 - R, &bar[buf]);   // 4-byte elements
        tma_load_2d(rawB(buf), &F.tm[TM_S1], x0 / 3 - 2, y0 / 3 - 1, &bar[buf]);
    };
    TileQueue<TW, TH, G::NT, 1, decltype(copies)> queue(s_queue, B, bar, copies);
    queue.load(nf);
    for (int i = threadIdx.x; i < nf; i += G::NT) {
        const FrameDev &F = B->f[i];
        s_out[i] = BlockOut{F.flt_depth, F.flt_valid, F.W, F.H};
        if (POINTS) {
            BlockPoints &P = s_pts[i];
            P.points = F.out_points;
            P.cap = F.points_cap;
            P.row = F.row_pre;
            P.seg = F.seg_pre;
#pragma unroll
            for (int e = 0; e < 12; ++e) P.c2w[e] = F.c2w32[e];
            P.ifx = 1.0f / F.fx;
            P.ify = 1.0f / F.fy;
            P.cx = F.cx;
            P.cy = F.cy;
        }
    }
    if (threadIdx.x == 0) {
        for (int f = 0; f < nf; ++f) {
            tmap_acquire(&B->f[f].tm[TM_RGB]);
            tmap_acquire(&B->f[f].tm[TM_S1]);
        }
    }
    __syncthreads();
    queue.start();
    __syncthreads();
    for (int it = 0;; ++it) {
        const int buf = it & 1;
        if (queue.done(buf)) break;
        const bool bad = queue.top(buf);
        const int fi = queue.frame(buf), x0 = queue.x0(buf), y0 = queue.y0(buf);
        const BlockOut &O = s_out[fi];
        const int gw = O.gw, gh = O.gh;
        float *const out_depth = O.depth;
        uint8_t *const out_valid = O.valid;
        if (!queue.copied(buf)) {   // no observation reaches the tile: every output is (0, invalid)
            queue.step();
            for (int ty = warp; ty < TH && y0 + ty < gh; ty += NW)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const int x = x0 + 32 * j + lane;
                    if (x >= gw) continue;
                    const int64_t o = (int64_t)(y0 + ty) * gw + x;
                    out_depth[o] = 0.0f;
                    out_valid[o] = 0;
                }
            __syncthreads();
            continue;
        }
        const uint8_t *const rgbraw = rawA(buf);
        const float2 *const craw = reinterpret_cast<const float2 *>(rawB(buf));
        if (!bad) block_convert<G>(rgbraw, sc);
        if (__syncthreads_or(bad)) {
            queue.leave();
            return;
        }
        queue.step();

        // the place of the first point of each of the warp's rows, copied into shared memory during the taps
        if (POINTS && lane < 6 && y0 + 6 * warp + lane < gh) {
            const BlockPoints &P = s_pts[fi];
            const int y = y0 + 6 * warp + lane;
            copy_word(&s_place[6 * warp + lane][0], P.row + y);
            copy_word(&s_place[6 * warp + lane][1], P.seg + (int64_t)y * ((gw + TW - 1) / TW) + x0 / TW);
        }
        BlockIn in;
        in.s0 = sc + 6 * warp * G::SW + G::LEAD - R + 3 * lane;
        in.s1 = in.s0 + 3 * G::SW;
        in.c0 = craw + 2 * warp * G::C_BX + lane + 1;
        in.c1 = in.c0 + G::C_BX;
        in.cols = gw - (x0 + 3 * lane - R);
        in.rows0 = gh - (y0 + 6 * warp - R);
        in.rows1 = in.rows0 - 3;
        // observed pooled neighbours of the two blocks (bit 3 b + i): rows 0 .. 2 and 1 .. 3
        uint32_t m = 0u;
#pragma unroll
        for (int i = 0; i < 12; ++i) m |= (in.c0[i / 3 * G::C_BX + i % 3].y > 0.0f ? 1u : 0u) << i;
        // depths of the warp's 6 rows of 96 through shared memory, so that its stores are whole rows
        float *const st = reinterpret_cast<float *>(smem + G::OFF_OUT) + warp * G::OUT;
        bool slow = false;
        auto filter = [&](auto edge) {
            float2 out[9];
            block_filter<G, decltype(edge)::value>(a, in, m & 0x1FFu, m >> 3, out);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                st[(i / 3) * TW + 3 * lane + i % 3] = out[i].x;
                st[(3 + i / 3) * TW + 3 * lane + i % 3] = out[i].y;
                slow |= out[i].x == -2.0f || out[i].y == -2.0f;
            }
        };
        if (!__any_sync(0xffffffffu, m != 0)) {
#pragma unroll
            for (int i = lane; i < G::OUT; i += 32) st[i] = -1.0f;
        } else if ((gw % 3 != 0 && x0 + TW + R > gw) || (gh % 3 != 0 && y0 + TH + R > gh)) {
            // a pooled pixel of the tile or its halo covers positions outside the image
            filter(std::true_type{});
        } else {
            filter(std::false_type{});
        }
        __syncwarp();
        if (__any_sync(0xffffffffu, slow)) {   // rare
#pragma unroll 1
            for (int i = lane; i < G::OUT; i += 32) {
                const int row = i / TW, tx = i - row * TW, ty = 6 * warp + row;
                if (st[i] == -2.0f && x0 + tx < gw && y0 + ty < gh)
                    st[i] = block_shifted<G>(a, sc, craw, tx, ty, gw - x0, gh - y0);
            }
            __syncwarp();
        }
        const BlockPoints &P = s_pts[POINTS ? fi : 0];
        if (POINTS) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
        }
#pragma unroll 2
        for (int row = 0; row < 6; ++row) {
            const int y = y0 + 6 * warp + row;
            if (y >= gh) break;
            const int64_t o = (int64_t)y * gw + x0 + lane;
            uint32_t at = POINTS ? s_place[6 * warp + row][0] + s_place[6 * warp + row][1] : 0u;
            float3 ray = make_float3(0.0f, 0.0f, 0.0f);
            if (POINTS) ray = ray_row(P.c2w, ray_coord((float)y + 0.5f, P.cy, P.ify));
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float d = st[row * TW + 32 * j + lane];
                const bool in = x0 + 32 * j + lane < gw, ok = in && d >= 0.0f;
                if (in) {
                    out_depth[o + 32 * j] = fmaxf(d, 0.0f);
                    out_valid[o + 32 * j] = ok;
                }
                if (POINTS) {
                    const uint32_t m = __ballot_sync(0xffffffffu, ok);
                    const uint32_t n = at + __popc(m & ((1u << lane) - 1u));
                    at += __popc(m);
                    if (ok && (int64_t)n < P.cap) {
                        const float u = ray_coord((float)(x0 + 32 * j + lane) + 0.5f, P.cx, P.ifx);
                        P.points[n] = ray_point(P.c2w, ray, u, d, sc[(6 * warp + row + R) * G::SW + G::LEAD + 32 * j + lane]);
                    }
                }
            }
        }
        __syncthreads();   // the staged words and raw[buf] are rewritten by the next tile
    }
}

template <int R, int NW>
void fill_info(TmaKernelInfo *o) {
    using G = BlockGeom<R, NW>;
    *o = TmaKernelInfo{};
    o->supported = 1;
    o->kp = 3;
    o->threads = NW * 32;
    o->tile_w = G::TW;
    o->tile_h = G::TH;
    o->smem = G::SMEM;
    o->rgb_elem = 4;
    o->rgb_box[0] = G::RGB_BX / 4; o->rgb_box[1] = G::RGB_BY;
    o->s1_box[0] = G::C_BX;        o->s1_box[1] = G::C_BY;
}

// (radius, warps per CTA). Tiles of 96 x 48 by 8 warps, two CTAs per SM (128 registers). Measured on
// eight 1080p three-scan frames (r = 2, autotuner's timing): 88 us, with 4 warps (96 x 24) 91, with 2
// 97; the column-paired expanded form 131 (its default, 64 x 48), the FP16 gather form 224. r = 1: 65
// against 115-123 for the gather forms, r = 3: 165 against 283-323. One 1080p frame: 21.5 against 28,
// one 960 x 540 frame 11.3 against 14.7; at 320 x 240 (20 tiles) 13.3 against 12.6.
// Bound: issue. ncu on four of those frames: 53 % of the issue slots (paired form 56 %, of 1.4 times
// the instructions), ahead of the FMA (40 %), ALU (34 %) and ex2 pipes (30 %); the top stall is the
// instruction fetch (the taps of 18 pixels are one straight run of some 2000 instructions), then
// fixed latency. With points (two frames, cold caches): 41 % of the issue slots, the fetch again the
// top stall (2.9 warps per issued instruction, fixed latency 1.3).
#define DZ_BLOCK_CASES(X) X(1, 8) X(2, 8) X(3, 8)

}  // namespace

int jbf_block_variants(int r, TmaVariant *out, int cap) {
    int n = 0;
#define DZ_X(R, NW) if (r == R && n < cap) out[n++] = TmaVariant{3, NW};
    DZ_BLOCK_CASES(DZ_X)
#undef DZ_X
    return n;
}

bool jbf_block_info(int r, TmaVariant v, TmaKernelInfo *out) {
#define DZ_X(R, NW) if (r == R && v.nw == NW) { fill_info<R, NW>(out); return true; }
    DZ_BLOCK_CASES(DZ_X)
#undef DZ_X
    return false;
}

cudaError_t jbf_block_prepare(int r, TmaVariant v) {
#define DZ_X(R, NW) \
    if (r == R && v.nw == NW) {                                                                                          \
        const cudaError_t e = cudaFuncSetAttribute(jbf_block_kernel<R, NW, false>,                                       \
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, BlockGeom<R, NW>::SMEM); \
        return e != cudaSuccess ? e                                                                                      \
                                : cudaFuncSetAttribute(jbf_block_kernel<R, NW, true>,                                    \
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, BlockGeom<R, NW>::SMEM); \
    }
    DZ_BLOCK_CASES(DZ_X)
#undef DZ_X
    return cudaErrorInvalidValue;
}

cudaError_t jbf_block_load(int r, TmaVariant v) {
    cudaFuncAttributes at;
#define DZ_X(R, NW)                                                                       \
    if (r == R && v.nw == NW) {                                                           \
        const cudaError_t e = cudaFuncGetAttributes(&at, jbf_block_kernel<R, NW, false>); \
        return e != cudaSuccess ? e : cudaFuncGetAttributes(&at, jbf_block_kernel<R, NW, true>); \
    }
    DZ_BLOCK_CASES(DZ_X)
#undef DZ_X
    return cudaErrorInvalidValue;
}

cudaError_t jbf_block_launch(int r, TmaVariant v, bool points, const BatchDev *b, const StageArgs &a, int grid, cudaStream_t s) {
#define DZ_X(R, NW)                                                                                         \
    if (r == R && v.nw == NW) {                                                                             \
        if (points) jbf_block_kernel<R, NW, true><<<grid, NW * 32, BlockGeom<R, NW>::SMEM, s>>>(b, a);      \
        else jbf_block_kernel<R, NW, false><<<grid, NW * 32, BlockGeom<R, NW>::SMEM, s>>>(b, a);            \
        return cudaGetLastError();                                                                          \
    }
    DZ_BLOCK_CASES(DZ_X)
#undef DZ_X
    return cudaErrorInvalidValue;
}

int jbf_block_occupancy(int r, TmaVariant v) {
    int n = 0;
#define DZ_X(R, NW) \
    if (r == R && v.nw == NW) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, jbf_block_kernel<R, NW, true>, NW * 32, BlockGeom<R, NW>::SMEM);
    DZ_BLOCK_CASES(DZ_X)
#undef DZ_X
    return n;
}

}  // namespace dz
