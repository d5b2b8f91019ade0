// The list form of the single stage (jbf_list.cuh): its persistent tile loop and instantiations.
#include "jbf_list.cuh"
#include "tile_queue.cuh"
#include "tma_info.h"

namespace dz {

namespace {

struct ListOut {
    float *depth;
    uint8_t *valid;
    int32_t gw, gh;
};

// Three CTAs of 8 warps per SM (80 registers). Measured: r = 7 on four 1080p three-scan frames 91 us
// (the sparse form, whose loop walked row masks and tested windows: 205), r = 4 on 32 frames of
// 320 x 240 38 us (the sparse form with half2 weights that FP16 contexts took: 82). Bound: issue, some
// 15 instructions per observation and warp (two pixels a lane), of whose evaluations 225 of 484
// (r = 7) fall inside their windows; where tiles gather (the line: kListDense, jbf_list.cuh), issue too.
template <int R, int BL>
__global__ void __launch_bounds__(256, 3) jbf_list_kernel(const BatchDev *__restrict__ B, const StageArgs a) {
    using G = ListGeom<R, BL>;
    constexpr int TW = G::TW, TH = G::TH;
    extern __shared__ __align__(128) uint8_t smem[];
    auto rawA = [&](int b) { return smem + b * (G::RAW_A + G::RAW_B); };
    auto rawB = [&](int b) { return smem + b * (G::RAW_A + G::RAW_B) + G::RAW_A; };
    float2 *const tab = reinterpret_cast<float2 *>(smem + G::OFF_TAB);
    float2 *const pair = reinterpret_cast<float2 *>(smem + G::OFF_PAIR);
    uint64_t *const rowmask = reinterpret_cast<uint64_t *>(smem + G::OFF_ROWS);
    uint64_t *const bar = reinterpret_cast<uint64_t *>(smem + G::OFF_BAR);
    __shared__ TileQueueMem s_queue;
    __shared__ ListOut s_out[kMaxBatch];
    const int nf = B->n_frames;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 *const list = reinterpret_cast<uint4 *>(smem + G::OFF_LIST) + warp * kListCap;
    auto copies = [&](int fi, int x0, int y0, int buf) {
        const FrameDev &F = B->f[fi];
        mbar_expect_tx(&bar[buf], G::TX_BYTES);
        tma_load_2d(rawA(buf), &F.tm[TM_RGB], 3 * x0 - G::RGB_LEAD, y0 - R, &bar[buf]);
        tma_load_2d(rawB(buf), &F.tm[TM_ZBUF], x0 - G::Z_LEAD, y0 - R, &bar[buf]);
    };
    TileQueue<TW, TH, G::NT, 0, decltype(copies)> queue(s_queue, B, bar, copies);
    queue.load(nf);
    for (int i = threadIdx.x; i < nf; i += G::NT) {
        const FrameDev &F = B->f[i];
        s_out[i] = ListOut{F.flt_depth, F.flt_valid, F.W, F.H};
    }
    if (threadIdx.x == 0)
        for (int f = 0; f < nf; ++f) {
            tmap_acquire(&B->f[f].tm[TM_RGB]);
            tmap_acquire(&B->f[f].tm[TM_ZBUF]);
        }
    __syncthreads();
    queue.start();
    list_table<G>(a, tab, pair);   // while the first tile's copies are on their way
    __syncthreads();
    for (int it = 0;; ++it) {
        const int buf = it & 1;
        if (queue.done(buf)) break;
        const bool bad = queue.top(buf);
        const int x0 = queue.x0(buf), y0 = queue.y0(buf);
        const ListOut &O = s_out[queue.frame(buf)];
        const int gw = O.gw, gh = O.gh;
        float *const out_depth = O.depth;
        uint8_t *const out_valid = O.valid;
        if (!queue.copied(buf)) {   // no observation reaches the tile: every output is (0, invalid)
            queue.step();
            if (x0 + lane < gw)
                for (int ty = warp; ty < TH && y0 + ty < gh; ty += G::NW) {
                    const int64_t o = (int64_t)(y0 + ty) * gw + x0 + lane;
                    out_depth[o] = 0.0f;
                    out_valid[o] = 0;
                }
            __syncthreads();
            continue;
        }
        const uint32_t *const zraw = reinterpret_cast<const uint32_t *>(rawB(buf));
        if (!bad) list_masks<G>(zraw, rowmask, x0, y0, gw, gh, warp, lane);
        if (__syncthreads_or(bad)) {
            queue.leave();
            return;
        }
        queue.step();
        float *const dp = out_depth + (int64_t)y0 * gw + x0;
        uint8_t *const vp = out_valid + (int64_t)y0 * gw + x0;
        const int cols = gw - x0, rows = gh - y0;
        auto store = [&](int tx, int ty, float d, bool v) {
            if (tx < cols && ty < rows) {
                dp[(int64_t)ty * gw + tx] = d;
                vp[(int64_t)ty * gw + tx] = v;
            }
        };
        if (list_count<G>(rowmask, lane) > G::DENSE)
            list_gather<G>(a, rawA(buf), zraw, rowmask, reinterpret_cast<uint32_t *>(smem + G::OFF_LIST), pair, cols, rows, warp,
                           lane, store);
        else
            list_blocks<G>(a, rawA(buf), zraw, rowmask, list, tab, cols, rows, warp, lane, store);
        __syncthreads();   // the masks and raw[buf] are rewritten by the next tile
    }
}

template <int R, int BL>
void fill_info(TmaKernelInfo *o) {
    using G = ListGeom<R, BL>;
    *o = TmaKernelInfo{};
    o->supported = 1;
    o->kp = BL;
    o->threads = G::NT;
    o->tile_w = G::TW;
    o->tile_h = G::TH;
    o->smem = G::SMEM;
    o->rgb_box[0] = G::RGB_BX; o->rgb_box[1] = G::RGB_BY;
    o->zbuf_box[0] = G::Z_BX;  o->zbuf_box[1] = G::Z_BY;
}

// (radius, 8 x 8 blocks of a warp); the first of a radius is the default before autotuning: at radius 4,
// whose workload is small frames, one block a warp (twice the tiles of a frame: 18.9 against 23.3 us for
// one 320 x 240 frame with its tile marks, 44 against 46 for 32; four 1080p frames 97 against 88), at 2
// and 7 two (76 against 89 us and 103 against 112 for four 1080p frames).
#define DZ_LIST_CASES(X) X(2, 2) X(4, 1) X(7, 2) X(4, 2) X(7, 1)

}  // namespace

int jbf_list_variants(int r, TmaVariant *out, int cap) {
    int n = 0;
#define DZ_X(R, BL) if (r == R && n < cap) out[n++] = TmaVariant{BL, 8};
    DZ_LIST_CASES(DZ_X)
#undef DZ_X
    return n;
}

bool jbf_list_info(int r, TmaVariant v, TmaKernelInfo *out) {
#define DZ_X(R, BL) if (r == R && v.kp == BL) { fill_info<R, BL>(out); return true; }
    DZ_LIST_CASES(DZ_X)
#undef DZ_X
    return false;
}

cudaError_t jbf_list_prepare(int r, TmaVariant v) {
#define DZ_X(R, BL)                                                                                               \
    if (r == R && v.kp == BL)                                                                                     \
        return cudaFuncSetAttribute(jbf_list_kernel<R, BL>, cudaFuncAttributeMaxDynamicSharedMemorySize, ListGeom<R, BL>::SMEM);
    DZ_LIST_CASES(DZ_X)
#undef DZ_X
    return cudaErrorInvalidValue;
}

cudaError_t jbf_list_load(int r, TmaVariant v) {
    cudaFuncAttributes at;
#define DZ_X(R, BL) if (r == R && v.kp == BL) return cudaFuncGetAttributes(&at, jbf_list_kernel<R, BL>);
    DZ_LIST_CASES(DZ_X)
#undef DZ_X
    return cudaErrorInvalidValue;
}

cudaError_t jbf_list_launch(int r, TmaVariant v, const BatchDev *b, const StageArgs &a, int grid, cudaStream_t s) {
#define DZ_X(R, BL)                                                                    \
    if (r == R && v.kp == BL) {                                                        \
        jbf_list_kernel<R, BL><<<grid, 256, ListGeom<R, BL>::SMEM, s>>>(b, a);         \
        return cudaGetLastError();                                                     \
    }
    DZ_LIST_CASES(DZ_X)
#undef DZ_X
    return cudaErrorInvalidValue;
}

int jbf_list_occupancy(int r, TmaVariant v) {
    int n = 0;
#define DZ_X(R, BL) \
    if (r == R && v.kp == BL) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, jbf_list_kernel<R, BL>, 256, ListGeom<R, BL>::SMEM);
    DZ_LIST_CASES(DZ_X)
#undef DZ_X
    return n;
}

}  // namespace dz
