// One tile of the joint bilateral filter (Eq. (1)-(4)) for a sparse input: the
// single stage on the z-buffer, where a few percent of the pixels hold an
// observation. FP32 differences on the colour bytes (exact squared distance by
// vabsdiff4 and dp4a, one rounding of the exponent, any sigma), as in
// jbf_block.cuh.
//
// A warp owns 8 x 8 blocks of output pixels (two per lane, rows ly and ly + 4 of
// column lx) and sums over the observed positions of a block's footprint (the
// block grown by R) only. Lane r takes footprint row r: the observed columns of
// its row (one 64-bit mask a staged row, by ballot) are counted, the counts
// scanned over the warp, and each lane copies its observations to their places
// in the warp's list: colour word, depth (twice, a two-lane operand) and the
// position's offset in the table of spatial weights. The loop over the list then
// has no rows, masks or bounds left: per observation one broadcast load of the
// record and, for both of the lane's pixels, one load of the spatial weights
//   S[dy][dx] = (2^(-kp |d|^2) for the upper pixel, for the lower), 0 outside the
// window, at least 2^-126 inside it, so that the sum of S says whether the window
// holds an observation. Colour weights, sums and products run as two-lane FP32.
// Records come straight from the raw boxes: no staged copy of the tile.
//
// A footprint with more than kListCap observations takes several lists in turn;
// the order is row-major either way, so results do not depend on the split.
//
// A list costs some 15 instructions per observation of the footprint, most of
// them for windows that do not hold it, so a tile of which more than a part
// G::DENSE is observed gathers instead (list_gather): a thread takes two pixels
// one above the other and walks their window positions in row-major order, an
// unobserved one with weight 0. The terms and their order are those of the
// lists, so a pixel's result is the same bits on either side of the line.
#pragma once

#include "jbf_core.cuh"
#include "tma_common.cuh"

namespace dz {

constexpr int kListCap = 96;   // records of a warp's list (a 1080p view holds some 15 to 30 in a footprint)

// Per cent of a tile's positions above which it gathers, by radius (2, 4 and 7 are instantiated), where
// the two cost the same on evenly spread observations. Four 1280 x 720 frames, lists against gather, us,
// at 10, 20, 30, 50 and 97 % observed: r = 2 54, 70, 91, 128, 257 against 64-67; r = 4 67, 98, 130, 212,
// 416 against 133; r = 7 93, 162, 228, 375, 730 against 294.
constexpr int kListDense[8] = {0, 0, 16, 0, 30, 0, 0, 39};

template <int R_, int BLOCKS_>   // BLOCKS_: 8 x 8 blocks of a warp (the tile is 32 x 16 BLOCKS_)
struct ListGeom {
    static_assert(R_ >= 1 && R_ <= 7, "a footprint row per lane, 64-bit row masks");
    static constexpr int R = R_, NW = 8, NT = NW * 32;
    static constexpr int TW = 32, TH = 16 * BLOCKS_, SW = TW + 2 * R, SH = TH + 2 * R;
    static constexpr int FR = 8 + 2 * R;   // footprint rows and columns
    // colour bytes from byte 3 x0 - RGB_LEAD, z-buffer words from column x0 - Z_LEAD
    static constexpr int RGB_LEAD = ceil_to(3 * R, 16);
    static constexpr int RGB_BX = ceil_to(3 * TW + 3 * R + RGB_LEAD, 16), RGB_BY = SH;
    static constexpr int Z_LEAD = ceil_to(R, 4);
    static constexpr int Z_BX = ceil_to(TW + R + Z_LEAD, 4), Z_BY = SH;
    static constexpr int RAW_A = ceil_to(RGB_BX * RGB_BY, 128), RAW_B = ceil_to(Z_BX * Z_BY * 4, 128);
    static constexpr int TX_BYTES = RGB_BX * RGB_BY + Z_BX * Z_BY * 4;
    // spatial weights: rows dy of the upper pixel + R + 3 (0 .. 10 + 2 R), columns dx + R + 7
    // (0 .. 14 + 2 R); a row stride of 8 modulo 16 entries puts the lanes' 8-byte loads on distinct banks
    static constexpr int SROWS = 11 + 2 * R, SCOLS = 15 + 2 * R, SPITCH = 40;
    static_assert(SCOLS <= SPITCH && SPITCH % 16 == 8, "table rows");
    static constexpr int OFF_LIST = 2 * (RAW_A + RAW_B);
    static constexpr int OFF_TAB = OFF_LIST + NW * kListCap * 16;
    // the gather's spatial weights: window row of the upper pixel (0 .. 2 R + 1), column (0 .. 2 R); its
    // colour words take the lists' place
    static constexpr int OFF_PAIR = OFF_TAB + SROWS * SPITCH * 8;
    static constexpr int OFF_ROWS = OFF_PAIR + (2 * R + 2) * (2 * R + 1) * 8;
    static_assert(SH * SW * 4 <= NW * kListCap * 16, "the colour words fit the lists");
    static constexpr int DENSE = SH * SW * kListDense[R] / 100;   // observations of a tile and its halo
    static constexpr int OFF_BAR = OFF_ROWS + SH * 8;
    static constexpr int SMEM = OFF_BAR + 16;
    static_assert(OFF_LIST % 16 == 0 && OFF_TAB % 16 == 0 && OFF_ROWS % 8 == 0, "layout");
};

// Spatial weight at (dx, dy): 0 outside the window, at least 2^-126 inside it.
template <int R>
__device__ __forceinline__ float list_spatial(const StageArgs &a, int dx, int dy) {
    const bool in = dy >= -R && dy <= R && dx >= -R && dx <= R;
    return in ? fmaxf(ex2_approx(-(float)(dy * dy + dx * dx) * a.kp), 0x1p-126f) : 0.0f;
}

// The tables of spatial weights (every thread of the CTA; followed by a barrier).
template <class G>
__device__ __forceinline__ void list_table(const StageArgs &a, float2 *tab, float2 *pair) {
    constexpr int R = G::R;
    for (int i = threadIdx.x; i < G::SROWS * G::SPITCH; i += G::NT) {
        const int dy = i / G::SPITCH - R - 3, dx = i % G::SPITCH - R - 7;
        tab[i] = make_float2(list_spatial<R>(a, dx, dy), list_spatial<R>(a, dx, dy - 4));
    }
    for (int i = threadIdx.x; i < (2 * R + 2) * (2 * R + 1); i += G::NT) {
        const int dy = i / (2 * R + 1) - R, dx = i % (2 * R + 1) - R;
        pair[i] = make_float2(list_spatial<R>(a, dx, dy), list_spatial<R>(a, dx, dy - 1));
    }
}

// One 64-bit mask of observed positions per staged row; warp w scans rows w, w + NW, ...
template <class G>
__device__ __forceinline__ void list_masks(const uint32_t *zraw, uint64_t *rowmask, int x0, int y0, int gw, int gh, int warp,
                                           int lane) {
    constexpr int R = G::R;
#pragma unroll 2
    for (int sy = warp; sy < G::SH; sy += G::NW) {
        uint64_t mask = 0;
#pragma unroll
        for (int c0 = 0; c0 < G::SW; c0 += 32) {
            const int sx = c0 + lane, gx = x0 - R + sx, gy = y0 - R + sy;
            bool o = false;
            if (sx < G::SW && gx >= 0 && gx < gw && gy >= 0 && gy < gh)
                o = zraw[sy * G::Z_BX + sx - R + G::Z_LEAD] != kEmpty;
            mask |= (uint64_t)__ballot_sync(0xffffffffu, o) << c0;
        }
        if (lane == 0) rowmask[sy] = mask;
    }
}

template <class G>
__device__ __forceinline__ uint32_t list_colour(const uint8_t *rgbraw, int sy, int sx) {
    const uint8_t *p = rgbraw + sy * G::RGB_BX + 3 * sx - 3 * G::R + G::RGB_LEAD;
    return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16);
}

// Observations of the tile and its halo (after the barrier behind list_masks; the same for every thread).
template <class G>
__device__ __forceinline__ int list_count(const uint64_t *rowmask, int lane) {
    int n = 0;
#pragma unroll
    for (int sy = lane; sy < G::SH; sy += 32) n += __popcll(rowmask[sy]);
    return __reduce_add_sync(0xffffffffu, n);
}

// Colour weights 2^(-kc |c_p - c_q|^2) of two pixels and one position, times their spatial weights.
__device__ __forceinline__ float2 list_weight(const StageArgs &a, uint32_t p0, uint32_t p1, uint32_t q, float2 s) {
    const uint32_t d0 = __vabsdiffu4(p0, q), d1 = __vabsdiffu4(p1, q);
    const float2 f = make_float2(__uint_as_float(__dp4a(d0, d0, 0x4B000000u)), __uint_as_float(__dp4a(d1, d1, 0x4B000000u)));
    const float2 x = __ffma2_rn(f, a.bkc, a.bkb);
    return __fmul2_rn(make_float2(ex2_approx(x.x), ex2_approx(x.y)), s);
}

// Depth of the valid pixel (px, py) of the tile from its sums; where the weight sum is too small (rare:
// every observation of the window far in colour), with the largest exponent shifted to 0.
template <class G>
__device__ __forceinline__ float list_depth(const StageArgs &a, const uint8_t *rgbraw, const uint32_t *zraw,
                                            const uint64_t *rowmask, int px, int py, float num, float den) {
    constexpr int R = G::R;
    if (den >= 0x1p-60f) return __fdividef(num, den);
    const uint32_t p = list_colour<G>(rgbraw, py + R, px + R);
    float amax = -__int_as_float(0x7F800000), sn = 0.0f, sd = 0.0f;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass)
#pragma unroll 1
        for (int sy = py; sy <= py + 2 * R; ++sy)
            for (uint64_t mm = (rowmask[sy] >> px) & ((uint64_t(1) << (2 * R + 1)) - 1u); mm; mm &= mm - 1u) {
                const int sx = px + __ffsll((long long)mm) - 1;
                const uint32_t d = __vabsdiffu4(p, list_colour<G>(rgbraw, sy, sx));
                const float z = __uint_as_float(zraw[sy * G::Z_BX + sx - R + G::Z_LEAD]);
                const int dx = sx - R - px, dy = sy - R - py;
                const float e = fmaf((float)__dp4a(d, d, 0u), -a.kc, -(float)(dx * dx + dy * dy) * a.kp);
                if (pass == 0) {
                    amax = fmaxf(amax, e);
                } else {
                    const float w = ex2_approx(e - amax);
                    sn = fmaf(w, z, sn);
                    sd += w;
                }
            }
    return sn / sd;
}

// A densely observed tile (every thread of the CTA): a thread takes rows y and y + 1 of column `lane`.
// Per position one colour word, one depth and one pair of spatial weights (the same for the warp) serve
// both pixels.
template <class G, class Store>
__device__ __forceinline__ void list_gather(const StageArgs &a, const uint8_t *rgbraw, const uint32_t *zraw,
                                            const uint64_t *rowmask, uint32_t *words, const float2 *pair, int cols, int rows,
                                            int warp, int lane, Store &&store) {
    constexpr int R = G::R, T = 2 * R + 1;
    static_assert(G::TH % (2 * G::NW) == 0 && 31 + T <= G::SW && G::TH - 2 + T < G::SH && 31 + R + G::Z_LEAD < G::Z_BX,
                  "every position of a thread's windows lies in the tile and its halo");
    for (int i = threadIdx.x; i < G::SH * G::SW; i += G::NT) words[i] = list_colour<G>(rgbraw, i / G::SW, i % G::SW);
    __syncthreads();
#pragma unroll 1
    for (int y = 2 * warp; y < G::TH && y < rows; y += 2 * G::NW) {
        const uint32_t *const w0 = words + y * G::SW + lane;
        const uint32_t *const z0 = zraw + y * G::Z_BX + lane - R + G::Z_LEAD;
        const uint32_t p0 = w0[R * G::SW + R], p1 = w0[(R + 1) * G::SW + R];
        float2 num = make_float2(0.0f, 0.0f), den = num;
        uint32_t hit0 = 0u, hit1 = 0u;
#pragma unroll 1
        for (int iy = 0; iy <= T; ++iy) {
            const uint32_t m = (uint32_t)(rowmask[y + iy] >> lane) & ((1u << T) - 1u);
            if (iy < T) hit0 |= m;
            if (iy > 0) hit1 |= m;
#pragma unroll
            for (int dx = 0; dx < T; ++dx) {
                const bool seen = (m >> dx) & 1u;
                const float d = seen ? __uint_as_float(z0[iy * G::Z_BX + dx]) : 0.0f, b = seen ? 1.0f : 0.0f;
                const float2 w = list_weight(a, p0, p1, w0[iy * G::SW + dx], pair[iy * T + dx]);
                num = __ffma2_rn(w, make_float2(d, d), num);
                den = __ffma2_rn(w, make_float2(b, b), den);
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool hit = (k ? hit1 : hit0) != 0u;
            float out = 0.0f;
            if (hit && lane < cols && y + k < rows)
                out = list_depth<G>(a, rgbraw, zraw, rowmask, lane, y + k, k ? num.y : num.x, k ? den.y : den.x);
            store(lane, y + k, out, hit);
        }
    }
}

// The tile's blocks (every warp; after the barrier behind list_masks). store(x, y, depth, valid)
// takes tile-relative pixel coordinates.
template <class G, class Store>
__device__ __forceinline__ void list_blocks(const StageArgs &a, const uint8_t *rgbraw, const uint32_t *zraw,
                                            const uint64_t *rowmask, uint4 *list, const float2 *tab, int cols, int rows, int warp,
                                            int lane, Store &&store) {
    constexpr int R = G::R, FR = G::FR;
    const int lx = lane & 7, ly = lane >> 3;
    const uint8_t *const tlane = reinterpret_cast<const uint8_t *>(tab + (3 - ly) * G::SPITCH + 7 - lx);
#pragma unroll 1
    for (int blk = warp; blk < (G::TW / 8) * (G::TH / 8); blk += G::NW) {
        const int bx = (blk % (G::TW / 8)) * 8, by = (blk / (G::TW / 8)) * 8;
        if (bx >= cols || by >= rows) continue;   // outside the image
        // lane r: the observations of footprint row r and their places in the list
        uint32_t m = 0u;
        if (lane < FR) m = (uint32_t)((rowmask[by + lane] >> bx) & ((uint64_t(1) << FR) - 1u));
        uint32_t first = __popc(m);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, first, o);
            if (lane >= o) first += u;
        }
        const int n = (int)__shfl_sync(0xffffffffu, first, 31);
        first -= __popc(m);
        float2 num = make_float2(0.0f, 0.0f), den = num, sum = num;
        if (n > 0) {
            const uint32_t p0 = list_colour<G>(rgbraw, by + ly + R, bx + lx + R),
                           p1 = list_colour<G>(rgbraw, by + ly + 4 + R, bx + lx + R);
#pragma unroll 1
            for (int c0 = 0; c0 < n; c0 += kListCap) {
                int at = (int)first - c0;
                for (uint32_t left = m; left; left &= left - 1u, ++at) {
                    if (at < 0 || at >= kListCap) continue;
                    const int c = __ffs(left) - 1, sy = by + lane, sx = bx + c;
                    const uint32_t z = zraw[sy * G::Z_BX + sx - R + G::Z_LEAD];
                    list[at] = make_uint4(list_colour<G>(rgbraw, sy, sx), (uint32_t)(lane * G::SPITCH + c) * 8u, z, z);
                }
                __syncwarp();
                const int e = min(kListCap, n - c0);
#pragma unroll 4
                for (int i = 0; i < e; ++i) {
                    const uint4 q = list[i];
                    const float2 s = *reinterpret_cast<const float2 *>(tlane + q.y);
                    const float2 w = list_weight(a, p0, p1, q.x, s);
                    num = __ffma2_rn(w, make_float2(__uint_as_float(q.z), __uint_as_float(q.w)), num);
                    den = __fadd2_rn(den, w);
                    sum = __fadd2_rn(sum, s);
                }
                __syncwarp();   // the list is rewritten
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int px = bx + lx, py = by + ly + 4 * k;
            const bool hit = (k ? sum.y : sum.x) > 0.0f;
            float out = 0.0f;
            if (hit && px < cols && py < rows)
                out = list_depth<G>(a, rgbraw, zraw, rowmask, px, py, k ? num.y : num.x, k ? den.y : den.x);
            store(px, py, out, hit);
        }
    }
}

}  // namespace dz
