// densify_frame_noalloc: the whole path for one frame without any device
// allocation, for callers that cannot call cudaMalloc (for example code that
// runs inside a real-time loop with a frozen memory footprint, or a host that
// shares the GPU under an allocator it does not own).
//
// The scratch the kernels need (batch descriptor, status word, z-buffer,
// pooled maps, first-stage result, compaction counts) lives in one file-scope
// __device__ array of kNoallocScratchBytes per device. Host code cannot use
// the array's name as a device address, so at set-up (once per device, on the
// first call made with that device current) the entry point asks the runtime
// for the array's device address with cudaGetSymbolAddress and passes that
// pointer to the kernels. Everything the kernels read is rewritten or cleared
// on every call: the descriptor by a one-block init kernel, the z-buffer by
// the clear kernel, the other maps before they are read. The status word, which
// the kernels only set (a bounded wait on tile copies that gave up, the frame's
// outputs then incomplete), keeps its bits until densify_noalloc_status reads
// them, so that a caller with several frames enqueued misses none.
#include <cstring>
#include <mutex>
#include <string>

#include "runtime_internal.h"

namespace dz {

namespace {

constexpr size_t kNoallocScratchBytes = size_t(16) << 20;   // enough for one 1920x1080 two-stage frame
constexpr int kMaxDevices = 64;

}  // namespace

// The scratch itself: one copy per device that loads the library, kept until exit.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

namespace {

struct DeviceSetup {
    bool ready = false;
    unsigned char *scratch = nullptr;   // device address of g_noalloc_scratch
    int sms = 0;
};

std::mutex g_setup_mu;
DeviceSetup g_setup[kMaxDevices];

// The scratch begins with the batch descriptor of one frame, then the status word.
constexpr size_t kOffStatus = (offsetof(BatchDev, f) + sizeof(FrameDev) + 255) & ~size_t(255);

thread_local bool g_inject_wait_failure = false;   // densify_inject_noalloc_wait_failure: armed for the thread's next call

// Frame descriptor passed by value as raw words (its tensor-map members are
// 64-byte aligned, which kernel parameters do not guarantee).
struct FrameWords {
    uint32_t w[sizeof(FrameDev) / 4];
};
static_assert(sizeof(FrameDev) % 4 == 0, "FrameDev is a whole number of words");

struct Prefix {
    int32_t zb, pt[kMaxScans], pool, t1, t2, bp, mk, rp;
    int32_t tw[2], th[2], r[2];   // tiles of the TMA stages (th 0: a plain kernel)
};

__global__ void noalloc_init_kernel(BatchDev *b, FrameWords f, Prefix p, int32_t *status) {
    uint32_t *dst = reinterpret_cast<uint32_t *>(&b->f[0]);
    for (int i = threadIdx.x; i < (int)(sizeof(FrameDev) / 4); i += blockDim.x) dst[i] = f.w[i];
    if (threadIdx.x == 0) {
        b->n_frames = 1;
        b->status = status;
        b->zb_pre[0] = 0;
        b->zb_pre[1] = p.zb;
        b->pt_pre[0] = 0;
        for (int s = 0; s < kMaxScans; ++s) b->pt_pre[s + 1] = b->pt_pre[s] + p.pt[s];
        b->pool_pre[0] = 0;
        b->pool_pre[1] = p.pool;
        b->t1_pre[0] = 0;
        b->t1_pre[1] = p.t1;
        b->t2_pre[0] = 0;
        b->t2_pre[1] = p.t2;
        b->bp_pre[0] = 0;
        b->bp_pre[1] = p.bp;
        b->mk_pre[0] = 0;
        b->mk_pre[1] = p.mk;
        b->rp_pre[0] = 0;
        b->rp_pre[1] = p.rp;
        b->tl_on = p.th[0] > 0 || p.th[1] > 0;
        for (int i = 0; i < 2; ++i) {
            b->tl_tw[i] = p.tw[i];
            b->tl_th[i] = p.th[i];
            b->tl_r[i] = p.r[i];
        }
    }
    // the tensor maps among the words, for the copies of the kernels that follow
    __syncthreads();
    asm volatile("fence.proxy.tensormap::generic.release.gpu;" ::: "memory");
}

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }
int cdiv(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Loads every kernel that some frame or parameters may take, whichever route they then go: code that is
// loaded lazily, at a kernel's first launch, takes device memory.
cudaError_t load_kernels() {
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, noalloc_init_kernel);
    if (e == cudaSuccess) e = load_points();
    if (e == cudaSuccess) e = load_pool_bp();
    if (e == cudaSuccess) e = load_tile_mark();
    for (int r = 1; r <= kMaxR && e == cudaSuccess; ++r) {
        e = load_jbf_single(r);
        if (e == cudaSuccess) e = load_jbf_coarse(r);
        if (e == cudaSuccess && r <= 3) e = load_jbf_up(r);
        // FP32 contexts' default kernels: the first variant of a form
        for (int src : {TMA_SRC_UP, TMA_SRC_ZBUF, TMA_SRC_COARSE})
            for (int form = 0; form <= TMA_FORM_LIST && e == cudaSuccess; ++form) {
                TmaVariant v;
                if (form != TMA_FORM_FP16 && jbf_tma_variants(src, r, form, &v, 1) == 1) e = jbf_tma_load(src, r, v, form);
            }
    }
    return e;
}

densify_status fail(densify_status s, const std::string &m) {
    set_thread_error(m);
    return s;
}

}  // namespace

}  // namespace dz

using namespace dz;

extern "C" DENSIFY_API densify_status densify_frame_noalloc(const densify_params *params, const densify_frame *f,
                                                            void *cuda_stream) {
    if (!params || !f) return fail(DENSIFY_E_INVALID, "params and frame must not be NULL");
    const std::string perr = check_params(*params);
    if (!perr.empty()) return fail(DENSIFY_E_INVALID, perr);
    if (f->memory != DENSIFY_MEM_DEVICE) return fail(DENSIFY_E_INVALID, "the no-allocation entry takes device frames");
    if (params->occlusion_radius > 0 || params->motion_threshold > 0.0f || params->contour_threshold > 0.0f)
        return fail(DENSIFY_E_INVALID, "the no-allocation entry runs without occlusion, afterimage or contour removal");
    const int W = f->K.width, H = f->K.height;
    if (W < 1 || H < 1 || W > 16384 || H > 16384) return fail(DENSIFY_E_INVALID, "image size must be in 1..16384");
    if (f->num_scans < 0 || f->num_scans > kMaxScans) return fail(DENSIFY_E_INVALID, "num_scans must be in 0..3");
    for (int s = 0; s < f->num_scans; ++s) {
        const densify_scan &S = f->scans[s];
        if (S.count < 0 || S.count > (int64_t)1 << 30) return fail(DENSIFY_E_INVALID, "scan count out of range");
        if (S.stride_bytes != 12 && S.stride_bytes != 16) return fail(DENSIFY_E_INVALID, "stride_bytes must be 12 or 16");
        if (S.count > 0 && (!S.xyz || ((uintptr_t)S.xyz & 15u)))
            return fail(DENSIFY_E_INVALID, "scan xyz must be a 16-byte aligned device pointer");
    }
    if (!f->rgb || f->rgb_pitch < 3 * (int64_t)W) return fail(DENSIFY_E_INVALID, "rgb missing or pitch < 3 * width");
    if (!f->out_depth || !f->out_valid)
        return fail(DENSIFY_E_INVALID, "the no-allocation entry needs out_depth and out_valid");
    if (params->emit_points && (!f->out_points_n || (f->out_points_cap > 0 && !f->out_points) ||
                                ((uintptr_t)f->out_points & 15u)))
        return fail(DENSIFY_E_INVALID, "points on: out_points_n needed, out_points 16-byte aligned");

    // scratch layout
    const int pool = params->num_stages == 2 ? params->pool : 1;
    const int Wc = (W + pool - 1) / pool, Hc = (H + pool - 1) / pool;
    const int zpitch = (W + 3) & ~3, cpitch = (Wc + 3) & ~3;
    const int64_t npx = (int64_t)W * H;
    const int n_bp = cdiv(npx, kBpChunk);
    size_t o = kOffStatus + 256;
    const size_t off_zbuf = o;
    o += up256((size_t)zpitch * H * 4);
    size_t off_cg = 0, off_cs = 0, off_s1 = 0;
    if (params->num_stages == 2) {
        off_cg = o;
        o += up256((size_t)cpitch * Hc * 16);
        off_cs = o;
        o += up256((size_t)cpitch * Hc * 4);
        off_s1 = o;
        o += up256((size_t)cpitch * Hc * 8);
    }
    const size_t off_cnt = o;
    o += up256((size_t)n_bp * kBpWarps * 4);
    // The filters run in the kernels that a context would take (TMA-staged tiles; the points from the
    // second filter where it can write them) when the colour rows start on 16-byte boundaries and the
    // tile flags and validity bits fit beside the rest; else in the plain shared-memory kernels. One
    // 1080p frame: 113 us in the plain kernels, 80 so.
    densify_params pf = *params;
    pf.precision = DENSIFY_FP32;   // what the plain kernels compute in
    const int nst = params->num_stages;
    StageKernel ker[2];
    size_t flag_words[2] = {0, 0};
    for (int i = 0; i < nst; ++i) {
        const int kind = nst == 1 ? 0 : i == 0 ? 1 : 2;
        ker[i] = default_stage_kernel(pf, kind, params->stage[i].radius);
        const int gw = kind == 1 ? Wc : W, gh = kind == 1 ? Hc : H;
        if (ker[i].tma) flag_words[i] = (size_t)cdiv(gw, ker[i].tile_w) * cdiv(gh, ker[i].tile_h);
    }
    // A single stage of few taps, or over more points than pixels, stays in the plain kernel: the list form
    // saves little there and its tile marks are one launch more. Pass times, list / plain, us: radius 2, one
    // lidar sweep to three, 320 x 240 46-50 / 39-41, 1280 x 720 52-56 / 46-48, 1920 x 1080 58.4 / 59.8 at 0.004
    // points a pixel, 68.2 / 68.2 at 0.09, 74.8 / 70.1 at 0.36; radius 4, 640 x 480 49.6 / 49.6 at 0.4,
    // 51.6 / 45.5 at 1.2; radius 7, 64.0 / 64.5 at 1.2, 76.3 / 66.4 at 2.4.
    int64_t points_in = 0;
    for (int s = 0; s < f->num_scans; ++s) points_in += f->scans[s].count;
    if (nst == 1 && ker[0].form == TMA_FORM_LIST &&
        (points_in > npx || (ker[0].radius == 2 && (npx < (1 << 20) || 10 * points_in > npx))))
        ker[0].tma = false;
    const size_t off_flags = o, off_bits = o + up256((flag_words[0] + flag_words[1]) * 4);
    const size_t bits_bytes = nst == 2 ? (size_t)cdiv(Wc, 32) * Hc * 4 : 0;
    const bool tma = (ker[0].tma || ker[1].tma) && !((uintptr_t)f->rgb & 15u) && !(f->rgb_pitch & 15) &&
                     off_bits + up256(bits_bytes) <= kNoallocScratchBytes;
    if (!tma) ker[0].tma = ker[1].tma = false;
    const bool points = tma && params->emit_points && nst == 2 && ker[1].tma && ker[1].form == TMA_FORM_BLOCK;
    if (o > kNoallocScratchBytes)
        return fail(DENSIFY_E_INVALID, "frame needs " + std::to_string(o) + " bytes of scratch; the no-allocation "
                                       "entry holds " + std::to_string(kNoallocScratchBytes) +
                                       " (one 1920x1080 two-stage frame fits)");

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(DENSIFY_E_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(DENSIFY_E_INVALID, "device index too large");
    DeviceSetup setup;
    {
        std::lock_guard<std::mutex> lock(g_setup_mu);
        DeviceSetup &S = g_setup[dev];
        if (!S.ready) {
            void *p = nullptr;
            if ((e = cudaGetSymbolAddress(&p, g_noalloc_scratch)) != cudaSuccess)
                return fail(DENSIFY_E_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            if ((e = cudaDeviceGetAttribute(&S.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
                return fail(DENSIFY_E_CUDA, std::string("device attribute: ") + cudaGetErrorString(e));
            if ((e = load_kernels()) != cudaSuccess)
                return fail(DENSIFY_E_CUDA, std::string("kernel load: ") + cudaGetErrorString(e));
            S.scratch = static_cast<unsigned char *>(p);
            S.ready = true;
        }
        setup = S;
    }
    unsigned char *base = setup.scratch;
    cudaStream_t s = (cudaStream_t)cuda_stream;

    // frame descriptor
    FrameDev d;
    std::memset(&d, 0, sizeof(d));
    d.W = W; d.H = H; d.Wc = Wc; d.Hc = Hc; d.cpitch = cpitch; d.zpitch = zpitch;
    d.fx = f->K.fx; d.fy = f->K.fy; d.cx = f->K.cx; d.cy = f->K.cy;
    std::memcpy(d.c2w, f->cam_to_world, sizeof(d.c2w));
    d.num_scans = f->num_scans;
    d.n_bp_chunks = n_bp;
    for (int k = 0; k < kMaxScans; ++k) {
        if (k < f->num_scans) {
            d.scans[k].xyz = f->scans[k].xyz;
            d.scans[k].count = f->scans[k].count;
            d.scans[k].stride_floats = f->scans[k].stride_bytes / 4;
            std::memcpy(d.scans[k].l2w, f->scans[k].lidar_to_world, sizeof(d.scans[k].l2w));
        } else {
            d.scans[k].stride_floats = 3;
        }
    }
    d.rgb = f->rgb;
    d.rgb_pitch = f->rgb_pitch;
    d.zbuf = reinterpret_cast<uint32_t *>(base + off_zbuf);
    d.zbuf_raw = d.zbuf;
    d.zclear = 1;   // the static scratch holds whatever the last call left: cleared every call
    d.newest_scan = -1;
    if (params->num_stages == 2) {
        d.cguide = reinterpret_cast<float4 *>(base + off_cg);
        d.cssum = reinterpret_cast<float *>(base + off_cs);
        d.s1 = reinterpret_cast<float2 *>(base + off_s1);
        d.out_coarse = f->out_coarse;
        d.out_coarse_valid = f->out_coarse_valid;
    }
    d.chunk_cnt = reinterpret_cast<uint32_t *>(base + off_cnt);
    d.out_depth = f->out_depth;
    d.out_valid = f->out_valid;
    d.flt_depth = f->out_depth;
    d.flt_valid = f->out_valid;
    if (params->emit_points) {
        d.out_points = reinterpret_cast<float4 *>(f->out_points);
        d.points_cap = f->out_points_cap;
        d.points_n = f->out_points_n;
    }
    for (int i = 0; i < nst; ++i)
        if (ker[i].tma && !encode_stage_maps(d, ker[i].src, ker[i].info))
            return fail(DENSIFY_E_CUDA, "tensor map encoding failed");
    if (tma) {
        d.tma = 1;
        d.tflags[0] = reinterpret_cast<int32_t *>(base + off_flags);
        d.tflags[1] = d.tflags[0] + (ker[0].tma ? flag_words[0] : 0);
        d.ntflags = (int32_t)((ker[0].tma ? flag_words[0] : 0) + (ker[1].tma ? flag_words[1] : 0));
    }
    if (points) {   // the prefixes take the pooled guide's place once the first filter is done with it
        d.vbits = reinterpret_cast<uint32_t *>(base + off_bits);
        d.row_pre = reinterpret_cast<uint32_t *>(d.cguide);
        d.seg_pre = d.row_pre + H;
    }
    FrameWords fw;
    std::memcpy(fw.w, &d, sizeof(d));
    Prefix pre{};
    pre.zb = cdiv((int64_t)zpitch * H, kZbWordsPerChunk);
    for (int k = 0; k < kMaxScans; ++k) pre.pt[k] = cdiv(d.scans[k].count, kPtsPerChunk);
    const int r1 = params->stage[0].radius, r2 = nst == 2 ? params->stage[1].radius : 0;
    for (int i = 0; i < nst; ++i) {
        const int plain_kp = ker[i].kind == 0 ? kp_jbf_single(r1) : ker[i].kind == 1 ? kp_jbf_coarse(r1) : kp_jbf_up(r2);
        const int tw = ker[i].tma ? ker[i].tile_w : 32, th = ker[i].tma ? ker[i].tile_h : 8 * plain_kp;
        const int gw = ker[i].kind == 1 ? Wc : W, gh = ker[i].kind == 1 ? Hc : H;
        (i == 0 ? pre.t1 : pre.t2) = cdiv(gw, tw) * cdiv(gh, th);
        pre.tw[i] = tw;
        pre.th[i] = ker[i].tma ? th : 0;
        pre.r[i] = ker[i].radius;
    }
    if (nst == 2) pre.pool = cdiv(Wc, kPoolPerChunk) * Hc;
    else pre.mk = cdiv(H, kMarkBand) * cdiv(W, 32);
    pre.rp = points ? cdiv(Hc, kRowsPerItem) : 0;
    pre.bp = params->emit_points ? n_bp : 0;

    StageArgs sa[2];
    if (params->num_stages == 1) {
        fill_stage_args(sa[0], params->stage[0], 1, 0);
    } else {
        fill_stage_args(sa[0], params->stage[0], params->pool, 0);
        fill_stage_args(sa[1], params->stage[1], params->pool, params->stage2_input);
    }

    BatchDev *b = reinterpret_cast<BatchDev *>(base);
    int32_t *status = reinterpret_cast<int32_t *>(base + kOffStatus);
    const int sms = setup.sms;
    noalloc_init_kernel<<<1, 128, 0, s>>>(b, fw, pre, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return fail(DENSIFY_E_CUDA, cudaGetErrorString(e));
#define NA_TRY(x)                                                             \
    do {                                                                      \
        if ((e = (x)) != cudaSuccess) return fail(DENSIFY_E_CUDA, cudaGetErrorString(e)); \
    } while (0)
    NA_TRY(launch_prep(b, sms * occupancy_points(K_PREP), s));
    NA_TRY(launch_project(b, sms * occupancy_points(K_PROJECT), s));
    auto filter = [&](int i) -> cudaError_t {
        const StageKernel &k = ker[i];
        if (k.tma) {
            cudaError_t e = jbf_tma_prepare(k.src, k.radius, k.v, k.form);
            if (e != cudaSuccess) return e;
            const int grid = sms * occupancy_jbf_tma(k.src, k.radius, k.v, k.form);
            if (i == 1 && points) return jbf_block_launch(k.radius, k.v, true, b, sa[i], grid, s);
            return launch_jbf_tma(k.src, k.radius, k.v, k.form, b, sa[i], grid, s);
        }
        if (k.kind == 0) return launch_jbf_single(r1, b, sa[i], sms * occupancy_jbf_single(r1), s);
        if (k.kind == 1) return launch_jbf_coarse(r1, b, sa[i], sms * occupancy_jbf_coarse(r1), s);
        return launch_jbf_up(r2, b, sa[i], sms * occupancy_jbf_up(r2), s);
    };
    if (nst == 2) {
        NA_TRY(launch_pool(b, params->pool, sms * occupancy_pool_bp(K_POOL), s));
        NA_TRY(filter(0));
        if (points) NA_TRY(launch_bp_rows(b, r2, sms * 4, s));
        NA_TRY(filter(1));
    } else {
        if (ker[0].tma) NA_TRY(launch_tile_mark(ker[0].src, b, 0, ker[0].tile_h, r1, sms * 8, s));
        NA_TRY(filter(0));
    }
    if (params->emit_points && !points) {
        NA_TRY(launch_bp_count(b, sms * occupancy_pool_bp(K_BP_COUNT), s));
        NA_TRY(launch_bp_write(b, sms * occupancy_pool_bp(K_BP_WRITE), s));
    }
    if (f->out_zbuf)
        NA_TRY(cudaMemcpy2DAsync(f->out_zbuf, (size_t)W * 4, d.zbuf, (size_t)zpitch * 4, (size_t)W * 4, (size_t)H,
                                 cudaMemcpyDeviceToDevice, s));
    if (g_inject_wait_failure) {   // test hook: the bit a kernel sets when a bounded wait gives up
        g_inject_wait_failure = false;
        NA_TRY(cudaMemsetAsync(status, 1, 1, s));
    }
#undef NA_TRY
    return DENSIFY_OK;
}

extern "C" DENSIFY_API densify_status densify_noalloc_status(void *cuda_stream) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(DENSIFY_E_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(DENSIFY_E_INVALID, "device index too large");
    unsigned char *base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_setup_mu);
        base = g_setup[dev].scratch;
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int32_t status = 0;
    if (base) {   // some call ran on this device
        e = cudaMemcpyAsync(&status, base + kOffStatus, sizeof(status), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e == cudaSuccess && status) {
            e = cudaMemsetAsync(base + kOffStatus, 0, sizeof(status), s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        }
    } else {
        e = cudaStreamSynchronize(s);
    }
    if (e != cudaSuccess) return fail(DENSIFY_E_CUDA, std::string("status: ") + cudaGetErrorString(e));
    if (status)
        return fail(DENSIFY_E_CUDA, "a kernel's bounded wait on its tile copies gave up (status " +
                                        std::to_string(status) + "): outputs are incomplete");
    return DENSIFY_OK;
}

extern "C" DENSIFY_API densify_status densify_inject_noalloc_wait_failure(void) {
    g_inject_wait_failure = true;
    return DENSIFY_OK;
}
