// C ABI of libelsa: host-side validation, dispatch and error reporting.  No kernel lives here.

#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <vector>

#include "elsa_internal.h"

namespace elsa {

static thread_local char g_error[512] = "";
static std::atomic<unsigned long long> g_launches{0};
static std::atomic<int> g_variant{(int)ELSA_VARIANT_AUTO};
static std::atomic<bool> g_grouping{true};

namespace {
struct ProfileRecord {
    int kernel, layer;
    cudaEvent_t start, stop;
};
std::atomic<bool> g_profile_on{false};
std::mutex g_profile_mutex;
std::vector<ProfileRecord> g_profile;
thread_local int g_profile_layer = -1;
}  // namespace

void set_profile_layer(int layer) { g_profile_layer = layer; }

ProfileScope::ProfileScope(int kernel, cudaStream_t stream) : slot_(-1), stream_(stream)
{
    if (!g_profile_on.load(std::memory_order_relaxed)) return;
    ProfileRecord r;
    r.kernel = kernel;
    r.layer = g_profile_layer;
    if (cudaEventCreate(&r.start) != cudaSuccess) { cudaGetLastError(); return; }
    if (cudaEventCreate(&r.stop) != cudaSuccess) { cudaGetLastError(); cudaEventDestroy(r.start); return; }
    cudaEventRecord(r.start, stream);
    std::lock_guard<std::mutex> lock(g_profile_mutex);
    g_profile.push_back(r);
    slot_ = (int)g_profile.size() - 1;
}

ProfileScope::~ProfileScope()
{
    if (slot_ < 0) return;
    std::lock_guard<std::mutex> lock(g_profile_mutex);
    if (slot_ < (int)g_profile.size()) cudaEventRecord(g_profile[slot_].stop, stream_);
}

elsa_status fail(elsa_status st, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_error, sizeof g_error, fmt, ap);
    va_end(ap);
    return st;
}

elsa_status launched(const char* what)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(ELSA_ERR_CUDA, "launch of %s failed: %s", what, cudaGetErrorString(e));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ELSA_OK;
}

elsa_status device_info(DeviceInfo* info)
{
    static DeviceInfo cache[64];
    static std::atomic<bool> have[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaError_t e = cudaGetLastError();
        return fail(ELSA_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    }
    const int slot = dev & 63;
    if (!have[slot].load(std::memory_order_acquire)) {
        DeviceInfo d;
        d.device = dev;
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) goto bad;
        d.sm_count = v;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) goto bad;
        d.cc_major = v;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) goto bad;
        d.smem_optin = (size_t)v;
        cache[slot] = d;
        have[slot].store(true, std::memory_order_release);
    }
    *info = cache[slot];
    if (info->cc_major != 10)
        return fail(ELSA_ERR_ARCH, "device %d has compute capability %d.x; this library is built for 10.x only",
                    dev, info->cc_major);
    return ELSA_OK;
bad:
    cudaError_t e = cudaGetLastError();
    return fail(ELSA_ERR_CUDA, "cudaDeviceGetAttribute: %s", cudaGetErrorString(e));
}

namespace {

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

elsa_status check_level(int out, int in, int N, int M, int dtype)
{
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return fail(ELSA_ERR_DTYPE, "dtype %d is neither ELSA_F16 nor ELSA_BF16", dtype);
    if (out <= 0 || in <= 0) return fail(ELSA_ERR_SHAPE, "non-positive dimension (out=%d, in=%d)", out, in);
    if (index_bits(M) < 0 || N < 1 || N > M) return fail(ELSA_ERR_NM, "unsupported level %d:%d (M in {4, 8, 16}, 1 <= N <= M)", N, M);
    if (in % M != 0) return fail(ELSA_ERR_SHAPE, "in=%d is not a multiple of M=%d", in, M);
    if (in % 8 != 0 || out % 8 != 0) return fail(ELSA_ERR_ALIGN, "in=%d and out=%d must be multiples of 8 (16-byte row pitch)", in, out);
    return ELSA_OK;
}

elsa_status check_linear(const void* X, int rows, const void* vals, const uint32_t* idx, const void* bias,
                         int out, int in, int N, int M, int dtype, const void* Y, const void* workspace,
                         size_t workspace_bytes)
{
    if (!X || !vals || !Y) return fail(ELSA_ERR_NULL, "X, vals and Y must not be NULL");
    elsa_status st = check_level(out, in, N, M, dtype);
    if (st != ELSA_OK) return st;
    if (rows <= 0) return fail(ELSA_ERR_SHAPE, "non-positive rows=%d", rows);
    if (N != M && !idx) return fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
    if (!aligned16(X) || !aligned16(vals) || !aligned16(Y) || (idx && !aligned16(idx)) ||
        (bias && !aligned16(bias)))
        return fail(ELSA_ERR_ALIGN, "X, vals, idx, bias and Y must be 16-byte aligned");
    const size_t need = elsa_workspace_bytes(rows, in, out, N, M, (elsa_dtype)dtype);
    if (need) {
        if (!workspace || workspace_bytes < need)
            return fail(ELSA_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, workspace ? workspace_bytes : (size_t)0);
        if (((uintptr_t)workspace & 255u) != 0) return fail(ELSA_ERR_ALIGN, "workspace must be 256-byte aligned");
    }
    return ELSA_OK;
}

// A side stream with its fork and join events, for the weight images that are built beside a call's other kernels.  A
// call takes one from the device's pool and hands it back when all it enqueued is joined into the caller's stream, so
// calls of several threads never share events; the pool holds as many as calls have ever overlapped.  A stream that was
// forked from a capturing one belongs to that capture until it ends: meanwhile only calls of the same capture take it.
struct SidePipe {
    int device;
    cudaStream_t stream;
    cudaEvent_t fork, join;
};
std::vector<SidePipe> g_side[64];
std::mutex g_side_mutex;

class SideStream {
public:
    ~SideStream()
    {
        if (!have_) return;
        std::lock_guard<std::mutex> lock(g_side_mutex);
        g_side[pipe_.device & 63].push_back(pipe_);
    }
    // Takes a pipe (once); the side stream then starts where `from` stands now.
    elsa_status fork(int device, cudaStream_t from)
    {
        if (!have_) {
            unsigned long long capture = 0;
            elsa_status st = capture_of(from, &capture);
            if (st != ELSA_OK) return st;
            std::lock_guard<std::mutex> lock(g_side_mutex);
            std::vector<SidePipe>& pool = g_side[device & 63];
            size_t at = pool.size();
            for (size_t i = pool.size(); i-- > 0 && at == pool.size();) {
                unsigned long long held = 0;
                if (pool[i].device == device && capture_of(pool[i].stream, &held) == ELSA_OK && (held == 0 || held == capture)) at = i;
            }
            if (at < pool.size()) {
                pipe_ = pool[at];
                pool.erase(pool.begin() + (long)at);
            } else {
                pipe_.device = device;
                const bool ok = cudaStreamCreateWithFlags(&pipe_.stream, cudaStreamNonBlocking) == cudaSuccess &&
                                cudaEventCreateWithFlags(&pipe_.fork, cudaEventDisableTiming) == cudaSuccess &&
                                cudaEventCreateWithFlags(&pipe_.join, cudaEventDisableTiming) == cudaSuccess;
                if (!ok) {
                    cudaError_t e = cudaGetLastError();
                    return fail(ELSA_ERR_CUDA, "creating the image stream: %s", cudaGetErrorString(e));
                }
            }
            have_ = true;
        }
        cudaError_t e = cudaEventRecord(pipe_.fork, from);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe_.stream, pipe_.fork, 0);
        if (e != cudaSuccess) { cudaGetLastError(); return fail(ELSA_ERR_CUDA, "forking the image stream: %s", cudaGetErrorString(e)); }
        forked_ = true;
        return ELSA_OK;
    }
    // `into` waits for what the side stream holds (nothing to do without a fork).  Also after a failed launch: a fork
    // must not dangle.
    elsa_status join(cudaStream_t into)
    {
        if (!forked_) return ELSA_OK;
        forked_ = false;
        cudaError_t e = cudaEventRecord(pipe_.join, pipe_.stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(into, pipe_.join, 0);
        if (e != cudaSuccess) { cudaGetLastError(); return fail(ELSA_ERR_CUDA, "joining the image stream: %s", cudaGetErrorString(e)); }
        return ELSA_OK;
    }
    bool forked() const { return forked_; }
    cudaStream_t stream() const { return pipe_.stream; }

private:
    // The capture a stream takes part in, 0 if none.  (One that was invalidated stays until its owner ends it.)
    static elsa_status capture_of(cudaStream_t s, unsigned long long* id)
    {
        cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
        const cudaError_t e = cudaStreamGetCaptureInfo(s, &status, id);
        if (e != cudaSuccess) { cudaGetLastError(); return fail(ELSA_ERR_CUDA, "asking for a stream's capture: %s", cudaGetErrorString(e)); }
        if (status == cudaStreamCaptureStatusNone) *id = 0;
        else if (status == cudaStreamCaptureStatusInvalidated) *id = ~0ull;
        return ELSA_OK;
    }

    bool have_ = false, forked_ = false;
    SidePipe pipe_;
};

// KIND_SMALL expands a packed weight itself; KIND_SMALL_IMAGE is the same kernel on the dense image of the weight.
enum LinearKind { KIND_SIMT, KIND_SMALL, KIND_SMALL_IMAGE, KIND_DENSE_ONE, KIND_DENSE_PAIR, KIND_SPARSE_ONE, KIND_SPARSE_PAIR, KIND_SPARSE_WS, KIND_SPARSE_ST };

// Form of the 2-of-4 weight image each sparse kernel reads (the weight-stationary one in the masked form only).
int sp24_layout_of(LinearKind kind)
{
    return kind == KIND_SPARSE_WS ? SP24_PERMUTED : kind == KIND_SPARSE_ST ? SP24_TILED : SP24_ROWS;
}

// The weight image that a layer's kernel reads, built in `region`.
ImageJob image_job(LinearKind kind, const void* vals, const uint32_t* idx, int out, int in, int N, int M, void* region)
{
    ImageJob j;
    j.src = (const uint16_t*)vals; j.idx = idx; j.dst = (uint16_t*)region; j.out = out; j.in = in; j.N = N; j.M = M;
    if (kind == KIND_SPARSE_PAIR || kind == KIND_SPARSE_ST) {
        j.kind = IMAGE_SP24;
        j.meta = (uint8_t*)region + sp24_meta_offset(out, in);
        j.layout = sp24_layout_of(kind);
    }
    return j;
}

// Whether a packed weight (N < M) goes through an image: the few-rows kernel and the weight-stationary one expand it themselves.
bool reads_image(LinearKind kind) { return kind != KIND_SIMT && kind != KIND_SMALL && kind != KIND_SPARSE_WS; }

// A layer of the sparse kernels: on the packed weight (weight-stationary kernel) or on its image.
SparseJob sparse_job(LinearKind kind, const void* X, int rows, const void* vals, const uint32_t* idx, const void* bias, int out, int in, int N,
                     int M, void* Y, const void* image)
{
    SparseJob j;
    j.X = (const uint16_t*)X; j.bias = (const uint16_t*)bias; j.Y = (uint16_t*)Y; j.workspace = image;
    j.rows = rows; j.in = in; j.out = out;
    if (kind == KIND_SPARSE_WS) { j.w = (const uint16_t*)vals; j.idx = idx; j.N = N; j.M = M; }
    return j;
}

// What a layer is part of: a call of its own, a table whose layers share persistent launches, or a chained block, where
// the images are built off the critical path and an epilogue that takes GELU or the residual saves a pass.
enum LinearUse { USE_SINGLE, USE_MASKED, USE_TABLE, USE_CHAIN };      // USE_MASKED: a call of its own on the shared weight

// Which kernel a layer runs on.  AUTO is the product rule; a forced variant is honoured where it applies.
// gelu: the layer's epilogue applies GELU (USE_CHAIN).
elsa_status pick_kind(LinearUse use, int rows, int out, int in, int N, int M, int sm_count, LinearKind* kind, bool gelu = false)
{
    const int variant = g_variant.load(std::memory_order_relaxed);
    const bool sparse_ok = N != M && linear_tc_sparse_suits(in, N);
    switch (variant) {
    case ELSA_VARIANT_SIMT: *kind = KIND_SIMT; return ELSA_OK;
    case ELSA_VARIANT_TC_DENSE: *kind = KIND_DENSE_ONE; return ELSA_OK;
    case ELSA_VARIANT_TC_SMALL: *kind = KIND_SMALL; return ELSA_OK;
    case ELSA_VARIANT_TC_PAIR: *kind = KIND_DENSE_PAIR; return ELSA_OK;
    case ELSA_VARIANT_TC_SPARSE:
    case ELSA_VARIANT_TC_SPARSE_PAIR:
        if (!sparse_ok)
            return fail(ELSA_ERR_NM, "the sparse-MMA variant needs N <= 2 < M and in %% 16 == 0 (got %d:%d, in=%d)", N, M, in);
        *kind = variant == ELSA_VARIANT_TC_SPARSE ? KIND_SPARSE_ONE : KIND_SPARSE_PAIR;
        return ELSA_OK;
    case ELSA_VARIANT_TC_SPARSE_WS:
        if (N == M || !linear_tc_sparse_ws_suits(in, out, N, sm_count))
            return fail(ELSA_ERR_NM, "the weight-stationary sparse variant needs N <= 2 < M, in %% 128 == 0 and in <= 1024 "
                        "(got %d:%d, in=%d)", N, M, in);
        *kind = KIND_SPARSE_WS;
        return ELSA_OK;
    case ELSA_VARIANT_TC_SPARSE_ST:
        if (N == M || !linear_tc_sparse_st_suits(in, N))
            return fail(ELSA_ERR_NM, "the streaming sparse variant needs N <= 2 < M and in %% 128 == 0 (got %d:%d, in=%d)", N, M, in);
        *kind = KIND_SPARSE_ST;
        return ELSA_OK;
    default: break;
    }
    // Times below: us back to back, weight image included, at 2:8 unless noted.
    const int k_blocks = (in + 63) / 64;
    const long long tiles_small = (long long)((rows + 127) / 128) * ((out + 63) / 64);
    const long long tiles_f = (out + 255) / 256, pairs = sm_count / 2;
    const bool pair_full = linear_tc_pair_suits(rows, out, sm_count);
    const bool ws_ok = sparse_ok && linear_tc_sparse_ws_suits(in, out, N, sm_count) && out >= 512;
    const bool st_ok = sparse_ok && linear_tc_sparse_st_suits(in, N);
    // With at least 900 rows per SM pair the weight-stationary kernel's set-up (its block goes to tensor memory first) is
    // paid back by activations being its only shared-memory traffic: 768 -> 3072, 6304 rows 23.2 against 23.1 on the
    // sparse pair kernel, 12608 rows 35.0 against 38.8, 3152 rows 17.3 against 16.4; 1024 -> 4096, 12608 rows 53.8
    // against 58.8 on the streaming kernel; 256 -> 1024 at the dense rate, 25216 rows 20.5 against 18.7.
    const bool ws_large = ws_ok && (long long)rows * tiles_f >= 900 * pairs;
    if (use == USE_TABLE) {
        // Layers of a table share launches, so a layer need not fill the chip by itself and what counts is throughput:
        // N <= 2 goes to the sparse MMA from K = 256 and a quarter wave of tiles up (K = 128 layers are pure streaming
        // problems), weight-stationary where the reduction fits beside wide accumulators, streaming where it does not.
        if (sparse_ok && in >= 256 && (long long)((rows + 223) / 224) * tiles_f >= sm_count / 4) {
            const bool ws = ws_large || (ws_ok && in <= 896 && rows >= 256 * pairs / tiles_f);
            *kind = ws ? KIND_SPARSE_WS : in > 768 && st_ok ? KIND_SPARSE_ST : KIND_SPARSE_PAIR;
        } else {
            // At the dense rate the pair kernel's tiles of a table's layers fill its launch together: from a wave of small
            // tiles up a layer goes there (24 linears of dim 256, 13987 rows: 242 us with its layers on the few-rows kernel
            // because 55 row tiles do not fill 74 pairs, 180 like this; 96 of a Swin at batch 4, 319 and 258), below it
            // where the table's small layers add up (see elsa_vit_linears).
            *kind = pair_full || tiles_small >= sm_count ? KIND_DENSE_PAIR : KIND_SMALL_IMAGE;
        }
        return ELSA_OK;
    }
    if (tiles_small <= sm_count) {
        // One wave of 128 x 64 tiles: latency.
        if (use == USE_CHAIN) { *kind = KIND_SMALL_IMAGE; return ELSA_OK; }
        int ranges = 1;
        {
            SmallJob j;
            j.rows = rows; j.out = out; j.in = in;
            ranges = linear_small_splits(&j, 1, sm_count);
        }
        // Expanding in the kernel saves a launch, but every row tile repeats it and a CTA's loads wait for one another, from HBM
        // above all.  Us with the weight in L2 and from HBM, expanded and by an image: packed 1:4 and 2:4, 197 x 768 -> 768
        // 6.6 and 6.9 against 7.1 and 7.9, 197 x 1024 -> 1024 7.4 and 7.7 against 8.4 and 11.1 (49 x 768 -> 2304 the other way
        // round, 9.6 and 9.8 against 8.0 and 9.2); 4:8 7.8 and 8.8 against 7.2 and 8.0, 394 rows 10.4 and 11.5 against 7.4
        // and 8.0; 3:8 9.8 and 12.0 against 7.6 and 8.1; 8:16 12.9 and 15.1 against 9.1 and 9.7; the shared weight at 2:4
        // 7.3 and 7.3 against 7.2 and 7.5, at 4:8 8.7 and 8.7 against 7.3 and 7.7.
        if (use == USE_SINGLE && M == 4 && N <= 2 && ranges >= 2 && k_blocks <= 6 * ranges) *kind = KIND_SMALL;
        // A cut reduction pays from 16 K blocks up (4:4, 197 rows: 3072 -> 768 7.4 against 12.2, 768 -> 768 5.3 both).
        else *kind = ranges >= 2 && k_blocks >= 16 ? KIND_SMALL_IMAGE : KIND_DENSE_ONE;
        return ELSA_OK;
    }
    // More than a wave of small tiles.  Up to K = 512 the sparse kernels do not beat the pair kernel until the
    // weight-stationary one does, from about 1200 rows per SM pair (pair, best sparse: 512 -> 1536, 6304 rows 13.0, 14.4, 12608
    // rows 19.6, 19.8, 18912 rows 25.0, 24.5; 512 -> 2048, 3136 rows 10.7, 11.7, 12544 rows 23.4, 22.6; 512 -> 512, 6304 rows
    // 9.3, 8.6, 12608 rows 10.7, 11.7; 256 -> 1024, 18912 rows 15.0, 15.8, 25088 rows 19.3, 18.5); above, the sparse pair
    // kernel leads, and from about 5M outputs the streaming one (3072 -> 768: 6304 rows 24.5 against 25.0, 12608 rows 38.7
    // against 36.6).
    // With GELU the epilogue weighs more: the weight-stationary kernel leads where an SM pair's rows times K pass 390000
    // (768 -> 3072, 3152 rows 16.8 against 17.0 on the pair kernel, 4925 rows 20.9 against 24.3; 384 -> 1536, 12608 rows
    // 19.9 against 21.7), the pair kernel below; the streaming one is slower than either up to K = 1024.
    if (gelu) {
        const bool ws = ws_ok && (long long)rows * tiles_f * (in < 768 ? in : 768) >= 390000LL * pairs;
        *kind = ws ? KIND_SPARSE_WS : in > 1024 && st_ok && (long long)rows * out >= 5000000LL ? KIND_SPARSE_ST : KIND_DENSE_PAIR;
        return ELSA_OK;
    }
    // A call of its own has no image to wait for on the weight-stationary kernel, which leads from 240 rows per SM pair, 128 up to
    // K = 256 (a block is small), 640 above K = 768 (accumulators get narrow).  Us there and on the best other kernel, image
    // included, at 2:4: 768 -> 3072, 1576 rows (255 per pair) 11.8, 12.7, 4925 rows 17.1, 20.0; 768 -> 768, 3152 rows (128) 11.2,
    // 10.2, 6304 rows 12.1, 12.6; 768 -> 2304, 1576 rows (192) 13.2, 12.6, 3152 rows 13.6, 14.4; 512 -> 1536, 6304 rows 12.1,
    // 13.4; 384 -> 1152 at 2:16, 2000 rows (135) 9.5, 8.4; 384 -> 1536, 3152 rows 9.3, 9.9, 12608 rows 14.6, 18.1; 256 -> 1024, 3152
    // rows (170) 7.2, 8.4; 896 -> 896, 6304 rows (341) 15.1, 13.6, 12608 rows 19.0, 19.7; 1024 -> 4096, 1576 rows (341) 16.9, 14.3,
    // 6304 rows 30.5, 34.7.
    const int ws_rows = in <= 256 ? 128 : in <= 768 ? 240 : 640;
    if (use == USE_SINGLE && ws_ok && (long long)rows * tiles_f >= ws_rows * pairs) *kind = KIND_SPARSE_WS;
    else if (in <= 512) *kind = ws_ok && (long long)rows * tiles_f >= 1200 * pairs ? KIND_SPARSE_WS : KIND_DENSE_PAIR;
    else if (ws_large) *kind = KIND_SPARSE_WS;
    else if (sparse_ok && st_ok && (long long)rows * out >= 5000000LL) *kind = KIND_SPARSE_ST;
    else if (sparse_ok) *kind = KIND_SPARSE_PAIR;
    else *kind = KIND_DENSE_PAIR;
    return ELSA_OK;
}

SmallJob small_job(const void* X, int rows, const void* w, const uint32_t* idx, const void* bias, int out, int in, int N, int M,
                   void* Y, bool masked = false)
{
    SmallJob j;
    j.X = (const uint16_t*)X; j.w = (const uint16_t*)w; j.idx = idx; j.bias = (const uint16_t*)bias; j.Y = (uint16_t*)Y;
    j.rows = rows; j.in = in; j.out = out; j.N = N; j.M = M; j.masked = masked;
    return j;
}

// The few-rows kernel on a weight that lies dense in memory (the dense level, or a weight image).
SmallJob small_dense_job(const void* X, int rows, const void* Wd, const void* bias, int out, int in, void* Y)
{
    return small_job(X, rows, Wd, nullptr, bias, out, in, 4, 4, Y);
}

// After validation: enqueue one layer.  small_splits: how the few-rows kernel cuts the reduction (0: its own choice).
elsa_status run_linear(LinearKind kind, const void* X, int rows, const void* vals, const uint32_t* idx, const void* bias, int out,
                       int in, int N, int M, elsa_dtype dtype, void* Y, void* workspace, uint32_t* dev_status,
                       cudaStream_t stream, int small_splits = 0)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    if (kind == KIND_SIMT)
        return launch_linear_simt((const uint16_t*)X, rows, (const uint16_t*)vals, idx, (const uint16_t*)bias, out,
                                  in, N, M, dtype, (uint16_t*)Y, stream);
    if (kind == KIND_SMALL) {
        const SmallJob job = small_job(X, rows, vals, idx, bias, out, in, N, M, Y);
        if (small_splits == 0) small_splits = linear_small_splits(&job, 1, dev.sm_count);
        return launch_linear_small_group(&job, 1, small_splits, false, dtype, dev_status, stream);
    }
    if (kind == KIND_SPARSE_ONE)
        return launch_linear_tc_sparse((const uint16_t*)X, rows, (const uint16_t*)vals, idx, (const uint16_t*)bias, out,
                                       in, N, M, dtype, (uint16_t*)Y, workspace, dev_status, stream);
    if (kind == KIND_SPARSE_PAIR)
        return launch_linear_tc_sparse_pair((const uint16_t*)X, rows, (const uint16_t*)vals, idx, (const uint16_t*)bias,
                                            out, in, N, M, dtype, (uint16_t*)Y, workspace, dev_status, stream);
    if (kind == KIND_SPARSE_WS) {
        const SparseJob job = sparse_job(kind, X, rows, vals, idx, bias, out, in, N, M, Y, nullptr);
        return launch_linear_tc_sparse_ws_group(&job, 1, dtype, dev_status, stream);
    }
    if (kind == KIND_SPARSE_ST)
        return launch_linear_tc_sparse_st((const uint16_t*)X, rows, (const uint16_t*)vals, idx, (const uint16_t*)bias,
                                          out, in, N, M, dtype, (uint16_t*)Y, workspace, dev_status, stream);
    // Dense-rate path.  The dense level multiplies the stored values as they are; every other level first
    // rebuilds the weight image the MMA reads, in the caller's scratch.
    const uint16_t* Wd = (const uint16_t*)vals;
    if (N != M) {
        if ((st = launch_unpack((const uint16_t*)vals, idx, out, in, N, M, (uint16_t*)workspace, stream)) != ELSA_OK)
            return st;
        Wd = (const uint16_t*)workspace;
    }
    if (kind == KIND_DENSE_PAIR)
        return launch_linear_tc_pair((const uint16_t*)X, rows, Wd, (const uint16_t*)bias, out, in, dtype,
                                     (uint16_t*)Y, dev_status, stream);
    if (kind == KIND_SMALL_IMAGE) {
        SmallJob job = small_dense_job(X, rows, Wd, bias, out, in, Y);
        job.after_image = N != M;
        if (small_splits == 0) small_splits = linear_small_splits(&job, 1, dev.sm_count);
        return launch_linear_small_group(&job, 1, small_splits, false, dtype, dev_status, stream);
    }
    return launch_linear_tc_dense((const uint16_t*)X, rows, Wd, (const uint16_t*)bias, out, in, dtype,
                                  (uint16_t*)Y, dev_status, stream);
}

}  // namespace
}  // namespace elsa

using namespace elsa;

extern "C" {

size_t elsa_nm_values_bytes(int out, int in, int N, int M, elsa_dtype dtype)
{
    if (out <= 0 || in <= 0 || index_bits(M) < 0 || N < 1 || N > M || in % M != 0) return 0;
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return 0;
    return (size_t)out * values_per_row(in, N, M) * 2;
}

size_t elsa_nm_index_bytes(int out, int in, int N, int M)
{
    if (out <= 0 || in <= 0 || index_bits(M) < 0 || N < 1 || N > M || in % M != 0) return 0;
    return (size_t)out * index_words_per_row(in, N, M) * 4;
}

size_t elsa_workspace_bytes(int rows, int in, int out, int N, int M, elsa_dtype dtype)
{
    (void)rows;
    if (out <= 0 || in <= 0 || index_bits(M) < 0 || N < 1 || N > M || in % M != 0) return 0;
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return 0;
    if (N == M) return 0;                              // the dense level needs no weight image
    size_t need = round_up((size_t)out * (size_t)in * 2, 256);  // dense image of the masked weight
    if (linear_tc_sparse_suits(in, N)) {                          // or its 2-of-4 image + metadata
        const size_t sp = round_up(linear_tc_sparse_workspace(out, in), 256);
        if (sp > need) need = sp;
    }
    return need;
}

elsa_status elsa_nm_compress(const void* W, int out, int in, int N, int M, elsa_dtype dtype, void* vals,
                             uint32_t* idx, void* stream)
{
    if (!W || !vals) return fail(ELSA_ERR_NULL, "W and vals must not be NULL");
    elsa_status st = check_level(out, in, N, M, dtype);
    if (st != ELSA_OK) return st;
    if (N != M && !idx) return fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
    if (!aligned16(W) || !aligned16(vals) || (idx && !aligned16(idx)))
        return fail(ELSA_ERR_ALIGN, "W, vals and idx must be 16-byte aligned");
    DeviceInfo dev;
    if ((st = device_info(&dev)) != ELSA_OK) return st;
    return launch_compress((const uint16_t*)W, out, in, N, M, (uint16_t*)vals, N == M ? nullptr : idx,
                           (cudaStream_t)stream);
}

elsa_status elsa_nm_unpack(const void* vals, const uint32_t* idx, int out, int in, int N, int M, elsa_dtype dtype,
                           void* W_masked, void* stream)
{
    if (!vals || !W_masked) return fail(ELSA_ERR_NULL, "vals and W_masked must not be NULL");
    elsa_status st = check_level(out, in, N, M, dtype);
    if (st != ELSA_OK) return st;
    if (N != M && !idx) return fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
    if (!aligned16(vals) || !aligned16(W_masked) || (idx && !aligned16(idx)))
        return fail(ELSA_ERR_ALIGN, "vals, idx and W_masked must be 16-byte aligned");
    DeviceInfo dev;
    if ((st = device_info(&dev)) != ELSA_OK) return st;
    return launch_unpack((const uint16_t*)vals, N == M ? nullptr : idx, out, in, N, M, (uint16_t*)W_masked,
                         (cudaStream_t)stream);
}

elsa_status elsa_nm_linear(const void* X, int rows, const void* vals, const uint32_t* idx, const void* bias,
                           int out, int in, int N, int M, elsa_dtype dtype, void* Y, void* workspace,
                           size_t workspace_bytes, uint32_t* dev_status, void* stream)
{
    elsa_status st = check_linear(X, rows, vals, idx, bias, out, in, N, M, dtype, Y, workspace, workspace_bytes);
    if (st != ELSA_OK) return st;
    DeviceInfo dev;
    if ((st = device_info(&dev)) != ELSA_OK) return st;
    LinearKind kind;
    if ((st = pick_kind(USE_SINGLE, rows, out, in, N, M, dev.sm_count, &kind)) != ELSA_OK) return st;
    return run_linear(kind, X, rows, vals, N == M ? nullptr : idx, bias, out, in, N, M, dtype, Y, workspace, dev_status,
                      (cudaStream_t)stream);
}

elsa_status elsa_nm_compress_levels(const void* W, int out, int in, int M, const int* N_list, int n_levels,
                                    elsa_dtype dtype, void* const* vals, uint32_t* const* idx, void* stream)
{
    if (!W || !N_list || !vals || !idx) return fail(ELSA_ERR_NULL, "W, N_list, vals and idx must not be NULL");
    if (n_levels < 1 || n_levels > kMaxLevels)
        return fail(ELSA_ERR_SHAPE, "n_levels=%d is outside 1..%d", n_levels, kMaxLevels);
    if (!aligned16(W)) return fail(ELSA_ERR_ALIGN, "W must be 16-byte aligned");
    CompressJob jobs[kMaxLevels];
    for (int l = 0; l < n_levels; ++l) {
        elsa_status st = check_level(out, in, N_list[l], M, dtype);
        if (st == ELSA_OK && !vals[l]) st = fail(ELSA_ERR_NULL, "vals must not be NULL");
        if (st == ELSA_OK && N_list[l] != M && !idx[l]) st = fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
        if (st == ELSA_OK && (!aligned16(vals[l]) || (idx[l] && !aligned16(idx[l]))))
            st = fail(ELSA_ERR_ALIGN, "vals and idx must be 16-byte aligned");
        if (st != ELSA_OK) {
            char msg[400];
            snprintf(msg, sizeof msg, "%s", elsa_last_error());
            return fail(st, "level %d: %s", l, msg);
        }
        jobs[l] = {(const uint16_t*)W, (uint16_t*)vals[l], N_list[l] == M ? nullptr : idx[l], out, in, N_list[l], M};
    }
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    return launch_compress_jobs(jobs, n_levels, (cudaStream_t)stream);
}

elsa_status elsa_nm_linear_masked(const void* X, int rows, const void* W_sup, const void* bias, int out, int in,
                                  int N, int M, elsa_dtype dtype, void* Y, void* workspace, size_t workspace_bytes,
                                  uint32_t* dev_status, void* stream_)
{
    // the dense weight takes the place of vals in the checks (same alignment rules), no index words
    uint32_t* no_idx = N == M ? nullptr : (uint32_t*)W_sup;
    elsa_status st = check_linear(X, rows, W_sup, no_idx, bias, out, in, N, M, dtype, Y, workspace, workspace_bytes);
    if (st != ELSA_OK) return st;
    DeviceInfo dev;
    if ((st = device_info(&dev)) != ELSA_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    LinearKind kind;
    if ((st = pick_kind(USE_MASKED, rows, out, in, N, M, dev.sm_count, &kind)) != ELSA_OK) return st;
    if (kind == KIND_SIMT || kind == KIND_SPARSE_ONE)
        return fail(ELSA_ERR_NM, "the forced variant has no mask-on-load form");
    if (kind == KIND_SMALL) {
        const SmallJob job = small_job(X, rows, W_sup, nullptr, bias, out, in, N, M, Y, N != M);
        return launch_linear_small_group(&job, 1, linear_small_splits(&job, 1, dev.sm_count), false, dtype, dev_status, stream);
    }
    ImageJob image;
    image.src = (const uint16_t*)W_sup; image.dst = (uint16_t*)workspace; image.out = out; image.in = in; image.N = N; image.M = M;
    if (kind == KIND_SPARSE_PAIR || kind == KIND_SPARSE_WS || kind == KIND_SPARSE_ST) {
        image.kind = IMAGE_MASK_SP24;
        image.meta = (uint8_t*)workspace + sp24_meta_offset(out, in);
        image.layout = sp24_layout_of(kind);
        if ((st = launch_images(&image, 1, stream)) != ELSA_OK) return st;
        SparseJob job;
        job.X = (const uint16_t*)X; job.bias = (const uint16_t*)bias; job.Y = (uint16_t*)Y; job.workspace = workspace;
        job.rows = rows; job.in = in; job.out = out;
        return kind == KIND_SPARSE_WS   ? launch_linear_tc_sparse_ws_group(&job, 1, dtype, dev_status, stream)
               : kind == KIND_SPARSE_ST ? launch_linear_tc_sparse_st_group(&job, 1, dtype, dev_status, stream)
                                        : launch_linear_tc_sparse_pair_group(&job, 1, dtype, dev_status, stream);
    }
    const uint16_t* Wd = (const uint16_t*)W_sup;     // the dense level multiplies the shared weight as it is
    if (N != M) {
        image.kind = IMAGE_MASK;
        if ((st = launch_images(&image, 1, stream)) != ELSA_OK) return st;
        Wd = (const uint16_t*)workspace;
    }
    if (kind == KIND_DENSE_PAIR)
        return launch_linear_tc_pair((const uint16_t*)X, rows, Wd, (const uint16_t*)bias, out, in, dtype, (uint16_t*)Y,
                                     dev_status, stream);
    if (kind == KIND_SMALL_IMAGE) {
        SmallJob job = small_dense_job(X, rows, Wd, bias, out, in, Y);
        job.after_image = N != M;
        return launch_linear_small_group(&job, 1, linear_small_splits(&job, 1, dev.sm_count), false, dtype, dev_status, stream);
    }
    return launch_linear_tc_dense((const uint16_t*)X, rows, Wd, (const uint16_t*)bias, out, in, dtype, (uint16_t*)Y,
                                  dev_status, stream);
}

elsa_status elsa_vit_compress(const elsa_weight* w, int n_weights, elsa_dtype dtype, void* stream)
{
    if (!w) return fail(ELSA_ERR_NULL, "w must not be NULL");
    if (n_weights <= 0) return fail(ELSA_ERR_SHAPE, "non-positive n_weights=%d", n_weights);
    for (int i = 0; i < n_weights; ++i) {
        const elsa_weight& c = w[i];
        elsa_status st = ELSA_OK;
        if (!c.W || !c.vals) st = fail(ELSA_ERR_NULL, "W and vals must not be NULL");
        else if ((st = check_level(c.out, c.in, c.N, c.M, dtype)) != ELSA_OK) {}
        else if (c.N != c.M && !c.idx) st = fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
        else if (!aligned16(c.W) || !aligned16(c.vals) || (c.idx && !aligned16(c.idx)))
            st = fail(ELSA_ERR_ALIGN, "W, vals and idx must be 16-byte aligned");
        if (st != ELSA_OK) {
            char msg[400];
            snprintf(msg, sizeof msg, "%s", elsa_last_error());
            return fail(st, "weight %d: %s", i, msg);
        }
    }
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    std::vector<CompressJob> jobs(n_weights);
    for (int i = 0; i < n_weights; ++i) {
        const elsa_weight& c = w[i];
        jobs[i] = {(const uint16_t*)c.W, (uint16_t*)c.vals, c.N == c.M ? nullptr : c.idx, c.out, c.in, c.N, c.M};
    }
    return launch_compress_jobs(jobs.data(), n_weights, (cudaStream_t)stream);
}

size_t elsa_vit_workspace_bytes(const elsa_layer* cfg, int n_layers, elsa_dtype dtype)
{
    // one region per layer, so that every weight image can be built before the grouped launches
    size_t need = 0;
    if (!cfg) return 0;
    for (int l = 0; l < n_layers; ++l)
        need += round_up(elsa_workspace_bytes(cfg[l].rows, cfg[l].in, cfg[l].out, cfg[l].N, cfg[l].M, dtype), 256);
    return need;
}

elsa_status elsa_vit_linears(const elsa_layer* cfg, int n_layers, elsa_dtype dtype, void* workspace,
                             size_t workspace_bytes, uint32_t* dev_status, void* stream_)
{
    if (!cfg) return fail(ELSA_ERR_NULL, "cfg must not be NULL");
    if (n_layers <= 0) return fail(ELSA_ERR_SHAPE, "non-positive n_layers=%d", n_layers);
    for (int l = 0; l < n_layers; ++l) {
        const elsa_layer& c = cfg[l];
        elsa_status st = check_linear(c.X, c.rows, c.vals, c.idx, c.bias, c.out, c.in, c.N, c.M, dtype, c.Y,
                                      workspace, workspace_bytes);
        if (st != ELSA_OK) {
            char msg[400];
            snprintf(msg, sizeof msg, "%s", elsa_last_error());
            return fail(st, "layer %d: %s", l, msg);
        }
    }
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    auto layer_fail = [](elsa_status code, int l) {
        set_profile_layer(-1);
        char msg[400];
        snprintf(msg, sizeof msg, "%s", elsa_last_error());
        return fail(code, "layer %d: %s", l, msg);
    };

    // With one scratch region per layer (elsa_vit_workspace_bytes) all weight images are built first and the
    // layers of each kernel family share persistent launches: the layers of a table do not depend on one
    // another, so their tiles may interleave.  With less scratch (at least the largest layer's, which
    // validation has checked) the layers run one after the other through the same region.
    const bool grouped = g_grouping.load(std::memory_order_relaxed) &&
                         g_variant.load(std::memory_order_relaxed) == ELSA_VARIANT_AUTO &&
                         workspace_bytes >= elsa_vit_workspace_bytes(cfg, n_layers, dtype);
    std::vector<LinearKind> kind(n_layers);
    std::vector<SmallJob> small;
    long long small_tiles = 0;
    for (int l = 0; l < n_layers; ++l) {
        const elsa_layer& c = cfg[l];
        if ((st = pick_kind(USE_TABLE, c.rows, c.out, c.in, c.N, c.M, dev.sm_count, &kind[l])) != ELSA_OK) return layer_fail(st, l);
        if (kind[l] == KIND_SMALL_IMAGE) small_tiles += (long long)((c.rows + 127) / 128) * ((c.out + 63) / 64);
    }
    // Layers too small for the pair kernel by themselves go to it together from 4.5 waves of small tiles up, us on the
    // few-rows kernel and there: 48 layers of dim 192 at batch 1 (2.5 waves) 28, 30, at batch 4 59, 45; 16 layers of dim 256 at
    // batch 2 (3.4) 25, 28; 48 of dim 384 at batch 1 (5) 68, 62; 48 of dim 768 at batch 1 193, 183.
    const bool together = 2 * small_tiles >= 9LL * dev.sm_count;
    for (int l = 0; l < n_layers; ++l) {
        const elsa_layer& c = cfg[l];
        if (together && kind[l] == KIND_SMALL_IMAGE) kind[l] = KIND_DENSE_PAIR;
        if (kind[l] == KIND_SMALL_IMAGE || kind[l] == KIND_SMALL)
            small.push_back(small_dense_job(c.X, c.rows, c.vals, c.bias, c.out, c.in, c.Y));
    }
    // cut as they are in shared launches, so that results do not depend on the scratch given
    const int small_splits = small.empty() ? 0 : linear_small_splits(small.data(), (int)small.size(), dev.sm_count);
    if (!grouped) {
        for (int l = 0; l < n_layers; ++l) {
            const elsa_layer& c = cfg[l];
            set_profile_layer(l);
            st = run_linear(kind[l], c.X, c.rows, c.vals, c.N == c.M ? nullptr : c.idx, c.bias, c.out, c.in, c.N, c.M, dtype,
                            c.Y, workspace, dev_status, stream, small_splits);
            if (st != ELSA_OK) return layer_fail(st, l);
        }
        set_profile_layer(-1);
        return ELSA_OK;
    }

    // The weight images are built on a side stream while the dense layers, which need none, already run on
    // the caller's: the image kernel is a small streaming kernel whose blocks fit beside the persistent GEMM's
    // one CTA per SM.  Everything else waits for the images.
    SideStream side;
    std::vector<uint8_t*> region(n_layers);
    size_t off = 0, n_small = 0;
    for (int l = 0; l < n_layers; ++l) {
        const elsa_layer& c = cfg[l];
        region[l] = (uint8_t*)workspace + off;
        if (kind[l] == KIND_SMALL_IMAGE && c.N != c.M) small[n_small].w = (const uint16_t*)region[l];
        n_small += kind[l] == KIND_SMALL_IMAGE;
        off += round_up(elsa_workspace_bytes(c.rows, c.in, c.out, c.N, c.M, dtype), 256);
    }
    // dense-rate layers that multiply the stored values as they are (N = M), on CTA pairs, in groups: launched
    // first, the weight images are built beside them
    {
        std::vector<PairJob> jobs;
        for (int l = 0; l <= n_layers; ++l) {
            if (l < n_layers && kind[l] == KIND_DENSE_PAIR && cfg[l].N == cfg[l].M) {
                const elsa_layer& c = cfg[l];
                PairJob j;
                j.X = (const uint16_t*)c.X; j.bias = (const uint16_t*)c.bias; j.Y = (uint16_t*)c.Y;
                j.Wd = (const uint16_t*)c.vals;
                j.rows = c.rows; j.in = c.in; j.out = c.out;
                jobs.push_back(j);
            }
            if (!jobs.empty() && (l == n_layers || (int)jobs.size() == linear_tc_pair_group_max())) {
                // the side stream starts where the caller's stream stands now (after the compress kernels)
                if (!side.forked() && (st = side.fork(dev.device, stream)) != ELSA_OK) return st;
                if ((st = launch_linear_tc_pair_group(jobs.data(), (int)jobs.size(), dtype, dev_status, stream)) != ELSA_OK) {
                    side.join(stream);
                    return st;
                }
                jobs.clear();
            }
        }
    }
    cudaStream_t image_stream = side.forked() ? side.stream() : stream;
    // weight images of all layers, one launch per 256 layers
    {
        std::vector<ImageJob> jobs;
        for (int l = 0; l < n_layers; ++l) {
            const elsa_layer& c = cfg[l];
            if (c.N != c.M && reads_image(kind[l]))
                jobs.push_back(image_job(kind[l], c.vals, c.idx, c.out, c.in, c.N, c.M, region[l]));
        }
        if (!jobs.empty()) st = launch_images(jobs.data(), (int)jobs.size(), image_stream);
    }
    {
        const elsa_status joined = side.join(stream);
        if (st != ELSA_OK) return st;
        if (joined != ELSA_OK) return joined;
    }
    // sparse-rate layers, in groups
    {
        std::vector<SparseJob> jobs;
        for (int l = 0; l <= n_layers; ++l) {
            if (l < n_layers && kind[l] == KIND_SPARSE_PAIR) {
                const elsa_layer& c = cfg[l];
                jobs.push_back(sparse_job(kind[l], c.X, c.rows, c.vals, c.idx, c.bias, c.out, c.in, c.N, c.M, c.Y, region[l]));
            }
            if (!jobs.empty() && (l == n_layers || (int)jobs.size() == linear_tc_sparse_pair_group_max())) {
                if ((st = launch_linear_tc_sparse_pair_group(jobs.data(), (int)jobs.size(), dtype, dev_status, stream)) != ELSA_OK)
                    return st;
                jobs.clear();
            }
        }
    }
    // sparse-rate layers whose weight block streams through tensor memory, in groups
    {
        std::vector<SparseJob> jobs;
        for (int l = 0; l <= n_layers; ++l) {
            if (l < n_layers && kind[l] == KIND_SPARSE_ST) {
                const elsa_layer& c = cfg[l];
                jobs.push_back(sparse_job(kind[l], c.X, c.rows, c.vals, c.idx, c.bias, c.out, c.in, c.N, c.M, c.Y, region[l]));
            }
            if (!jobs.empty() && (l == n_layers || (int)jobs.size() == linear_tc_sparse_st_group_max())) {
                if ((st = launch_linear_tc_sparse_st_group(jobs.data(), (int)jobs.size(), dtype, dev_status, stream)) != ELSA_OK)
                    return st;
                jobs.clear();
            }
        }
    }
    // sparse-rate layers whose weight block fits tensor memory, in groups
    {
        std::vector<SparseJob> jobs;
        for (int l = 0; l <= n_layers; ++l) {
            if (l < n_layers && kind[l] == KIND_SPARSE_WS) {
                const elsa_layer& c = cfg[l];
                jobs.push_back(sparse_job(kind[l], c.X, c.rows, c.vals, c.idx, c.bias, c.out, c.in, c.N, c.M, c.Y, region[l]));
            }
            if (!jobs.empty() && (l == n_layers || (int)jobs.size() == linear_tc_sparse_ws_group_max())) {
                if ((st = launch_linear_tc_sparse_ws_group(jobs.data(), (int)jobs.size(), dtype, dev_status, stream)) != ELSA_OK)
                    return st;
                jobs.clear();
            }
        }
    }
    // dense-rate layers that read a weight image (N < M), on CTA pairs, in groups
    {
        std::vector<PairJob> jobs;
        for (int l = 0; l <= n_layers; ++l) {
            if (l < n_layers && kind[l] == KIND_DENSE_PAIR && cfg[l].N != cfg[l].M) {
                const elsa_layer& c = cfg[l];
                PairJob j;
                j.X = (const uint16_t*)c.X; j.bias = (const uint16_t*)c.bias; j.Y = (uint16_t*)c.Y;
                j.Wd = c.N == c.M ? (const uint16_t*)c.vals : (const uint16_t*)region[l];
                j.rows = c.rows; j.in = c.in; j.out = c.out;
                jobs.push_back(j);
            }
            if (!jobs.empty() && (l == n_layers || (int)jobs.size() == linear_tc_pair_group_max())) {
                if ((st = launch_linear_tc_pair_group(jobs.data(), (int)jobs.size(), dtype, dev_status, stream)) != ELSA_OK)
                    return st;
                jobs.clear();
            }
        }
    }
    // layers with few rows, in groups
    for (size_t at = 0; at < small.size(); at += (size_t)linear_small_group_max()) {
        const int n = (int)(small.size() - at) < linear_small_group_max() ? (int)(small.size() - at) : linear_small_group_max();
        if ((st = launch_linear_small_group(small.data() + at, n, small_splits, false, dtype, dev_status, stream)) != ELSA_OK) return st;
    }
    return ELSA_OK;
}

// Device memory plan of the host-memory variant: two slots, used by alternate layers so that the
// copies of one layer overlap the kernels of its neighbours; each slot holds regions sized for the
// largest layer: X | Y | W | bias | vals | idx | linear workspace.
namespace {
struct HostPlan {
    size_t x, y, w, bias, vals, idx, ws, slot, total;
};

// Copy streams and ordering events of the host-memory variant, created once per device.
struct HostPipe {
    cudaStream_t in, out;
    cudaEvent_t start, in_done[2], compute_done[2], out_done[2];
    bool ready;
};
HostPipe g_pipe[64];
std::mutex g_pipe_mutex;

elsa_status host_pipe(int device, HostPipe** pipe)
{
    std::lock_guard<std::mutex> lock(g_pipe_mutex);
    HostPipe& p = g_pipe[device & 63];
    if (!p.ready) {
        bool ok = cudaStreamCreateWithFlags(&p.in, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&p.out, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaEventCreateWithFlags(&p.start, cudaEventDisableTiming) == cudaSuccess;
        for (int i = 0; ok && i < 2; ++i)
            ok = cudaEventCreateWithFlags(&p.in_done[i], cudaEventDisableTiming) == cudaSuccess &&
                 cudaEventCreateWithFlags(&p.compute_done[i], cudaEventDisableTiming) == cudaSuccess &&
                 cudaEventCreateWithFlags(&p.out_done[i], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) {
            cudaError_t e = cudaGetLastError();
            return fail(ELSA_ERR_CUDA, "creating the copy streams: %s", cudaGetErrorString(e));
        }
        p.ready = true;
    }
    *pipe = &p;
    return ELSA_OK;
}
bool host_plan(const elsa_host_layer* cfg, int n_layers, elsa_dtype dtype, HostPlan* plan)
{
    size_t mx = 0, my = 0, mw = 0, mb = 0, mv = 0, mi = 0, ms = 0;
    for (int l = 0; l < n_layers; ++l) {
        const elsa_host_layer& c = cfg[l];
        if (c.rows <= 0 || c.in <= 0 || c.out <= 0) return false;
        auto up = [](size_t& m, size_t v) { if (v > m) m = v; };
        up(mx, (size_t)c.rows * c.in * 2);
        up(my, (size_t)c.rows * c.out * 2);
        up(mw, (size_t)c.out * c.in * 2);
        up(mb, (size_t)c.out * 2);
        up(mv, elsa_nm_values_bytes(c.out, c.in, c.N, c.M, dtype));
        up(mi, elsa_nm_index_bytes(c.out, c.in, c.N, c.M));
        up(ms, elsa_workspace_bytes(c.rows, c.in, c.out, c.N, c.M, dtype));
    }
    size_t off = 0;
    plan->x = off; off += round_up(mx, 256);
    plan->y = off; off += round_up(my, 256);
    plan->w = off; off += round_up(mw, 256);
    plan->bias = off; off += round_up(mb, 256);
    plan->vals = off; off += round_up(mv, 256);
    plan->idx = off; off += round_up(mi, 256);
    plan->ws = off; off += round_up(ms, 256);
    plan->slot = off;
    plan->total = 2 * off;
    return true;
}
}  // namespace

size_t elsa_vit_host_device_bytes(const elsa_host_layer* cfg, int n_layers, elsa_dtype dtype)
{
    HostPlan plan;
    if (!cfg || n_layers <= 0 || !host_plan(cfg, n_layers, dtype, &plan)) return 0;
    return plan.total;
}

elsa_status elsa_vit_linears_host(const elsa_host_layer* cfg, int n_layers, elsa_dtype dtype, void* device_mem,
                                  size_t device_bytes, uint32_t* dev_status, void* stream_)
{
    if (!cfg) return fail(ELSA_ERR_NULL, "cfg must not be NULL");
    if (n_layers <= 0) return fail(ELSA_ERR_SHAPE, "non-positive n_layers=%d", n_layers);
    HostPlan plan;
    if (!host_plan(cfg, n_layers, dtype, &plan)) return fail(ELSA_ERR_SHAPE, "a layer has a non-positive dimension");
    for (int l = 0; l < n_layers; ++l) {
        const elsa_host_layer& c = cfg[l];
        if (!c.X || !c.Y || !c.W) return fail(ELSA_ERR_NULL, "layer %d: X, Y and W must not be NULL", l);
        elsa_status st = check_level(c.out, c.in, c.N, c.M, dtype);
        if (st != ELSA_OK) {
            char msg[400];
            snprintf(msg, sizeof msg, "%s", elsa_last_error());
            return fail(st, "layer %d: %s", l, msg);
        }
    }
    if (!device_mem || device_bytes < plan.total)
        return fail(ELSA_ERR_WORKSPACE, "device memory of %zu bytes needed, %zu given", plan.total,
                    device_mem ? device_bytes : (size_t)0);
    if (((uintptr_t)device_mem & 255u) != 0) return fail(ELSA_ERR_ALIGN, "device_mem must be 256-byte aligned");
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;

    cudaStream_t stream = (cudaStream_t)stream_;
    HostPipe* pipe = nullptr;
    if ((st = host_pipe(dev.device, &pipe)) != ELSA_OK) return st;
    // Three queues: host-to-device copies, kernels (the caller's stream), device-to-host copies.  Layer l
    // uses slot l % 2; events order a slot's copy-in after the kernels that last read it, its kernels after
    // its copy-in and after the copy-out that last read its Y, and its copy-out after its kernels.
    auto cuda_fail = [](cudaError_t e, int l, const char* what) {
        cudaGetLastError();
        set_profile_layer(-1);
        return fail(ELSA_ERR_CUDA, "layer %d: %s: %s", l, what, cudaGetErrorString(e));
    };
    cudaError_t e = cudaEventRecord(pipe->start, stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe->in, pipe->start, 0);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe->out, pipe->start, 0);
    if (e != cudaSuccess) return cuda_fail(e, 0, "ordering the copy streams");
    for (int l = 0; l < n_layers; ++l) {
        const elsa_host_layer& c = cfg[l];
        const int slot = l & 1;
        uint8_t* base = (uint8_t*)device_mem + (size_t)slot * plan.slot;
        set_profile_layer(l);
        void* dX = base + plan.x; void* dY = base + plan.y; void* dW = base + plan.w;
        void* dB = c.bias ? base + plan.bias : nullptr;
        void* dV = base + plan.vals; uint32_t* dI = c.N == c.M ? nullptr : (uint32_t*)(base + plan.idx);
        // copy-in
        e = cudaSuccess;
        if (l >= 2) e = cudaStreamWaitEvent(pipe->in, pipe->compute_done[slot], 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dW, c.W, (size_t)c.out * c.in * 2, cudaMemcpyHostToDevice, pipe->in);
        if (e == cudaSuccess && c.bias) e = cudaMemcpyAsync(dB, c.bias, (size_t)c.out * 2, cudaMemcpyHostToDevice, pipe->in);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dX, c.X, (size_t)c.rows * c.in * 2, cudaMemcpyHostToDevice, pipe->in);
        if (e == cudaSuccess) e = cudaEventRecord(pipe->in_done[slot], pipe->in);
        if (e != cudaSuccess) return cuda_fail(e, l, "host-to-device copy");
        // kernels
        e = cudaStreamWaitEvent(stream, pipe->in_done[slot], 0);
        if (e == cudaSuccess && l >= 2) e = cudaStreamWaitEvent(stream, pipe->out_done[slot], 0);
        if (e != cudaSuccess) return cuda_fail(e, l, "ordering the kernels");
        if ((st = launch_compress((const uint16_t*)dW, c.out, c.in, c.N, c.M, (uint16_t*)dV, dI, stream)) != ELSA_OK) return st;
        LinearKind kind;
        if ((st = pick_kind(USE_SINGLE, c.rows, c.out, c.in, c.N, c.M, dev.sm_count, &kind)) != ELSA_OK) return st;
        if ((st = run_linear(kind, dX, c.rows, dV, dI, dB, c.out, c.in, c.N, c.M, dtype, dY, base + plan.ws, dev_status,
                             stream)) != ELSA_OK)
            return st;
        e = cudaEventRecord(pipe->compute_done[slot], stream);
        // copy-out
        if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe->out, pipe->compute_done[slot], 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(c.Y, dY, (size_t)c.rows * c.out * 2, cudaMemcpyDeviceToHost, pipe->out);
        if (e == cudaSuccess) e = cudaEventRecord(pipe->out_done[slot], pipe->out);
        if (e != cudaSuccess) return cuda_fail(e, l, "device-to-host copy");
    }
    set_profile_layer(-1);
    // the caller's stream is complete only when the last copies out are
    e = cudaStreamWaitEvent(stream, pipe->out_done[(n_layers - 1) & 1], 0);
    if (e == cudaSuccess && n_layers >= 2) e = cudaStreamWaitEvent(stream, pipe->out_done[n_layers & 1], 0);
    if (e != cudaSuccess) return cuda_fail(e, n_layers - 1, "joining the copy streams");
    return ELSA_OK;
}

}  // extern "C"

/* ---------------------------------------------------------------------------------------------- */
/* The chained block                                                                              */
/* ---------------------------------------------------------------------------------------------- */
namespace elsa {
namespace {

struct BlockLinear {
    const elsa_block_linear* w;
    int in, out;
    LinearKind kind;
    void* ws;          // this linear's part of region WORKSPACE
    bool image_ready;  // its weight image has been enqueued already
    bool first;        // no kernel of the same call runs before it
    const BlockLinear* next;   // the linear that runs after it in the same call, or NULL
};

struct BlockPlan {
    size_t off[ELSA_BLOCK_REGIONS];
    size_t ws_off[4];   // qkv, proj, fc1, fc2 inside region WORKSPACE
    size_t total;
};

bool block_plan(int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype, BlockPlan* p)
{
    if (!w || rows <= 0 || dim <= 0 || mlp_dim <= 0 || dim % 8 != 0 || mlp_dim % 8 != 0) return false;
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return false;
    const size_t row = (size_t)rows * 2;
    const size_t sizes[7] = {row * dim, row * dim * 3, row * dim, row * dim, row * dim, row * mlp_dim, row * dim};
    size_t at = 0;
    for (int r = 0; r < 7; ++r) {
        p->off[r] = at;
        at += round_up(sizes[r], 256);
    }
    p->off[ELSA_BLOCK_WORKSPACE] = at;
    const elsa_block_linear* lin[4] = {&w->qkv, &w->proj, &w->fc1, &w->fc2};
    const int ins[4] = {dim, dim, dim, mlp_dim}, outs[4] = {3 * dim, dim, mlp_dim, dim};
    for (int l = 0; l < 4; ++l) {
        if (index_bits(lin[l]->M) < 0 || lin[l]->N < 1 || lin[l]->N > lin[l]->M || ins[l] % lin[l]->M != 0) return false;
        p->ws_off[l] = at;
        at += round_up(elsa_workspace_bytes(rows, ins[l], outs[l], lin[l]->N, lin[l]->M, dtype), 256);
    }
    p->total = at;
    return true;
}

// Validation shared by the entry points; fills the four linears' descriptions.  images: where their weight images go
// when not in region WORKSPACE of the scratch.
elsa_status block_check(const void* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype,
                        const void* y, bool need_y, void* scratch, size_t scratch_bytes, BlockPlan* plan,
                        BlockLinear (&lin)[4], const DeviceInfo& dev, uint8_t* images = nullptr)
{
    if (!x || !w || !scratch || (need_y && !y)) return fail(ELSA_ERR_NULL, "x, w, y and scratch must not be NULL");
    if (rows <= 0 || dim <= 0 || mlp_dim <= 0) return fail(ELSA_ERR_SHAPE, "non-positive size (rows=%d, dim=%d, mlp_dim=%d)", rows, dim, mlp_dim);
    if (!w->ln1_gain || !w->ln1_bias || !w->ln2_gain || !w->ln2_bias)
        return fail(ELSA_ERR_NULL, "the LayerNorm gains and biases must not be NULL");
    if (!(w->eps >= 0.f)) return fail(ELSA_ERR_SHAPE, "eps must not be negative");
    const elsa_block_linear* src[4] = {&w->qkv, &w->proj, &w->fc1, &w->fc2};
    const char* names[4] = {"qkv", "proj", "fc1", "fc2"};
    const int ins[4] = {dim, dim, dim, mlp_dim}, outs[4] = {3 * dim, dim, mlp_dim, dim};
    for (int l = 0; l < 4; ++l) {
        elsa_status st = check_level(outs[l], ins[l], src[l]->N, src[l]->M, dtype);
        if (st == ELSA_OK && !src[l]->vals) st = fail(ELSA_ERR_NULL, "vals must not be NULL");
        if (st == ELSA_OK && src[l]->N != src[l]->M && !src[l]->idx) st = fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
        if (st == ELSA_OK && (!aligned16(src[l]->vals) || (src[l]->idx && !aligned16(src[l]->idx)) ||
                              (src[l]->bias && !aligned16(src[l]->bias))))
            st = fail(ELSA_ERR_ALIGN, "vals, idx and bias must be 16-byte aligned");
        if (st != ELSA_OK) {
            char msg[400];
            snprintf(msg, sizeof msg, "%s", elsa_last_error());
            return fail(st, "%s: %s", names[l], msg);
        }
    }
    if (!aligned16(x) || (y && !aligned16(y)) || !aligned16(w->ln1_gain) || !aligned16(w->ln1_bias) ||
        !aligned16(w->ln2_gain) || !aligned16(w->ln2_bias))
        return fail(ELSA_ERR_ALIGN, "x, y and the LayerNorm parameters must be 16-byte aligned");
    if (y && y == x) return fail(ELSA_ERR_ALIGN, "y may not alias x");
    if (!block_plan(rows, dim, mlp_dim, w, dtype, plan)) return fail(ELSA_ERR_SHAPE, "dim and mlp_dim must be multiples of 8");
    if (((uintptr_t)scratch & 255u) != 0) return fail(ELSA_ERR_ALIGN, "scratch must be 256-byte aligned");
    if (scratch_bytes < plan->total)
        return fail(ELSA_ERR_WORKSPACE, "scratch of %zu bytes needed, %zu given", plan->total, scratch_bytes);
    for (int l = 0; l < 4; ++l) {
        lin[l].w = src[l];
        lin[l].in = ins[l];
        lin[l].out = outs[l];
        lin[l].ws = images ? images + (plan->ws_off[l] - plan->off[ELSA_BLOCK_WORKSPACE]) : (uint8_t*)scratch + plan->ws_off[l];
        lin[l].image_ready = false;
        lin[l].first = false;
        lin[l].next = l < 3 ? &lin[l + 1] : nullptr;
        elsa_status st = pick_kind(USE_CHAIN, rows, outs[l], ins[l], src[l]->N, src[l]->M, dev.sm_count, &lin[l].kind, l == 2);
        if (st != ELSA_OK) return st;
    }
    return ELSA_OK;
}

// Whether a linear's kernel takes a ready-made weight image (the others build theirs when they run, or need none).
bool takes_image(const BlockLinear& L)
{
    return L.w->N != L.w->M && (L.kind == KIND_DENSE_PAIR || L.kind == KIND_SMALL_IMAGE || L.kind == KIND_SPARSE_PAIR || L.kind == KIND_SPARSE_ST);
}

// Adds the images that n linears take to `jobs`.
void add_images(const BlockLinear* lin, int n, std::vector<ImageJob>* jobs)
{
    for (int l = 0; l < n; ++l)
        if (takes_image(lin[l]) && !lin[l].image_ready)
            jobs->push_back(image_job(lin[l].kind, lin[l].w->vals, lin[l].w->idx, lin[l].out, lin[l].in, lin[l].w->N, lin[l].w->M, lin[l].ws));
}

// The images of n linears that take one, in one launch.
elsa_status block_images(BlockLinear* lin, int n, cudaStream_t stream)
{
    std::vector<ImageJob> jobs;
    add_images(lin, n, &jobs);
    if (jobs.empty()) return ELSA_OK;
    const elsa_status st = launch_images(jobs.data(), (int)jobs.size(), stream);
    if (st == ELSA_OK)
        for (int l = 0; l < n; ++l) lin[l].image_ready = takes_image(lin[l]);
    return st;
}

// Y = act(X Wm^T + bias) [+ residual].  Returns in *residual_left whether the residual is still to be added:
// then the linear's output went to `tmp` instead of Y, rounded to 16 bits.
elsa_status block_linear(BlockLinear& L, const uint16_t* X, int rows, elsa_dtype dtype, uint16_t* Y, int act,
                         const uint16_t* residual, uint16_t* tmp, bool* residual_left, uint32_t* dev_status,
                         cudaStream_t stream)
{
    const elsa_block_linear& w = *L.w;
    elsa_status st = ELSA_OK;
    *residual_left = false;
    if (L.kind == KIND_DENSE_PAIR) {
        if ((st = block_images(&L, 1, stream)) != ELSA_OK) return st;
        PairJob job;
        job.X = X; job.Wd = w.N == w.M ? (const uint16_t*)w.vals : (const uint16_t*)L.ws;
        job.bias = (const uint16_t*)w.bias; job.Y = Y;
        job.rows = rows; job.in = L.in; job.out = L.out;
        job.act = act; job.residual = residual;
        return launch_linear_tc_pair_group(&job, 1, dtype, dev_status, stream);
    }
    if (L.kind == KIND_SMALL || L.kind == KIND_SMALL_IMAGE) {
        const bool ready = L.image_ready;       // enqueued before an earlier kernel of this call, which waited for it
        if ((st = block_images(&L, 1, stream)) != ELSA_OK) return st;
        SmallJob job = L.kind == KIND_SMALL ? small_job(X, rows, w.vals, w.N == w.M ? nullptr : w.idx, w.bias, L.out, L.in, w.N, w.M, Y)
                                            : small_dense_job(X, rows, w.N == w.M ? w.vals : L.ws, w.bias, L.out, L.in, Y);
        job.act = act; job.residual = residual; job.chained = true;
        if (L.next != nullptr && L.next->kind == KIND_SMALL_IMAGE) {
            const elsa_block_linear& n = *L.next->w;
            job.ahead = n.N == n.M ? n.vals : L.next->ws;
            job.ahead_bytes = (size_t)L.next->out * L.next->in * 2;
        }
        DeviceInfo dev;
        if ((st = device_info(&dev)) != ELSA_OK) return st;
        // after another kernel of the same call the weights are older than that kernel's start (KIND_SMALL: only where the
        // variant is forced, a chain picks KIND_SMALL_IMAGE)
        const bool early = !L.first && (L.kind == KIND_SMALL || w.N == w.M || ready);
        return launch_linear_small_group(&job, 1, linear_small_splits(&job, 1, dev.sm_count), early, dtype, dev_status, stream);
    }
    // GELU and a residual never come together; where they did, or the kernel has no residual, the next row-wise kernel adds it
    const bool adds = residual != nullptr && act == 0 && (L.kind == KIND_SPARSE_WS || L.kind == KIND_SPARSE_ST);
    *residual_left = residual != nullptr && !adds;
    uint16_t* dst = *residual_left ? tmp : Y;
    if (L.kind == KIND_SPARSE_WS || L.kind == KIND_SPARSE_ST || (L.kind == KIND_SPARSE_PAIR && act == 0)) {
        if ((st = block_images(&L, 1, stream)) != ELSA_OK) return st;
        SparseJob job = sparse_job(L.kind, X, rows, w.vals, w.idx, w.bias, L.out, L.in, w.N, w.M, dst, L.ws);
        job.act = act;
        if (adds) job.residual = residual;
        return L.kind == KIND_SPARSE_WS   ? launch_linear_tc_sparse_ws_group(&job, 1, dtype, dev_status, stream)
               : L.kind == KIND_SPARSE_ST ? launch_linear_tc_sparse_st_group(&job, 1, dtype, dev_status, stream)
                                          : launch_linear_tc_sparse_pair_group(&job, 1, dtype, dev_status, stream);
    }
    st = run_linear(L.kind, X, rows, w.vals, w.N == w.M ? nullptr : w.idx, w.bias, L.out, L.in, w.N, w.M, dtype, dst, L.ws,
                    dev_status, stream);
    if (st != ELSA_OK) return st;
    return launch_act_inplace(dst, (long long)rows * L.out, act, dtype, stream);
}

// What a block leaves to its successor when the residual of its last linear has not been added yet: the block's
// output is t + r, and the successor's first LayerNorm adds, stores and normalises it in one pass.
struct BlockCarry {
    const uint16_t* t = nullptr;   // fc2's output, rounded to 16 bits
    const uint16_t* r = nullptr;   // x2
};

// carry (or NULL) + x_sum: the block's input is carry->t + carry->r, written to x_sum; otherwise it is x.
elsa_status block_qkv(const uint16_t* x, int rows, int dim, const elsa_block_weights* w, elsa_dtype dtype,
                      uint8_t* scratch, const BlockPlan& plan, BlockLinear (&lin)[4], uint32_t* dev_status,
                      cudaStream_t stream, const BlockCarry* carry = nullptr, uint16_t* x_sum = nullptr,
                      const elsa_swin_attn* swin = nullptr)
{
    uint16_t* x1 = (uint16_t*)(scratch + plan.off[ELSA_BLOCK_X1]);
    uint16_t* qkv = (uint16_t*)(scratch + plan.off[ELSA_BLOCK_QKV]);
    const bool add = carry != nullptr && carry->t != nullptr;
    RowMap out_map = {0, 0, 0, 0, 0, 1};      // Swin: x1 is written in window order, so that windows are runs of rows
    if (swin) { out_map.H = swin->H; out_map.W = swin->W; out_map.ws = swin->window; out_map.shift = swin->shift; }
    elsa_status st = launch_layer_norm(add ? carry->t : x, add ? carry->r : nullptr, add ? x_sum : nullptr,
                                       (const uint16_t*)w->ln1_gain, (const uint16_t*)w->ln1_bias,
                                       x1, rows, dim, w->eps, dtype, stream, swin ? &out_map : nullptr);
    if (st != ELSA_OK) return st;
    bool left = false;
    return block_linear(lin[0], x1, rows, dtype, qkv, 0, nullptr, nullptr, &left, dev_status, stream);
}

elsa_status block_rest(const uint16_t* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype,
                       uint16_t* y, uint8_t* scratch, const BlockPlan& plan, BlockLinear (&lin)[4],
                       uint32_t* dev_status, cudaStream_t stream, BlockCarry* defer = nullptr,
                       const elsa_swin_attn* swin = nullptr)
{
    (void)mlp_dim;
    const uint16_t* a = (const uint16_t*)(scratch + plan.off[ELSA_BLOCK_A]);
    uint16_t* x2 = (uint16_t*)(scratch + plan.off[ELSA_BLOCK_X2]);
    uint16_t* x3 = (uint16_t*)(scratch + plan.off[ELSA_BLOCK_X3]);
    uint16_t* h = (uint16_t*)(scratch + plan.off[ELSA_BLOCK_H]);
    uint16_t* t = (uint16_t*)(scratch + plan.off[ELSA_BLOCK_T]);
    const uint16_t* g2 = (const uint16_t*)w->ln2_gain;
    const uint16_t* b2 = (const uint16_t*)w->ln2_bias;
    bool left = false;
    elsa_status st;
    if (swin) {
        // proj runs on rows in window order; the add that follows reads them back in the grid's order
        RowMap in_map = {swin->H, swin->W, swin->window, swin->shift, 1, 0};
        if ((st = block_linear(lin[1], a, rows, dtype, t, 0, nullptr, nullptr, &left, dev_status, stream)) != ELSA_OK) return st;
        st = launch_layer_norm(t, x, x2, g2, b2, x3, rows, dim, w->eps, dtype, stream, &in_map);
    } else {
        if ((st = block_linear(lin[1], a, rows, dtype, x2, 0, x, t, &left, dev_status, stream)) != ELSA_OK) return st;
        // x2 = x + proj(a) and x3 = LayerNorm2(x2): one pass where the residual is still to be added
        st = left ? launch_layer_norm(t, x, x2, g2, b2, x3, rows, dim, w->eps, dtype, stream)
                  : launch_layer_norm(x2, nullptr, nullptr, g2, b2, x3, rows, dim, w->eps, dtype, stream);
    }
    if (st != ELSA_OK) return st;
    if ((st = block_linear(lin[2], x3, rows, dtype, h, 1, nullptr, nullptr, &left, dev_status, stream)) != ELSA_OK) return st;
    if ((st = block_linear(lin[3], h, rows, dtype, y, 0, x2, t, &left, dev_status, stream)) != ELSA_OK) return st;
    if (left && defer != nullptr) {          // the successor's first LayerNorm adds the residual
        defer->t = t;
        defer->r = x2;
        return ELSA_OK;
    }
    if (left) st = launch_layer_norm(t, x2, y, nullptr, nullptr, nullptr, rows, dim, w->eps, dtype, stream);
    return st;
}

}  // namespace
}  // namespace elsa

extern "C" {

size_t elsa_vit_block_scratch_bytes(int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype,
                                    size_t* offsets)
{
    BlockPlan plan;
    if (!block_plan(rows, dim, mlp_dim, w, dtype, &plan)) return 0;
    if (offsets)
        for (int r = 0; r < ELSA_BLOCK_REGIONS; ++r) offsets[r] = plan.off[r];
    return plan.total;
}

elsa_status elsa_vit_block_qkv(const void* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w,
                               elsa_dtype dtype, void* scratch, size_t scratch_bytes, uint32_t* dev_status, void* stream)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    BlockPlan plan;
    BlockLinear lin[4];
    if ((st = block_check(x, rows, dim, mlp_dim, w, dtype, nullptr, false, scratch, scratch_bytes, &plan, lin, dev)) != ELSA_OK)
        return st;
    return block_qkv((const uint16_t*)x, rows, dim, w, dtype, (uint8_t*)scratch, plan, lin, dev_status, (cudaStream_t)stream);
}

elsa_status elsa_vit_block_rest(const void* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w,
                                elsa_dtype dtype, void* y, void* scratch, size_t scratch_bytes, uint32_t* dev_status,
                                void* stream)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    BlockPlan plan;
    BlockLinear lin[4];
    if ((st = block_check(x, rows, dim, mlp_dim, w, dtype, y, true, scratch, scratch_bytes, &plan, lin, dev)) != ELSA_OK)
        return st;
    lin[1].first = true;
    return block_rest((const uint16_t*)x, rows, dim, mlp_dim, w, dtype, (uint16_t*)y, (uint8_t*)scratch, plan, lin,
                      dev_status, (cudaStream_t)stream);
}

}  // extern "C"

namespace elsa {
namespace {

struct PreparedBlock {
    BlockPlan plan;
    BlockLinear lin[4];
};

// A validated block's kernels; tokens == 0 runs the stand-in a = V, otherwise the attention kernel over images of
// `tokens` rows.  The block's images have been enqueued already, or are built where they are used.
elsa_status run_prepared(const void* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype,
                         void* y, void* scratch, PreparedBlock& block, uint32_t* dev_status, cudaStream_t stream,
                         int tokens, int heads, const BlockCarry* carry = nullptr, uint16_t* x_sum = nullptr,
                         BlockCarry* defer = nullptr, const elsa_swin_attn* swin = nullptr)
{
    const BlockPlan& plan = block.plan;
    BlockLinear (&lin)[4] = block.lin;
    elsa_status st;
    uint8_t* s8 = (uint8_t*)scratch;
    if ((st = block_qkv((const uint16_t*)x, rows, dim, w, dtype, s8, plan, lin, dev_status, stream, carry, x_sum, swin)) != ELSA_OK)
        return st;
    if (carry != nullptr && carry->t != nullptr) x = x_sum;      // the block's input, as just stored
    if (swin) {
        const int pack = swin->pack < 1 ? 1 : swin->pack;
        const int T = swin->window * swin->window * pack;
        st = launch_attention((const uint16_t*)(s8 + plan.off[ELSA_BLOCK_QKV]), rows / T, T, heads, dim, dtype,
                              (uint16_t*)(s8 + plan.off[ELSA_BLOCK_A]), dev_status, stream, swin->rel_bias,
                              swin->shift > 0 ? swin->mask : nullptr, (swin->H / swin->window) * (swin->W / swin->window) / pack,
                              swin->bias_pitch);
    } else if (tokens == 0) {
        // the stated stand-in for attention: a = V
        st = launch_copy_columns((const uint16_t*)(s8 + plan.off[ELSA_BLOCK_QKV]), (uint16_t*)(s8 + plan.off[ELSA_BLOCK_A]),
                                 rows, 3 * dim, 2 * dim, dim, stream);
    } else {
        st = launch_attention((const uint16_t*)(s8 + plan.off[ELSA_BLOCK_QKV]), rows / tokens, tokens, heads, dim, dtype,
                              (uint16_t*)(s8 + plan.off[ELSA_BLOCK_A]), dev_status, stream);
    }
    if (st != ELSA_OK) return st;
    return block_rest((const uint16_t*)x, rows, dim, mlp_dim, w, dtype, (uint16_t*)y, s8, plan, lin, dev_status, stream, defer, swin);
}

// One block on its own.  Its images are one launch ahead of the first LayerNorm: a fork to a side stream and back costs
// about 7 us in events and lost launch overlap, the launch 3 to 6.
elsa_status run_block(const void* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype,
                      void* y, void* scratch, size_t scratch_bytes, uint32_t* dev_status, void* stream_, int tokens, int heads,
                      const elsa_swin_attn* swin = nullptr)
{
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    PreparedBlock block;
    if ((st = block_check(x, rows, dim, mlp_dim, w, dtype, y, true, scratch, scratch_bytes, &block.plan, block.lin, dev)) != ELSA_OK)
        return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    if ((st = block_images(block.lin, 4, stream)) != ELSA_OK) return st;
    return run_prepared(x, rows, dim, mlp_dim, w, dtype, y, scratch, block, dev_status, stream, tokens, heads, nullptr, nullptr,
                        nullptr, swin);
}

struct EncoderPlan {
    size_t block_bytes;   // scratch of the largest block
    size_t buf[2];        // byte offsets of the two activation buffers the blocks alternate between
    size_t images;        // the weight images of every block, behind what the chain cannot do without
    size_t total;
};

bool encoder_plan(int rows, int dim, int mlp_dim, const elsa_block_weights* blocks, int n_blocks, elsa_dtype dtype, EncoderPlan* p)
{
    if (!blocks || n_blocks <= 0) return false;
    p->block_bytes = 0;
    size_t image_bytes = 0;
    for (int b = 0; b < n_blocks; ++b) {
        BlockPlan plan;
        if (!block_plan(rows, dim, mlp_dim, blocks + b, dtype, &plan)) return false;
        if (plan.total > p->block_bytes) p->block_bytes = plan.total;
        image_bytes += plan.total - plan.off[ELSA_BLOCK_WORKSPACE];
    }
    size_t at = round_up(p->block_bytes, 256);
    for (int i = 0; i < 2; ++i) {
        p->buf[i] = at;
        at += round_up((size_t)rows * dim * 2, 256);
    }
    p->images = at;
    at += image_bytes;
    p->total = at;
    return true;
}

}  // namespace
}  // namespace elsa

extern "C" {

size_t elsa_vit_encoder_scratch_bytes(int images, int tokens, int dim, int mlp_dim, const elsa_block_weights* blocks,
                                      int n_blocks, elsa_dtype dtype)
{
    EncoderPlan p;
    if (images <= 0 || tokens <= 0 || (long long)images * tokens > 0x7fffffffLL) return 0;
    return encoder_plan(images * tokens, dim, mlp_dim, blocks, n_blocks, dtype, &p) ? p.total : 0;
}

elsa_status elsa_vit_encoder(const void* x, int images, int tokens, int heads, int dim, int mlp_dim,
                             const elsa_block_weights* blocks, int n_blocks, const void* final_gain, const void* final_bias,
                             float final_eps, elsa_dtype dtype, void* y, void* scratch, size_t scratch_bytes,
                             uint32_t* dev_status, void* stream)
{
    if (!x || !y || !blocks || !scratch) return fail(ELSA_ERR_NULL, "x, y, blocks and scratch must not be NULL");
    if (images <= 0 || tokens <= 0 || n_blocks <= 0)
        return fail(ELSA_ERR_SHAPE, "non-positive images=%d, tokens=%d or n_blocks=%d", images, tokens, n_blocks);
    if (!attention_suits(tokens, heads, dim))
        return fail(ELSA_ERR_SHAPE, "attention needs at most 256 tokens per image and dim = 64 * heads (tokens=%d, heads=%d, dim=%d)",
                    tokens, heads, dim);
    if ((long long)images * tokens > 0x7fffffffLL) return fail(ELSA_ERR_SHAPE, "images * tokens does not fit an int");
    if ((final_gain == nullptr) != (final_bias == nullptr)) return fail(ELSA_ERR_NULL, "final_gain and final_bias go together");
    if (final_gain && (!aligned16(final_gain) || !aligned16(final_bias)))
        return fail(ELSA_ERR_ALIGN, "final_gain and final_bias must be 16-byte aligned");
    if (final_gain && !(final_eps >= 0.f)) return fail(ELSA_ERR_SHAPE, "final_eps must not be negative");
    const int rows = images * tokens;
    EncoderPlan plan;
    if (!encoder_plan(rows, dim, mlp_dim, blocks, n_blocks, dtype, &plan))
        return fail(ELSA_ERR_SHAPE, "dim and mlp_dim must be multiples of 8 and every level valid");
    if (((uintptr_t)scratch & 255u) != 0) return fail(ELSA_ERR_ALIGN, "scratch must be 256-byte aligned");
    // With less than the whole the images of a block go to its own scratch, built before it runs: same results.
    if (scratch_bytes < plan.images) return fail(ELSA_ERR_WORKSPACE, "scratch of %zu bytes needed, %zu given", plan.images, scratch_bytes);
    const bool ahead = scratch_bytes >= plan.total;
    DeviceInfo dev;
    elsa_status st = device_info(&dev);
    if (st != ELSA_OK) return st;
    uint8_t* s8 = (uint8_t*)scratch;
    uint16_t* buf[2] = {(uint16_t*)(s8 + plan.buf[0]), (uint16_t*)(s8 + plan.buf[1])};
    // every block is validated before the first launch
    std::vector<PreparedBlock> prepared(n_blocks);
    std::vector<ImageJob> image_jobs;
    uint8_t* image_at = ahead ? s8 + plan.images : nullptr;
    for (int b = 0; b < n_blocks; ++b) {
        PreparedBlock& p = prepared[b];
        if ((st = block_check(x, rows, dim, mlp_dim, blocks + b, dtype, buf[0], true, scratch, plan.block_bytes, &p.plan, p.lin, dev,
                              image_at)) != ELSA_OK) {
            char msg[400];
            snprintf(msg, sizeof msg, "%s", elsa_last_error());
            return fail(st, "block %d: %s", b, msg);
        }
        if (!ahead) continue;
        image_at += p.plan.total - p.plan.off[ELSA_BLOCK_WORKSPACE];
        add_images(p.lin, 4, &image_jobs);
        for (int l = 0; l < 4; ++l) p.lin[l].image_ready = takes_image(p.lin[l]);
    }
    // The weight images of all blocks in one launch ahead of the chain (170 MB for a dense DeiT-B: 25 us once, against
    // about 7 us a block for building them beside the block before on a side stream).
    if (!image_jobs.empty() && (st = launch_images(image_jobs.data(), (int)image_jobs.size(), (cudaStream_t)stream)) != ELSA_OK) return st;
    // Block b reads its input from buf[b % 2] (block 0: from x) and writes its output to buf[(b + 1) % 2]; where a
    // block's last residual is still to be added, the next block's first LayerNorm does it while it normalises.
    BlockCarry carry;
    const void* in = x;
    for (int b = 0; b + 1 < n_blocks; ++b) prepared[b].lin[3].next = &prepared[b + 1].lin[0];
    for (int b = 0; b < n_blocks; ++b) {
        const bool last = b + 1 == n_blocks;
        void* out = (last && final_gain == nullptr) ? y : (void*)buf[(b + 1) & 1];
        BlockCarry next;
        if (!ahead && (st = block_images(prepared[b].lin, 4, (cudaStream_t)stream)) != ELSA_OK) return st;
        st = run_prepared(in, rows, dim, mlp_dim, blocks + b, dtype, out, scratch, prepared[b], dev_status, (cudaStream_t)stream,
                          tokens, heads, &carry, buf[b & 1], last && final_gain == nullptr ? nullptr : &next);
        if (st != ELSA_OK) return st;
        carry = next;
        in = buf[(b + 1) & 1];
    }
    if (final_gain != nullptr) {
        const bool add = carry.t != nullptr;
        st = launch_layer_norm(add ? carry.t : buf[n_blocks & 1], add ? carry.r : nullptr, add ? buf[n_blocks & 1] : nullptr,
                               (const uint16_t*)final_gain, (const uint16_t*)final_bias, (uint16_t*)y, rows, dim, final_eps, dtype,
                               (cudaStream_t)stream);
    }
    return st;
}

elsa_status elsa_vit_block(const void* x, int rows, int dim, int mlp_dim, const elsa_block_weights* w, elsa_dtype dtype,
                           void* y, void* scratch, size_t scratch_bytes, uint32_t* dev_status, void* stream)
{
    return run_block(x, rows, dim, mlp_dim, w, dtype, y, scratch, scratch_bytes, dev_status, stream, 0, 0);
}

elsa_status elsa_attention(const void* qkv, int images, int tokens, int heads, int dim, elsa_dtype dtype, void* a,
                           uint32_t* dev_status, void* stream)
{
    if (!qkv || !a) return fail(ELSA_ERR_NULL, "qkv and a must not be NULL");
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return fail(ELSA_ERR_DTYPE, "dtype %d is neither ELSA_F16 nor ELSA_BF16", (int)dtype);
    if (images <= 0) return fail(ELSA_ERR_SHAPE, "non-positive images=%d", images);
    if (!aligned16(qkv) || !aligned16(a)) return fail(ELSA_ERR_ALIGN, "qkv and a must be 16-byte aligned");
    return launch_attention((const uint16_t*)qkv, images, tokens, heads, dim, dtype, (uint16_t*)a, dev_status, (cudaStream_t)stream);
}

int elsa_swin_mask(int H, int W, int window, int shift, int pack, int pitch, float* mask)
{
    if (H <= 0 || W <= 0 || window <= 0 || H % window != 0 || W % window != 0 || shift <= 0 || shift >= window || pack < 1 ||
        pitch < pack * window * window || !mask)
        return -1;
    const int T = window * window, nww = W / window, n_windows = (H / window) * nww;
    if (n_windows % pack != 0) return -1;
    // region of a position of the rolled grid: the bands [0, n - window), [n - window, n - shift), [n - shift, n) of each axis
    auto band = [&](int v, int n) { return v < n - window ? 0 : v < n - shift ? 1 : 2; };
    auto region = [&](int win, int t) {
        const int wi = win / nww, wj = win % nww;
        return 3 * band(wi * window + t / window, H) + band(wj * window + t % window, W);
    };
    for (int g = 0; g < n_windows / pack; ++g) {
        float* m = mask + (size_t)g * pack * T * pitch;
        for (int p = 0; p < pack * T; ++p)
            for (int q = 0; q < pitch; ++q) {
                float v = 0.f;
                // tokens of different windows of a group are kept apart by the bias table; here: the seam inside a window
                if (q < pack * T && p / T == q / T) v = region(g * pack + p / T, p % T) != region(g * pack + q / T, q % T) ? -100.f : 0.f;
                m[(size_t)p * pitch + q] = v;
            }
    }
    return n_windows / pack;
}

int elsa_swin_pack_bias(const float* rel_bias, int heads, int window, int pack, int pitch, float* packed)
{
    if (!rel_bias || !packed || heads <= 0 || window <= 0 || pack < 1 || pitch < pack * window * window) return -1;
    const int T = window * window;
    for (int h = 0; h < heads; ++h)
        for (int p = 0; p < pack * T; ++p)
            for (int q = 0; q < pitch; ++q) {
                float v = 0.f;
                if (q < pack * T) v = p / T == q / T ? rel_bias[((size_t)h * T + p % T) * T + q % T] : -30000.f;
                packed[((size_t)h * pack * T + p) * pitch + q] = v;
            }
    return 0;
}

elsa_status elsa_swin_block(const void* x, int images, int heads, int dim, int mlp_dim, const elsa_block_weights* w,
                            const elsa_swin_attn* attn, elsa_dtype dtype, void* y, void* scratch, size_t scratch_bytes,
                            uint32_t* dev_status, void* stream)
{
    if (!attn) return fail(ELSA_ERR_NULL, "attn must not be NULL");
    if (images <= 0 || attn->H <= 0 || attn->W <= 0 || attn->window <= 0 || attn->H % attn->window != 0 ||
        attn->W % attn->window != 0 || attn->shift < 0 || attn->shift >= attn->window)
        return fail(ELSA_ERR_SHAPE, "windows of %d do not tile a %d x %d grid, or shift=%d is outside [0, window)", attn->window,
                    attn->H, attn->W, attn->shift);
    const int pack = attn->pack < 1 ? 1 : attn->pack;
    const int T = attn->window * attn->window * pack;         // tokens of one attention item: `pack` windows
    if (!attention_suits(T, heads, dim))
        return fail(ELSA_ERR_SHAPE, "window attention needs at most 256 tokens per group of windows and dim = 32 or 64 times heads "
                    "(window=%d, pack=%d, heads=%d, dim=%d)", attn->window, pack, heads, dim);
    if (((long long)images * (attn->H / attn->window) * (attn->W / attn->window)) % pack != 0)
        return fail(ELSA_ERR_SHAPE, "the windows do not divide into groups of %d", pack);
    if (attn->shift > 0 && ((attn->H / attn->window) * (attn->W / attn->window)) % pack != 0)
        return fail(ELSA_ERR_SHAPE, "with a shift the windows of one image must divide into groups of %d", pack);
    if (!attn->rel_bias || (attn->shift > 0 && !attn->mask)) return fail(ELSA_ERR_NULL, "rel_bias (and mask when shift > 0) must not be NULL");
    if (attn->bias_pitch < T) return fail(ELSA_ERR_SHAPE, "bias_pitch=%d is below the %d tokens of a window", attn->bias_pitch, T);
    if ((long long)images * attn->H * attn->W > 0x7fffffffLL) return fail(ELSA_ERR_SHAPE, "images * H * W does not fit an int");
    return run_block(x, images * attn->H * attn->W, dim, mlp_dim, w, dtype, y, scratch, scratch_bytes, dev_status, stream, T, heads,
                     attn);
}

elsa_status elsa_window_attention(const void* qkv, int windows, int tokens, int heads, int dim, const float* bias,
                                  int bias_pitch, const float* mask, int n_masks, elsa_dtype dtype, void* a,
                                  uint32_t* dev_status, void* stream)
{
    if (!qkv || !a || !bias) return fail(ELSA_ERR_NULL, "qkv, a and bias must not be NULL");
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return fail(ELSA_ERR_DTYPE, "dtype %d is neither ELSA_F16 nor ELSA_BF16", (int)dtype);
    if (windows <= 0) return fail(ELSA_ERR_SHAPE, "non-positive windows=%d", windows);
    if (!aligned16(qkv) || !aligned16(a) || ((uintptr_t)bias & 3u) || ((uintptr_t)mask & 3u))
        return fail(ELSA_ERR_ALIGN, "qkv and a must be 16-byte aligned, the tables 4-byte aligned");
    return launch_attention((const uint16_t*)qkv, windows, tokens, heads, dim, dtype, (uint16_t*)a, dev_status, (cudaStream_t)stream,
                            bias, mask, n_masks, bias_pitch);
}

elsa_status elsa_vit_block_attn(const void* x, int images, int tokens, int heads, int dim, int mlp_dim,
                                const elsa_block_weights* w, elsa_dtype dtype, void* y, void* scratch, size_t scratch_bytes,
                                uint32_t* dev_status, void* stream)
{
    if (images <= 0 || tokens <= 0) return fail(ELSA_ERR_SHAPE, "non-positive images=%d or tokens=%d", images, tokens);
    if (!attention_suits(tokens, heads, dim))
        return fail(ELSA_ERR_SHAPE, "attention needs at most 256 tokens per image and dim = 64 * heads (tokens=%d, heads=%d, dim=%d)",
                    tokens, heads, dim);
    if ((long long)images * tokens > 0x7fffffffLL) return fail(ELSA_ERR_SHAPE, "images * tokens does not fit an int");
    return run_block(x, images * tokens, dim, mlp_dim, w, dtype, y, scratch, scratch_bytes, dev_status, stream, tokens, heads);
}

}  // extern "C"

/* ---------------------------------------------------------------------------------------------- */
/* Backward pass                                                                                  */
/* ---------------------------------------------------------------------------------------------- */
namespace elsa {
namespace {

struct BackwardPlan {
    size_t wmt, partial, sums, total;   // byte offsets of the regions
    int parts;                          // rows of `out` floats in `partial`
};

// Upper bound, from host arithmetic alone, of the ranges the dW product may be cut into: what a device of 256 SMs
// would use.  The call clamps its choice to it.
int wgrad_splits_bound(int in, int out)
{
    const long long tiles = (long long)((out + 255) / 256) * ((in + 255) / 256);
    long long s = 128 / tiles;
    if (s > 8) s = 8;
    return s < 1 ? 1 : (int)s;
}

BackwardPlan backward_plan(int rows, int in, int out)
{
    BackwardPlan p;
    size_t at = 0;
    p.wmt = at;     at += round_up((size_t)out * in * 2, 256);                      // transposed masked weight [in][out]
    const int bound = wgrad_splits_bound(in, out);
    int parts = (rows + 511) / 512;                                                 // parts of the column sums of dY:
    const int product = bound > 1 ? bound * ((in + 255) / 256) : 0;                 // 512 rows each, or from dW's product
    if (parts < (in + 127) / 128) parts = (in + 127) / 128;
    if (parts < product) parts = product;
    p.parts = parts;
    p.partial = at; at += round_up((size_t)parts * out * 4, 256);
    // fp32 sums of dW per range of rows
    p.sums = at;    at += bound > 1 ? round_up((size_t)bound * out * in * 4, 256) : 0;
    p.total = at;
    return p;
}

// Y [m][n] = A [m][k] . B [n][k]^T on the dense tensor-core kernels (no bias).
elsa_status dense_product(const uint16_t* A, int m, const uint16_t* B, int n, int k, elsa_dtype dtype, uint16_t* Y,
                          uint32_t* dev_status, cudaStream_t stream, int sm_count)
{
    const int variant = g_variant.load(std::memory_order_relaxed);
    SmallJob job = small_dense_job(A, m, B, nullptr, n, k, Y);
    job.after_image = true;      // B is what a transpose has just written
    LinearKind kind;       // the dense level's rule
    const elsa_status st = pick_kind(USE_SINGLE, m, n, k, 4, 4, sm_count, &kind);
    if (st != ELSA_OK || variant == ELSA_VARIANT_TC_DENSE || kind == KIND_DENSE_ONE)
        return launch_linear_tc_dense(A, m, B, nullptr, n, k, dtype, Y, dev_status, stream);
    if (kind == KIND_SMALL || kind == KIND_SMALL_IMAGE)
        return launch_linear_small_group(&job, 1, linear_small_splits(&job, 1, sm_count), false, dtype, dev_status, stream);
    return launch_linear_tc_pair(A, m, B, nullptr, n, k, dtype, Y, dev_status, stream);
}

}  // namespace
}  // namespace elsa

extern "C" {

size_t elsa_backward_workspace_bytes(int rows, int in, int out, int N, int M, elsa_dtype dtype)
{
    if (rows <= 0 || out <= 0 || in <= 0 || index_bits(M) < 0 || N < 1 || N > M || in % M != 0) return 0;
    if (dtype != ELSA_F16 && dtype != ELSA_BF16) return 0;
    return backward_plan(rows, in, out).total;
}

elsa_status elsa_nm_linear_backward(const void* dY, const void* X, int rows, const void* vals, const uint32_t* idx,
                                    int out, int in, int N, int M, elsa_dtype dtype, void* dX, void* dW, void* db,
                                    void* workspace, size_t workspace_bytes, uint32_t* dev_status, void* stream_)
{
    if (!dY) return fail(ELSA_ERR_NULL, "dY must not be NULL");
    elsa_status st = check_level(out, in, N, M, dtype);
    if (st != ELSA_OK) return st;
    if (rows <= 0) return fail(ELSA_ERR_SHAPE, "non-positive rows=%d", rows);
    if (dX && !vals) return fail(ELSA_ERR_NULL, "vals must not be NULL when dX is wanted");
    if (dW && !X) return fail(ELSA_ERR_NULL, "X must not be NULL when dW is wanted");
    if ((dX || dW) && N != M && !idx) return fail(ELSA_ERR_NULL, "idx must not be NULL when N < M");
    if (!aligned16(dY) || (X && !aligned16(X)) || (vals && !aligned16(vals)) || (idx && !aligned16(idx)) ||
        (dX && !aligned16(dX)) || (dW && !aligned16(dW)) || (db && !aligned16(db)))
        return fail(ELSA_ERR_ALIGN, "dY, X, vals, idx, dX, dW and db must be 16-byte aligned");
    const BackwardPlan plan = backward_plan(rows, in, out);
    if (!workspace || workspace_bytes < plan.total)
        return fail(ELSA_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", plan.total, workspace ? workspace_bytes : (size_t)0);
    if (((uintptr_t)workspace & 255u) != 0) return fail(ELSA_ERR_ALIGN, "workspace must be 256-byte aligned");
    DeviceInfo dev;
    if ((st = device_info(&dev)) != ELSA_OK) return st;
    cudaStream_t stream = (cudaStream_t)stream_;
    uint8_t* ws = (uint8_t*)workspace;
    const uint16_t* dy = (const uint16_t*)dY;
    if (dX) {
        // dX = dY Wm: the forward GEMM with the transposed masked weight, reduction over `out`
        uint16_t* wmt = (uint16_t*)(ws + plan.wmt);
        if ((st = launch_transpose_packed((const uint16_t*)vals, idx, wmt, out, in, N, M, stream)) != ELSA_OK) return st;
        if ((st = dense_product(dy, rows, wmt, in, out, dtype, (uint16_t*)dX, dev_status, stream, dev.sm_count)) != ELSA_OK) return st;
    }
    float* db_sums = (float*)(ws + plan.partial);
    int db_parts = 0;
    if (dW) {
        // dW = dY^T X, reduction over the token rows: both operands are read as they are stored (reduction index
        // outermost), then the mask
        // when tiles alone leave SM pairs idle, the rows are cut into ranges summed afterwards
        const TnShape shape = linear_tc_pair_tn_shape(out, in, rows, wgrad_splits_bound(in, out), db ? plan.parts : 0, dev.sm_count);
        float* sums = (float*)(ws + plan.sums);
        // (the sums of dY find room: plan.parts covers 256 columns in every number of ranges, and the shape's choice minds it at 128)
        if ((st = launch_linear_tc_pair_tn(dy, (const uint16_t*)X, out, in, rows, dtype, (uint16_t*)dW, shape, sums,
                                           db ? db_sums : nullptr, &db_parts, dev_status, stream)) != ELSA_OK)
            return st;
        if (shape.splits > 1) {
            st = launch_wgrad_finish(sums, shape.splits, idx, out, in, N, M, dtype, (uint16_t*)dW, db_sums, db_parts, (uint16_t*)db, stream);
            if (st != ELSA_OK || db_parts > 0) return st;
        } else if ((st = launch_mask_apply((uint16_t*)dW, idx, out, in, N, M, stream)) != ELSA_OK) {
            return st;
        }
    }
    if (!db) return ELSA_OK;
    return db_parts > 0 ? launch_colsum_finish(db_sums, db_parts, out, (uint16_t*)db, dtype, stream)
                        : launch_colsum(dy, rows, out, db_sums, (uint16_t*)db, dtype, stream);
}

}  // extern "C"

extern "C" {

elsa_status elsa_set_linear_variant(elsa_variant v)
{
    if (v != ELSA_VARIANT_AUTO && v != ELSA_VARIANT_SIMT && v != ELSA_VARIANT_TC_DENSE && v != ELSA_VARIANT_TC_PAIR &&
        v != ELSA_VARIANT_TC_SPARSE && v != ELSA_VARIANT_TC_SPARSE_PAIR && v != ELSA_VARIANT_TC_SPARSE_WS &&
        v != ELSA_VARIANT_TC_SPARSE_ST && v != ELSA_VARIANT_TC_SMALL)
        return fail(ELSA_ERR_SHAPE, "unknown variant %d", (int)v);
    g_variant.store((int)v, std::memory_order_relaxed);
    return ELSA_OK;
}

void elsa_set_grouping(int on) { g_grouping.store(on != 0, std::memory_order_relaxed); }

elsa_variant elsa_get_linear_variant(void) { return (elsa_variant)g_variant.load(std::memory_order_relaxed); }

elsa_status elsa_profile_start(void)
{
    std::lock_guard<std::mutex> lock(g_profile_mutex);
    for (auto& r : g_profile) { cudaEventDestroy(r.start); cudaEventDestroy(r.stop); }
    g_profile.clear();
    g_profile_on.store(true, std::memory_order_relaxed);
    return ELSA_OK;
}

int elsa_profile_stop(elsa_kernel_time* records, int capacity)
{
    g_profile_on.store(false, std::memory_order_relaxed);
    std::lock_guard<std::mutex> lock(g_profile_mutex);
    const int n = (int)g_profile.size();
    for (int i = 0; i < n; ++i) {
        ProfileRecord& r = g_profile[i];
        float ms = -1.f;
        if (cudaEventSynchronize(r.stop) != cudaSuccess || cudaEventElapsedTime(&ms, r.start, r.stop) != cudaSuccess) {
            cudaGetLastError();
            ms = -1.f;
        }
        if (records && i < capacity) {
            records[i].kernel = r.kernel;
            records[i].layer = r.layer;
            records[i].ms = ms;
        }
        cudaEventDestroy(r.start);
        cudaEventDestroy(r.stop);
    }
    g_profile.clear();
    return n;
}

unsigned long long elsa_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char* elsa_last_error(void) { return g_error; }

}  // extern "C"
