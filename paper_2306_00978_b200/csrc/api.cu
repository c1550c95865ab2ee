// C ABI of the library: argument checks, dispatch, workspace and status bookkeeping.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include <cuda.h>

#include "common.cuh"

namespace awq {

namespace {

constexpr int kMaxDevices = 64;
std::atomic<unsigned long long> g_launches{0};
thread_local char t_cuda_error[256] = "";

// A stream, and the capture that it is in (0: none).  A handle that comes back after cudaStreamDestroy is no harm: the new stream's
// first launch waits once for nothing.  (cudaStreamGetId would tell them apart, but it invalidates a capture.)
struct StreamKey {
    unsigned long long stream, capture;
    bool operator==(const StreamKey& o) const { return stream == o.stream && capture == o.capture; }
};
// Streams on which one of this library's kernels that write packed arrays or 1 / s (quantizer, 3-bit packing and expansion) has been
// enqueued and no layer call since.  Most layer kernels copy weights before the launch in front of them has completed, so the
// first one behind such a writer on the same stream is launched fully serialized; what runs on other streams changes nothing.
// Between streams an event waits for the writer's end - but not inside a capture: there a launch joined behind a writer by an event gets
// a programmatic edge to it like one on its own stream (read from captured graphs), at any time up to the capture's end and also where a
// call on the writer's stream has waited.  So a capture's entries stay, `taken` by their own stream's reader, and calls on the
// capture's other streams are serialized.
struct PendingWriters {
    static constexpr int kMost = 64;
    struct Entry { StreamKey key; unsigned long long serial; bool taken; };
    Entry list[kMost];
    int count = 0;
    unsigned long long serial = 0;         // of the last writer
    unsigned long long forgotten = 0;      // the largest of the captures whose entries made room for others: up to it every captured launch is serialized
    bool overflow = false;                 // more streams than fit: every launch is serialized until the device has been waited for

    void add(const StreamKey& key) {
        const Entry entry = {key, ++serial, false};
        int room = -1;
        for (int i = 0; i < count; ++i) {
            // a stream is in one capture at a time: a writer in an earlier one can have no reader any more
            if (list[i].key.stream == key.stream && (list[i].key.capture != 0) == (key.capture != 0)) { list[i] = entry; return; }
            if (list[i].taken && (room < 0 || list[i].serial < list[room].serial)) room = i;
        }
        if (count < kMost) {
            list[count++] = entry;
        } else if (room >= 0) {
            if (list[room].key.capture > forgotten) forgotten = list[room].key.capture;
            list[room] = entry;
        } else {
            overflow = true;
        }
    }
    unsigned long long pending(const StreamKey& key) const {         // the writer's serial, 0: none
        for (int i = 0; i < count; ++i) if (list[i].key == key && !list[i].taken) return list[i].serial;
        return 0;
    }
    bool elsewhere_in_capture(const StreamKey& key) const {
        if (key.capture == 0) return false;
        for (int i = 0; i < count; ++i) if (list[i].key.capture == key.capture && list[i].key.stream != key.stream) return true;
        return key.capture <= forgotten;
    }
    void remove(const StreamKey& key, unsigned long long upto) {
        for (int i = 0; i < count; ++i)
            if (list[i].key == key && list[i].serial <= upto) {
                if (key.capture != 0) list[i].taken = true; else list[i] = list[--count];
                return;
            }
    }
    void completed(unsigned long long upto) {                        // all work enqueued before this serial's writer, and it, has ended
        for (int i = 0; i < count;) if (list[i].key.capture == 0 && list[i].serial <= upto) list[i] = list[--count]; else ++i;
        if (upto == serial) overflow = false;
    }
};

struct DeviceState {
    void* workspace = nullptr;
    size_t workspace_bytes = 0;
    unsigned int* status_word = nullptr;   // device address of g_status on this device
    int cc_major = -1;
    int sms = 0;
    int tx_surplus_once = 0;               // time-out test: see awq_test_stall_next_gemv
    PendingWriters writers;
};
DeviceState g_dev[kMaxDevices];
std::mutex g_mutex;                        // DeviceState's fields

// [0]: 0, or a code written by a kernel that gave up a wait; [1]: limit of a device-side wait in
// microseconds (0 = the built-in default)
__device__ unsigned int g_status[2];

int note_cuda(cudaError_t e) {
    if (e == cudaSuccess) return AWQ_OK;
    std::snprintf(t_cuda_error, sizeof(t_cuda_error), "%s: %s", cudaGetErrorName(e), cudaGetErrorString(e));
    return AWQ_ERR_CUDA;
}

// A thread that has not used the GPU has no context until the runtime makes one current, which a kernel launch does; tensor maps are
// encoded by the driver in front of it, and that fails without one.
int bind_context(int dev) {
    typedef CUresult (*GetCurrentFn)(CUcontext*);
    static const GetCurrentFn get_current = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuCtxGetCurrent", &p, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<GetCurrentFn>(p);
    }();
    CUcontext current = nullptr;
    if (!get_current || (get_current(&current) == CUDA_SUCCESS && current)) return AWQ_OK;
    return note_cuda(cudaSetDevice(dev));
}

// Per-device set-up on first use: compute capability and the status word's device address.
int device_state(DeviceState** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return note_cuda(e);
    if (dev < 0 || dev >= kMaxDevices) return AWQ_ERR_WRONG_DEVICE;
    if (int rc = bind_context(dev)) return rc;
    std::lock_guard<std::mutex> lock(g_mutex);
    DeviceState& d = g_dev[dev];
    if (d.cc_major < 0) {
        int major = 0;
        e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (e != cudaSuccess) return note_cuda(e);
        if (major == 10) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_status);
            if (e != cudaSuccess) return note_cuda(e);
            e = cudaMemset(p, 0, 2 * sizeof(unsigned int));
            if (e != cudaSuccess) return note_cuda(e);
            d.status_word = reinterpret_cast<unsigned int*>(p);
        }
        e = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return note_cuda(e);
        d.cc_major = major;
    }
    if (d.cc_major != 10) return AWQ_ERR_WRONG_DEVICE;
    *out = &d;
    return AWQ_OK;
}

thread_local char t_per_thread_stream;     // its address stands for the calling thread's cudaStreamPerThread

StreamKey stream_key(cudaStream_t st) {
    StreamKey key = {(unsigned long long)(uintptr_t)st, 0};
    if (st == cudaStreamLegacy) key.stream = 0;
    if (st == cudaStreamPerThread) key.stream = (unsigned long long)(uintptr_t)&t_per_thread_stream;
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) (void)cudaGetLastError();
    else if (status != cudaStreamCaptureStatusNone) key.capture = id;
    return key;
}

// Called after a writer of packed arrays has been enqueued.  (Not before: another thread's layer call on the same stream could take
// the entry and be enqueued in front of the writer.)
void note_packed_writer(DeviceState* d, void* stream) {
    const StreamKey key = stream_key((cudaStream_t)stream);
    std::lock_guard<std::mutex> lock(g_mutex);
    d->writers.add(key);
}

// How a layer's launch is ordered behind the work in front of it.
struct LaunchOrder {
    DeviceState* d;
    StreamKey key;
    unsigned long long writer;             // serial of the writer that it waits for, 0: none is known
    bool serialize;
    // the kernel is in the stream: the launches behind it need not wait for that writer any more
    cudaError_t launched(cudaError_t e) const {
        if (e == cudaSuccess && writer != 0) {
            std::lock_guard<std::mutex> lock(g_mutex);
            d->writers.remove(key, writer);
        }
        return e;
    }
};
// behind_writer: the call itself has just enqueued a kernel that writes what this launch reads
LaunchOrder launch_order(DeviceState* d, void* stream, bool behind_writer = false) {
    LaunchOrder o = {d, {0, 0}, 0, behind_writer};
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (d->writers.overflow) o.serialize = true;
        if (d->writers.count == 0 && d->writers.forgotten == 0) return o;
    }
    o.key = stream_key((cudaStream_t)stream);
    std::lock_guard<std::mutex> lock(g_mutex);
    o.writer = d->writers.pending(o.key);
    if (o.writer != 0 || d->writers.elsewhere_in_capture(o.key)) o.serialize = true;
    return o;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Scales and zero points are stored per group up to 128 columns and per 128 columns above (each
// group's entry group / 128 times), so the layer kernels see groups of 64 or 128 only.
int stored_group(int group) { return group > 128 ? 128 : group; }

int check_shape(int N, int K, int group) {
    if (group != 64 && group != 128 && group != 256 && group != 512 && group != 1024) return AWQ_ERR_BAD_GROUP;
    if (N < 128 || K < 128 || N % 128 != 0 || K % 128 != 0 || K % group != 0) return AWQ_ERR_BAD_SHAPE;
    if (N / 128 > kMaxSlabs) return AWQ_ERR_BAD_SHAPE;
    if ((long long)N * K > (1LL << 33)) return AWQ_ERR_BAD_SHAPE;
    return AWQ_OK;
}

}  // namespace

void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

}  // namespace awq

using namespace awq;

extern "C" {

size_t awq_qweight_bytes(int N, int K) {
    return check_shape(N, K, 128) == AWQ_OK ? (size_t)N * K / 2 : 0;
}
size_t awq_scales_bytes(int N, int K, int group) {
    return check_shape(N, K, group) == AWQ_OK ? (size_t)(K / stored_group(group)) * N * 2 : 0;
}
size_t awq_zeros_bytes(int N, int K, int group) {
    return check_shape(N, K, group) == AWQ_OK ? (size_t)(K / stored_group(group)) * N / 2 : 0;
}

int awq_channel_scale(const float* act_mean_abs, float alpha, float* s, int K, void* stream) {
    if (!(alpha >= 0.0f && alpha <= 1.0f)) return AWQ_ERR_BAD_ALPHA;
    if (!s || (!act_mean_abs && alpha != 0.0f)) return AWQ_ERR_NULL_POINTER;
    if (K < 1) return AWQ_ERR_BAD_SHAPE;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    return note_cuda(launch_channel_scale(act_mean_abs, alpha, s, K, (cudaStream_t)stream));
}

int awq_quantize_pack_ex(const void* W, const float* act_mean_abs, float alpha, int group, int bits,
                         int symmetric, const float* clip_ratio, void* qweight, void* scales, void* zeros,
                         int N, int K, void* stream) {
    if (!(alpha >= 0.0f && alpha <= 1.0f)) return AWQ_ERR_BAD_ALPHA;
    if (int rc = check_shape(N, K, group)) return rc;
    if ((bits != 3 && bits != 4) || (symmetric != 0 && symmetric != 1)) return AWQ_ERR_BAD_ARGUMENT;
    if (!W || !qweight || !scales || !zeros || (!act_mean_abs && alpha != 0.0f)) return AWQ_ERR_NULL_POINTER;
    if (!aligned16(W) || !aligned16(qweight) || !aligned16(scales) || !aligned16(zeros) ||
        (reinterpret_cast<uintptr_t>(act_mean_abs) & 3u) || (reinterpret_cast<uintptr_t>(clip_ratio) & 3u))
        return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    const int rc = note_cuda(launch_quantize_pack(reinterpret_cast<const __half*>(W), act_mean_abs, alpha, group, bits,
                                                  symmetric != 0, clip_ratio, reinterpret_cast<uint32_t*>(qweight),
                                                  reinterpret_cast<__half*>(scales),
                                                  reinterpret_cast<uint8_t*>(zeros), N, K, d->sms, (cudaStream_t)stream));
    note_packed_writer(d, stream);
    return rc;
}

int awq_quantize_pack(const void* W, const float* act_mean_abs, float alpha, int group,
                      void* qweight, void* scales, void* zeros, int N, int K, void* stream) {
    return awq_quantize_pack_ex(W, act_mean_abs, alpha, group, 4, 0, nullptr, qweight, scales, zeros, N, K, stream);
}

int awq_search_clip(const void* W, const float* act_mean_abs, float alpha, int group, int bits,
                    const float* ratios, int n_ratios, float* clip_ratio, int N, int K, void* stream) {
    if (!(alpha >= 0.0f && alpha <= 1.0f)) return AWQ_ERR_BAD_ALPHA;
    if (int rc = check_shape(N, K, group)) return rc;
    if (group > 128) return AWQ_ERR_BAD_GROUP;
    if ((bits != 3 && bits != 4) || n_ratios < 1 || n_ratios > kMaxClipRatios) return AWQ_ERR_BAD_ARGUMENT;
    if (!W || !ratios || !clip_ratio || (!act_mean_abs && alpha != 0.0f)) return AWQ_ERR_NULL_POINTER;
    if ((reinterpret_cast<uintptr_t>(W) & 1u) || (reinterpret_cast<uintptr_t>(act_mean_abs) & 3u) ||
        (reinterpret_cast<uintptr_t>(clip_ratio) & 3u))
        return AWQ_ERR_MISALIGNED;
    for (int i = 0; i < n_ratios; ++i)
        if (!(ratios[i] > 0.0f && ratios[i] <= 1.0f)) return AWQ_ERR_BAD_ARGUMENT;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    return note_cuda(launch_clip_search(reinterpret_cast<const __half*>(W), act_mean_abs, alpha, group, bits,
                                        ratios, n_ratios, clip_ratio, N, K, (cudaStream_t)stream));
}

// Up to 8 tokens: where kernels that share their partial sums through the workspace beat the band kernel.  Their time hardly depends
// on M, while the band kernel's grows with the tokens that travel through its stages.  Chunked / band, us (one machine):
//   8192 -> 28672   3 tokens 27.4 / 31.5   5: 27.7 / 36.7   8: 28.3 / 46.6
//   8192 -> 16384   3: 17.1 / 18.5   4: 17.1 / 18.7   8: 17.3 / 27.5
//   8192 -> 8192    3: 10.9 / 11.3   4: 10.9 / 11.5   8: 11.0 / 17.2
//   13824 -> 5120   3: 11.8 / 14.1   4: 11.8 / 15.1   8: 12.1 / 21.2
//   5120 -> 13824   3: 11.1 / 11.9   4: 11.1 / 12.3   5: 11.2 / 13.8
//   11008 -> 4096   4: 10.4 / 9.8   5: 10.6 / 11.5   6: 10.6 / 13.1   8: 10.6 / 14.0
// With 4096 input channels the band kernel keeps x in registers and beats the chunked one up to 8 tokens
// (4096 -> 11008 at 8 tokens: 11.7 / 9.8; 4096 -> 4096: 6.5 / 6.9).
// (The stream kernel would win from 5 tokens on shorter rows too, 5120 -> 5120 at 8 tokens 6.6 / 10.2; the calls that the band kernel
// serves touch no workspace and may run on several streams at once, so the line stays.)
static bool mid_kernel_preferred(int M, int N, int K) {
    const long long nk = (long long)N * K;
    if (M < 2) return false;
    if (M == 2) return K >= 12288 && nk >= (1LL << 26);   // 13824 -> 5120: 11.6 / 12.9 us, 28672 -> 8192: 29.1 / 30.9 us
    return M <= 8 && K > 4096 && nk >= (M <= 4 ? (1LL << 26) : (1LL << 25));
}

// Of those calls the stream kernel takes the ones with rows of at least 5/4 of the outputs and up to 2^28 weights: its ranges are equal
// whatever the sizes, while the chunked kernel's blocks cross from one slice of x to the next and end on whole units.  Stream / chunked,
// us, 3 and 8 tokens, groups of 128:
//   11008 -> 4096  8.9 / 10.5   9.1 / 10.6      13824 -> 5120  11.4 / 11.8   11.5 / 12.1     28672 -> 8192  28.1 / 29.5   28.3 / 30.3
//   10240 -> 8192  12.7 / 13.6   12.6 / 13.8    13824 -> 11008  19.6 / 21.6   19.7 / 22.2    65536 -> 512  10.0 / 11.8   9.8 / 12.0
//   12288 -> 8192  14.2 / 14.2   14.3 / 14.6    16384 -> 6144  14.2 / 14.6   14.3 / 14.9
// and beyond the lines: 9216 -> 8192 11.7 / 11.2   11.7 / 11.4, 8192 -> 8192 10.8 / 10.9   10.9 / 11.0, 8192 -> 28672 28.7 / 27.4   29.4 / 28.3,
// 18944 -> 14336 31.9 / 31.2   32.2 / 32.2, 28672 -> 11008 at 2 tokens 37.0 / 36.0, 28672 -> 22016 66.6 / 61.7   67.8 / 64.4.
// (Groups of 64 the same way: 28672 -> 8192 32.9 / 32.9   33.1 / 33.7, 11008 -> 4096 9.8 / 11.4   10.1 / 11.6.)
static bool stream_beats_chunked(int M, int N, int K, int group) {
    return mid_kernel_preferred(M, N, K) && 4LL * K >= 5LL * N && (long long)N * K <= (1LL << 28) && gemm_stream_applies(M, N, K, group);
}

// Where the stream kernel runs up to 64 tokens: from 9, and below where the output rows are too few for the band kernel
// (1024 -> 8192 at 3 / 8 tokens 4.8 / 4.9 us; the split-K kernel 8 and 10 us).  Calls of several matrices with rows enough stay on the
// band kernel up to 8 tokens, although on long rows it is the slower one from 4 (stream / band, us: 8192 -> 28672 at 4 / 8 tokens
// 32.1 / 32.7 against 34.7 / 49.1): it gives the bits that each matrix gets by itself, and it touches no workspace, so such calls may run
// on several streams at once.
static bool stream_kernel_preferred(int M, int total_n, int K, int group, int sms) {
    return M <= 64 && (M > 8 || !gemv_uses_band_kernel(M, total_n, sms)) && gemm_stream_applies(M, total_n, K, group);
}

// Above 64 tokens the stream kernel is taken where its estimate is below the prefill kernels' (few tiles for many pairs, long
// rows).  Stream / SM-pair kernel, us: 4096 -> 4096 at 65 / 100 / 128 tokens 10.1 / 11.2 / 11.9 against 14.1 / 14.3 / 14.3,
// 11008 -> 4096 at 100 / 256 tokens 16.8 / 27.7 against 23.8 / 31.8, 8192 -> 3072 at 256 tokens 19.9 against 25.9; but 4096 -> 11008
// at 100 tokens 18.3 against 16.2, 4096 -> 4096 at 256 tokens 17.1 against 15.9, 8192 -> 8192 38.2 against 28.8.  Beyond two tiles of
// 128 tokens the latter won everywhere.  The one-SM kernel keeps the shapes that it had.
static bool stream_beats_prefill(const DeviceState* d, const AwqLinearProblem* problems, int count, int M, int K, int group) {
    if (M <= 64 || M > 256) return false;
    size_t have = 0;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        have = d->workspace_bytes;
    }
    if (have < gemm_stream_workspace_bytes(M, d->sms)) return false;
    double others = 0.0;
    int slabs = 0;
    for (int i = 0; i < count; ++i) {
        bool one_sm = false;
        if (!gemm_stream_applies(M, problems[i].N, K, group)) return false;
        others += gemm_prefill_estimate(M, problems[i].N, K, group, d->sms, have, &one_sm);
        if (one_sm) return false;
        slabs += (problems[i].N + 255) / 256;
    }
    return gemm_stream_estimate(M, slabs, K, d->sms) < others;
}

static int resolve_path(int M, int K, int path) {
    if (path == AWQ_PATH_AUTO) return (M <= 8 && K <= 65536) ? AWQ_PATH_GEMV : AWQ_PATH_GEMM;
    return path;
}

size_t awq_workspace_bytes(int M, int N, int K, int group) {
    if (check_shape(N, K, group) != AWQ_OK || M < 1) return 0;
    group = stored_group(group);
    // optional for the tensor-core kernels: with it they spread their work evenly over the SMs
    static std::atomic<int> known[kMaxDevices];           // SM counts, asked for once per device
    int dev = 0, sms = 0;
    const bool device = cudaGetDevice(&dev) == cudaSuccess;
    if (device && dev >= 0 && dev < kMaxDevices) sms = known[dev].load(std::memory_order_relaxed);
    if (sms == 0) {
        if (!device || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            sms = 160;                       // no device to ask: an upper bound for this GPU family
        } else if (dev >= 0 && dev < kMaxDevices) {
            known[dev].store(sms, std::memory_order_relaxed);
        }
    }
    size_t gemm = gemm_workspace_bytes(M, N, sms);
    const size_t mid = (M <= 8 && gemv_mid_applies(M, N, K, group, sms)) ? gemv_mid_workspace_bytes(M, N, K) : 0;
    const size_t parts = stream_kernel_preferred(M, N, K, group, sms) || stream_beats_chunked(M, N, K, group)
                             ? gemm_stream_workspace_bytes(M, sms) : 0;
    if (parts > gemm) gemm = parts;
    if (M > 16) return gemm;
    size_t gemv = gemv_workspace_bytes(M);         // required by the split-K matrix-vector kernel
    if (M > 8) return gemv > gemm ? gemv : gemm;
    if (mid > gemv) gemv = mid;                    // awq_linear takes no prefill kernel here
    return gemv > parts ? gemv : parts;
}

int awq_set_workspace(void* dev_ptr, size_t bytes) {
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    if ((dev_ptr == nullptr) != (bytes == 0)) return AWQ_ERR_BAD_ARGUMENT;
    if (dev_ptr) {
        if (!aligned16(dev_ptr)) return AWQ_ERR_MISALIGNED;
        if (bytes < kCounterBytes) return AWQ_ERR_BAD_ARGUMENT;
        if (int rc = note_cuda(cudaMemset(dev_ptr, 0, kCounterBytes))) return rc;
    }
    std::lock_guard<std::mutex> lock(g_mutex);
    d->workspace = dev_ptr;
    d->workspace_bytes = bytes;
    return AWQ_OK;
}

// behind_writer: the caller has just enqueued a kernel that writes these packed arrays
static int linear_path(const void* x, const void* qweight, const void* scales, const void* zeros,
                       void* y, int M, int N, int K, int group, int path, void* stream, bool behind_writer) {
    if (int rc = check_shape(N, K, group)) return rc;
    group = stored_group(group);
    if (M < 1 || (long long)M * K > (1LL << 40) || (long long)M * N > (1LL << 40)) return AWQ_ERR_BAD_SHAPE;
    if (!x || !qweight || !scales || !zeros || !y) return AWQ_ERR_NULL_POINTER;
    if (!aligned16(x) || !aligned16(qweight) || !aligned16(scales) || !aligned16(zeros) || !aligned16(y))
        return AWQ_ERR_MISALIGNED;
    if (path != AWQ_PATH_AUTO && path != AWQ_PATH_GEMV && path != AWQ_PATH_GEMM && path != AWQ_PATH_GEMV_SPLITK &&
        path != AWQ_PATH_GEMM_1SM && path != AWQ_PATH_GEMV_MID && path != AWQ_PATH_GEMM_SKINNY)
        return AWQ_ERR_BAD_ARGUMENT;
    const bool automatic = path == AWQ_PATH_AUTO;
    path = resolve_path(M, K, path);
    if (path == AWQ_PATH_GEMV_MID) {
        if (M > 32 || K > 65536) return AWQ_ERR_BAD_SHAPE;
    } else if (path == AWQ_PATH_GEMM_SKINNY) {
        if ((M > 64 || !gemm_stream_applies(M, N, K, group))) return AWQ_ERR_BAD_SHAPE;
    } else if (path != AWQ_PATH_GEMM && path != AWQ_PATH_GEMM_1SM && (M > 16 || K > 65536)) {
        return AWQ_ERR_BAD_SHAPE;
    }
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    int without_stream = path;               // (automatic) taken where the stream kernel cannot be launched
    if (automatic && stream_kernel_preferred(M, N, K, group, d->sms)) {
        const size_t need = gemm_stream_workspace_bytes(M, d->sms);
        std::lock_guard<std::mutex> lock(g_mutex);
        if (d->workspace_bytes >= need) path = AWQ_PATH_GEMM_SKINNY;
    }
    if (automatic && path == AWQ_PATH_GEMV && mid_kernel_preferred(M, N, K) && gemv_mid_applies(M, N, K, group, d->sms)) {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (d->workspace_bytes >= gemv_mid_workspace_bytes(M, N, K)) {
            path = without_stream = AWQ_PATH_GEMV_MID;
            if (stream_beats_chunked(M, N, K, group) && d->workspace_bytes >= gemm_stream_workspace_bytes(M, d->sms)) path = AWQ_PATH_GEMM_SKINNY;
        }
    }
    if (automatic && path == AWQ_PATH_GEMM) {          // (asked for by name it is the prefill kernels)
        const AwqLinearProblem one = {qweight, scales, zeros, y, N};
        if (stream_beats_prefill(d, &one, 1, M, K, group)) path = AWQ_PATH_GEMM_SKINNY;
    }
    if (path == AWQ_PATH_GEMV_MID && M > 8 && gemm_stream_applies(M, N, K, group)) path = AWQ_PATH_GEMM_SKINNY;
    const cudaStream_t st = (cudaStream_t)stream;
    const LaunchOrder order = launch_order(d, stream, behind_writer);
    if (path == AWQ_PATH_GEMM_SKINNY) {
        const size_t need = gemm_stream_workspace_bytes(M, d->sms);
        void* ws = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            if (d->workspace_bytes < need) return AWQ_ERR_NO_WORKSPACE;
            ws = d->workspace;
        }
        const GemvMatrix one = {qweight, scales, zeros, y, N};
        const cudaError_t e = order.launched(launch_gemm_stream(x, &one, 1, M, K, group, nullptr, ws, d->status_word,
                                                                d->sms, order.serialize, st));
        if (!automatic || e != cudaErrorNotSupported) return note_cuda(e);
        path = without_stream;               // no pair of SMs to be had (a partition of the device): nothing was launched
    }
    if (path == AWQ_PATH_GEMV_MID) {
        if (!gemv_mid_applies(M, N, K, group, d->sms)) return AWQ_ERR_BAD_SHAPE;
        void* ws = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            if (d->workspace_bytes < gemv_mid_workspace_bytes(M, N, K)) return AWQ_ERR_NO_WORKSPACE;
            ws = d->workspace;
        }
        return note_cuda(order.launched(launch_gemv_mid(x, qweight, scales, zeros, y, M, N, K, group, ws, d->status_word, d->sms,
                                                        order.serialize, st)));
    }
    if (path == AWQ_PATH_GEMV && gemv_uses_band_kernel(M, N, d->sms)) {
        const GemvMatrix one = {qweight, scales, zeros, y, N};
        return note_cuda(order.launched(launch_gemv_band(x, &one, 1, M, K, group, d->status_word, d->sms, order.serialize, st)));
    }
    // (split-K and one-SM kernels are plainly stream-ordered)
    if (path == AWQ_PATH_GEMV || path == AWQ_PATH_GEMV_SPLITK) {
        void* ws = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            if (d->workspace_bytes < gemv_workspace_bytes(M)) return AWQ_ERR_NO_WORKSPACE;
            ws = d->workspace;
        }
        int surplus = 0;
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            surplus = d->tx_surplus_once;
            d->tx_surplus_once = 0;
        }
        return note_cuda(order.launched(launch_gemv_splitk(x, qweight, scales, zeros, y, M, N, K, group, ws, d->status_word,
                                                           d->sms, st, surplus)));
    }
    void* ws = nullptr;
    size_t ws_bytes = 0;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        ws = d->workspace;
        ws_bytes = d->workspace_bytes;
    }
    return note_cuda(order.launched(launch_gemm(x, qweight, scales, zeros, y, M, N, K, group, path != AWQ_PATH_GEMM_1SM,
                                                ws, ws_bytes, d->status_word, order.serialize, st)));
}

int awq_linear_path(const void* x, const void* qweight, const void* scales, const void* zeros,
                    void* y, int M, int N, int K, int group, int path, void* stream) {
    return linear_path(x, qweight, scales, zeros, y, M, N, K, group, path, stream, false);
}

int awq_linear_gemv_static(const void* x, const void* qweight, const void* scales, const void* zeros,
                            void* y, int M, int N, int K, int group, void* stream) {
    if (int rc = check_shape(N, K, group)) return rc;
    group = stored_group(group);
    if (M < 1) return AWQ_ERR_BAD_SHAPE;
    if (M > gemv_static_max_m() || K > 65536) return AWQ_ERR_STATIC_LIMIT;
    if (!x || !qweight || !scales || !zeros || !y) return AWQ_ERR_NULL_POINTER;
    if (!aligned16(x) || !aligned16(qweight) || !aligned16(scales) || !aligned16(zeros) || !aligned16(y))
        return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    void* scratch = nullptr;
    if (int rc = note_cuda(gemv_static_scratch(&scratch))) return rc;
    const cudaStream_t st = (cudaStream_t)stream;
    // the arrival counters must start at zero whatever an earlier call left behind
    if (int rc = note_cuda(cudaMemsetAsync(scratch, 0, kCounterBytes, st))) return rc;
    return note_cuda(launch_gemv_splitk(x, qweight, scales, zeros, y, M, N, K, group, scratch,
                                        d->status_word, d->sms, st));
}

int awq_set_wait_limit_us(unsigned int microseconds) {
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    if (int rc = note_cuda(cudaDeviceSynchronize())) return rc;
    return note_cuda(cudaMemcpy(d->status_word + 1, &microseconds, sizeof(microseconds), cudaMemcpyHostToDevice));
}

int awq_test_stall_next_gemv(void) {
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    std::lock_guard<std::mutex> lock(g_mutex);
    d->tx_surplus_once = 16;
    return AWQ_OK;
}

int awq_static_scratch_fill(int value, void* stream) {
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    void* scratch = nullptr;
    if (int rc = note_cuda(gemv_static_scratch(&scratch))) return rc;
    return note_cuda(cudaMemsetAsync(scratch, value & 0xFF, kCounterBytes, (cudaStream_t)stream));
}

// All matrices in one launch of the stream kernel, if the workspace holds their partial sums and the kernel can run.
static int linear_multi_stream(DeviceState* d, const void* x, const float* inv_s, const AwqLinearProblem* problems,
                               int count, int M, int K, int group, void* stream, bool* launched) {
    const size_t need = gemm_stream_workspace_bytes(M, d->sms);
    void* ws = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (d->workspace_bytes < need) return AWQ_OK;
        ws = d->workspace;
    }
    GemvMatrix mats[kMaxMulti];
    for (int i = 0; i < count; ++i)
        mats[i] = GemvMatrix{problems[i].qweight, problems[i].scales, problems[i].zeros, problems[i].y, problems[i].N};
    const LaunchOrder order = launch_order(d, stream);
    const cudaError_t e = order.launched(launch_gemm_stream(x, mats, count, M, K, group, inv_s, ws, d->status_word, d->sms,
                                                            order.serialize, (cudaStream_t)stream));
    if (e == cudaErrorNotSupported) return AWQ_OK;           // as in linear_path
    *launched = true;
    return note_cuda(e);
}

int awq_linear_multi(const void* x, const AwqLinearProblem* problems, int count,
                     int M, int K, int group, void* stream) {
    if (!problems || !x) return AWQ_ERR_NULL_POINTER;
    if (count < 1 || count > kMaxMulti) return AWQ_ERR_BAD_ARGUMENT;
    int total_n = 0;
    for (int i = 0; i < count; ++i) {
        const AwqLinearProblem& p = problems[i];
        if (int rc = check_shape(p.N, K, group)) return rc;
        if (!p.qweight || !p.scales || !p.zeros || !p.y) return AWQ_ERR_NULL_POINTER;
        if (!aligned16(p.qweight) || !aligned16(p.scales) || !aligned16(p.zeros) || !aligned16(p.y))
            return AWQ_ERR_MISALIGNED;
        total_n += p.N;
    }
    group = stored_group(group);
    if (M < 1) return AWQ_ERR_BAD_SHAPE;
    if (!aligned16(x)) return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    if (stream_kernel_preferred(M, total_n, K, group, d->sms) || (count > 1 && stream_beats_prefill(d, problems, count, M, K, group))) {
        bool launched = false;
        const int rc = linear_multi_stream(d, x, nullptr, problems, count, M, K, group, stream, &launched);
        if (rc != AWQ_OK || launched) return rc;
    }
    if (M <= 8 && K <= 65536 && gemv_uses_band_kernel(M, total_n, d->sms)) {
        GemvMatrix mats[kMaxMulti];
        for (int i = 0; i < count; ++i)
            mats[i] = GemvMatrix{problems[i].qweight, problems[i].scales, problems[i].zeros, problems[i].y,
                                 problems[i].N};
        const LaunchOrder order = launch_order(d, stream);
        return note_cuda(order.launched(launch_gemv_band(x, mats, count, M, K, group, d->status_word, d->sms, order.serialize,
                                                         (cudaStream_t)stream)));
    }
    // otherwise one call per matrix, as awq_linear would run it
    for (int i = 0; i < count; ++i) {
        const AwqLinearProblem& p = problems[i];
        if (int rc = awq_linear(x, p.qweight, p.scales, p.zeros, p.y, M, p.N, K, group, stream)) return rc;
    }
    return AWQ_OK;
}

int awq_linear(const void* x, const void* qweight, const void* scales, const void* zeros,
               void* y, int M, int N, int K, int group, void* stream) {
    return awq_linear_path(x, qweight, scales, zeros, y, M, N, K, group, AWQ_PATH_AUTO, stream);
}

// ---- the layer with diag(s)^-1 folded in (Sec. 3.2: the inverse scale goes into the operator in front)
static bool scaled_call_folds(int M, int total_n, int K, int group, int sms) {
    return M <= 8 && K <= 65536 && gemv_uses_band_kernel(M, total_n, sms) && gemv_band_folds_scale(M, K, group);
}

int awq_linear_scaled_needs_scratch(int M, int N, int K, int group) {
    if (check_shape(N, K, group) != AWQ_OK || M < 1) return 1;
    group = stored_group(group);
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return 1;
    }
    return scaled_call_folds(M, N, K, group, sms) ? 0 : 1;
}

int awq_linear_multi_scaled(const void* x, const float* inv_s, void* x_scratch, const AwqLinearProblem* problems,
                            int count, int M, int K, int group, void* stream) {
    if (!problems || !x || !inv_s) return AWQ_ERR_NULL_POINTER;
    if (count < 1 || count > kMaxMulti) return AWQ_ERR_BAD_ARGUMENT;
    int total_n = 0;
    for (int i = 0; i < count; ++i) {
        const AwqLinearProblem& p = problems[i];
        if (int rc = check_shape(p.N, K, group)) return rc;
        if (!p.qweight || !p.scales || !p.zeros || !p.y) return AWQ_ERR_NULL_POINTER;
        if (!aligned16(p.qweight) || !aligned16(p.scales) || !aligned16(p.zeros) || !aligned16(p.y))
            return AWQ_ERR_MISALIGNED;
        total_n += p.N;
    }
    group = stored_group(group);
    if (M < 1 || (long long)M * K > (1LL << 40)) return AWQ_ERR_BAD_SHAPE;
    if (!aligned16(x) || !aligned16(inv_s) || !aligned16(x_scratch)) return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    if (scaled_call_folds(M, total_n, K, group, d->sms)) {
        GemvMatrix mats[kMaxMulti];
        for (int i = 0; i < count; ++i)
            mats[i] = GemvMatrix{problems[i].qweight, problems[i].scales, problems[i].zeros, problems[i].y,
                                 problems[i].N};
        const LaunchOrder order = launch_order(d, stream);
        return note_cuda(order.launched(launch_gemv_band(x, mats, count, M, K, group, d->status_word, d->sms, order.serialize,
                                                         (cudaStream_t)stream, inv_s)));
    }
    if (!x_scratch) return AWQ_ERR_NULL_POINTER;
    if (stream_kernel_preferred(M, total_n, K, group, d->sms) || stream_beats_prefill(d, problems, count, M, K, group)) {
        bool launched = false;
        const int rc = linear_multi_stream(d, x, inv_s, problems, count, M, K, group, stream, &launched);
        if (rc != AWQ_OK || launched) return rc;
    }
    // no kernel to fold it into: scale first (one more launch), then the plain calls
    if (int rc = note_cuda(launch_multiply_by_inverse(x, inv_s, x_scratch, M, K, (cudaStream_t)stream))) return rc;
    return awq_linear_multi(x_scratch, problems, count, M, K, group, stream);
}

int awq_linear_scaled(const void* x, const float* inv_s, void* x_scratch, const void* qweight, const void* scales,
                      const void* zeros, void* y, int M, int N, int K, int group, void* stream) {
    const AwqLinearProblem one = {qweight, scales, zeros, y, N};
    return awq_linear_multi_scaled(x, inv_s, x_scratch, &one, 1, M, K, group, stream);
}

// ---- 3-bit storage
size_t awq_qweight_bytes_int3(int N, int K) {
    return check_shape(N, K, 128) == AWQ_OK ? (size_t)N * K / 8 * 3 : 0;
}

int awq_pack_int3(const void* qweight, void* qweight3, int N, int K, void* stream) {
    if (int rc = check_shape(N, K, 128)) return rc;
    if (!qweight || !qweight3) return AWQ_ERR_NULL_POINTER;
    if (!aligned16(qweight) || !aligned16(qweight3)) return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    const int rc = note_cuda(launch_pack_int3(qweight, qweight3, N, K, (cudaStream_t)stream));
    note_packed_writer(d, stream);
    return rc;
}

int awq_unpack_int3(const void* qweight3, void* qweight, int N, int K, void* stream) {
    if (int rc = check_shape(N, K, 128)) return rc;
    if (!qweight || !qweight3) return AWQ_ERR_NULL_POINTER;
    if (!aligned16(qweight) || !aligned16(qweight3)) return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    const int rc = note_cuda(launch_unpack_int3(qweight3, qweight, N, K, (cudaStream_t)stream));
    note_packed_writer(d, stream);
    return rc;
}

int awq_linear_int3(const void* x, const void* qweight3, const void* scales, const void* zeros, void* y,
                    void* qweight_scratch, int M, int N, int K, int group, void* stream) {
    if (int rc = check_shape(N, K, group)) return rc;
    group = stored_group(group);
    if (M < 1 || (long long)M * K > (1LL << 40) || (long long)M * N > (1LL << 40)) return AWQ_ERR_BAD_SHAPE;
    if (!x || !qweight3 || !scales || !zeros || !y) return AWQ_ERR_NULL_POINTER;
    if (!aligned16(x) || !aligned16(qweight3) || !aligned16(scales) || !aligned16(zeros) || !aligned16(y) ||
        !aligned16(qweight_scratch))
        return AWQ_ERR_MISALIGNED;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    if (M <= 8 && K <= 65536 && gemv_uses_band_kernel(M, N, d->sms)) {
        const GemvMatrix one = {qweight3, scales, zeros, y, N};
        const LaunchOrder order = launch_order(d, stream);
        return note_cuda(order.launched(launch_gemv_band(x, &one, 1, M, K, group, d->status_word, d->sms, order.serialize,
                                                         (cudaStream_t)stream, nullptr, 3)));
    }
    // Up to 64 tokens, where awq_linear takes the stream kernel, that kernel reads the 3-bit storage as it is (expanding and then it / it
    // alone, us: 4096 -> 11008 at 16 / 64 tokens 16.6 / 20.3 against 11.3 / 14.9, 4096 -> 4096 at 16 10.6 against 8.1, 8192 -> 28672 at 16
    // 62.1 against 32.1).  The stream kernel is plainly ordered here: an expansion waited for whatever wrote the 3-bit words in front of
    // it, a caller's own kernel too, and such calls stay right.  That costs about 2 us against awq_linear's launches on 4-bit words.
    if (stream_kernel_preferred(M, N, K, group, d->sms)) {
        void* ws = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            if (d->workspace_bytes >= gemm_stream_workspace_bytes(M, d->sms)) ws = d->workspace;
        }
        if (ws) {
            const GemvMatrix one = {qweight3, scales, zeros, y, N};
            const LaunchOrder order = launch_order(d, stream, true);
            const cudaError_t e = order.launched(launch_gemm_stream(x, &one, 1, M, K, group, nullptr, ws, d->status_word, d->sms,
                                                                    true, (cudaStream_t)stream, 3));
            if (e != cudaErrorNotSupported) return note_cuda(e);
        }
    }
    // every other kernel reads the 4-bit layout: expand first (one more launch), then the plain call
    if (!qweight_scratch) return AWQ_ERR_NULL_POINTER;
    if (int rc = awq_unpack_int3(qweight3, qweight_scratch, N, K, stream)) return rc;
    return linear_path(x, qweight_scratch, scales, zeros, y, M, N, K, group, AWQ_PATH_AUTO, stream, true);
}

int awq_inverse_channel_scale(const float* act_mean_abs, float alpha, float* inv_s, int K, void* stream) {
    if (int rc = awq_channel_scale(act_mean_abs, alpha, inv_s, K, stream)) return rc;
    const int rc = note_cuda(launch_inverse_scale(inv_s, inv_s, K, (cudaStream_t)stream));
    DeviceState* d;
    if (int bad = device_state(&d)) return bad;
    note_packed_writer(d, stream);           // the band kernel loads 1 / s as early as the packed arrays
    return rc;
}

size_t awq_search_scratch_bytes(int M, int N, int K, int group) {
    if (check_shape(N, K, group) != AWQ_OK || M < 1 || group > 128) return 0;
    return search_plan(nullptr, 0, M, N, K, group, 1).total;
}

size_t awq_search_scratch_bytes_points(int M, int N, int K, int group, int points) {
    if (check_shape(N, K, group) != AWQ_OK || M < 1 || group > 128 || points < 1 || points > kMaxSearchAlphas) return 0;
    return search_plan(nullptr, SIZE_MAX, M, N, K, group, points).total;
}

int awq_search_alpha(const void* W, const float* act_mean_abs, const void* X, int M, int N, int K, int group,
                     const float* alphas, int n_alphas, float* losses, int* best_index,
                     void* scratch, size_t scratch_bytes, void* stream) {
    if (int rc = check_shape(N, K, group)) return rc;
    if (group > 128) return AWQ_ERR_BAD_GROUP;
    if (M < 1) return AWQ_ERR_BAD_SHAPE;
    if (!W || !act_mean_abs || !X || !alphas || !losses || !best_index || !scratch) return AWQ_ERR_NULL_POINTER;
    if (n_alphas < 1 || n_alphas > kMaxSearchAlphas) return AWQ_ERR_BAD_ARGUMENT;
    for (int i = 0; i < n_alphas; ++i)
        if (!(alphas[i] >= 0.0f && alphas[i] <= 1.0f)) return AWQ_ERR_BAD_ARGUMENT;
    const SearchPlan p = search_plan(scratch, scratch_bytes, M, N, K, group, n_alphas);
    if (scratch_bytes < p.total) return AWQ_ERR_BAD_ARGUMENT;
    if (!aligned16(W) || !aligned16(X) || (reinterpret_cast<uintptr_t>(scratch) & 255u) != 0) return AWQ_ERR_MISALIGNED;
    if (reinterpret_cast<uintptr_t>(act_mean_abs) & 3u) return AWQ_ERR_MISALIGNED;
    const cudaStream_t st = (cudaStream_t)stream;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    void* ws = nullptr;
    size_t ws_bytes = 0;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        ws = d->workspace;
        ws_bytes = d->workspace_bytes;
    }
    if (int rc = note_cuda(launch_reference_product(W, X, p.yref, M, N, K, d->status_word, st))) return rc;
    const int batches = (n_alphas + p.batch - 1) / p.batch, most = (n_alphas + batches - 1) / batches;
    for (int i0 = 0; i0 < n_alphas; i0 += most) {
        const int b = n_alphas - i0 < most ? n_alphas - i0 : most;
        if (int rc = note_cuda(launch_channel_scales(act_mean_abs, alphas + i0, b, p.s, K, st))) return rc;
        if (int rc = note_cuda(launch_quantize_pack_many(reinterpret_cast<const __half*>(W), p.s, b, group,
                                                         reinterpret_cast<uint32_t*>(p.qweight), reinterpret_cast<__half*>(p.scales),
                                                         p.zeros, N, K, d->sms, st)))
            return rc;
        // (the plainly ordered division stands between this writer and its readers)
        if (int rc = note_cuda(launch_divide_by_scale(X, p.s, b, p.xs, M, p.rows, K, st))) return rc;
        // all products at once where the layer's kernel rounds (q - z) * Delta to fp16 too (above 64 tokens)
        bool launched = false;
        if (M > 64)
            if (int rc = note_cuda(launch_gemm_blocks(p.xs, p.qweight, p.scales, p.zeros, p.yq, b, M, p.rows, N, K, group, ws, ws_bytes,
                                                      d->status_word, d->sms, st, &launched)))
                return rc;
        const size_t groups = (size_t)(K / group);
        for (int i = 0; i < b && !launched; ++i)
            if (int rc = awq_linear(p.xs + (size_t)i * p.rows * K, p.qweight + (size_t)i * N * K / 2, p.scales + i * groups * N * 2,
                                    p.zeros + i * groups * N / 2, p.yq + (size_t)i * p.rows * N, M, N, K, group, stream))
                return rc;
        if (int rc = note_cuda(launch_squared_difference(p.yq, p.yref, b, M, p.rows, N, p.partials, st))) return rc;
        if (int rc = note_cuda(launch_losses(p.partials, b, (size_t)M * N, p.losses + i0, st))) return rc;
    }
    if (int rc = note_cuda(cudaMemcpyAsync(losses, p.losses, (size_t)n_alphas * sizeof(float),
                                           cudaMemcpyDeviceToHost, st)))
        return rc;
    if (int rc = note_cuda(cudaStreamSynchronize(st))) return rc;
    int best = 0;
    bool have = false;
    for (int i = 0; i < n_alphas; ++i) {
        if (!std::isfinite(losses[i])) continue;
        if (!have || losses[i] < losses[best]) { best = i; have = true; }
    }
    *best_index = best;
    return AWQ_OK;
}

int awq_unpack_canonical(const void* qweight, const void* scales, const void* zeros,
                         int N, int K, int group,
                         uint8_t* codes, uint16_t* scales_nk, uint8_t* zeros_nk, void* stream) {
    if (int rc = check_shape(N, K, group)) return rc;
    if (!qweight || !scales || !zeros || !codes || !scales_nk || !zeros_nk) return AWQ_ERR_NULL_POINTER;
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    return note_cuda(launch_unpack(reinterpret_cast<const uint32_t*>(qweight),
                                   reinterpret_cast<const __half*>(scales),
                                   reinterpret_cast<const uint8_t*>(zeros), N, K, group,
                                   codes, scales_nk, zeros_nk, (cudaStream_t)stream));
}

int awq_poll_status(void) {
    DeviceState* d;
    if (int rc = device_state(&d)) return rc;
    unsigned long long upto = 0;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        upto = d->writers.serial;
    }
    if (int rc = note_cuda(cudaDeviceSynchronize())) return rc;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        d->writers.completed(upto);
    }
    unsigned int v = 0;
    if (int rc = note_cuda(cudaMemcpy(&v, d->status_word, sizeof(v), cudaMemcpyDeviceToHost))) return rc;
    if (v != 0) {
        if (int rc = note_cuda(cudaMemset(d->status_word, 0, sizeof(v)))) return rc;
        // a kernel that gave up may have left arrival counters half-way: start them afresh
        void* ws = nullptr;
        size_t ws_bytes = 0;
        {
            std::lock_guard<std::mutex> lock(g_mutex);
            ws = d->workspace;
            ws_bytes = d->workspace_bytes;
        }
        if (ws && ws_bytes >= kCounterBytes)
            if (int rc = note_cuda(cudaMemset(ws, 0, kCounterBytes))) return rc;
        return AWQ_ERR_TIMEOUT;
    }
    return AWQ_OK;
}

const char* awq_status_string(int status) {
    switch (status) {
        case AWQ_OK: return "ok";
        case AWQ_ERR_NULL_POINTER: return "null pointer";
        case AWQ_ERR_BAD_SHAPE: return "bad shape (N, K multiples of 128; K % group == 0; M >= 1)";
        case AWQ_ERR_BAD_GROUP: return "group must be 64 or 128";
        case AWQ_ERR_BAD_ALPHA: return "alpha must lie in [0, 1]";
        case AWQ_ERR_MISALIGNED: return "pointer not 16-byte aligned";
        case AWQ_ERR_NO_WORKSPACE: return "registered workspace too small (see awq_workspace_bytes)";
        case AWQ_ERR_WRONG_DEVICE: return "current device is not compute capability 10.x";
        case AWQ_ERR_CUDA: return "CUDA call failed (see awq_last_cuda_error)";
        case AWQ_ERR_TIMEOUT: return "a device-side wait ran out";
        case AWQ_ERR_BAD_ARGUMENT: return "bad argument";
        case AWQ_ERR_STATIC_LIMIT: return "problem exceeds the built-in scratch of awq_linear_gemv_static (M <= 8, K <= 65536)";
        default: return "unknown status";
    }
}

const char* awq_last_cuda_error(void) { return t_cuda_error; }
int awq_layout_version(void) { return 3; }
unsigned long long awq_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

}  // extern "C"
