// api.cu — host-side plumbing of libqnn: pointer-kind checks, the per-device status word and
// scratch buffers, and the status calls of the C ABI.
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "qnn_host.h"

namespace qnn {

struct Held {  // a stream's scratch: grown in its order
    unsigned long long stream = 0;
    void *p = nullptr;
    size_t bytes = 0;
    int calls = 0;  // being made with it
};

namespace {

constexpr int kMaxDevices = 64;

struct DeviceState {
    Held held[kHeldStreams];
    int held_streams = 0;
    cudaMemPool_t pool = nullptr;
    size_t pool_keeps = 0;
    char *reduce = nullptr;  // kReduceStreams slots
    unsigned long long reduce_stream[kReduceStreams] = {};
    int reduce_streams = 0;
    int *status = nullptr;
    int sms = 0;
};

std::mutex g_mu;
DeviceState g_dev[kMaxDevices];

qnn_status current(int *dev) {
    QNN_CUDA_TRY(cudaGetDevice(dev));
    if (*dev < 0 || *dev >= kMaxDevices) return QNN_ERR_CUDA;
    return QNN_OK;
}

}  // namespace

bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

void *host_mapped_ptr(void *p) {
    if (!p) return nullptr;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
}

qnn_status Scratch::take(size_t bytes, cudaStream_t st) {
    int dev = 0;
    QNN_TRY(current(&dev));
    cudaMemPool_t pool = nullptr;
    unsigned long long id = 0;  // (of the process's life: a later stream at the same address has another)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    QNN_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    if (cap == cudaStreamCaptureStatusNone) QNN_CUDA_TRY(cudaStreamGetId(st, &id));
    {
        std::lock_guard<std::mutex> lk(g_mu);
        DeviceState &d = g_dev[dev];
        if (!d.pool) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            QNN_CUDA_TRY(cudaMemPoolCreate(&d.pool, &props));
        }
        const size_t keeps = bytes > (size_t)1 << 30 ? bytes : (size_t)1 << 30;
        if (keeps > d.pool_keeps) {
            unsigned long long v = keeps;
            QNN_CUDA_TRY(cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &v));
            d.pool_keeps = keeps;
        }
        pool = d.pool;
        int i = 0;
        while (i < d.held_streams && d.held[i].stream != id) ++i;
        // (not while another thread launches with it: two calls' kernels could follow one another in any order)
        if (cap == cudaStreamCaptureStatusNone && bytes <= kHeldBytes && i < kHeldStreams && d.held[i].calls == 0) {
            Held &h = d.held[i];
            if (h.bytes < bytes) {
                if (h.p) QNN_CUDA_TRY(cudaFreeAsync(h.p, st));  // (what used it is on the stream already)
                h.p = nullptr, h.bytes = 0;
                QNN_CUDA_TRY(cudaMallocFromPoolAsync(&h.p, bytes, pool, st));
                h.bytes = bytes;
            }
            if (i == d.held_streams) h.stream = id, ++d.held_streams;
            ++h.calls;
            p_ = h.p, held_ = &h;
            return QNN_OK;
        }
    }
    QNN_CUDA_TRY(cudaMallocFromPoolAsync(&p_, bytes, pool, st));
    pooled_ = true, st_ = st;
    return QNN_OK;
}

qnn_status Scratch::take_reduce(cudaStream_t st) {
    int dev = 0;
    QNN_TRY(current(&dev));
    const size_t slot = kReduceHeader + (sizeof(float) * 2 * kReduceBlocks * (size_t)sm_count() + 255) / 256 * 256;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    QNN_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    if (cap == cudaStreamCaptureStatusNone) {
        unsigned long long id = 0;
        QNN_CUDA_TRY(cudaStreamGetId(st, &id));
        std::lock_guard<std::mutex> lk(g_mu);
        DeviceState &d = g_dev[dev];
        int i = 0;
        while (i < d.reduce_streams && d.reduce_stream[i] != id) ++i;
        if (i < kReduceStreams) {
            if (!d.reduce) {
                void *p = nullptr;
                QNN_CUDA_TRY(cudaMalloc(&p, slot * kReduceStreams));
                if (cudaMemset(p, 0, slot * kReduceStreams) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
                    cudaFree(p);
                    return QNN_FAIL(QNN_ERR_CUDA);
                }
                d.reduce = static_cast<char *>(p);
            }
            if (i == d.reduce_streams) d.reduce_stream[d.reduce_streams++] = id;
            p_ = d.reduce + (size_t)i * slot;
            return QNN_OK;
        }
    }
    QNN_TRY(take(slot, st));
    QNN_CUDA_TRY(cudaMemsetAsync(p_, 0, sizeof(unsigned), st));
    return QNN_OK;
}

Scratch::~Scratch() {
    if (held_) {
        std::lock_guard<std::mutex> lk(g_mu);
        --held_->calls;
    }
    if (pooled_ && cudaFreeAsync(p_, st_) != cudaSuccess) cudaGetLastError();
}

void scratch_trim() {
    int dev = 0;
    if (current(&dev) != QNN_OK) return;
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceState &d = g_dev[dev];
    if (!d.pool || cudaDeviceSynchronize() != cudaSuccess) return;
    for (Held &h : d.held)
        if (h.p && h.calls == 0) {
            cudaFree(h.p);
            h.p = nullptr, h.bytes = 0;
        }
    cudaMemPoolTrimTo(d.pool, 0);
}

qnn_status status_word(int **out) {
    int dev = 0;
    QNN_TRY(current(&dev));
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceState &d = g_dev[dev];
    if (!d.status) {
        QNN_CUDA_TRY(cudaMalloc(&d.status, sizeof(int)));
        QNN_CUDA_TRY(cudaMemset(d.status, 0, sizeof(int)));
    }
    *out = d.status;
    return QNN_OK;
}

int sm_count() {
    int dev = 0;
    if (current(&dev) != QNN_OK) return 1;
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceState &d = g_dev[dev];
    if (!d.sms) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 1;
        d.sms = v;
    }
    return d.sms;
}

}  // namespace qnn

using namespace qnn;

extern "C" const char *qnn_status_string(qnn_status s) {
    switch (s) {
        case QNN_OK: return "QNN_OK";
        case QNN_ERR_INVALID_ARG: return "QNN_ERR_INVALID_ARG: invalid argument";
        case QNN_ERR_NONFINITE: return "QNN_ERR_NONFINITE: a quantization unit held NaN or Inf";
        case QNN_ERR_K_TOO_LARGE: return "QNN_ERR_K_TOO_LARGE: K exceeds 33025 (int32 accumulator limit)";
        case QNN_ERR_CUDA: return "QNN_ERR_CUDA: CUDA runtime error or no device";
        case QNN_ERR_TIMEOUT: return "QNN_ERR_TIMEOUT: a persistent-kernel grid wait timed out";
        case QNN_ERR_NO_COOP: return "QNN_ERR_NO_COOP: persistent grid cannot be co-resident";
        case QNN_ERR_NO_MEMORY: return "QNN_ERR_NO_MEMORY: device allocation failed";
    }
    return "unknown qnn_status";
}

extern "C" qnn_status qnn_device_status(void *stream) {
    int *w = nullptr;
    QNN_TRY(status_word(&w));
    QNN_CUDA_TRY(cudaStreamSynchronize(as_stream(stream)));
    int v = 0;
    QNN_CUDA_TRY(cudaMemcpy(&v, w, sizeof(int), cudaMemcpyDeviceToHost));
    if (v) QNN_CUDA_TRY(cudaMemset(w, 0, sizeof(int)));
    return static_cast<qnn_status>(v);
}

// ------------------------------------------------------------------------------------------------
// Kernel timing (diagnostics): CUDA events around every launch while enabled.
// ------------------------------------------------------------------------------------------------

namespace qnn {
namespace {

struct ProfPending {
    const char *name;
    cudaEvent_t a, b;
};
struct ProfAgg {
    const char *name;
    double ms;
    int64_t n;
};
std::mutex g_pmu;
bool g_prof_on = false;
std::vector<ProfPending> g_pending;
std::vector<cudaEvent_t> g_pool;
std::vector<ProfAgg> g_agg;

cudaEvent_t take_event() {
    if (!g_pool.empty()) {
        cudaEvent_t e = g_pool.back();
        g_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

}  // namespace

ProfScope::ProfScope(const char *name, cudaStream_t st) : st_(st), idx_(-1) {
    std::lock_guard<std::mutex> lk(g_pmu);
    if (!g_prof_on) return;
    ProfPending p{name, take_event(), take_event()};
    if (!p.a || !p.b) return;
    cudaEventRecord(p.a, st);
    g_pending.push_back(p);
    idx_ = (int)g_pending.size() - 1;
}

ProfScope::~ProfScope() {
    if (idx_ < 0) return;
    std::lock_guard<std::mutex> lk(g_pmu);
    if (idx_ < (int)g_pending.size()) cudaEventRecord(g_pending[idx_].b, st_);
}

}  // namespace qnn

extern "C" qnn_status qnn_profile_enable(int on) {
    std::lock_guard<std::mutex> lk(g_pmu);
    g_prof_on = on != 0;
    return QNN_OK;
}

extern "C" qnn_status qnn_profile_read(int capacity, const char **names, double *total_ms, int64_t *launches,
                                       int *count) {
    std::lock_guard<std::mutex> lk(g_pmu);
    for (ProfPending &p : g_pending) {
        float ms = 0.0f;
        QNN_CUDA_TRY(cudaEventSynchronize(p.b));
        QNN_CUDA_TRY(cudaEventElapsedTime(&ms, p.a, p.b));
        bool found = false;
        for (ProfAgg &g : g_agg)
            if (g.name == p.name || std::strcmp(g.name, p.name) == 0) {
                g.ms += ms;
                g.n += 1;
                found = true;
                break;
            }
        if (!found) g_agg.push_back({p.name, (double)ms, 1});
        g_pool.push_back(p.a);
        g_pool.push_back(p.b);
    }
    g_pending.clear();
    int n = (int)g_agg.size();
    for (int i = 0; i < n && i < capacity; ++i) {
        if (names) names[i] = g_agg[i].name;
        if (total_ms) total_ms[i] = g_agg[i].ms;
        if (launches) launches[i] = g_agg[i].n;
    }
    if (count) *count = n;
    g_agg.clear();
    return QNN_OK;
}
