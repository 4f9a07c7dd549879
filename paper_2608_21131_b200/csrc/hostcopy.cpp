// Copies between ordinary (pageable) host memory and the device for the client calls.
//
// The driver stages such a copy through one thread: 20 GB/s up and 13 GB/s down on a host whose bus does 54.  Here up to four threads
// share the pieces out, each with two page-locked slots of its own: a thread fills one slot while the copy engine empties the other.
#include <atomic>
#include <cstring>
#include <string>
#include <thread>

#include "internal.h"

namespace {

constexpr int kThreads = 4, kSlots = 2;
constexpr int64_t kPiece = 512 << 10;
static_assert(kThreads * kSlots == sizeof(hann_ctx::pin_ev) / sizeof(cudaEvent_t), "an event per slot");

bool pageable(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeUnregistered;
}

// the page-locked slots of a context and their events, on first use; false if they cannot be had
bool slots(hann_ctx* c) {
    if (c->pin) return true;
    for (cudaEvent_t& ev : c->pin_ev)
        if (!ev && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            ev = nullptr;
            return false;
        }
    if (cudaHostAlloc(&c->pin, kThreads * kSlots * kPiece, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        c->pin = nullptr;
        return false;
    }
    return true;
}

struct Job {
    hann_ctx* c;
    const HostCopy* list;
    int n;
    bool up;
    cudaStream_t stream;
    std::atomic<int64_t> next{0};
    std::atomic<int> error{(int)cudaSuccess};

    static int64_t pieces_of(const HostCopy& h) { return (h.bytes + kPiece - 1) / kPiece; }
    int64_t pieces() const {
        int64_t k = 0;
        for (int i = 0; i < n; i++) k += pieces_of(list[i]);
        return k;
    }
    cudaError_t piece(int64_t k, int worker, int& turn) {
        int i = 0;
        for (; k >= pieces_of(list[i]); i++) k -= pieces_of(list[i]);
        const HostCopy& h = list[i];
        const int64_t off = k * kPiece, bytes = h.bytes - off < kPiece ? h.bytes - off : kPiece;
        if (h.from) {
            memcpy((char*)h.host + off, (const char*)h.from + off, (size_t)bytes);
            return cudaSuccess;
        }
        const int s = worker * kSlots + (turn++ % kSlots);
        char* slot = (char*)c->pin + s * kPiece;
        cudaError_t e = cudaEventSynchronize(c->pin_ev[s]);  // the slot's last copy is over
        if (e != cudaSuccess) return e;
        if (up) {
            memcpy(slot, (const char*)h.host + off, (size_t)bytes);
            e = cudaMemcpyAsync((char*)h.dev + off, slot, (size_t)bytes, cudaMemcpyHostToDevice, stream);
            if (e == cudaSuccess) e = cudaEventRecord(c->pin_ev[s], stream);
            return e;
        }
        e = cudaMemcpyAsync(slot, (const char*)h.dev + off, (size_t)bytes, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaEventRecord(c->pin_ev[s], stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(c->pin_ev[s]);
        if (e == cudaSuccess) memcpy((char*)h.host + off, slot, (size_t)bytes);
        return e;
    }
    void work(int worker) {
        cudaError_t e = cudaSetDevice(c->device);
        const int64_t total = pieces();
        int turn = 0;
        for (int64_t k; e == cudaSuccess && error == (int)cudaSuccess && (k = next++) < total;) e = piece(k, worker, turn);
        if (e != cudaSuccess) error = (int)e;
    }
};

}  // namespace

int host_copy(hann_ctx* c, const HostCopy* list, int n, bool up, cudaStream_t stream) {
    int64_t total = 0;
    bool plain = false;
    for (int i = 0; i < n; i++) {
        total += list[i].bytes;
        plain = plain || !pageable(list[i].host);
    }
    cudaError_t e = cudaSuccess;
    if (plain || total < 2 * kPiece || !slots(c)) {
        // page-locked or device memory, small copies, no memory for the slots: the driver's own copy
        for (int i = 0; i < n && e == cudaSuccess; i++) {
            if (list[i].from) memcpy(list[i].host, list[i].from, (size_t)list[i].bytes);
            else if (up) e = cudaMemcpyAsync(list[i].dev, list[i].host, (size_t)list[i].bytes, cudaMemcpyDefault, stream);
            else e = cudaMemcpyAsync(list[i].host, list[i].dev, (size_t)list[i].bytes, cudaMemcpyDefault, stream);
        }
    } else {
        Job job;
        job.c = c;
        job.list = list;
        job.n = n;
        job.up = up;
        job.stream = stream;
        std::thread helper[kThreads - 1];
        const int64_t pieces = job.pieces();
        const unsigned cores = std::thread::hardware_concurrency();
        for (int w = 1; w < kThreads && w < pieces && (cores == 0 || w < (int)cores); w++) {
            try {
                helper[w - 1] = std::thread([&job, w] { job.work(w); });
            } catch (...) {
                break;  // fewer threads share the same pieces out
            }
        }
        job.work(0);
        for (std::thread& t : helper)
            if (t.joinable()) t.join();
        e = (cudaError_t)job.error.load();
    }
    if (e != cudaSuccess) {
        c->err = std::string("host copy: ") + cudaGetErrorString(e);
        return HANN_ECUDA;
    }
    return HANN_OK;
}

void host_copy_release(hann_ctx* c) {
    for (cudaEvent_t& ev : c->pin_ev)
        if (ev) {
            cudaEventSynchronize(ev);
            cudaEventDestroy(ev);
            ev = nullptr;
        }
    if (c->pin) cudaFreeHost(c->pin);
    c->pin = nullptr;
}
