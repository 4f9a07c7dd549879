// Uploads from ordinary (pageable) host memory for a decryption.
//
// The driver stages such a copy through one thread at 20 GB/s, on a host whose bus does 54.  Here the calling thread and a helper share the
// pieces out, each with two page-locked slots of its own: a thread fills one slot while the copy engine empties the other.
//
// The helper starts with the list and ends with it, which costs as much as a few MiB of copying and more where the host's cores were
// asleep.  Decryption of k ciphertexts at N = 2^16, L = 4 (4 MiB each), us with the driver's copy / with the helper:
//   called in a loop: k = 1 365 / 409, 2 601 / 635, 3 844 / 830, 4 1078 / 1016, 5 1328 / 1203, 7 1809 / 1591, 8 2054 / 1789
//   after 5 ms without a call: 1 384 / 411, 4 1116 / 1053, 7 2079 / 1598;  after 50 ms: 4 1677 / 1281, 7 3075 / 1939
// hence from 16 MiB on.  (Where another library's threads still spin on every core the two wait for one: right after a multi-threaded
// factorisation seven take 1874 / 2261.)  Three helpers gave 1591 at seven in a loop, and 690 in place of 384 for one after 5 ms.
// Downloads and the copies of an encryption, 4 MiB and less, go through the driver: with helpers an encryption took 665 in place of 523
// after 5 ms, and the scores of seven ciphertexts 100 more.
#include <atomic>
#include <cstring>
#include <string>
#include <thread>

#include "internal.h"

namespace {

constexpr int kThreads = 2, kSlots = 2;
constexpr int64_t kPiece = 512 << 10, kShared = 16 << 20;
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
    cudaStream_t stream;
    std::atomic<int64_t> next{0};
    std::atomic<int> error{(int)cudaSuccess};

    static int64_t pieces_of(const HostCopy& h) { return (h.bytes + kPiece - 1) / kPiece; }
    // false when the list has no piece k
    bool piece(int64_t k, int worker, int& turn, cudaError_t& e) {
        int i = 0;
        for (; i < n && k >= pieces_of(list[i]); i++) k -= pieces_of(list[i]);
        if (i == n) return false;
        const HostCopy& h = list[i];
        const int64_t off = k * kPiece, bytes = h.bytes - off < kPiece ? h.bytes - off : kPiece;
        const int s = worker * kSlots + (turn++ % kSlots);
        char* slot = (char*)c->pin + s * kPiece;
        e = cudaEventSynchronize(c->pin_ev[s]);  // the slot's last copy is over
        if (e != cudaSuccess) return true;
        memcpy(slot, (const char*)h.host + off, (size_t)bytes);
        e = cudaMemcpyAsync((char*)h.dev + off, slot, (size_t)bytes, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaEventRecord(c->pin_ev[s], stream);
        return true;
    }
    void work(int worker) {
        cudaError_t e = cudaSetDevice(c->device);
        int turn = 0;
        while (e == cudaSuccess && error == (int)cudaSuccess && piece(next++, worker, turn, e)) {
        }
        if (e != cudaSuccess) error = (int)e;
    }
};

}  // namespace

int host_upload(hann_ctx* c, const HostCopy* list, int n, cudaStream_t stream) {
    int64_t total = 0;
    for (int i = 0; i < n; i++) total += list[i].bytes;
    bool shared = total >= kShared;
    for (int i = 0; i < n && shared; i++) shared = pageable(list[i].host);
    cudaError_t e = cudaSuccess;
    if (!shared || !slots(c)) {
        // small lists, page-locked or device memory, no memory for the slots: the driver's own copy
        for (int i = 0; i < n && e == cudaSuccess; i++) e = cudaMemcpyAsync(list[i].dev, list[i].host, (size_t)list[i].bytes, cudaMemcpyDefault, stream);
    } else {
        Job job;
        job.c = c;
        job.list = list;
        job.n = n;
        job.stream = stream;
        std::thread helper;
        try {
            helper = std::thread([&job] { job.work(1); });
        } catch (...) {
            // no thread to be had: this one copies every piece
        }
        job.work(0);
        if (helper.joinable()) helper.join();
        e = (cudaError_t)job.error.load();
    }
    if (e != cudaSuccess) {
        c->err = std::string("host upload: ") + cudaGetErrorString(e);
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
