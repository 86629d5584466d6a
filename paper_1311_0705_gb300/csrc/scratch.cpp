// Stream-ordered device scratch that survives the call.
//
// The device's stream-ordered pool hands its memory back to the system whenever the host waits for the GPU, so a
// program that waits after every call paid for mapping the next call's scratch anew: a call of 255 rays took
// 267 us alone against 49 among others, now 82; a step of 1e6 rays with staged emission (1 GB of scratch) 4.37 ms
// against 1.23, now 1.22.  Blocks of finished calls are therefore kept, at most kKeep bytes per device, while a grid or
// ray plan of that device is alive, and reused.
//   * A kept block is only given to a call on the stream that used it last (no call ever waits for another
//     stream's work because of its scratch), and the stream waits for the event recorded at its release, so
//     that a new stream that got a destroyed one's handle is ordered too.
//   * Under stream capture blocks come from and go to the allocator, as graph nodes: a graph's scratch is its own.
//   * When an allocation fails the kept blocks are released and it is tried again.
// (Kept blocks are freed by cudaFreeAsync throughout: after cudaFree the pool went on counting them as used.)
#include "scratch.h"

#include <mutex>
#include <vector>

namespace hg {
namespace {

constexpr size_t kKeep = (size_t)2 << 30;

struct Idle {
    Scratch s;
    int device;
    cudaStream_t stream;
};
std::mutex g_mtx;
std::vector<Idle> g_idle;  // oldest first
constexpr int kDevices = 64;
size_t g_kept[kDevices] = {};
int g_users[kDevices] = {};

bool capturing(cudaStream_t stream) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(stream, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone;
}

// Take the idle blocks of a device out of the list (under the lock).
std::vector<Idle> take_all(int device) {
    std::vector<Idle> out, rest;
    for (const Idle &i : g_idle) (i.device == device ? out : rest).push_back(i);
    g_idle.swap(rest);
    g_kept[device] = 0;
    return out;
}

// Free a block once its last use has ended, in `stream`'s order.
void release_in(const Scratch &s, cudaStream_t stream) {
    cudaStreamWaitEvent(stream, s.done, 0);
    cudaFreeAsync(s.p, stream);
    cudaEventDestroy(s.done);
}

}  // namespace

cudaError_t scratch_get(Scratch &s, size_t bytes, cudaStream_t stream) {
    s = Scratch();
    int device = -1;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (bytes < 256) bytes = 256;
    if (device >= kDevices || capturing(stream)) {
        e = cudaMallocAsync(&s.p, bytes, stream);
        s.bytes = e == cudaSuccess ? bytes : 0;
        if (e != cudaSuccess) s.p = nullptr;
        return e;
    }
    {
        std::lock_guard<std::mutex> lock(g_mtx);
        size_t best = g_idle.size();
        for (size_t i = 0; i < g_idle.size(); i++) {
            const Idle &c = g_idle[i];
            // not a block that several smaller ones could be made of
            if (c.device == device && c.stream == stream && c.s.bytes >= bytes && c.s.bytes / 4 <= bytes + ((size_t)1 << 20) &&
                (best == g_idle.size() || c.s.bytes < g_idle[best].s.bytes))
                best = i;
        }
        if (best < g_idle.size()) {
            s = g_idle[best].s;
            g_kept[device] -= s.bytes;
            g_idle.erase(g_idle.begin() + (std::ptrdiff_t)best);
        }
    }
    if (s.p) {
        e = cudaStreamWaitEvent(stream, s.done, 0);
        if (e != cudaSuccess) scratch_put(s, stream);
        return e;
    }
    e = cudaMallocAsync(&s.p, bytes, stream);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        std::vector<Idle> all;
        {
            std::lock_guard<std::mutex> lock(g_mtx);
            all = take_all(device);
        }
        for (const Idle &i : all) release_in(i.s, stream);
        if (!all.empty()) cudaStreamSynchronize(stream);
        e = cudaMallocAsync(&s.p, bytes, stream);
    }
    if (e != cudaSuccess) {
        s = Scratch();
        return e;
    }
    s.bytes = bytes;
    if (cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        s.done = nullptr;  // not kept, then
    }
    return cudaSuccess;
}

void scratch_put(Scratch &s, cudaStream_t stream) {
    if (!s.p) return;
    int device = -1;
    std::vector<Scratch> drop;
    bool keep = s.done && !capturing(stream) && cudaGetDevice(&device) == cudaSuccess && device < kDevices &&
                s.bytes <= kKeep && cudaEventRecord(s.done, stream) == cudaSuccess;
    if (keep) {
        std::lock_guard<std::mutex> lock(g_mtx);
        keep = g_users[device] > 0;
        if (keep) {
            for (size_t i = 0; i < g_idle.size() && g_kept[device] + s.bytes > kKeep;) {
                if (g_idle[i].device != device) {
                    i++;
                    continue;
                }
                drop.push_back(g_idle[i].s);
                g_kept[device] -= g_idle[i].s.bytes;
                g_idle.erase(g_idle.begin() + (std::ptrdiff_t)i);
            }
            g_idle.push_back({s, device, stream});
            g_kept[device] += s.bytes;
        }
    }
    if (!keep) {
        cudaFreeAsync(s.p, stream);
        if (s.done) cudaEventDestroy(s.done);
    }
    for (const Scratch &d : drop) release_in(d, stream);
    s = Scratch();
}

void scratch_users(int device, int delta) {
    if (device < 0 || device >= kDevices) return;
    std::vector<Idle> all;
    {
        std::lock_guard<std::mutex> lock(g_mtx);
        g_users[device] += delta;
        if (g_users[device] <= 0) all = take_all(device);
    }
    if (all.empty()) return;
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != device) cudaSetDevice(device);
    for (const Idle &i : all) {
        cudaEventSynchronize(i.s.done);
        cudaFreeAsync(i.s.p, 0);
        cudaEventDestroy(i.s.done);
    }
    if (cur != device) cudaSetDevice(cur);
}

}  // namespace hg
