// Stream-ordered device scratch that survives the call.
//
// The device's stream-ordered pool hands its memory back to the system whenever the host waits for the GPU, so a
// program that waits after every call paid for mapping the next call's scratch anew: a call of 255 rays took
// 267 us alone against 49 among others, now 82; a step of 1e6 rays with staged emission (1 GB of scratch) 4.37 ms
// against 1.23, now 1.22.  Blocks of finished calls are therefore kept, at most kKeep bytes in kBlocks blocks per
// device, while a grid or ray plan of that device is alive, and reused.
//   * A kept block is only given to a call on the stream that used it last.  It makes room for blocks of
//     that stream, and for those of others when it was not used during the last kStale releases and its work
//     has ended (a stream at rest, or destroyed): no call waits for another stream's work because of its scratch, and
//     streams that take turns do not displace each other's blocks.  What finds no room goes back to the
//     pool, as all blocks did before.  The stream waits for the event recorded at a block's release, so
//     that a new stream that got a destroyed one's handle is ordered too.
//   * Under stream capture blocks come from and go to the allocator, as graph nodes: a graph's scratch is its own.
//   * The list of kept blocks is a fixed array: nothing here allocates on the host or throws.
//   * When an allocation of this library fails the kept blocks are released and it is tried again; for other
//     allocators of the program there is hg_release_scratch.
// (Kept blocks are freed by cudaFreeAsync throughout: after cudaFree the pool went on counting them as used.)
#include "scratch.h"

#include "hg_internal.h"

#include <cstdint>
#include <mutex>

namespace hg {
namespace {

constexpr size_t kKeep = (size_t)2 << 30;

constexpr int kBlocks = 64;  // kept blocks of a device
constexpr int kStale = 128;  // releases (some tens of calls)

struct Idle {
    Scratch s;
    cudaStream_t stream;
    uint64_t turn;  // the device's count of releases when it came
};
// Blocks of a device, oldest first.
struct Blocks {
    Idle v[kBlocks];
    int n = 0;
    Scratch remove(int i) {
        const Scratch s = v[i].s;
        for (n--; i < n; i++) v[i] = v[i + 1];
        return s;
    }
};
struct Device {
    Blocks idle;
    size_t kept = 0;
    uint64_t turn = 0;  // blocks released so far
    int users = 0;
};
std::mutex g_mtx;
constexpr int kDevices = 64;
Device g_dev[kDevices];

// (A failed query leaves an error behind that the next launch's check would take for its own: cleared, here and below.)
bool ok(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
}

bool capturing(cudaStream_t stream) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return !ok(cudaStreamIsCapturing(stream, &st)) || st != cudaStreamCaptureStatusNone;
}

// Queries and waits inside do not break a capture that another thread has under way.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Whether the work of a block's last use has ended.
bool ended(const Scratch &s) {
    const RelaxedCapture relaxed;
    return ok(cudaEventQuery(s.done));
}

// Take a device's idle blocks (under the lock).
Blocks take_all(Device &d) {
    const Blocks out = d.idle;
    d.idle.n = 0;
    d.kept = 0;
    return out;
}

// Free a block in the order of `stream`, whose own it was or whose work has ended.
void release_in(const Scratch &s, cudaStream_t stream) {
    cudaStreamWaitEvent(stream, s.done, 0);
    cudaFreeAsync(s.p, stream);
    cudaEventDestroy(s.done);
}

// Free a device's kept blocks once their last uses have ended (the host waits), and have the pool give their memory back to
// the system, on a stream of its own; false when there were none.
bool release_kept(int device) {
    Blocks all;
    {
        std::lock_guard<std::mutex> lock(g_mtx);
        all = take_all(g_dev[device]);
    }
    if (all.n == 0) return false;
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != device) cudaSetDevice(device);
    {
        const RelaxedCapture relaxed;
        cudaStream_t stream = nullptr;
        if (!ok(cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking))) stream = nullptr;
        for (int i = 0; i < all.n; i++) {
            ok(cudaEventSynchronize(all.v[i].s.done));
            release_in(all.v[i].s, stream);
        }
        ok(cudaStreamSynchronize(stream));
        if (stream) cudaStreamDestroy(stream);
    }
    if (cur != device) cudaSetDevice(cur);
    return true;
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
        if (!ok(e)) s.p = nullptr;
        return e;
    }
    {
        std::lock_guard<std::mutex> lock(g_mtx);
        Device &d = g_dev[device];
        int best = -1;
        for (int i = 0; i < d.idle.n; i++) {
            const Idle &c = d.idle.v[i];
            // not a block that several smaller ones could be made of
            if (c.stream == stream && c.s.bytes >= bytes && c.s.bytes / 4 <= bytes + ((size_t)1 << 20) &&
                (best < 0 || c.s.bytes < d.idle.v[best].s.bytes))
                best = i;
        }
        if (best >= 0) {
            s = d.idle.remove(best);
            d.kept -= s.bytes;
        }
    }
    if (s.p) {
        e = cudaStreamWaitEvent(stream, s.done, 0);
        if (!ok(e)) scratch_put(s, stream);
        return e;
    }
    e = cudaMallocAsync(&s.p, bytes, stream);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        if (release_kept(device)) e = cudaMallocAsync(&s.p, bytes, stream);
    }
    if (!ok(e)) {
        s = Scratch();
        return e;
    }
    s.bytes = bytes;
    if (!ok(cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming))) s.done = nullptr;  // not kept, then
    return cudaSuccess;
}

void scratch_put(Scratch &s, cudaStream_t stream) {
    if (!s.p) return;
    int device = -1;
    Blocks drop;
    bool keep = s.done && !capturing(stream) && cudaGetDevice(&device) == cudaSuccess && device < kDevices &&
                s.bytes <= kKeep && ok(cudaEventRecord(s.done, stream));
    if (keep) {
        std::lock_guard<std::mutex> lock(g_mtx);
        Device &d = g_dev[device];
        keep = d.users > 0;
        if (keep) {
            d.turn++;
            for (int i = 0; i < d.idle.n && (d.idle.n == kBlocks || d.kept + s.bytes > kKeep);) {
                const Idle &c = d.idle.v[i];
                if (c.stream != stream && !(d.turn - c.turn > kStale && ended(c.s))) {
                    i++;
                    continue;
                }
                drop.v[drop.n].s = d.idle.remove(i);
                d.kept -= drop.v[drop.n++].s.bytes;
            }
            keep = d.idle.n < kBlocks && d.kept + s.bytes <= kKeep;
        }
        if (keep) {
            d.idle.v[d.idle.n++] = {s, stream, d.turn};
            d.kept += s.bytes;
        }
    }
    if (!keep) {
        cudaFreeAsync(s.p, stream);
        if (s.done) cudaEventDestroy(s.done);
    }
    for (int i = 0; i < drop.n; i++) release_in(drop.v[i].s, stream);
    s = Scratch();
}

void scratch_users(int device, int delta) {
    if (device < 0 || device >= kDevices) return;
    bool last;
    {
        std::lock_guard<std::mutex> lock(g_mtx);
        g_dev[device].users += delta;
        last = g_dev[device].users <= 0;
    }
    if (last) release_kept(device);
}

cudaError_t device_malloc(void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    int device = -1;
    if (e == cudaErrorMemoryAllocation && cudaGetDevice(&device) == cudaSuccess && device < kDevices) {
        cudaGetLastError();
        if (release_kept(device)) e = cudaMalloc(p, bytes);
    }
    ok(e);
    return e;
}

}  // namespace hg

extern "C" hg_status hg_release_scratch(void) {
    int device = -1;
    const cudaError_t e = cudaGetDevice(&device);
    if (!hg::ok(e)) {
        hg::set_error("hg_release_scratch: %s", cudaGetErrorString(e));
        return HG_ECUDA;
    }
    if (device < hg::kDevices) hg::release_kept(device);
    return HG_OK;
}
