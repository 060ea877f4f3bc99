// What the plans of a process share: device memory for their tables and packed weights, and the streams of
// gdws_forward_host.
//
// Device memory:  A cudaMalloc beyond a megabyte maps new memory, about a
// millisecond; a network builds dozens of plans.  Plans up to kPlanMemLargest bytes therefore share slabs: ranges of a slab
// are handed out first fit and come back when a plan is destroyed (after its device is idle).  A slab that holds no plan is
// kept only while it is the device's only empty one, and the last one goes with the device's last plan.  Plans up to
// kPlanMemAlone bytes make no slab: the driver serves them from what it has mapped already (a plan built and destroyed by
// itself, 16 -> 16 to 128 -> 128 channels: 450 us with a slab of its own), and a small layer does not hold 32 MB.
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "gdws_internal.h"

namespace gdws {

namespace {

constexpr size_t kSlabBytes = (size_t)32 << 20, kPlanMemLargest = (size_t)16 << 20, kPlanMemAlone = (size_t)512 << 10;

struct Slab {
    int device = 0;
    char *base = nullptr;
    std::map<size_t, size_t> free_ranges;      // offset -> bytes, merged
    bool empty() const { return free_ranges.size() == 1 && free_ranges.begin()->second == kSlabBytes; }
};

std::mutex g_lock;
std::vector<Slab> g_slabs;
std::vector<HostPipe *> g_pipes;               // those not in use
std::map<int, int> g_plans;                    // per device
constexpr int kKeepPipes = 2;

void destroy(HostPipe *p)
{
    if (p->in) cudaStreamDestroy(p->in);
    if (p->out) cudaStreamDestroy(p->out);
    if (p->begin) cudaEventDestroy(p->begin);
    for (cudaEvent_t e : p->copied) if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : p->computed) if (e) cudaEventDestroy(e);
    delete p;
}

char *take(Slab &s, size_t bytes)
{
    for (auto it = s.free_ranges.begin(); it != s.free_ranges.end(); ++it) {
        if (it->second < bytes) continue;
        const size_t off = it->first, rest = it->second - bytes;
        if (rest) s.free_ranges.emplace(off + bytes, rest);      // before anything is taken away: emplace may throw
        s.free_ranges.erase(off);
        return s.base + off;
    }
    return nullptr;
}

}  // namespace

// On the current device, which is `device`; `bytes` a multiple of 256.
cudaError_t plan_mem_alloc(int device, size_t bytes, void **out)
{
    *out = nullptr;
    if (bytes > kPlanMemLargest) return cudaMalloc(out, bytes);
    std::lock_guard<std::mutex> hold(g_lock);
    try {
        for (Slab &s : g_slabs)
            if (s.device == device && (*out = take(s, bytes))) return cudaSuccess;
        if (bytes <= kPlanMemAlone) return cudaMalloc(out, bytes);
        g_slabs.reserve(g_slabs.size() + 1);
        Slab s;
        s.device = device;
        s.free_ranges.emplace(0, kSlabBytes);
        const cudaError_t e = cudaMalloc((void **)&s.base, kSlabBytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return cudaMalloc(out, bytes);     // no room for a slab: the plan alone may fit
        }
        g_slabs.push_back(std::move(s));
        *out = take(g_slabs.back(), bytes);
        return cudaSuccess;
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

// The device (current) has finished all work that uses the memory.
void plan_mem_free(int device, void *ptr, size_t bytes)
{
    if (!ptr) return;
    std::lock_guard<std::mutex> hold(g_lock);
    for (size_t i = 0; i < g_slabs.size(); ++i) {
        Slab &s = g_slabs[i];
        if (s.device != device || (char *)ptr < s.base || (char *)ptr >= s.base + kSlabBytes) continue;
        const size_t off = (size_t)((char *)ptr - s.base);
        try {
            auto it = s.free_ranges.emplace(off, bytes).first;
            auto next = std::next(it);
            if (next != s.free_ranges.end() && off + bytes == next->first) {
                it->second += next->second;
                s.free_ranges.erase(next);
            }
            if (it != s.free_ranges.begin()) {
                auto prev = std::prev(it);
                if (prev->first + prev->second == off) {
                    prev->second += it->second;
                    s.free_ranges.erase(it);
                }
            }
        } catch (const std::bad_alloc &) {
            return;                            // the range stays unused until the process ends
        }
        int used = 0, empties = 0;
        for (const Slab &o : g_slabs)
            if (o.device == device) { if (o.empty()) ++empties; else ++used; }
        const int keep = used ? 1 : 0;
        for (size_t j = g_slabs.size(); j-- > 0 && empties > keep;)
            if (g_slabs[j].device == device && g_slabs[j].empty()) {
                cudaFree(g_slabs[j].base);
                g_slabs.erase(g_slabs.begin() + (long)j);
                --empties;
            }
        return;
    }
    cudaFree(ptr);
}

HostPipe *host_pipe_take(int device)
{
    {
        std::lock_guard<std::mutex> hold(g_lock);
        for (size_t i = 0; i < g_pipes.size(); ++i)
            if (g_pipes[i]->device == device) {
                HostPipe *p = g_pipes[i];
                g_pipes.erase(g_pipes.begin() + (long)i);
                return p;
            }
    }
    HostPipe *p = new (std::nothrow) HostPipe;
    if (!p) return nullptr;
    p->device = device;
    bool ok = cudaStreamCreateWithFlags(&p->in, cudaStreamNonBlocking) == cudaSuccess && cudaStreamCreateWithFlags(&p->out, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&p->begin, cudaEventDisableTiming) == cudaSuccess;
    for (cudaEvent_t &e : p->copied) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    for (cudaEvent_t &e : p->computed) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    if (ok) return p;
    cudaGetLastError();
    destroy(p);
    return nullptr;
}

void host_pipe_give(HostPipe *p)
{
    std::lock_guard<std::mutex> hold(g_lock);
    int kept = 0;
    for (const HostPipe *o : g_pipes) kept += o->device == p->device;
    try {
        if (kept < kKeepPipes && g_plans[p->device] > 0) {
            g_pipes.push_back(p);
            return;
        }
    } catch (const std::bad_alloc &) {
    }
    destroy(p);
}

void plan_count(int device, int change)
{
    std::lock_guard<std::mutex> hold(g_lock);
    try {
        if ((g_plans[device] += change) > 0) return;
    } catch (const std::bad_alloc &) {
        return;
    }
    for (size_t i = g_pipes.size(); i-- > 0;)
        if (g_pipes[i]->device == device) {
            destroy(g_pipes[i]);
            g_pipes.erase(g_pipes.begin() + (long)i);
        }
}

}  // namespace gdws
