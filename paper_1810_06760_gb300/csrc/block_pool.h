// Idle blocks.  A released device or pinned block goes to a process-wide pool, per device, and serves a later
// request of nearly its size: cudaMalloc, cudaMallocHost and their frees took 1.2 of the 1.8 ms of a small solve
// and 10-25 ms of a large one (about 30 buffers, some of gigabytes).  Like cudaFree, whose implicit device
// synchronisation ordered every reuse, a block released since the device was last known to be idle is handed out
// only after a device synchronisation (one for all such blocks), so any stream and thread may release and take.
// Idle blocks are bounded (the largest go first), are given back when an allocation fails or would pass the caller's
// bound, when the bound is set, on request, and when the last model or beam set is destroyed.  Calls that need neither (the transform
// alone) release their scratch with no such end in sight: then the bound is a small one.
//
// Host code without CUDA types, so that several devices can be tested on a machine without any.  Rt is the runtime:
//   static int device(); static bool synchronize(); static void free_device(void *); static void free_host(void *);
// where synchronize waits for the current device.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <iterator>
#include <map>
#include <mutex>

namespace fga {

template <class Rt> class BlockPool {
    struct Block {
        void *p;
        bool dirty;
        int dev;   // device whose work may still use a dirty block
    };
    using Blocks = std::multimap<size_t, Block>;
    struct Device {
        Blocks blocks;
        size_t bytes = 0;
    };
    const size_t dev_max, alone_max, host_max;   // alone: with no model or beam set alive
    std::mutex mu;
    std::map<int, Device> dev;
    Blocks host;
    size_t host_bytes = 0;
    std::atomic<int64_t> &in_use;   // device bytes in use, kept with the idle ones under the lock
    int objects = 0;                // models and beam sets alive

    size_t total() const {
        size_t t = 0;
        for (const auto &d : dev) t += d.second.bytes;
        return t;
    }
    // a block of at least need bytes, at most an eighth larger
    void *take(Blocks &c, size_t &bytes, size_t need, size_t *size) {
        auto it = c.lower_bound(need);
        if (it == c.end() || it->first > need + need / 8 + 4096) return nullptr;
        if (it->second.dirty) {
            const int d = Rt::device();
            if (it->second.dev != d || !Rt::synchronize()) return nullptr;   // no reuse
            for (auto &kv : dev[d].blocks) kv.second.dirty = false;
            for (auto &kv : host)
                if (kv.second.dev == d) kv.second.dirty = false;
        }
        void *p = it->second.p;
        *size = it->first;
        bytes -= it->first;
        c.erase(it);
        return p;
    }
    void free_largest(Device &d) {
        auto it = std::prev(d.blocks.end());
        Rt::free_device(it->second.p);
        d.bytes -= it->first;
        d.blocks.erase(it);
    }
    // free idle device blocks, largest first, until at most keep bytes are left on all devices together
    void trim_locked(size_t keep) {
        while (total() > keep) {
            Device *best = nullptr;
            for (auto &d : dev)
                if (!d.second.blocks.empty() &&
                    (!best || std::prev(d.second.blocks.end())->first > std::prev(best->blocks.end())->first))
                    best = &d.second;
            if (!best) break;
            free_largest(*best);
        }
    }
    void release_locked() {
        trim_locked(0);
        for (auto &kv : host) Rt::free_host(kv.second.p);
        host.clear();
        host_bytes = 0;
    }

public:
    BlockPool(size_t dev_max_, size_t alone_max_, size_t host_max_, std::atomic<int64_t> &used)
        : dev_max(dev_max_), alone_max(alone_max_), host_max(host_max_), in_use(used) {}

    // idle bytes of one device: a reserve for allocations on that device only
    size_t idle_bytes(int d) {
        std::lock_guard<std::mutex> lk(mu);
        auto it = dev.find(d);
        return it == dev.end() ? 0 : it->second.bytes;
    }
    void *take_device(int d, size_t need, size_t *size) {
        std::lock_guard<std::mutex> lk(mu);
        Device &D = dev[d];
        void *p = take(D.blocks, D.bytes, need, size);
        if (p) in_use += (int64_t)*size;
        return p;
    }
    void *take_host(size_t need, size_t *size) {
        std::lock_guard<std::mutex> lk(mu);
        return take(host, host_bytes, need, size);
    }
    void put_device(void *p, size_t bytes, int d) {
        std::lock_guard<std::mutex> lk(mu);
        const size_t max = objects > 0 ? dev_max : alone_max;
        if (bytes > max) {
            Rt::free_device(p);
        } else {
            trim_locked(max - bytes);
            Device &D = dev[d];
            D.blocks.emplace(bytes, Block{p, true, d});
            D.bytes += bytes;
        }
        in_use -= (int64_t)bytes;
    }
    void put_host(void *p, size_t bytes, int d) {
        std::lock_guard<std::mutex> lk(mu);
        if (host_bytes + bytes > host_max) {
            Rt::free_host(p);
            return;
        }
        host.emplace(bytes, Block{p, true, d});
        host_bytes += bytes;
    }
    void trim(size_t keep) {
        std::lock_guard<std::mutex> lk(mu);
        trim_locked(keep);
    }
    // all idle blocks of one device (an allocation on it failed; blocks of others would not help it)
    void trim_device(int d) {
        std::lock_guard<std::mutex> lk(mu);
        Device &D = dev[d];
        while (!D.blocks.empty()) free_largest(D);
    }
    // a model or beam set created (1) or destroyed (-1); with the last one the pool is emptied
    void object(int d) {
        std::lock_guard<std::mutex> lk(mu);
        objects += d;
        if (objects <= 0) release_locked();
    }
    // every idle block, whatever is alive
    void release() {
        std::lock_guard<std::mutex> lk(mu);
        release_locked();
    }
};

}  // namespace fga
