// Device memory kept by a context between calls (MemPool in common.cuh).
#include <algorithm>

#include "common.cuh"

namespace sw {

namespace {
thread_local MemPool* t_pool = nullptr;
size_t rounded(size_t n) {
    const size_t unit = n >= (1u << 20) ? (size_t)1 << 16 : 512;
    return (n + unit - 1) / unit * unit;
}

// Every pool of the process, so that a context that runs out of memory can ask back what the others keep. Neither lock is
// held while the other is waited for in the opposite order: a pool never looks at the list under its own lock.
std::mutex g_pools_lock;
std::vector<MemPool*>& pools() {
    static auto* v = new std::vector<MemPool*>;  // never destroyed: a context may outlive the library's statics
    return *v;
}

}  // namespace

MemPool::MemPool() {
    std::lock_guard<std::mutex> l(g_pools_lock);
    pools().push_back(this);
}

MemPool::~MemPool() {
    {
        std::lock_guard<std::mutex> l(g_pools_lock);
        std::vector<MemPool*>& v = pools();
        v.erase(std::find(v.begin(), v.end(), this));
    }
    trim(0);
    for (const Block& b : live_) cudaFree(b.p);
}

size_t MemPool::cached() {
    std::lock_guard<std::mutex> l(m_);
    return cached_;
}

cudaError_t MemPool::allocate(void** p, size_t n) {
    cudaError_t e = cudaMalloc(p, n);
    const auto again = [&] {
        cudaGetLastError();
        e = cudaMalloc(p, n);
    };
    if (e == cudaErrorMemoryAllocation) {
        trim(0);
        again();
    }
    if (e == cudaErrorMemoryAllocation && spare()) {
        trim(0);
        again();
    }
    if (e == cudaErrorMemoryAllocation) {
        {
            std::lock_guard<std::mutex> l(g_pools_lock);
            for (MemPool* q : pools()) q->trim(0);
        }
        again();
    }
    return e;
}

cudaError_t MemPool::alloc(void** p, size_t bytes) {
    const size_t n = rounded(bytes > 0 ? bytes : 1);
    {
        std::lock_guard<std::mutex> l(m_);
        size_t best = free_.size();
        for (size_t i = 0; i < free_.size(); ++i)
            if (free_[i].bytes >= n && free_[i].bytes / 5 * 4 <= n && (best == free_.size() || free_[i].bytes < free_[best].bytes)) best = i;
        if (best < free_.size()) {
            *p = free_[best].p;
            cached_ -= free_[best].bytes;
            live_.push_back(free_[best]);
            free_.erase(free_.begin() + (std::ptrdiff_t)best);
            return cudaSuccess;
        }
    }
    const cudaError_t e = allocate(p, n);
    if (e != cudaSuccess) {
        *p = nullptr;
        return e;
    }
    std::lock_guard<std::mutex> l(m_);
    live_.push_back(Block{*p, n, 0});
    return cudaSuccess;
}

void MemPool::free(void* p) {
    if (!p) return;
    {
        std::lock_guard<std::mutex> l(m_);
        for (size_t i = 0; i < live_.size(); ++i) {
            if (live_[i].p != p) continue;
            Block b = live_[i];
            live_.erase(live_.begin() + (std::ptrdiff_t)i);
            if (b.bytes > LIMIT - cached_) break;
            b.epoch = epoch_;
            cached_ += b.bytes;
            free_.push_back(b);
            return;
        }
    }
    cudaFree(p);
}

void MemPool::trim(int keep) {
    std::lock_guard<std::mutex> l(m_);
    size_t n = 0;
    for (const Block& b : free_) {
        if (keep > 0 && epoch_ - b.epoch < keep) {
            free_[n++] = b;
        } else {
            cached_ -= b.bytes;
            cudaFree(b.p);  // waits for the device: work that still uses the block's former contents is done by then
        }
    }
    free_.resize(n);
}

void MemPool::end_of_call() {
    {
        std::lock_guard<std::mutex> l(m_);
        ++epoch_;
    }
    trim(KEEP);
}

PoolScope::PoolScope(MemPool* p) : before_(t_pool) { t_pool = p; }
PoolScope::~PoolScope() { t_pool = before_; }

cudaError_t dev_alloc_bytes(void** p, size_t bytes) { return t_pool ? t_pool->alloc(p, bytes) : cudaMalloc(p, bytes); }
void dev_free(void* p) {
    if (!p) return;
    if (t_pool) t_pool->free(p);
    else cudaFree(p);
}
bool dev_room(size_t bytes, bool give_up) {
    const auto fits = [&] {
        size_t free_b = 0, total_b = 0;
        cudaMemGetInfo(&free_b, &total_b);
        return bytes <= free_b + (t_pool ? t_pool->cached() : 0);
    };
    return fits() || (give_up && t_pool && t_pool->spare() && fits());
}

}  // namespace sw
