// Process-wide resources of the host code, free of CUDA so that they can be tested without a GPU.
#pragma once
#include <stddef.h>

#include <atomic>
#include <mutex>

namespace gb300lbm {

// A fixed number of int words on one page that a kernel can write and the host read (mapped host memory),
// handed to contexts and taken back.  The page is allocated on the first take (a context of its own
// page would cost lbm_create a quarter of a millisecond) and kept: kWords words, never more.  A failed
// allocation is tried again on the next take.  Safe to call from several threads.
class StatusWords {
public:
    static constexpr int kWords = 1024;
    typedef int* (*AllocFn)(size_t bytes);   // nullptr on failure

    explicit constexpr StatusWords(AllocFn alloc) : alloc_(alloc) {}

    // a word no one else holds, or nullptr (all taken, or no page): the caller does without
    int* take() {
        std::lock_guard<std::mutex> hold(m_);
        if (!page_) page_ = alloc_(kWords * sizeof(int));
        if (!page_) return nullptr;
        for (int q = 0; q < kWords; ++q) {
            const int k = (next_ + q) % kWords;
            if (used_[k]) continue;
            used_[k] = true;
            next_ = (k + 1) % kWords;
            return page_ + k;
        }
        return nullptr;
    }
    void give(int* word) {
        if (!word) return;
        std::lock_guard<std::mutex> hold(m_);
        used_[word - page_] = false;
    }

private:
    AllocFn alloc_;
    std::mutex m_;
    int* page_ = nullptr;
    bool used_[kWords] = {};
    int next_ = 0;
};

// The result of a lookup (a pointer), kept once it is found: a lookup that fails (nullptr) is made again by
// the next caller.
template <class Fn, class Lookup> Fn kept_lookup(std::atomic<Fn>& kept, Lookup lookup) {
    Fn fn = kept.load(std::memory_order_acquire);
    if (!fn && (fn = lookup())) kept.store(fn, std::memory_order_release);
    return fn;
}

}  // namespace gb300lbm
