// vbq_error_words.h — how the calls that validate on the device (vbq_quantize,
// vbq_pack) hear of an error. Host code only.
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <cuda_runtime_api.h>

namespace vbq {

// Two error words of one call, in pinned host memory: a validating kernel
// stores to them only on an error, and the host reads them once it has
// synchronised, without a copy or an allocation per call. The words come from
// one page per device, shared by all threads (64 calls at a time, one 64-byte
// line each, given back when the call ends); a call beyond those allocates its
// own. A page belongs to its device's context, so a reset of one device takes
// no other device's words away.
class ErrorWords {
public:
    ErrorWords() = default;
    ErrorWords(const ErrorWords&) = delete;
    ErrorWords& operator=(const ErrorWords&) = delete;
    // The words may be another call's next: a kernel of this one that has not
    // been synchronised with (an error on the way out) is waited for first.
    ~ErrorWords() {
        if (armed_) cudaStreamSynchronize(stream_);
        if (slot_ >= 0) {
            std::lock_guard<std::mutex> lock(mu_);
            pages_[dev_].used &= ~(1ull << slot_);
        } else if (w_) {
            cudaFreeHost(w_);
        }
    }
    cudaError_t get(cudaStream_t stream) {
        stream_ = stream;
        const cudaError_t ed = cudaGetDevice(&dev_);
        if (ed != cudaSuccess) return ed;
        if (dev_ >= 0 && dev_ < MAX_DEVICES) {
            std::lock_guard<std::mutex> lock(mu_);
            Page& page = pages_[dev_];
            if (!page.words) {
                const cudaError_t e = host_words(&page.words, LINES * LINE_WORDS * sizeof(uint32_t));
                if (e != cudaSuccess) return e;
            }
            for (int i = 0; i < LINES && slot_ < 0; ++i)
                if (!(page.used >> i & 1)) slot_ = i;
            if (slot_ >= 0) {
                page.used |= 1ull << slot_;
                w_ = page.words + LINE_WORDS * slot_;
            }
        }
        if (!w_) {
            const cudaError_t e = host_words(&w_, LINE_WORDS * sizeof(uint32_t));
            if (e != cudaSuccess) return e;
        }
        w_[0] = w_[1] = 0;
        return cudaSuccess;
    }
    uint32_t* arm(int i) {                  // for a kernel about to be launched on the stream
        armed_ = true;
        return w_ + i;
    }
    cudaError_t settle() {                  // wait for the stream; the words can be read
        const cudaError_t e = cudaStreamSynchronize(stream_);
        armed_ = false;
        return e;
    }
    bool set(int i) const { return static_cast<volatile uint32_t*>(w_)[i] != 0; }

private:
    static constexpr int MAX_DEVICES = 64, LINES = 64, LINE_WORDS = 16;
    struct Page {
        uint32_t* words;
        uint64_t used;                      // bit i: line i is taken
    };
    static cudaError_t host_words(uint32_t** p, size_t bytes) {
        return cudaHostAlloc(reinterpret_cast<void**>(p), bytes, cudaHostAllocPortable | cudaHostAllocMapped);
    }
    inline static std::mutex mu_;
    inline static Page pages_[MAX_DEVICES] = {};
    uint32_t* w_ = nullptr;
    int slot_ = -1, dev_ = 0;
    cudaStream_t stream_ = nullptr;
    bool armed_ = false;
};

}  // namespace vbq
