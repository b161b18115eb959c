// staging.h -- host memory for descriptors that a call copies to the device asynchronously.
#pragma once

#include <cstddef>
#include <memory>
#include <vector>

namespace qs {

// Blocks of host memory, one per copy.  cudaMemcpyAsync from pageable memory may still read its source after
// it returned (always so where the GPU reads host memory itself), so a block is handed out again only
// after wait(), which waits for every copy issued so far: when all are in use, and when the ring goes
// away, unless idle() has said that the caller has waited.
template <typename Wait> class StagingRing {
public:
    StagingRing(size_t bytes, size_t blocks, Wait wait) : bytes_(bytes), wait_(wait) { ring_.reserve(blocks); }
    StagingRing(const StagingRing &) = delete;
    StagingRing &operator=(const StagingRing &) = delete;
    ~StagingRing()
    {
        if (used_) wait_();
    }
    // A block that no copy is reading.
    void *next()
    {
        if (used_ == ring_.capacity()) {
            wait_();
            used_ = 0;
        }
        if (used_ == ring_.size()) ring_.emplace_back(new unsigned char[bytes_]);
        return ring_[used_++].get();
    }
    void idle() { used_ = 0; }

private:
    const size_t bytes_;
    Wait wait_;
    size_t used_ = 0;
    std::vector<std::unique_ptr<unsigned char[]>> ring_;
};

}  // namespace qs
