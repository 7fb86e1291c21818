// Blocks of device or page-locked host memory kept between calls: a call that
// needs working memory for its own duration takes a block and gives it back
// when its work has completed, instead of paying for an allocation (a
// one-segment inflation spent a third of its time in thirty of them). A pool
// keeps at most kKeep blocks and kBytes bytes, the ones given back last and only
// of sizes up to kMaxBlock, hands a block out on the device it was made on and
// to one taker at a time, and frees what it holds when the last robot, obstacle
// set and batch are gone. A block whose work may not have completed is freed,
// not kept. Obstacle sets take their memory here too.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <mutex>
#include <vector>

namespace ezo {

// While in scope, this thread's allocations and event queries are allowed
// beside a stream capture that any thread has begun in global mode; without
// it they fail and invalidate that capture, which they have no part in.
class RelaxedCapture {
 public:
  RelaxedCapture() { ok_ = cudaThreadExchangeStreamCaptureMode(&mode_) == cudaSuccess; }
  ~RelaxedCapture() {
    if (ok_) cudaThreadExchangeStreamCaptureMode(&mode_);
  }
  RelaxedCapture(const RelaxedCapture&) = delete;
  RelaxedCapture& operator=(const RelaxedCapture&) = delete;

 private:
  cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
  bool ok_;
};

// Waits for everything queued on device `dev`, whichever device is current;
// false when that could not be done.
inline bool device_idle(int dev) {
  int current = -1;
  bool ok = cudaGetDevice(&current) == cudaSuccess && (current == dev || cudaSetDevice(dev) == cudaSuccess);
  if (ok) {
    RelaxedCapture relaxed;
    ok = cudaDeviceSynchronize() == cudaSuccess;
  }
  if (current >= 0 && current != dev) cudaSetDevice(current);
  if (!ok) (void)cudaGetLastError();
  return ok;
}

class BlockPool {
 public:
  explicit BlockPool(bool host) : host_(host) {}

  // at least `bytes`, of the smallest that fit the one given back last; null
  // when there is no memory
  void* take(size_t bytes, cudaError_t* err) {
    int dev = 0;
    *err = cudaGetDevice(&dev);
    if (*err != cudaSuccess) return nullptr;
    size_t size = kMinBlock;
    while (size < bytes) size *= 2;
    {
      std::lock_guard<std::mutex> lock(mu_);
      size_t best = held_.size();
      for (size_t i = 0; i < held_.size(); ++i)
        if (held_[i].dev == dev && held_[i].bytes >= bytes && held_[i].bytes <= 4 * size &&
            (best == held_.size() || held_[i].bytes <= held_[best].bytes))
          best = i;
      if (best < held_.size()) {
        const Block b = held_[best];
        held_.erase(held_.begin() + best);
        total_ -= b.bytes;
        out_.push_back(b);
        return b.p;
      }
    }
    if (bytes > kMaxBlock) size = bytes;
    void* p = nullptr;
    RelaxedCapture relaxed;
    *err = host_ ? cudaMallocHost(&p, size) : cudaMalloc(&p, size);
    if (*err != cudaSuccess) {
      (void)cudaGetLastError();
      trim();
      *err = host_ ? cudaMallocHost(&p, size) : cudaMalloc(&p, size);
      if (*err != cudaSuccess) return nullptr;
    }
    std::lock_guard<std::mutex> lock(mu_);
    out_.push_back(Block{p, size, dev});
    return p;
  }

  // a block from take(); idle: its work has completed
  void give(void* p, bool idle) {
    if (!p) return;
    std::vector<Block> gone;
    {
      std::lock_guard<std::mutex> lock(mu_);
      size_t i = 0;
      while (i < out_.size() && out_[i].p != p) ++i;
      Block b{p, kMaxBlock + 1, 0};
      if (i < out_.size()) {
        b = out_[i];
        out_.erase(out_.begin() + i);
      }
      if (idle && b.bytes <= kMaxBlock) {
        held_.push_back(b);
        total_ += b.bytes;
        while (held_.size() > kKeep || total_ > kBytes) {  // the longest unused go
          total_ -= held_.front().bytes;
          gone.push_back(held_.front());
          held_.erase(held_.begin());
        }
      } else {
        gone.push_back(b);
      }
    }
    for (const Block& b : gone) release(b.p);
  }

  void trim() {
    std::vector<Block> gone;
    {
      std::lock_guard<std::mutex> lock(mu_);
      gone.swap(held_);
      total_ = 0;
    }
    for (const Block& b : gone) release(b.p);
  }

 private:
  struct Block {
    void* p;
    size_t bytes;
    int dev;
  };
  static constexpr size_t kMinBlock = 1 << 16, kMaxBlock = 32 << 20, kBytes = 64 << 20, kKeep = 8;
  void release(void* p) {
    RelaxedCapture relaxed;
    if (host_) cudaFreeHost(p);
    else cudaFree(p);
  }
  const bool host_;
  std::mutex mu_;
  std::vector<Block> held_, out_;
  size_t total_ = 0;
};

}  // namespace ezo
