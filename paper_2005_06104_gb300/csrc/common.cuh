// Shared device/host helpers of libgsetdvp: complex FP64 arithmetic, error
// handling, a caching device allocator and launch helpers.
#pragma once
#include <atomic>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <cstdint>
#include <cstdio>
#include <map>
#include <mutex>
#include <stdexcept>
#include <string>
#include <vector>

#include "../../include/gse_tdvp.h"

typedef double2 cplx;

__host__ __device__ __forceinline__ cplx mkc(double r, double i) { return make_double2(r, i); }
__host__ __device__ __forceinline__ cplx cadd(cplx a, cplx b) { return mkc(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ cplx csub(cplx a, cplx b) { return mkc(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ cplx cmul(cplx a, cplx b) {
  return mkc(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ cplx cconj(cplx a) { return mkc(a.x, -a.y); }
__host__ __device__ __forceinline__ cplx cscale(cplx a, double s) { return mkc(a.x * s, a.y * s); }
#ifdef __CUDACC__
// |a|^2 and a b with the fused operations written out, for kernels whose results have to keep their
// bits whatever the compiler contracts around them
__device__ __forceinline__ double cabs2_fma(cplx a) { return fma(a.x, a.x, __dmul_rn(a.y, a.y)); }
__device__ __forceinline__ cplx cmul_fma(cplx a, cplx b) {
  return mkc(fma(a.x, b.x, -__dmul_rn(a.y, b.y)), fma(a.x, b.y, __dmul_rn(a.y, b.x)));
}
#endif
// a += b * c
__host__ __device__ __forceinline__ void cfma(cplx& a, cplx b, cplx c) {
  a.x = fma(b.x, c.x, fma(-b.y, c.y, a.x));
  a.y = fma(b.x, c.y, fma(b.y, c.x, a.y));
}
// a += conj(b) * c
__host__ __device__ __forceinline__ void cfma_conj(cplx& a, cplx b, cplx c) {
  a.x = fma(b.x, c.x, fma(b.y, c.y, a.x));
  a.y = fma(b.x, c.y, fma(-b.y, c.x, a.y));
}
__host__ __device__ __forceinline__ double cabs2(cplx a) { return a.x * a.x + a.y * a.y; }

// Internal error type; converted to a tdvp_status at the C-ABI boundary.
struct TdvpError : public std::runtime_error {
  tdvp_status status;
  TdvpError(tdvp_status s, const std::string& m) : std::runtime_error(m), status(s) {}
};

#define TDVP_CUDA(call)                                                              \
  do {                                                                               \
    cudaError_t e_ = (call);                                                         \
    if (e_ != cudaSuccess) {                                                         \
      throw TdvpError(e_ == cudaErrorMemoryAllocation ? TDVP_ERR_OUT_OF_MEMORY        \
                                                      : TDVP_ERR_CUDA,               \
                      std::string(#call) + ": " + cudaGetErrorString(e_) + " at " +  \
                          __FILE__ + ":" + std::to_string(__LINE__));                \
    }                                                                                \
  } while (0)

// Process-wide count of kernel launches made by this library.  Every launch
// site is followed by exactly one TDVP_CHECK_LAUNCH, which bumps it.
extern std::atomic<long long> g_kernel_launches;
#define TDVP_CHECK_LAUNCH()                                             \
  do {                                                                  \
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);          \
    TDVP_CUDA(cudaGetLastError());                                      \
  } while (0)

inline void tdvp_require(bool ok, tdvp_status s, const std::string& msg) {
  if (!ok) throw TdvpError(s, msg);
}

// ---------------------------------------------------------------------------
// Caching device allocator: blocks are rounded up to a power of two (>= 4 KiB)
// and recycled per size class, so steady-state sweeps never call cudaMalloc.
// Blocks up to 256 KiB are cut from 4 MiB slabs: a new handle needs some hundred of them, and
// a cudaMalloc is 2 us alone but over 100 us while other threads launch (four chains created,
// stepped and destroyed: 170 ms of cudaMalloc in a pass).  Slabs go back with the pool.
class DevicePool {
 public:
  static constexpr size_t kSlab = size_t(4) << 20, kSlabBlock = size_t(256) << 10;
  void* get(size_t bytes) {
    size_t cls = size_class(bytes);
    auto& fl = free_[cls];
    if (!fl.empty()) {
      void* p = fl.back();
      fl.pop_back();
      return p;
    }
    if (cls <= kSlabBlock) {
      if (slab_left_ < cls) {
        // the rest of the old slab (multiples of 4 KiB) stays in use as smaller blocks
        for (size_t c = kSlabBlock; c >= 4096; c >>= 1)
          while (slab_left_ >= c) {
            free_[c].push_back(slab_);
            slab_ += c;
            slab_left_ -= c;
          }
        slab_ = static_cast<char*>(from_device(kSlab));
        slabs_.push_back(slab_);
        slab_left_ = kSlab;
      }
      void* p = slab_;
      slab_ += cls;
      slab_left_ -= cls;
      return p;
    }
    return from_device(cls);
  }
  void put(void* p, size_t bytes) {
    if (p) free_[size_class(bytes)].push_back(p);
  }
  // returns the cached blocks that are allocations of their own to the device
  void trim() {
    for (auto& kv : free_) {
      if (kv.first <= kSlabBlock) continue;
      for (void* p : kv.second) cudaFree(p);
      kv.second.clear();
    }
  }
  DevicePool() = default;
  DevicePool(const DevicePool&) = delete;
  DevicePool& operator=(const DevicePool&) = delete;
  ~DevicePool() {
    trim();
    for (void* p : slabs_) cudaFree(p);
  }
  // bytes held in the free lists (allocated from the device, not in use)
  size_t cached_bytes() const {
    size_t b = 0;
    for (const auto& kv : free_) b += kv.first * kv.second.size();
    return b;
  }
  // powers of two up to 256 MiB; above, multiples of 1/16 of the next power of two (at most
  // 6.25 % unused), so that the large environments of a high bond dimension do not waste
  // up to half of their block
  static size_t size_class(size_t bytes) {
    size_t c = 4096;
    while (c < bytes) c <<= 1;
    if (c > (size_t(256) << 20)) {
      const size_t step = c >> 4;
      c = (bytes + step - 1) / step * step;
    }
    return c;
  }

 private:
  void* from_device(size_t bytes) {
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
      (void)cudaGetLastError();
      trim();
      TDVP_CUDA(cudaMalloc(&p, bytes));
    }
    return p;
  }
  std::map<size_t, std::vector<void*>> free_;
  std::vector<void*> slabs_;
  char* slab_ = nullptr;
  size_t slab_left_ = 0;
};

// A device array of complex numbers drawn from a pool (RAII).
class DArr {
 public:
  DArr() = default;
  DArr(DevicePool* pool, size_t n) { reset(pool, n); }
  DArr(const DArr&) = delete;
  DArr& operator=(const DArr&) = delete;
  DArr(DArr&& o) noexcept { swap(o); }
  DArr& operator=(DArr&& o) noexcept {
    if (this != &o) {
      release();
      swap(o);
    }
    return *this;
  }
  ~DArr() { release(); }
  void reset(DevicePool* pool, size_t n) {
    release();
    pool_ = pool;
    n_ = n;
    if (n) p_ = static_cast<cplx*>(pool->get(n * sizeof(cplx)));
  }
  // keeps the buffer when it is large enough
  void ensure(DevicePool* pool, size_t n) {
    if (p_ && DevicePool::size_class(n * sizeof(cplx)) ==
                  DevicePool::size_class(n_ * sizeof(cplx))) {
      n_ = n;
      return;
    }
    reset(pool, n);
  }
  void release() {
    if (p_ && pool_) pool_->put(p_, n_ * sizeof(cplx));
    p_ = nullptr;
    n_ = 0;
  }
  void swap(DArr& o) {
    std::swap(p_, o.p_);
    std::swap(n_, o.n_);
    std::swap(pool_, o.pool_);
  }
  cplx* data() const { return p_; }
  size_t size() const { return n_; }

 private:
  cplx* p_ = nullptr;
  size_t n_ = 0;
  DevicePool* pool_ = nullptr;
};

// A raw device buffer (bytes) drawn from a pool (RAII).
class RawBuf {
 public:
  RawBuf() = default;
  RawBuf(const RawBuf&) = delete;
  RawBuf& operator=(const RawBuf&) = delete;
  RawBuf(RawBuf&& o) noexcept { swap(o); }
  RawBuf& operator=(RawBuf&& o) noexcept {
    if (this != &o) {
      release();
      swap(o);
    }
    return *this;
  }
  ~RawBuf() { release(); }
  void swap(RawBuf& o) {
    std::swap(p_, o.p_);
    std::swap(bytes_, o.bytes_);
    std::swap(pool_, o.pool_);
  }
  void ensure(DevicePool* pool, size_t bytes) {
    if (p_ && DevicePool::size_class(bytes) == DevicePool::size_class(bytes_)) {
      bytes_ = bytes;
      return;
    }
    release();
    pool_ = pool;
    bytes_ = bytes;
    if (bytes) p_ = pool->get(bytes);
  }
  void release() {
    if (p_ && pool_) pool_->put(p_, bytes_);
    p_ = nullptr;
    bytes_ = 0;
  }
  template <class T>
  T* as() const { return static_cast<T*>(p_); }
  size_t bytes() const { return bytes_; }

 private:
  void* p_ = nullptr;
  size_t bytes_ = 0;
  DevicePool* pool_ = nullptr;
};

// Host data of several arrays for one device buffer: parts at 256-byte offsets, one copy.  The
// copy is from pageable memory, so the host data may go once upload() has returned.
class Packed {
 public:
  template <class T>
  size_t add(const T* p, size_t n) {
    const size_t at = bytes_.size();
    bytes_.resize(at + ((n * sizeof(T) + 255) & ~size_t(255)));
    if (n) std::memcpy(bytes_.data() + at, p, n * sizeof(T));
    return at;
  }
  template <class T>
  size_t add(const std::vector<T>& v) {
    return add(v.data(), v.size());
  }
  size_t zeros(size_t n) {  // n zero bytes
    const size_t at = bytes_.size();
    bytes_.resize(at + ((n + 255) & ~size_t(255)));
    return at;
  }
  size_t size() const { return bytes_.size(); }
  char* upload(cudaStream_t st, DevicePool* pool, RawBuf& buf) const {
    buf.ensure(pool, std::max<size_t>(bytes_.size(), 256));
    if (!bytes_.empty())
      TDVP_CUDA(cudaMemcpyAsync(buf.as<char>(), bytes_.data(), bytes_.size(), cudaMemcpyHostToDevice, st));
    return buf.as<char>();
  }

 private:
  std::vector<char> bytes_;
};

// f() once per device and call site (each lambda is a type of its own); returns what it returned there.
// Function attributes and launch limits belong to a device: set once per process they would be missing
// on the second one.  A call that throws is tried again next time.
constexpr int kMaxDevices = 64;
template <class F>
int once_per_device(int dev, F&& f) {
  struct Slot {
    std::once_flag once;
    int value = 0;
  };
  static Slot slots[kMaxDevices];
  tdvp_require(dev >= 0 && dev < kMaxDevices, TDVP_ERR_INVALID_ARG, "device index out of range");
  Slot& s = slots[dev];
  std::call_once(s.once, [&] { s.value = (int)f(); });
  return s.value;
}
template <class F>
int per_device(F&& f) {
  int dev = 0;
  TDVP_CUDA(cudaGetDevice(&dev));
  return once_per_device(dev, f);
}

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }
