// The limit of dynamic shared memory of each kernel, raised when a launch first needs it.  Apart from
// the CUDA calls (`Api`), so that its behaviour with several threads and contexts can be tested on a host
// without a GPU.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>

namespace m2rnn {

// Api: bool context(uint64_t *id)           the current context's number, unique for the life of the process
//      int most(const void *kernel, int *n) the most dynamic shared memory the device lets the kernel have
//      int set(const void *kernel, int n)   sets its limit in the current context
// (0 = success; other values go back to the caller)
template <typename Api>
class SmemLimits {
 public:
  explicit SmemLimits(int too_much) : too_much_(too_much) {}

  // Lets `kernel` be launched with `bytes`, in the current context, from now on.  The limit is always set
  // to the most there is: whichever of several threads sets it, in whatever order, it is the same, and no
  // launch can find less than an earlier call has granted.  The attribute lives and dies with the
  // context (a reset of the device ends it), so a context is part of what is remembered; a call whose context
  // cannot be told, or that finds no room in the table, sets the limit again.
  int allow(Api &api, const void *kernel, size_t bytes) {
    Entry *e = find(api, kernel);
    if (e) {
      const int n = e->limit.load(std::memory_order_acquire);
      if (n) return bytes <= (size_t)n ? 0 : too_much_;
    }
    int most = 0;
    int rc = api.most(kernel, &most);
    if (rc) return rc;
    if (bytes > (size_t)most) return too_much_;
    rc = api.set(kernel, most);
    if (rc) return rc;
    if (!e) e = find(api, kernel);   // (the calls above make a context current where there was none)
    if (e) e->limit.store(most, std::memory_order_release);
    return 0;
  }

 private:
  static constexpr int kSlots = 1024, kProbes = 64;   // far more (kernel, context) pairs than the library has kernels
  struct Entry { std::atomic<uint64_t> key; std::atomic<int> limit; };
  Entry table_[kSlots] = {};
  const int too_much_;

  Entry *find(Api &api, const void *kernel) {
    uint64_t ctx = 0;
    if (!api.context(&ctx) || ctx >= 0xffff) return nullptr;
    // addresses of host functions have 48 bits, the context's number takes the other 16
    const uint64_t key = (uint64_t)reinterpret_cast<uintptr_t>(kernel) ^ ((ctx + 1) << 48);
    size_t h = (size_t)((key * 0x9e3779b97f4a7c15ull) >> 54);
    for (int i = 0; i < kProbes; ++i, h = (h + 1) % kSlots) {
      uint64_t seen = table_[h].key.load(std::memory_order_acquire);
      if (seen == 0 && table_[h].key.compare_exchange_strong(seen, key, std::memory_order_acq_rel)) seen = key;
      if (seen == key) return &table_[h];
    }
    return nullptr;
  }
};

}  // namespace m2rnn
