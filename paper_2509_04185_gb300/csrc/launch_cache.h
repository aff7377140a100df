// What the host path of a launch keeps about its kernels on one device: how many
// clusters of a shape the device holds, and how much dynamic shared memory a
// kernel has been allowed.  No CUDA in here: the driver's calls are arguments.
#ifndef SBD_LAUNCH_CACHE_H
#define SBD_LAUNCH_CACHE_H

#include <stddef.h>
#include <stdint.h>

#include <mutex>

namespace sbd {

class LaunchCache {
 public:
  // Entries of one device: about 60 for the bf16 attention (4 kernels x cluster
  // sizes 2 to 16), 54 for the fp32 attention (6 x 9), 70 for sbd_linear (10
  // sizes of shared memory x 7), 6 CTA-pair kernels and one a kernel for its
  // shared memory.
  static constexpr int kEntries = 512;

  // query(): clusters the device holds at once, or < 0 when it could not be
  // asked; that is returned as 0 and not kept, so that the next call asks again.
  template <class Query>
  int clusters(const void* fn, int threads, size_t smem, int cluster_x, Query query) {
    {
      std::lock_guard<std::mutex> lock(mu_);
      const Entry* e = slot(fn, threads, smem, cluster_x);
      if (e && e->fn) return (int)e->value;
    }
    const int n = query();
    if (n < 0) return 0;
    std::lock_guard<std::mutex> lock(mu_);
    if (Entry* e = slot(fn, threads, smem, cluster_x)) *e = Entry{fn, smem, threads, cluster_x, n};
    return n;
  }

  // set(bytes) allows `fn` that much dynamic shared memory.  Threads launch one
  // kernel with different sizes, and what is allowed is the kernel's, not the
  // thread's: it is only ever raised, by one thread at a time.  Returns set's
  // status (0: done).
  template <class Set>
  int allow_smem(const void* fn, size_t smem, Set set) {
    std::lock_guard<std::mutex> lock(mu_);
    Entry* e = slot(fn, 0, 0, 0);
    const size_t most = e && e->fn && (size_t)e->value > smem ? (size_t)e->value : smem;
    const int st = set(most);
    if (st == 0 && e) *e = Entry{fn, 0, 0, 0, (long long)most};
    return st;
  }

 private:
  struct Entry {
    const void* fn;      // nullptr: free
    size_t smem;
    int threads, cluster_x;
    long long value;
  };

  // The entry of this key, or the free one it would take; nullptr when full.
  Entry* slot(const void* fn, int threads, size_t smem, int cluster_x) {
    const uint64_t h = ((uint64_t)(uintptr_t)fn >> 4) * 1000003u + (uint64_t)smem * 31u +
                       (uint64_t)threads * 7u + (uint64_t)cluster_x * 131u;
    for (int i = 0; i < kEntries; ++i) {
      Entry& e = entries_[(h + (uint64_t)i) % kEntries];
      if (!e.fn || (e.fn == fn && e.smem == smem && e.threads == threads && e.cluster_x == cluster_x))
        return &e;
    }
    return nullptr;
  }

  std::mutex mu_;
  Entry entries_[kEntries] = {};
};

}  // namespace sbd

#endif  // SBD_LAUNCH_CACHE_H
