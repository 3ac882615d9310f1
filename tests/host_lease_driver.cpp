// Drives csrc/host_lease.h against a stand-in for the CUDA calls it makes (no GPU, no CUDA
// library): prints one line per check, "ok" or what went wrong.
#include <cstdio>
#include <cstdlib>
#include <set>
#include <string>

#include "host_lease.h"

static int g_allocs = 0, g_frees = 0, g_syncs = 0;
static cudaError_t g_sync_result = cudaSuccess;
static bool g_no_memory = false;
static cudaStream_t g_synced = nullptr;

extern "C" {
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) {
  if (g_no_memory) return cudaErrorMemoryAllocation;
  ++g_allocs;
  *p = std::malloc(n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  ++g_frees;
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  ++g_syncs;
  g_synced = s;
  return g_sync_result;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
}

using kss_rt::HostLease;

static void check(const char* what, bool ok) { std::printf("%s: %s\n", what, ok ? "ok" : "FAILED"); }

int main() {
  cudaStream_t const s = reinterpret_cast<cudaStream_t>(8);
  unsigned char* first = nullptr;
  {
    HostLease a(s);
    first = a.p;
    a.settled();
  }
  check("a call that waited is not waited for again", first && g_syncs == 0);
  { HostLease a(s); }  // the call returned before it waited
  check("a call that returned early is waited for", g_syncs == 1 && g_synced == s);
  {
    HostLease a(s);
    check("its buffer is handed on after the wait", a.p == first);
    g_sync_result = cudaErrorLaunchFailure;
  }
  g_sync_result = cudaSuccess;
  {
    HostLease a(s);
    check("a buffer that cannot be waited for is not handed on", a.p && a.p != first);
    a.settled();
  }
  {
    HostLease a(s, false);
    check("no lease, no room", !a.p && !a.room(1));
  }
  {
    HostLease a(s);
    check("room beside the status block",
          a.room(HostLease::kBytes - HostLease::kMailBytes) == a.p + HostLease::kMailBytes &&
              !a.room(HostLease::kBytes - HostLease::kMailBytes + 1));
    a.settled();
  }
  // more calls at once than the pool has buffers, three times over
  constexpr int kCalls = 40;
  for (int round = 0; round < 3; ++round) {
    HostLease* lease[kCalls];
    std::set<unsigned char*> lent;
    int without = 0;
    for (auto& l : lease) {
      l = new HostLease(s);
      if (l->p) lent.insert(l->p);
      else ++without;
      l->settled();
    }
    const std::string what = "no buffer is lent twice (" + std::to_string(round) + ")";
    check(what.c_str(), int(lent.size()) + without == kCalls && without < kCalls);
    for (auto& l : lease) delete l;
  }
  check("calls beyond the pool's size make and free no memory", g_allocs <= 16 && g_frees == 0);
  g_no_memory = true;
  {
    HostLease a(s);
    check("kept buffers need no new memory", a.p != nullptr);
    a.settled();
  }
  return 0;
}
