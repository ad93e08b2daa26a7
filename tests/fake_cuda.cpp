// A CUDA runtime that launches nothing, for tests of the host side on a machine without a GPU: what the library asks of the
// runtime succeeds, and every kernel launch is written down.  Loaded before libacc.so with its symbols global, its
// definitions are the ones the library finds.
#include <cxxabi.h>
#include <dlfcn.h>

#include <atomic>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <thread>

struct dim3 { unsigned x, y, z; };

static int sms = 148, cooperative = 1, capturing = 0;
static std::string launches;                 // a line per launch: "name|grid|block|C" (C: cooperative)
static char* pages[64];                      // pinned host memory handed out
static size_t page_bytes[64];
static int n_pages = 0;
static uint32_t* status_words = nullptr;     // of the last launch: where its arguments say that it reports, and as which run
static uint32_t status_run = 0;
static int32_t second[8];                    // of the last launch of k_hist: its second argument's first words
static size_t seg_shared = 0;                // of the last launch of k_segfold: bytes of shared memory asked for

static int note(const void* kernel, dim3 grid, dim3 block, void** args, bool coop) {
  if (launches.size() > (1u << 20)) launches.clear();
  Dl_info info;
  std::string name = "?";
  if (dladdr(kernel, &info) && info.dli_sname) {
    int failed = 0;
    char* plain = abi::__cxa_demangle(info.dli_sname, nullptr, nullptr, &failed);
    name = failed ? info.dli_sname : plain;
    free(plain);
  }
  name = name.substr(0, name.find('('));
  char rest[64];
  snprintf(rest, sizeof rest, "|%u|%u|%s\n", grid.x, block.x, coop ? "C" : "");
  launches += name + rest;
  if (name.find("k_hist<") != std::string::npos) memcpy(second, args[1], 6 * sizeof second[0]);
  // the first argument of a cluster's kernel holds a pointer to status words, the run's number behind it
  const char* a = static_cast<const char*>(args[0]);
  status_words = nullptr;
  for (int at = 0; at < 4000 && !status_words; at += 8) {
    char* p;
    memcpy(&p, a + at, 8);
    for (int k = 0; k < n_pages; ++k)
      if (p >= pages[k] && p < pages[k] + page_bytes[k]) {
        status_words = reinterpret_cast<uint32_t*>(p);
        memcpy(&status_run, a + at + 8, 4);
      }
  }
  return 0;
}

namespace acc {
int sm_count() { return sms; }
bool cooperative_launch_ok() { return cooperative != 0; }
}  // namespace acc

struct Held { void (*destroy)(void*); void* p; };
static Held held_by_graph[4096];             // user objects of the graph that is being captured
static int n_held = 0;

extern "C" {
void fake_device(int sm_count, int can_launch_cooperatively) { sms = sm_count; cooperative = can_launch_cooperatively; }
void fake_capturing(int on) { capturing = on; }
void fake_destroy_graph() {
  while (n_held > 0) { --n_held; held_by_graph[n_held].destroy(held_by_graph[n_held].p); }
}
void fake_clear() { launches.clear(); }
const char* fake_launches() { return launches.c_str(); }
const int32_t* fake_second_argument() { return second; }
size_t fake_seg_shared() { return seg_shared; }
int fake_pages() { return n_pages; }
uint32_t* fake_status(uint32_t* run) { *run = status_run; return status_words; }

// Two threads over one handle: one enqueues `runs` runs over workspaces of their own, the other waits for those before it;
// how many calls failed.
int fake_run_and_wait(int (*run)(void*, void*, size_t, void*, int), int (*finish)(void*, void*, void*), void* handle, int executor, int runs) {
  std::atomic<int> begun{0}, failed{0};
  const auto workspace = [](int k) { return reinterpret_cast<void*>((uintptr_t(1) << 50) + (uintptr_t(k) << 20)); };
  std::thread waits([&] {
    for (int k = 0; k < runs; ++k) {
      while (begun.load() <= k) {}
      if (finish(handle, workspace(k), nullptr) != 0) ++failed;
      if (finish(handle, workspace(k / 2), nullptr) != 0) ++failed;
    }
  });
  for (int k = 0; k < runs; ++k) {
    if (run(handle, workspace(k), size_t(1) << 40, nullptr, executor) != 0) ++failed;
    begun = k + 1;
  }
  waits.join();
  return failed;
}

int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 1; return 0; }
int cudaGetLastError() { return 0; }
int cudaFuncSetAttribute(const void*, int, int) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 2; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return 0; }
int cudaMemsetAsync(void* p, int v, size_t bytes, void*) {           // host memory only: device addresses are not mapped
  for (int k = 0; k < n_pages; ++k)
    if (!capturing && static_cast<char*>(p) >= pages[k] && static_cast<char*>(p) < pages[k] + page_bytes[k]) memset(p, v, bytes);
  return 0;
}
int cudaMemcpyAsync(void*, const void*, size_t, int, void*) { return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaStreamIsCapturing(void*, int* status) { *status = capturing; return 0; }
int cudaStreamGetCaptureInfo_v2(void*, int* status, unsigned long long*, void** graph, const void***, size_t*) {
  *status = capturing;
  *graph = capturing ? &held_by_graph : nullptr;
  return 0;
}
int cudaUserObjectCreate(void** object, void* p, void (*destroy)(void*), unsigned, unsigned) {
  *object = new Held{destroy, p};
  return 0;
}
int cudaGraphRetainUserObject(void*, void* object, unsigned, unsigned) {
  if (n_held == 4096) return 1;
  held_by_graph[n_held++] = *static_cast<Held*>(object);
  delete static_cast<Held*>(object);
  return 0;
}
int cudaThreadExchangeStreamCaptureMode(int*) { return 0; }
int cudaHostAlloc(void** p, size_t bytes, unsigned) {
  if (n_pages == 64) return 2;
  *p = pages[n_pages] = static_cast<char*>(calloc(1, bytes));
  page_bytes[n_pages++] = bytes;
  return 0;
}
static int fake_encode(char* map, int, int, void*, const uint64_t*, const uint64_t*, const uint32_t*, const uint32_t*, int, int, int, int) {
  memset(map, 0, 128);
  return 0;
}
int cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, int* found) {
  *fn = reinterpret_cast<void*>(&fake_encode);
  if (found) *found = 0;
  return 0;
}
int cudaLaunchKernel(const void* kernel, dim3 grid, dim3 block, void** args, size_t shared, void*) {
  note(kernel, grid, block, args, false);
  const size_t line = launches.rfind('\n', launches.size() - 2) + 1;      // (npos + 1: the first)
  if (launches.find("k_segfold<", line) != std::string::npos) seg_shared = shared;
  return 0;
}
int cudaLaunchCooperativeKernel(const void* kernel, dim3 grid, dim3 block, void** args, size_t, void*) { return note(kernel, grid, block, args, true); }
}
