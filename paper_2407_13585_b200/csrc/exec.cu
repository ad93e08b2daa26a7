// Execution of a program: clusters run by ascending cluster number (Section 4.1), one kernel
// launch each (or one per pass) on the caller's stream.  The unfused executor is the same
// machinery with every combinator its own cluster.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <deque>
#include <map>
#include <memory>
#include <mutex>

#include "cluster.h"
#include "exec.h"
#include "graph.h"
#include "registry.h"

namespace acc {

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Cuts the cluster formed by `members` (ascending) out of the graph, mirroring the
// build-time extract(): externals appear just before their first use.
static bool extract_runtime(const Graph& g, const std::vector<int>& members, const std::vector<uint8_t>& man, CCluster& c) {
  c = CCluster{};
  std::map<int, int> local;
  std::vector<uint8_t> in_cluster(g.nodes.size(), 0);
  for (int m : members) in_cluster[m] = 1;
  for (int m : members) {
    const acc_node_desc& d = g.nodes[m].d;
    for (int s = 0; s < d.n_inputs; ++s) {
      const int a = d.inputs[s];
      if (!in_cluster[a] && !local.count(a)) {
        if (c.n >= kMaxCluster) return false;
        CNode e{ACC_INPUT, g.nodes[a].d.dtype, g.nodes[a].d.rank, 0, 0, 0, 0, {-1, -1, -1, -1, -1, -1}, false, true};
        local[a] = c.n;
        c.source[c.n] = a;
        c.nodes[c.n++] = e;
      }
    }
    if (c.n >= kMaxCluster) return false;
    CNode n{d.kind, d.dtype, d.rank, d.fn_id, d.idx_fn_id, d.n_inputs, d.n_array_inputs, {-1, -1, -1, -1, -1, -1}, true, man[m] != 0};
    if (d.kind != ACC_BACKPERMUTE) n.idxfn = 0;
    if (d.kind == ACC_BACKPERMUTE || d.kind == ACC_GATHER) n.fn = 0;
    if (d.kind == ACC_BACKPERMUTE && d.idx_fn_id == ACC_IDX_SHIFT_CLAMP && d.iparam[0] >= -1 && d.iparam[0] <= 1 &&
        d.iparam[1] >= -1 && d.iparam[1] <= 1) {
      n.p0 = (int)d.iparam[0];                         // kernels built for these very offsets are looked up first
      n.p1 = (int)d.iparam[1];
    }
    if ((d.kind == ACC_SCANL || d.kind == ACC_SCANR) && (d.flags & ACC_FLAG_SCAN_EXCLUSIVE)) n.p0 = 1;   // other code, not another argument
    if (d.kind == ACC_MAP && d.fn_id == ACC_FN_MUL_MOD && d.iparam[1] > 0 && (d.iparam[1] & (d.iparam[1] - 1)) == 0)
      n.p0 = kPow2;                                    // a kernel built for power-of-two moduli is looked up first
    for (int s = 0; s < d.n_inputs; ++s) n.in[s] = local[d.inputs[s]];
    local[m] = c.n;
    c.source[c.n] = m;
    c.nodes[c.n++] = n;
  }
  return true;
}

static dev::NodeArg node_arg(const Node& n, const void* ptr) {
  dev::NodeArg a{};
  a.ptr = ptr;
  a.ip0 = (int32_t)(uint32_t)(n.d.iparam[0] & 0xFFFFFFFFll);
  a.ip1 = (int32_t)(uint32_t)(n.d.iparam[1] & 0xFFFFFFFFll);
  a.fp0 = (float)n.d.fparam[0];
  a.fp1 = (float)n.d.fparam[1];
  // branch-free division by d (Granlund and Montgomery's round-up multiplier, 33 bits with the
  // add-and-shift fix-up): l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1,
  // v / d = (t + ((v - t) >> min(l, 1))) >> max(l - 1, 0) with t = umulhi(v, m); d = 1 gives v
  const uint32_t d = (uint32_t)(n.d.fn_id == ACC_FN_MUL_MOD ? a.ip1 : a.ip0);
  if (d >= 1) {
    uint32_t l = 0;
    while (l < 32 && (1ull << l) < d) ++l;
    a.div_mul = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
    a.div_sh1 = l < 1 ? l : 1;
    a.div_sh2 = l - a.div_sh1;
    a.div_mask = (d & (d - 1)) == 0 ? d - 1 : 0;
  }
  a.R = n.d.rank == 2 ? (int32_t)n.d.shape[0] : 1;
  a.C = n.d.rank == 2 ? (int32_t)n.d.shape[1] : (n.d.rank == 1 ? (int32_t)n.d.shape[0] : 1);
  return a;
}

// The kernel instantiated for a cluster: for its very constants, else the one that takes them at run time.
static const KernelEntry* lookup(CCluster& cc, std::string& sig) {
  sig = signature(cc);
  const KernelEntry* k = find_kernel(sig);
  if (!k) {
    for (int li = 0; li < cc.n; ++li)
      if (cc.nodes[li].kind == ACC_BACKPERMUTE || (cc.nodes[li].kind == ACC_MAP && cc.nodes[li].fn == ACC_FN_MUL_MOD))
        cc.nodes[li].p0 = cc.nodes[li].p1 = kRunTime;
    sig = signature(cc);
    k = find_kernel(sig);
  }
  return k;
}

int refine_to_kernels(const Graph& g, std::vector<int32_t>& pi, int recompute_depth, int& splits) {
  const int n = (int)g.nodes.size();
  splits = 0;
  for (;;) {
    std::vector<uint8_t> man;
    manifest_of(g, pi.data(), man);
    std::map<int, std::vector<int>> clusters;
    for (int i = 0; i < n; ++i)
      if (!is_input(g.nodes[i])) clusters[pi[i]].push_back(i);
    const std::vector<int>* bad = nullptr;
    std::string sig;
    for (auto& kv : clusters) {
      CCluster cc;
      if (!extract_runtime(g, kv.second, man, cc) || !lookup(cc, sig)) { bad = &kv.second; break; }
    }
    if (!bad) return ACC_OK;
    if (bad->size() == 1)
      return set_error(ACC_ERR_NO_KERNEL, "no kernel instantiated for node %d alone [%s]", bad->front(), sig.c_str());
    // the latest member that may leave and still leave a legal clustering becomes a cluster of its own;
    // failing that the whole cluster falls apart into its nodes
    const int n_blocks = (int)clusters.size();
    std::vector<int> block_of(pi.begin(), pi.end());
    std::vector<int32_t> trial;
    bool done = false;
    for (auto it = bad->rbegin(); it != bad->rend() && !done; ++it) {
      std::vector<int> b(block_of);
      b[*it] = n_blocks;
      done = canonical_numbering(g, b, n_blocks + 1, trial) && check_partition(g, trial.data(), nullptr, true, recompute_depth) == ACC_OK;
    }
    if (!done) {
      std::vector<int> b(block_of);
      int next = n_blocks;
      for (size_t k = 1; k < bad->size(); ++k) b[(*bad)[k]] = next++;
      if (!canonical_numbering(g, b, next, trial) || check_partition(g, trial.data(), nullptr, true, recompute_depth) != ACC_OK)
        return set_error(ACC_ERR_NO_KERNEL, "the cluster at node %d has no kernel and cannot be split legally [%s]", bad->front(), sig.c_str());
    }
    clear_error();
    pi = trial;
    ++splits;
  }
}

int build_schedule(Graph& g, int executor, Schedule& sch) {
  const int n = (int)g.nodes.size();
  sch = Schedule{};
  std::vector<int32_t> pi;
  if (executor == ACC_EXEC_FUSED) {
    if (!g.has_pi) return set_error(ACC_ERR_NO_PARTITION, "no clustering set: call acc_set_partition or acc_plan first");
    pi = g.pi;
  } else if (executor == ACC_EXEC_UNFUSED) {
    pi.assign(n, -1);
    int c = 0;
    for (int i = 0; i < n; ++i)
      if (!is_input(g.nodes[i])) pi[i] = c++;
  } else {
    return set_error(ACC_ERR_ARG, "unknown executor %d", executor);
  }
  std::vector<uint8_t> man;
  manifest_of(g, pi.data(), man);

  // buffers: bound ones stay where they are, other manifest arrays go into the workspace
  sch.array_off.assign(n, SIZE_MAX);
  size_t off = 0;
  for (int i = 0; i < n; ++i) {
    const Node& nd = g.nodes[i];
    if (is_input(nd) || nd.output) {
      if (!nd.dev && nd.count > 0)
        return set_error(ACC_ERR_UNBOUND, "node %d (%s) has no device buffer", i, is_input(nd) ? "input" : "output");
      continue;
    }
    if (!man[i] || nd.dev) continue;
    sch.array_off[i] = off;
    off += align_up((size_t)std::max<int64_t>(nd.count, 1) * 4, 256);
  }
  sch.array_bytes = off;

  std::map<int, std::vector<int>> clusters;
  for (int i = 0; i < n; ++i)
    if (!is_input(g.nodes[i])) clusters[pi[i]].push_back(i);
  size_t ctrl = 256;                                    // (first the word that acc_check_gather_indices reports to)
  for (auto& kv : clusters) {
    ClusterStep st;
    st.first_node = kv.second.front();
    st.n_members = (int)kv.second.size();
    if (!extract_runtime(g, kv.second, man, st.cc))
      return set_error(ACC_ERR_NO_KERNEL, "cluster at node %d has more than %d local nodes", st.first_node, kMaxCluster);
    std::string sig;
    st.kernel = lookup(st.cc, sig);
    if (!st.kernel)
      return set_error(ACC_ERR_NO_KERNEL, "no kernel instantiated for the cluster of %d nodes starting at node %d [%s]",
                       st.n_members, st.first_node, sig.c_str());
    st.launch.n = st.cc.n;
    for (int li = 0; li < st.cc.n; ++li) st.launch.nodes[li] = node_arg(g.nodes[st.cc.source[li]], nullptr);
    const int64_t sb = st.kernel->scratch_bytes(st.launch);
    if (sb < 0) return set_error((int)sb, "cluster at node %d: no scratch layout", st.first_node);
    const int64_t zb = st.kernel->zeroed_bytes(st.launch);
    st.scratch_off = ctrl;
    st.scratch_bytes = (size_t)sb;
    st.zero_bytes = (size_t)std::min<int64_t>(std::max<int64_t>(zb, 0), sb);
    ctrl += align_up((size_t)sb, 256);
    sch.steps.push_back(st);
  }
  sch.ctrl_bytes = ctrl;
  sch.to_clear.clear();
  for (const ClusterStep& st : sch.steps) {
    if (st.zero_bytes == 0) continue;
    if (!sch.to_clear.empty() && sch.to_clear.back().first + align_up(sch.to_clear.back().second, 256) == st.scratch_off)
      sch.to_clear.back().second = st.scratch_off - sch.to_clear.back().first + st.zero_bytes;   // one piece
    else sch.to_clear.emplace_back(st.scratch_off, st.zero_bytes);
  }
  sch.total_bytes = ctrl + sch.array_bytes;
  for (const ClusterStep& st : sch.steps) {
    char item[48];
    snprintf(item, sizeof item, "%s%d:%d", sch.text.empty() ? "" : " ", st.first_node, st.n_members);
    sch.text += item;
  }
  sch.manifest = man;
  sch.pi = pi;
  return ACC_OK;
}

static void* buffer_of(const Graph& g, const Schedule& sch, char* ws, int node) {
  const Node& nd = g.nodes[node];
  if (nd.dev) return nd.dev;
  if (sch.array_off[node] == SIZE_MAX) return nullptr;
  return ws + sch.ctrl_bytes + sch.array_off[node];
}

// Status words of the runs (see raise_status in device/eval.cuh): pinned host memory that the kernels write to, a cache
// line for every workspace that a handle runs over (runs over different workspaces may be in flight together), in pages
// that stay with the process; a destroyed handle's lines go to other handles, those of runs that nobody has waited for last.
// Run numbers are unique in the process, so a kernel that outlives its handle cannot speak for another run.  A run that is
// being captured into a CUDA graph will be replayed under one number: its line is cleared in the stream, like the control
// region, and stays with the graph (a user object of it) after the handle is gone.
// With the words in device memory a run paid for clearing them (3 us to enqueue) and a waited-for one for a copy back
// (7 us to enqueue, 8 us of waiting): a chain of 2^16, waited for, 29.6 -> 16.6 us with the rest of the host path.
namespace {
constexpr int kStatusLines = 512;                          // lines of one page of status words
constexpr int kSettled = 15;                               // word of a line: its last run was waited for and had nothing to report
constexpr size_t kManyReports = 64;                        // lines of one handle beyond which it looks for one it can use again
std::atomic<uint32_t> last_run{0};
struct StatusPool {
  std::mutex guard;
  std::deque<uint32_t*> free;
};
StatusPool& status_pool() {
  static StatusPool* pool = new StatusPool();              // (never destroyed: a CUDA graph may outlive everything static)
  return *pool;
}

void hand_back(uint32_t* words) {
  StatusPool& pool = status_pool();
  std::lock_guard<std::mutex> lock(pool.guard);
  if (words[kSettled]) pool.free.push_front(words);
  else pool.free.push_back(words);
}

// `words` stay in use as long as the graph that `stream` is being captured into, or an executable made of it (for good, if
// the graph does not take them).
void keep_with_captured_graph(const std::shared_ptr<uint32_t>& words, cudaStream_t stream) {
  auto* held = new std::shared_ptr<uint32_t>(words);
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  cudaGraph_t graph = nullptr;
  cudaUserObject_t object = nullptr;
  if (cudaStreamGetCaptureInfo(stream, &status, nullptr, &graph) != cudaSuccess || !graph ||
      cudaUserObjectCreate(&object, held, [](void* p) { delete static_cast<std::shared_ptr<uint32_t>*>(p); }, 1, cudaUserObjectNoDestructorSync) != cudaSuccess ||
      cudaGraphRetainUserObject(graph, object, 1, cudaGraphUserObjectMove) != cudaSuccess)
    cudaGetLastError();
}

// (the one used last is looked at first)
RunReport* report_for(Graph& handle, const void* workspace) {
  for (RunReport& r : handle.reports)
    if (r.workspace == workspace) {
      std::swap(r, handle.reports.front());
      return &handle.reports.front();
    }
  return nullptr;
}

std::shared_ptr<uint32_t> take_status_words() {
  StatusPool& pool = status_pool();
  std::lock_guard<std::mutex> lock(pool.guard);
  if (pool.free.size() <= kStatusLines / 2) {              // (so many others are handed on before a line put last)
    void* page = nullptr;
    // (allocating is not allowed while a stream is being captured, unless the thread says that it does not matter)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaHostAlloc(&page, kStatusLines * 64, cudaHostAllocPortable | cudaHostAllocMapped);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) {
      cudaGetLastError();
      set_error(ACC_ERR_CUDA, "no pinned memory for the status words: %s", cudaGetErrorString(e));
      return nullptr;
    }
    for (int k = kStatusLines - 1; k >= 0; --k) pool.free.push_front(static_cast<uint32_t*>(page) + k * 16);
  }
  uint32_t* words = pool.free.front();
  pool.free.pop_front();
  memset(words, 0, 64);
  return std::shared_ptr<uint32_t>(words, hand_back);
}

// The report of a new run over `workspace`, as it is now.
int begin_run(Graph& handle, const void* workspace, cudaStream_t stream, RunReport& out) {
  std::lock_guard<std::mutex> lock(handle.reports_guard);
  RunReport* r = report_for(handle, workspace);
  if (!r && handle.reports.size() >= kManyReports) {       // the line of a run with nothing to report, waited for the longest ago
    for (RunReport& c : handle.reports)
      if (!c.captured && c.words.get()[kSettled] && (!r || (int32_t)(c.run_id - r->run_id) < 0)) r = &c;
  }
  if (!r) {
    std::shared_ptr<uint32_t> words = take_status_words();
    if (!words) return ACC_ERR_CUDA;
    handle.reports.emplace_back();
    r = &handle.reports.back();
    r->words = words;
  }
  r->workspace = workspace;
  r->words.get()[kSettled] = 0;
  do r->run_id = ++last_run;
  while (r->run_id == 0);
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) cudaGetLastError();
  if (capturing == cudaStreamCaptureStatusActive) {
    r->captured = true;
    keep_with_captured_graph(r->words, stream);
  }
  if (r->captured && cudaMemsetAsync(r->words.get(), 0, dev::kStatusConditions * 4, stream) != cudaSuccess)
    return set_error(ACC_ERR_CUDA, "clearing the status words failed: %s", cudaGetErrorString(cudaGetLastError()));
  out = *r;
  return ACC_OK;
}
}  // namespace

static bool mark(std::vector<cudaEvent_t>* marks, cudaStream_t stream) {
  if (!marks) return true;
  cudaEvent_t e;
  if (cudaEventCreate(&e) != cudaSuccess) return false;
  marks->push_back(e);
  return cudaEventRecord(e, stream) == cudaSuccess;
}

// Fills in the addresses of the steps' arrays and scratch regions in this workspace.  Bindings are part of the
// schedule (a new one is built when they change), so a run over the workspace of the run before has nothing to fill in.
static int resolve_pointers(const Graph& g, Schedule& sch, char* ws) {
  sch.resolved_for = nullptr;
  for (ClusterStep& st : sch.steps) {
    for (int li = 0; li < st.cc.n; ++li) {
      const int node = st.cc.source[li];
      const CNode& cn = st.cc.nodes[li];
      void* p = (!cn.member || cn.manifest) ? buffer_of(g, sch, ws, node) : nullptr;
      if ((!cn.member || cn.manifest) && !p && g.nodes[node].count > 0)
        return set_error(ACC_ERR_UNBOUND, "node %d is read or written by the cluster at node %d but has no buffer", node, st.first_node);
      st.launch.nodes[li].ptr = p;
    }
    st.launch.scratch = reinterpret_cast<uint32_t*>(ws + st.scratch_off);
  }
  sch.resolved_for = ws;
  return ACC_OK;
}

int run_schedule(Graph& handle, Graph& g, Schedule& sch, void* workspace, size_t ws_bytes, cudaStream_t stream, std::vector<cudaEvent_t>* marks) {
  if (!workspace) return set_error(ACC_ERR_WORKSPACE, "workspace is null, %zu bytes needed", sch.total_bytes);
  if (reinterpret_cast<uintptr_t>(workspace) & 255) return set_error(ACC_ERR_WORKSPACE, "workspace is not 256-byte aligned");
  if (ws_bytes < sch.total_bytes) return set_error(ACC_ERR_WORKSPACE, "workspace has %zu bytes, %zu needed", ws_bytes, sch.total_bytes);
  char* ws = static_cast<char*>(workspace);
  if (sch.resolved_for != ws) {
    const int rc = resolve_pointers(g, sch, ws);
    if (rc != ACC_OK) return rc;
  }
  RunReport report;
  const int begun = begin_run(handle, workspace, stream, report);
  if (begun != ACC_OK) return begun;
  for (const auto& piece : sch.to_clear)
    if (cudaMemsetAsync(ws + piece.first, 0, piece.second, stream) != cudaSuccess)
      return set_error(ACC_ERR_CUDA, "clearing the control region failed: %s", cudaGetErrorString(cudaGetLastError()));
  g.launches = 0;
  g.schedule = sch.text;
  if (!mark(marks, stream)) return set_error(ACC_ERR_CUDA, "recording an event failed: %s", cudaGetErrorString(cudaGetLastError()));
  for (ClusterStep& st : sch.steps) {
    st.launch.stream = stream;
    st.launch.spin_limit = g.spin_limit;
    st.launch.status = report.words.get();
    st.launch.run_id = report.run_id;
    st.launch.extra_launches = 0;
    const int rc = st.kernel->launch(st.launch);
    if (rc != ACC_OK) return rc;
    if (!mark(marks, stream)) return set_error(ACC_ERR_CUDA, "recording an event failed: %s", cudaGetErrorString(cudaGetLastError()));
    g.launches += st.kernel->passes + st.launch.extra_launches;
  }
  return ACC_OK;
}

// One word per index: out of range (as unsigned, so negative ones too) sets the index bit of the status word.
__global__ void k_index_range(const uint32_t* idx, int64_t n, uint32_t bound, uint32_t* status) {
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) bad = bad || idx[i] >= bound;
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, 2u);
}

int check_gather_indices(const Graph& g, void* workspace, size_t ws_bytes, cudaStream_t stream) {
  if (!workspace || ws_bytes < 256 || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return set_error(ACC_ERR_WORKSPACE, "the check needs a 256-byte aligned workspace of 256 bytes");
  if (cudaMemsetAsync(workspace, 0, 256, stream) != cudaSuccess)
    return set_error(ACC_ERR_CUDA, "clearing the status word failed: %s", cudaGetErrorString(cudaGetLastError()));
  for (const Node& nd : g.nodes) {
    if (nd.d.kind != ACC_GATHER) continue;
    const Node& idx = g.nodes[nd.d.inputs[0]];
    const Node& src = g.nodes[nd.d.inputs[1]];
    if (!is_input(idx) || !idx.dev || idx.count == 0) continue;
    const uint32_t bound = (uint32_t)std::min<int64_t>(src.count, 0x7FFFFFFF);
    const int grid = (int)std::min<int64_t>((idx.count + 255) / 256, (int64_t)sm_count() * 8);
    k_index_range<<<grid, 256, 0, stream>>>(static_cast<const uint32_t*>(idx.dev), idx.count, bound, static_cast<uint32_t*>(workspace));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
  }
  uint32_t status = 0;
  if (cudaMemcpyAsync(&status, workspace, 4, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
    return set_error(ACC_ERR_CUDA, "reading the status word failed: %s", cudaGetErrorString(cudaGetLastError()));
  const cudaError_t e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "stream failed: %s", cudaGetErrorString(e));
  return status ? set_error(ACC_ERR_INDEX_RANGE, "a gather index falls outside its source") : ACC_OK;
}

int finish(Graph& g, void* workspace, cudaStream_t stream) {
  RunReport r;                                             // the run to wait for; another thread may begin others meanwhile
  {
    std::lock_guard<std::mutex> lock(g.reports_guard);
    if (const RunReport* known = workspace ? report_for(g, workspace) : nullptr) r = *known;
  }
  const cudaError_t e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return set_error(ACC_ERR_CUDA, "stream failed: %s", cudaGetErrorString(e));
  if (!r.words) return ACC_OK;
  const volatile uint32_t* words = r.words.get();
  const auto raised = [&](int condition) { return r.captured ? words[condition] != 0 : words[condition] == r.run_id; };
  if (raised(dev::kStatusTimeout)) return set_error(ACC_ERR_DEVICE_TIMEOUT, "a device-side wait ran out of iterations");
  if (raised(dev::kStatusIndex)) return set_error(ACC_ERR_INDEX_RANGE, "a scatter index or a segment offset fell outside its array");
  if (raised(dev::kStatusEmptySegment)) return set_error(ACC_ERR_SHAPE, "an empty segment has no value: segment offsets must increase");
  std::lock_guard<std::mutex> lock(g.reports_guard);
  const RunReport* now = report_for(g, workspace);
  if (now && now->run_id == r.run_id) r.words.get()[kSettled] = 1;
  return ACC_OK;
}

}  // namespace acc
