// Checks of the host runtime without a GPU: pcs_runtime.cpp is compiled into
// this program over a stand-in CUDA runtime (device memory is host memory,
// nothing runs, events are done at once or on demand one call late) and stand-in kernel launchers,
// which keep the order and the arguments of what a call enqueues.
// Usage: runtime_check <check>; prints "ok" or the first failure.
#include <cstdlib>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "pcs_runtime.cpp"

// ---- what the calls enqueued ------------------------------------------------

struct Op {
  std::string what;
  bool upload;  // a kernel that writes descriptors and lets the next one start before
  bool early;   // a kernel that may start before the one ahead has finished
};
static std::map<cudaStream_t, std::vector<Op>> g_ops;
static std::string g_fail_at;  // a launcher that returns an error
static bool g_behind = false;  // the event recorded last is not done yet
static cudaEvent_t g_last_event = nullptr;

static cudaError_t op(cudaStream_t s, const char* what, bool early = false) {
  g_ops[s].push_back({what, false, early});
  return g_fail_at == what ? cudaErrorInvalidValue : cudaSuccess;
}

// ---- CUDA runtime stand-ins -------------------------------------------------

extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in error"; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::aligned_alloc(256, (n + 255) / 256 * 256); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(new int); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<int*>(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { g_last_event = e; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) { return g_behind && e == g_last_event ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  std::memcpy(d, s, n);
  return op(st, "memcpy");
}
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  std::memset(d, v, n);
  return op(st, "memset");
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  *a = cudaPointerAttributes{};
  a->type = cudaMemoryTypeDevice;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*) {
  return cudaErrorNotSupported;
}
}  // extern "C"

// ---- kernel launcher stand-ins ------------------------------------------------
// A launcher without an `early` argument launches its kernel early always
// (k_finalize, k_reduce_nodes, k_gsmall) or never (the others).

namespace pcs {
cudaError_t launch_upload(void* d, const void* s, uint64_t n, cudaStream_t st) {
  std::memcpy(d, s, n);
  g_ops[st].push_back({"upload", true, true});
  return cudaSuccess;
}
cudaError_t launch_stream(int, bool early, bool, const SecDesc*, WorkList, int, uint64_t*, uint32_t*,
                          int, int, cudaStream_t st) { return op(st, "stream", early); }
cudaError_t launch_bulk(int, bool, bool early, const SecDesc*, WorkList, uint64_t*, uint32_t*,
                        uint32_t*, int, cudaStream_t st) { return op(st, "bulk", early); }
cudaError_t launch_small(int, bool early, const uint8_t* host_plan, uint64_t, const SmallArgs&, int,
                         int, cudaStream_t st) { return op(st, host_plan ? "small" : "small(ws)", early); }
cudaError_t launch_reduce_nodes(const NodeLevel*, int, uint64_t*, uint32_t, uint32_t, int,
                                cudaStream_t st) { return op(st, "reduce", true); }
cudaError_t launch_finalize(int, const SecDesc*, const SessDesc*, int, const Entry*, uint64_t*,
                            uint64_t*, const uint64_t*, uint8_t*, uint32_t*, int, cudaStream_t st) {
  return op(st, "finalize", true);
}
cudaError_t launch_score(const Banks& b, uint64_t entries, int, int, float*, int, cudaStream_t st,
                         GHist gh, bool* fused) {
  if (fused) *fused = gh.st != nullptr;
  return entries ? op(st, "score", b.early) : cudaSuccess;
}
cudaError_t launch_topk(const Banks& b, const float*, int32_t*, int32_t*, int32_t, cudaStream_t st) {
  return op(st, "topk", b.early);
}
cudaError_t launch_gsmall(const Banks&, uint64_t, const float*, uint64_t, bool, bool, int32_t*,
                          int32_t*, cudaStream_t st) { return op(st, "gsmall", true); }
cudaError_t launch_gselect(const GPlan&, int, int, cudaStream_t st) { return op(st, "gselect"); }
cudaError_t launch_gfinish(const GPlan&, int, int, cudaStream_t st) { return op(st, "gfinish"); }
cudaError_t launch_mismatch(bool, const MmPair*, const uint64_t*, const uint64_t*, int32_t, uint64_t,
                            uint64_t*, uint64_t*, uint32_t*, int, cudaStream_t st) { return op(st, "mismatch"); }
cudaError_t launch_classify_reads(bool, ReadPlan, const uint64_t*, const uint64_t*, int64_t,
                                  uint8_t*, int, cudaStream_t st) { return op(st, "reads"); }
cudaError_t launch_pool_alloc(const PoolDev&, int32_t*, int32_t, cudaStream_t st) { return op(st, "pool"); }
cudaError_t launch_pool_share(const PoolDev&, const int32_t*, int32_t*, int32_t, cudaStream_t st) { return op(st, "pool"); }
cudaError_t launch_pool_cow(const PoolDev&, int32_t*, int64_t, const int32_t*, int32_t, int, cudaStream_t st) { return op(st, "pool"); }
cudaError_t launch_pool_release(const PoolDev&, const int32_t*, int32_t, cudaStream_t st) { return op(st, "pool"); }
cudaError_t launch_selftest_wait(int, const uint32_t*, uint32_t*, cudaStream_t st) { return op(st, "selftest"); }
cudaError_t launch_fingerprint_static(const StaticPlan&, uint64_t*, uint64_t*, cudaStream_t st) { return op(st, "static"); }
cudaError_t static_scratch(uint64_t**) { return cudaErrorNotSupported; }
int stream_blocks_per_sm() { return 2; }
}  // namespace pcs

// ---- helpers ------------------------------------------------------------------

#define NEED(cond)                                                    \
  do {                                                                \
    if (!(cond)) {                                                    \
      std::printf("line %d: %s (%s)\n", __LINE__, #cond, g_err.c_str()); \
      std::exit(1);                                                   \
    }                                                                 \
  } while (0)

static std::vector<uint8_t> g_mem(64 << 20);
static uint8_t* mem(uint64_t at) {
  const uintptr_t p = reinterpret_cast<uintptr_t>(g_mem.data());
  return g_mem.data() + ((256 - p % 256) % 256) + at;
}

// n sessions of `secs` contiguous sections of `bytes`, `off` bytes past a boundary.
struct Sessions {
  std::vector<std::vector<pcs_section>> secs;
  std::vector<pcs_session> s;
  Sessions(int n, int k, uint64_t bytes, uint64_t off = 0) : secs(n, std::vector<pcs_section>(k)), s(n) {
    uint64_t at = 0;
    for (int i = 0; i < n; ++i) {
      for (auto& x : secs[i]) {
        x = pcs_section{};
        x.type = 1;
        x.layout = PCS_LAYOUT_CONTIG;
        x.base = mem(at + off);
        x.bytes = bytes;
        at = (at + bytes + 31) / 16 * 16;
      }
      s[i] = pcs_session{};
      s[i].session_id = static_cast<uint32_t>(i);
      s[i].sections = secs[i].data();
      s[i].n_sections = k;
    }
  }
  int n() const { return static_cast<int>(s.size()); }
};

static void drop(pcs_ctx* c, std::vector<pcs_snapshot*>& h) {
  for (auto* x : h) NEED(pcs_delete(c, x) == PCS_OK);
  h.clear();
}

// ---- checks -------------------------------------------------------------------

// k_upload lets the next kernel start before it has written the descriptors:
// the kernel enqueued right after it must wait for it to finish.
static std::string upload_order(size_t* uploads) {
  for (auto& kv : g_ops) {
    const auto& v = kv.second;
    for (size_t i = 0; i < v.size(); ++i) {
      *uploads += v[i].upload;
      if (i > 0 && v[i - 1].upload && v[i].early) return v[i].what + " starts early after an upload";
    }
  }
  return {};
}

// Uploads are for calls that find the stream's last one unfinished.
static void upload_order_of_calls(bool behind) {
  g_behind = behind;
  pcs_ctx* c = nullptr;
  NEED(pcs_create(0, &c) == PCS_OK);
  size_t uploads = 0;
  bool in_ws = false;
  // Small calls with descriptors under and over what a launch can carry, calls
  // of the bulk kernel, of the register kernel and of both.
  const struct { int n, secs; uint64_t bytes, off; } shapes[] = {
      {1, 1, 100, 0}, {64, 2, 16, 0}, {53, 3, 16, 0}, {54, 3, 16, 0}, {64, 3, 16, 0}, {64, 32, 16, 1},
      {1, 171, 16, 0}, {1, 400, 16, 0}, {3, 1000, 16, 3}, {65, 2, 16, 0}, {8, 1, 1 << 20, 0},
      {8, 1, 1 << 20, 1}, {300, 2, 40000, 0}, {2000, 4, 1000, 0}};
  for (auto& sh : shapes) {
    Sessions S(sh.n, sh.secs, sh.bytes, sh.off);
    for (uint32_t place : {PCS_PLACE_DEVICE, PCS_PLACE_PINNED_HOST}) {
      for (int verify = 0; verify < 3; ++verify) {
        g_ops.clear();
        std::vector<pcs_snapshot*> h(sh.n), k(sh.n);
        NEED(pcs_checkpoint(c, S.s.data(), sh.n, place, h.data(), nullptr) == PCS_OK);
        const size_t at = g_ops[nullptr].size();
        NEED(pcs_restore(c, h.data(), sh.n, S.s.data(), verify, nullptr) == PCS_OK);
        for (size_t i = at; i < g_ops[nullptr].size(); ++i)
          NEED(!(verify == 1 && g_ops[nullptr][i].upload));  // (copied: it waits for its end)
        NEED(pcs_fork_many(c, h.data(), sh.n, k.data(), nullptr) == PCS_OK);
        for (auto& o : g_ops[nullptr]) in_ws |= o.what == "small(ws)";
        const std::string e = upload_order(&uploads);
        if (!e.empty()) {
          std::printf("%d sessions of %d sections of %llu bytes, verify %d: %s\n", sh.n, sh.secs,
                      static_cast<unsigned long long>(sh.bytes), verify, e.c_str());
          std::exit(1);
        }
        drop(c, h);
        drop(c, k);
      }
    }
  }
  NEED(in_ws);  // the shapes reach a small call with its descriptors in the workspace
  for (int n : {1, 60, 61, 300, 1025}) {  // banks that travel with a launch and that do not
    for (int entries : {0, 3, 200}) {
      g_ops.clear();
      std::vector<pcs_bank> b(n);
      for (auto& x : b) {
        x = pcs_bank{};
        x.keys = x.query = mem(0);
        x.n_entries = entries;
        x.key_dim = 64;
        x.key_dtype = PCS_DT_F16;
        x.entry_bytes = 100;
      }
      auto* f = reinterpret_cast<float*>(mem(1 << 20));
      auto* i = reinterpret_cast<int32_t*>(mem(8 << 20));
      pcs_prune_params p{};
      p.rule = PCS_K_FIXED;
      p.k_max = 2;
      for (float* scores : {f, static_cast<float*>(nullptr)}) {
        NEED(pcs_prune(c, b.data(), n, &p, scores, i, i, nullptr) == PCS_OK);
        NEED(pcs_prune_global(c, b.data(), n, 1000, scores, i, i, nullptr) == PCS_OK);
      }
      std::vector<int32_t> cnt(n, entries), k(n, std::min(entries, 1));
      NEED(pcs_topk(c, f, cnt.data(), k.data(), n, i, i, nullptr) == PCS_OK);
      std::vector<pcs_buf> bufs(n);
      for (int j = 0; j < n; ++j) bufs[j] = {mem(64 * j + j % 3), 60};
      auto* w = reinterpret_cast<uint64_t*>(mem(1 << 20));
      NEED(pcs_fingerprint(c, bufs.data(), n, w, nullptr) == PCS_OK);
      NEED(pcs_mismatch(c, bufs.data(), bufs.data(), n, w, nullptr) == PCS_OK);
      NEED(pcs_classify_reads(c, bufs.data(), n, w, w, 5, mem(0), nullptr) == PCS_OK);
      const std::string e = upload_order(&uploads);
      if (!e.empty()) {
        std::printf("%d banks or buffers, %d entries: %s\n", n, entries, e.c_str());
        std::exit(1);
      }
    }
  }
  NEED((uploads > 0) == behind);
  NEED(pcs_destroy(c) == PCS_OK);
}

static void check_upload_order() {
  upload_order_of_calls(true);
  g_ops.clear();
  upload_order_of_calls(false);
}

// A forked child keeps its own section table and no other: a block's tables are
// those its snapshots point into, each once, however its parents were made.
static void check_fork_tables() {
  pcs_ctx* c = nullptr;
  NEED(pcs_create(0, &c) == PCS_OK);
  // One old session forked again and again together with a new one, the
  // parents and the new one's child dropped: the number does not grow.
  Sessions A(1, 3, 1000), B(1, 2, 500), M(40, 2, 300);
  pcs_snapshot* old = nullptr;
  NEED(pcs_checkpoint(c, A.s.data(), 1, PCS_PLACE_DEVICE, &old, nullptr) == PCS_OK);
  for (int it = 0; it < 50; ++it) {
    pcs_snapshot *fresh = nullptr, *kid[2];
    NEED(pcs_checkpoint(c, B.s.data(), 1, PCS_PLACE_DEVICE, &fresh, nullptr) == PCS_OK);
    pcs_snapshot* par[2] = {old, fresh};
    NEED(pcs_fork_many(c, par, 2, kid, nullptr) == PCS_OK);
    std::vector<pcs_snapshot*> gone = {old, fresh, kid[1]};
    drop(c, gone);
    old = kid[0];
    NEED(old->block->tables.size() <= 2);
  }
  NEED(old->n_sections == 3 && old->table()[2].bytes == 1000);
  // Parents of several calls and both placements, in any order and more than once.
  std::vector<pcs_snapshot*> dev(40), host(40), one(40), par, kid(400);
  NEED(pcs_checkpoint(c, M.s.data(), 40, PCS_PLACE_DEVICE, dev.data(), nullptr) == PCS_OK);
  NEED(pcs_checkpoint(c, M.s.data(), 40, PCS_PLACE_PINNED_HOST, host.data(), nullptr) == PCS_OK);
  for (int i = 0; i < 40; ++i)
    NEED(pcs_checkpoint(c, &M.s[i], 1, PCS_PLACE_DEVICE, &one[i], nullptr) == PCS_OK);
  uint64_t rnd = 1;
  for (int i = 0; i < 400; ++i) {
    rnd = rnd * 6364136223846793005ull + 1442695040888963407ull;
    const uint32_t r = static_cast<uint32_t>(rnd >> 33);
    par.push_back((r & 1 ? dev : r & 2 ? host : one)[(r >> 2) % 40]);
  }
  NEED(pcs_fork_many(c, par.data(), 400, kid.data(), nullptr) == PCS_OK);
  std::vector<uint32_t> ids;
  for (auto* p : par) ids.push_back(p->session_id);
  drop(c, dev);
  drop(c, host);
  drop(c, one);
  for (int i = 0; i < 400; ++i) {
    std::set<const void*> have;
    size_t holds = 0;
    for (auto& t : kid[i]->block->tables) {
      NEED(have.insert(t.get()).second);
      const Entry* e = t->data();
      holds += kid[i]->entries >= e && kid[i]->entries + 2 <= e + t->size();
    }
    NEED(holds == 1);
    std::set<const void*> used;
    for (auto* k : kid)
      if (k->block == kid[i]->block)
        for (auto& t : k->block->tables)
          if (k->entries >= t->data() && k->entries < t->data() + t->size()) used.insert(t.get());
    NEED(used == have);
    NEED(kid[i]->session_id == ids[i] && kid[i]->table()[1].bytes == 300);
  }
  drop(c, kid);
  NEED(pcs_delete(c, old) == PCS_OK);
  NEED(pcs_destroy(c) == PCS_OK);
}

// A call that fails after its descriptors were sent from a pinned slot leaves
// that slot held, since what it enqueued may still read it.  No later call may
// give it back, whichever way that call's own descriptors travel.
static void check_failed_call() {
  Sessions big(8, 1, 1 << 20), few(2, 2, 100);
  std::vector<pcs_buf> bufs(200);
  for (int j = 0; j < 200; ++j) bufs[j] = {mem(64 * j), 60};
  auto* w = reinterpret_cast<uint64_t*>(mem(1 << 20));
  auto* f = reinterpret_cast<float*>(mem(1 << 20));
  auto* ix = reinterpret_cast<int32_t*>(mem(8 << 20));
  std::vector<pcs_bank> b(2);
  for (auto& x : b) {
    x = pcs_bank{};
    x.keys = x.query = mem(0);
    x.n_entries = 9;
    x.key_dim = 64;
    x.key_dtype = PCS_DT_F16;
    x.entry_bytes = 100;
  }
  pcs_prune_params p{};
  p.rule = PCS_K_FIXED;
  p.k_max = 2;
  cudaStream_t s2 = reinterpret_cast<cudaStream_t>(8);
  for (int after = 0; after < 8; ++after) {
    pcs_ctx* c = nullptr;
    NEED(pcs_create(0, &c) == PCS_OK);
    std::vector<pcs_snapshot*> h(8), k(2);
    g_fail_at = "finalize";
    NEED(pcs_checkpoint(c, big.s.data(), 8, PCS_PLACE_DEVICE, h.data(), nullptr) == PCS_E_CUDA);
    g_fail_at.clear();
    NEED(c->plan_slot_busy[0] && !c->plan_slot_busy[0]->done());
    switch (after) {
      case 0: NEED(pcs_fingerprint(c, bufs.data(), 3, w, s2) == PCS_OK); break;
      case 1: NEED(pcs_fingerprint(c, bufs.data(), 200, w, s2) == PCS_OK); break;
      case 2: NEED(pcs_mismatch(c, bufs.data(), bufs.data(), 3, w, s2) == PCS_OK); break;
      case 3: NEED(pcs_classify_reads(c, bufs.data(), 3, w, w, 5, mem(0), s2) == PCS_OK); break;
      case 4: NEED(pcs_prune(c, b.data(), 2, &p, nullptr, ix, ix, s2) == PCS_OK); break;
      case 5: NEED(pcs_prune_global(c, b.data(), 2, 500, nullptr, ix, ix, s2) == PCS_OK); break;
      case 6: NEED(pcs_prune(c, b.data(), 2, &p, f, ix, ix, s2) == PCS_OK); break;
      default:
        NEED(pcs_checkpoint(c, few.s.data(), 2, PCS_PLACE_DEVICE, k.data(), s2) == PCS_OK);
        NEED(pcs_restore(c, k.data(), 2, few.s.data(), 2, s2) == PCS_OK);
    }
    if (c->plan_slot_busy[0]->done()) {
      std::printf("call %d gave back the slot of a failed one\n", after);
      std::exit(1);
    }
    NEED(pcs_destroy(c) == PCS_OK);
  }
}

int main(int argc, char** argv) {
  const std::map<std::string, void (*)()> checks = {{"upload_order", check_upload_order},
                                                    {"fork_tables", check_fork_tables},
                                                    {"failed_call", check_failed_call}};
  auto it = checks.find(argc > 1 ? argv[1] : "");
  if (it == checks.end()) return 2;
  it->second();
  std::puts("ok");
}
