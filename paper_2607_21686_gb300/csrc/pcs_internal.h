// pcs_internal.h -- descriptors shared by the host runtime (pcs_runtime.cpp)
// and the sm_103a kernels (pcs_kernels.cu).  Plain structs copied to the
// device once per call; no torch types.
#pragma once

#include <atomic>
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

namespace pcs {

constexpr uint32_t kChunkBytes = 4096;   // fingerprint chunk
constexpr uint32_t kRecordAlign = 256;   // record / payload alignment
constexpr uint32_t kHeaderBytes = 64;
constexpr uint32_t kEntryBytes = 64;
constexpr uint32_t kMagic = 0x31534350u;  // "PCS1"
constexpr uint32_t kVersion = 1;
constexpr int kMaxGroupLog2 = 5;         // static fingerprints: at most 32 chunks per warp task

// Errors a kernel records (OR-ed into the context's device error word).
constexpr uint32_t kDevErrIndex = 1u;    // a row / page id out of range
constexpr uint32_t kDevErrTimeout = 2u;  // a bounded wait inside a kernel gave up
constexpr uint32_t kDevErrNoPage = 4u;   // a page pool had no free page
constexpr uint32_t kDevErrRefcount = 8u; // a page released, shared or written while held by nobody

enum Layout : uint32_t { kContig = 0, kRows = 1, kRing = 2 };

// Work modes of the streaming kernel.
enum Mode : int {
  kModeHash = 0,       // read a contiguous buffer, fingerprint it
  kModePack = 1,       // gather layout side -> payload, fingerprint
  kModeRestore = 2,    // payload -> scatter layout side (no hashing)
  kModeRestoreV = 3,   // payload -> scatter layout side, fingerprint payload
};

// One fingerprinted stream of bytes (a buffer, or a section payload).
// "Layout side" = where the bytes live in the session (source of a pack,
// target of a restore, the buffer itself when hashing); the other side is
// the contiguous payload inside a record.
struct alignas(16) SecDesc {
  uint8_t* lbase;          // layout-side base
  uint8_t* payload;        // contiguous side (record payload), or null
  const int32_t* index;    // ROWS row ids / RING page table
  uint64_t bytes;          // logical bytes L
  uint64_t row_bytes;      // ROWS / RING
  uint64_t base_rows;      // bound on index values
  uint32_t layout;
  int32_t rb_shift;        // log2(row_bytes) if a power of two, else -1
  uint32_t ring_start;
  uint32_t window;
  uint32_t page_rows;
  int32_t pr_shift;        // log2(page_rows) if a power of two, else -1
  uint32_t task_begin;     // first warp task (= node slot) of this stream
  uint32_t n_tasks;
  uint64_t n_chunks;
  uint32_t align;          // CONTIG layout side: 16, 4 or 1 (largest that divides lbase)
  uint32_t fin_count;      // nodes the finaliser trees: [fin_begin, fin_begin + fin_count)
  uint32_t fin_begin;      // (the task nodes, or their 32-to-1 reduction)
  uint32_t sess;           // checkpoint / restore: the session of this stream
  uint64_t row_shift;      // bytes of row 0 before the stream's first byte (a ring
                           // walked by whole pages: see make_desc), else 0
};
static_assert(sizeof(SecDesc) == 112, "SecDesc layout");

// One session: a record and the contiguous range of its sections.
struct alignas(16) SessDesc {
  uint8_t* record;         // record base (pack: written; restore: read)
  uint64_t total_bytes;
  uint64_t payload_start;  // header + table, rounded up to 256
  uint32_t sec_begin;
  uint32_t n_sections;
  uint32_t session_id;
  uint32_t kind;
  uint32_t n_tasks;        // tasks of all its sections
  uint32_t pad;
};
static_assert(sizeof(SessDesc) == 48, "SessDesc layout");

// Section entry exactly as stored in a record (64 bytes, little-endian).
struct alignas(16) Entry {
  uint32_t type, dtype, layer, layout;
  uint64_t offset, bytes, fp, dim0, dim1, aux;
};
static_assert(sizeof(Entry) == 64, "Entry layout");

// One memory bank to score / prune.
struct alignas(16) BankDesc {
  const uint16_t* keys;    // [n][D] fp16 / bf16 bits
  const uint16_t* query;   // [D]
  uint64_t entry_begin;    // CSR offset of this bank's scores
  uint64_t kept_begin;     // CSR offset of this bank's kept indices
  int32_t n;
  int32_t D;
  int32_t k;
  uint32_t is_bf16;
  uint64_t entry_bytes;    // bytes one kept entry costs (global threshold)
  uint64_t pad;
};
static_assert(sizeof(BankDesc) == 64, "BankDesc layout");

// The streams one streaming kernel processes: item j is stream secs[ids[j]],
// owning this kernel's tasks [begin[j], begin[j+1]) (the last up to n_tasks).
// Task t of item j writes node secs[ids[j]].task_begin + (t - begin[j]).
struct WorkList {
  const uint32_t* ids;
  const uint32_t* begin;
  int n_items;
  uint32_t n_tasks;
};

// Chunks per task of the TMA-staged kernel (an 8 KiB tile).
constexpr int kBulkTileChunks = 2;
constexpr uint32_t kFinRegNodes = 1024;  // nodes a finalising warp trees from registers
// Smallest row size the TMA-staged kernel takes for ROWS / RING streams.
constexpr uint64_t kBulkMinRowBytes = 512;

// Kernel launchers (pcs_kernels.cu).  All enqueue on `stream`, return the
// CUDA error of the launch.  `early`: the kernel may be scheduled before the
// one ahead on the stream has finished; false right after launch_upload, whose
// kernel lets it start before the descriptors are written.

// Register kernel: warp tasks of 2^group_log2 chunks, 128-bit loads/stores.
// `beside`: the launch just before it on the stream is the same call's
// launch_bulk, and the two run side by side.
cudaError_t launch_stream(int mode, bool early, bool beside, const SecDesc* secs, WorkList wl,
                          int group_log2, uint64_t* nodes, uint32_t* dev_err, int sm_count,
                          int blocks_per_sm, cudaStream_t stream);

// TMA-staged kernel: tasks of kBulkTileChunks chunks staged through shared
// memory with cp.async.bulk; one persistent block per SM.  `sched`: two
// device words of the call (zero on entry, left zero) that share out the
// launch's last tiles at run time; launches using the same words must be
// ordered.  (Hash mode runs k_hash and does not use them.)  `shift`: some
// stream has a row_shift.
cudaError_t launch_bulk(int mode, bool shift, bool early, const SecDesc* secs, WorkList wl, uint64_t* nodes,
                        uint32_t* dev_err, uint32_t* sched, int sm_count, cudaStream_t stream);

// One launch for a small call: the register streaming pass over its tasks (no
// node reduction) and the finalisation of `mode` (hash: n_items buffers; pack
// / restore_verify: n_items sessions of at most max_secs sections), each item
// by the warp that completes it.  `ticket` and `done` (a word per item, at
// most kSmallMaxItems) are zero on entry and on exit.
constexpr int kSmallMaxItems = 64;
constexpr uint64_t kSmallPlanMax = 31744;  // descriptors that travel as a kernel parameter
struct SmallArgs {
  const uint8_t* plan;     // the descriptors on the device (not read if they are a parameter)
  uint32_t o_secs, o_sess, o_entries, o_ids, o_begin;  // offsets in the descriptors
  int32_t n_list;          // work list items
  uint32_t n_tasks;
  int32_t glog2;
  uint64_t* nodes;
  uint32_t* err;
  uint32_t* ticket;
  uint32_t* done;
  int32_t n_items, max_secs;
  uint64_t* fp_out;
  const uint64_t* fp_before;
  uint8_t* flags;
  uint32_t* bad;
};
// host_plan: the descriptors (`bytes` of them, at most kSmallPlanMax, in
// memory readable to kSmallPlanMax), sent with the launch; null: a.plan.
cudaError_t launch_small(int mode, bool early, const uint8_t* host_plan, uint64_t bytes,
                         const SmallArgs& a, int sm_count, int blocks_per_sm, cudaStream_t stream);

// One level of the node reduction of stream i: count nodes at src, reduced
// by aligned groups of 32 to ceil(count / 32) nodes at dst.
struct NodeLevel {
  uint32_t src, count, dst, pad;
};

// Streams with many task nodes: reduce each aligned group of 32 nodes of
// stream i (nodes[lv[i].src ...]) to one node at nodes[lv[i].dst + g].
// Groups of all streams are numbered by dst - base (monotone).
cudaError_t launch_reduce_nodes(const NodeLevel* lv, int n_secs, uint64_t* nodes, uint32_t base,
                                uint32_t n_groups, int sm_count, cudaStream_t stream);

// Section fps from the nodes [fin_begin, fin_begin + fin_count) (in place), then per mode:
//   kModeHash: fp_out[i] = fp; if fp_before: flags[i] = fp != fp_before[i]
//   kModePack: header + section table of each session's record
//   kModeRestoreV: compare with the record's stored fps; corrupt[s] = 1 and
//                  ++*bad on mismatch
cudaError_t launch_finalize(int mode, const SecDesc* secs, const SessDesc* sess, int n_sess,
                            const Entry* entries, uint64_t* nodes, uint64_t* fp_out,
                            const uint64_t* fp_before, uint8_t* flags, uint32_t* bad,
                            int max_secs, cudaStream_t stream);



// The banks of a call: on the device, or (dev null, at most kBankBlob of them)
// in host memory, to travel with the launch.
constexpr int kBankBlob = 60;  // 3,840 bytes
struct Banks {
  const BankDesc* host;
  const BankDesc* dev;
  int n;
  bool early = true;  // the next launch may be scheduled early (launch_upload's was not the last)
};
// Kept indices per bank; with kept_off, also the offsets of the lists
// (kept_off[n] = kept_total).
cudaError_t launch_topk(const Banks& banks, const float* scores, int32_t* kept_idx,
                        int32_t* kept_off, int32_t kept_total, cudaStream_t stream);
// One thread waits for what never happens (which = 0: an mbarrier's second
// arrival; 1: *never_set >= 1), gives up after the kernels' wait bound and
// sets the timeout bit in *err.
cudaError_t launch_selftest_wait(int which, const uint32_t* never_set, uint32_t* err,
                                 cudaStream_t stream);


// ---- One relevance threshold across all banks (pcs_prune_global) ---------
constexpr int kGTile = 4096;    // entries per tile of the global passes
constexpr int kGPasses = 6;     // digits of the 64-bit key: 11, 11, 10, 11, 11, 10 bits
constexpr int kGBins = 2048;    // bins of the widest digit

// Select state: the kept set is every entry whose ranking key exceeds
// `threshold`.  Set by the host, advanced by the last block of each pass.
struct alignas(16) GState {
  uint64_t prefix, mask;  // key bits fixed so far
  uint64_t remaining;     // budget left for keys inside the prefix
  uint64_t threshold;
  uint32_t done, ticket, total_kept, n_cand;
  uint32_t bar_count, bar_gen, pad[2];  // k_gfinish: arrivals, last barrier released
  uint64_t whist[kGBins]; // entry bytes per digit (mixed entry sizes)
  uint32_t chist[kGBins]; // entries per digit
};

// Summed bins of one later digit pass inside k_gfinish.
struct GBinSet {
  uint64_t w[kGBins];
  uint32_t c[kGBins];
};

// The score kernel's optional epilogue: the first digit pass of the global
// threshold (a histogram of the top key bits, then the digit choice).
struct GHist {
  GState* st;             // NULL: no histogram
  uint64_t uniform_bytes; // entry bytes when every bank costs the same
  int32_t mode;           // 1: uniform entry bytes, 2: per-bank entry bytes
  int32_t pad;
};

// Passed by value as a kernel parameter.
struct GPlan {
  const float* scores;        // [entries], bank-major
  const uint64_t* ebeg;       // [n_banks + 1]: first entry of each bank; ebeg[n_banks] = entries
  const uint64_t* ebytes;     // [n_banks]: bytes one entry of the bank costs
  const uint32_t* tile_bank;  // [tiles + 1]: bank of entry min(t * kGTile, entries - 1)
  uint32_t* tile_cnt;         // [tiles]: kept per tile
  GState* st;
  int32_t* kept_idx;          // [<= entries], CSR by bank
  int32_t* kept_off;          // [n_banks + 1]
  uint64_t entries;
  uint64_t uniform_bytes;     // entry bytes when every bank costs the same
  int32_t n_banks;
  int32_t tiles;
  int32_t uniform;
  int32_t local;              // 1: histogram only, the host sums the parts and picks
  uint64_t pos_base;          // position of entry 0 in the whole (split) population
  int32_t vec;                // 1: scores 16-byte aligned (whole runs read as float4)
  int32_t pad;
  // k_gfinish scratch
  uint32_t* ucand;            // [tiles * 8]: candidates of each 512-entry unit
  uint64_t* ckey;             // [tiles * kGTile]: their keys, unit u's from 512 u
  uint32_t* cbank;            // the same slots: their banks (mixed entry sizes only)
  GBinSet* hb;                // [kGPasses]: summed bins of the passes after the first
  uint32_t* err;              // the context's error word (a barrier that timed out)
};

// Scores of every entry; with gh.st set (and a fixed-width kernel), also the
// first digit pass of the global threshold.  Returns through *fused whether
// that pass was done.
cudaError_t launch_score(const Banks& banks, uint64_t n_entries, int max_dim, int key_types,
                         float* scores, int sm_count, cudaStream_t stream,
                         GHist gh = GHist{}, bool* fused = nullptr);

// The bins of pass `pass` (0..kGPasses-1) of the byte-weighted radix select
// over a part of a split population (local plan: the host sums and picks);
// a no-op once the threshold is known.
cudaError_t launch_gselect(const GPlan& p, int pass, int sm_count, cudaStream_t stream);
// The digit passes from `first_pass` on (none once the state is done) and
// the compaction: kept indices and bank offsets.  One cooperative launch.
cudaError_t launch_gfinish(const GPlan& p, int first_pass, int sm_count, cudaStream_t stream);

// The whole threshold and compaction of a population of at most
// kGSmallEntries entries in at most kGSmallBanks banks, from its scores, in
// one block.  keep_all: the budget does not bind.
constexpr uint64_t kGSmallEntries = 16384;
constexpr int kGSmallBanks = 1024;
cudaError_t launch_gsmall(const Banks& banks, uint64_t entries, const float* scores, uint64_t budget,
                          bool uniform, bool keep_all, int32_t* kept_idx,
                          int32_t* kept_off, cudaStream_t stream);

// ---- Copy-on-write page pool (pcs_pool_*) ---------------------------------
// Reference counts and a free stack over caller memory.  A kernel either only
// takes pages off the stack (alloc, copy leg) or only puts pages back
// (release), never both, so the stack needs no lock.
struct PoolDev {
  uint8_t* base;       // n_pages * page_bytes, caller memory
  uint32_t* rc;        // [n_pages] table slots holding each page
  int32_t* free_ids;   // [n_pages] stack of free pages; [0, *top) valid
  int32_t* top;
  uint32_t* err;       // the context's error word
  uint64_t page_bytes; // multiple of 16
  int32_t n_pages;
  int32_t pad;
};

cudaError_t launch_pool_alloc(const PoolDev& p, int32_t* ids, int32_t n, cudaStream_t stream);
cudaError_t launch_pool_share(const PoolDev& p, const int32_t* src, int32_t* dst, int32_t n,
                              cudaStream_t stream);
// The copy leg before a write of table[entries[j]] (j < n; entries NULL: j).
cudaError_t launch_pool_cow(const PoolDev& p, int32_t* table, int64_t n_table,
                            const int32_t* entries, int32_t n, int sm_count, cudaStream_t stream);
cudaError_t launch_pool_release(const PoolDev& p, const int32_t* ids, int32_t n,
                                cudaStream_t stream);

// ---- Byte-mismatch distance (pcs_mismatch) --------------------------------
constexpr uint32_t kMmUnit = 2048;  // bytes of each pair per warp iteration

struct MmPair {
  const uint8_t* a;     // the first 16-byte vector (16-byte aligned)
  const uint8_t* b;     // the same byte of the second buffer
  uint64_t n_vec;       // 16-byte vectors from there
  uint16_t head, tail;  // single bytes before the first vector and after the last
  uint32_t shift;       // offset of b from a 16-byte boundary
};

// The plan of a call as k_mismatch's parameter: up to N pairs, or where they
// are on the device.  extra: the bytes only one buffer of a pair has.
constexpr int kMmBlob = 512;  // pairs that travel with a launch at most (24.6 KB)
template <int N>
struct MmBlob {
  MmPair pair[N];
  uint64_t unit_begin[N + 1];
  uint64_t extra[N];
  __host__ __device__ const MmPair* pairs() const { return pair; }
  __host__ __device__ const uint64_t* begins() const { return unit_begin; }
  __host__ __device__ uint64_t more(int i) const { return extra[i]; }
};
template <>
struct MmBlob<0> {
  const MmPair* pair;
  const uint64_t* unit_begin;
  __host__ __device__ const MmPair* pairs() const { return pair; }
  __host__ __device__ const uint64_t* begins() const { return unit_begin; }
  __host__ __device__ uint64_t more(int) const { return 0; }
};

// Pair i owns units [unit_begin[i], unit_begin[i+1]) (units of kMmUnit bytes
// after its head; at least one if it compares any byte); counts[i] = its
// mismatches and extra bytes.  host (at most kMmBlob pairs): the arrays are in
// host memory and travel with the launch; sums are zero on entry and on exit.
// Else they are on the device and sums[i] = extra[i] on entry.  `ticket`: a
// device word, zero on entry and on exit.
cudaError_t launch_mismatch(bool host, const MmPair* pairs, const uint64_t* unit_begin,
                            const uint64_t* extra, int32_t n, uint64_t units, uint64_t* sums,
                            uint64_t* counts, uint32_t* ticket, int sm_count, cudaStream_t stream);

// ---- Reads against buffers (pcs_classify_reads) ---------------------------
// The non-empty buffers sorted by start; maxend[i] = max(end[0..i]).
struct ReadPlan {
  const uint64_t* start;
  const uint64_t* end;
  const uint64_t* maxend;
  const uint32_t* orig;   // [n_all] caller index of each buffer: the sorted ones, then the empty
  uint32_t* bitmap;       // [ceil(n / 32)] device words, zero on entry
  uint32_t* ticket;       // a device word, zero on entry and on exit
  int32_t n;              // non-empty buffers (at least 1)
  int32_t n_all;
  uint64_t base, top;     // the first start and the largest end
  int32_t slices;         // set by the launcher: slices of the address range
  int32_t slice_shift;    // and log2 of their bytes
};
// A plan's arrays as k_classify_reads' parameter: up to N buffers, or nothing
// (they are where the plan points, on the device).
// Buffers that travel with a launch at most (3.6 KB): every block stages the
// arrays, from the constant bank an element at a time (765 buffers and 2,268
// blocks took 30.7 us that way, 15.9 us from the workspace; 128 and fewer gain
// at every length of the log).
constexpr int kReadBlob = 128;
template <int N>
struct ReadBlob {
  uint64_t start[N], end[N], maxend[N];
  uint32_t orig[N];
  void fill(const ReadPlan& p) {
    std::memcpy(start, p.start, 8 * p.n);
    std::memcpy(end, p.end, 8 * p.n);
    std::memcpy(maxend, p.maxend, 8 * p.n);
    std::memcpy(orig, p.orig, 4 * p.n_all);
  }
  __host__ __device__ const uint64_t* starts(const ReadPlan&) const { return start; }
  __host__ __device__ const uint64_t* ends(const ReadPlan&) const { return end; }
  __host__ __device__ const uint64_t* maxends(const ReadPlan&) const { return maxend; }
  __host__ __device__ const uint32_t* origs(const ReadPlan&) const { return orig; }
};
template <>
struct ReadBlob<0> {
  void fill(const ReadPlan&) {}
  __host__ __device__ const uint64_t* starts(const ReadPlan& p) const { return p.start; }
  __host__ __device__ const uint64_t* ends(const ReadPlan& p) const { return p.end; }
  __host__ __device__ const uint64_t* maxends(const ReadPlan& p) const { return p.maxend; }
  __host__ __device__ const uint32_t* origs(const ReadPlan& p) const { return p.orig; }
};
// flags[i] = a read overlaps buffer i; every flag is written.  m > 0.  host
// (at most kReadBlob buffers): the plan's arrays are in host memory and travel
// with the launch; the bitmap is zero on exit too.
cudaError_t launch_classify_reads(bool host, ReadPlan p, const uint64_t* addr,
                                  const uint64_t* bytes, int64_t m, uint8_t* flags, int sm_count,
                                  cudaStream_t stream);

// A call's descriptors from pinned host memory to device memory (both 16-byte
// aligned, readable and writable to a multiple of 16 bytes).
cudaError_t launch_upload(void* dst, const void* src, uint64_t bytes, cudaStream_t stream);

// Occupancy of the streaming kernel (blocks per SM) for the launch shape.
int stream_blocks_per_sm();

// ---- Fingerprints with no allocation (pcs_fingerprint_static) -------------
constexpr int kStaticMaxBufs = 64;         // buffers per call
constexpr uint32_t kStaticMaxNodes = 65536;  // tree nodes per call (512 KiB)

struct StaticBuf {
  const uint8_t* ptr;
  uint64_t bytes;
  uint64_t n_chunks;
  uint32_t task_begin;  // first node slot of this buffer
  uint32_t n_tasks;
  uint32_t align;       // 16, 4 or 1
  uint32_t pad;
};

// Passed by value as a kernel parameter (no device copy of the plan).
struct StaticPlan {
  StaticBuf b[kStaticMaxBufs];
  int32_t n;
  uint32_t n_tasks;
  int32_t glog2;
  int32_t pad;
};

// Device address of the fixed node scratch on the current device; the first
// call on a device looks it up (cudaGetSymbolAddress) with that device current.
cudaError_t static_scratch(uint64_t** nodes);
cudaError_t launch_fingerprint_static(const StaticPlan& plan, uint64_t* nodes, uint64_t* fp_out,
                                      cudaStream_t stream);

}  // namespace pcs
