// pcs_kernels.cu -- sm_103a kernels of the PCS hot path.
//
// k_stream<MODE>  one pass over 4 KiB chunks of many byte streams: a warp walks
//                 a range of tasks of one or two chunks; lane l moves the
//                 16-byte segments l + 32k of each chunk (every warp access is
//                 512 contiguous bytes), puts them together from the aligned
//                 vectors of a buffer off a 16-byte boundary or gathers /
//                 scatters them through a row or paged-ring layout, and folds
//                 them into the PCSFP64-v1 lane chain; a shuffle tree makes
//                 the task's node (Sec. 4 FINGERPRINT, step 1).
// k_bulk<MODE>    the moving passes (pack, restore) of aligned streams: per-warp
//                 TMA pipelines of 8 KiB tiles through shared memory, the
//                 fingerprint of each tile fused into the copy
//                 (k_bulk_shared: the same for small launches, the last
//                 tiles handed out at run time).
// k_hash          the read-only fingerprint pass of aligned buffers: a warp per
//                 8 KiB tile, plain loads into registers, 20 warps per SM.
// k_finalize<MODE> trees the task nodes of each stream into its fingerprint and
//                 writes outputs: fps / classification flags, record headers
//                 and section tables (checkpoint, Sec. 3 "The contract", I4),
//                 or the verification verdict of a restore (I1).
// k_score         cos(query, key) per bank entry, fp32, fixed order (Sec. 5).
// k_topk          per-bank radix select of the k largest (score, -index),
//                 kept indices written in ascending order (Sec. 7.5).
//
// k_gfinish       the global threshold's later digit passes and its
//                 compaction, in one cooperative launch (Sec. 7.5 variant).
//
// Only k_gfinish has blocks that wait on one another, at grid barriers of a
// cooperative launch (all blocks resident); every wait here, there and on an
// mbarrier, gives up after about two seconds and sets the timeout bit.
// Index values read from device memory are bounds-checked; a bad one is
// reported through the error word and skipped.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <mutex>

#include "pcs_internal.h"

namespace pcs {
namespace {

constexpr uint64_t kP = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kSeed = 0x5043534650363401ull;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// PCSFP64-v1 primitives
// ---------------------------------------------------------------------------

// SplitMix64 finaliser (Steele, Lea & Flood 2014).
__device__ __forceinline__ uint64_t fmix(uint64_t z) {
  z ^= z >> 30;
  z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27;
  z *= 0x94D049BB133111EBull;
  z ^= z >> 31;
  return z;
}

__device__ __forceinline__ uint64_t rotl64(uint64_t x, int r) {
  return (x << r) | (x >> (64 - r));
}

__device__ __forceinline__ uint64_t comb(uint64_t a, uint64_t b) {
  return fmix(a * kP + rotl64(b, 31));
}

__device__ __forceinline__ uint64_t ld_l2(const uint64_t* p) {
  return __ldcg(reinterpret_cast<const unsigned long long*>(p));
}

// A word of a call's descriptors: from the workspace (GLOBAL), through the
// read-only path, or from where else they are (a kernel parameter).
template <bool GLOBAL, typename T>
__device__ __forceinline__ T fetch(const T* p) {
  if constexpr (GLOBAL) return __ldg(p);
  else return *p;
}

// A hint to bring the 128-byte line holding `p` into this SM's L1.
__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// Programmatic dependent launch (sm_90 and later).  The streaming, finalising,
// scoring and top-k kernels are launched with programmatic stream
// serialisation (launch_after), so the GPU may schedule one while the kernel
// before it on the stream is still finishing.  Each calls this before it
// touches anything another kernel may write: wait until that kernel has
// completed and its writes are visible, then let the next kernel be
// scheduled.  Before this point a kernel reads only the call's descriptors
// (work lists, sections, sessions and banks): kernel parameters, words that a
// copy put into the workspace, or words that k_upload writes there.  k_upload
// releases its dependents before it writes, so the call's first kernel after
// it is launched without that attribute and starts when the words are there;
// the later ones start no sooner than the first has.
__device__ __forceinline__ void grid_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void grid_release() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency() {
  grid_wait();
  grid_release();
}

// Absorb one 16-byte segment (two little-endian words) into a lane chain.
__device__ __forceinline__ uint64_t absorb(uint64_t h, uint4 v) {
  const uint64_t w0 = static_cast<uint64_t>(v.x) | (static_cast<uint64_t>(v.y) << 32);
  const uint64_t w1 = static_cast<uint64_t>(v.z) | (static_cast<uint64_t>(v.w) << 32);
  h = (rotl64(h, 23) ^ w0) * kP;
  h = (rotl64(h, 23) ^ w1) * kP;
  return h;
}

// Fixed-order pairwise tree over the values of lanes [0, n), n <= 32; an odd
// last item is carried up.  The root ends in lane 0.
__device__ __forceinline__ uint64_t warp_tree(uint64_t v, int n, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_down_sync(kFull, v, d);
    if ((lane & (2 * d - 1)) == 0 && lane + d < n) v = comb(v, o);
  }
  return v;
}

// Tree over a[0..n) (global or shared), reduced in place by aligned groups
// of 32; every lane returns the root.  Called by one whole warp.
__device__ uint64_t warp_tree_inplace(uint64_t* a, uint32_t n, int lane) {
  while (n > 1) {
    const uint32_t groups = (n + 31) / 32;
    for (uint32_t g = 0; g < groups; ++g) {
      const uint32_t i = 32 * g + lane;
      const uint64_t v = i < n ? a[i] : 0;
      const uint32_t m = min(32u, n - 32 * g);
      const uint64_t r = warp_tree(v, static_cast<int>(m), lane);
      __syncwarp();
      if (lane == 0) a[g] = r;
      __syncwarp();
    }
    n = groups;
  }
  return a[0];
}

// The same tree for n <= 1024, nothing written; called by one whole warp,
// every lane returns the root.  L2: the items are read past L1 (a small call's
// are written by other blocks of the same launch; elsewhere L1 serves seven
// of a lane's eight loads: without it the step of 32 KV contexts lost 0.5 %).  Up to 32 items: one warp tree.  Beyond,
// in blocks of 256 items: lane l reads items 8l .. 8l+7 of the block and
// reduces them in its registers (the tree's first three levels over that
// aligned group of eight, an odd last item carried up), the warp then
// reduces the 32 group roots (five more levels), and the roots of up to four
// blocks end the tree.  Aligned groups of 2^m items reduce to the nodes of
// the global pairwise tree, so the root is the same; all 32 lanes combine
// at once, where trees of 32-item groups leave half the lanes idle at each
// level (a 256-item tree took 1,790 warp instructions that way).
template <bool L2>
__device__ uint64_t warp_tree_regs(const uint64_t* a, uint32_t n, int lane) {
  auto item = [&](uint32_t i) { return L2 ? ld_l2(a + i) : a[i]; };
  if (n <= 32) {
    const uint64_t v = lane < static_cast<int>(n) ? item(lane) : 0;
    return __shfl_sync(kFull, warp_tree(v, static_cast<int>(n), lane), 0);
  }
  const uint32_t blocks = (n + 255) / 256;
  uint64_t block_root = 0;  // root of block b, kept in lane b
  for (uint32_t b = 0; b < blocks; ++b) {
    const uint32_t base = 256 * b;
    const uint32_t nb = min(256u, n - base);
    const int m = max(0, min(8, static_cast<int>(nb) - 8 * lane));  // this lane's items
    uint64_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = i < m ? item(base + 8 * lane + i) : 0;
#pragma unroll
    for (int w = 1; w < 8; w <<= 1)
#pragma unroll
      for (int i = 0; i + w < 8; i += 2 * w)
        if (i + w < m) v[i] = comb(v[i], v[i + w]);
    const uint64_t r = __shfl_sync(kFull, warp_tree(v[0], static_cast<int>((nb + 7) / 8), lane), 0);
    if (lane == static_cast<int>(b)) block_root = r;
  }
  const uint64_t root = blocks > 1 ? warp_tree(block_root, static_cast<int>(blocks), lane) : block_root;
  return __shfl_sync(kFull, root, 0);
}

// Tree of a 2-chunk tile, both chunks at once.  Lane l holds a0 = lane value
// l of chunk 0 and a1 = lane value l of chunk 1.  Level 1 puts chunk q's pair
// (2i, 2i+1) in lane 16q + i; from then on the pair of every level is in lanes
// (2L, 2L+1), so each level is one comb across the warp.  After five levels
// lane q holds chunk q's hash; with nc == 2 one more level gives the tile's
// node comb(x0, x1) (the pairwise tree over its chunks).  Result in lane 0.
__device__ __forceinline__ uint64_t tile_tree2(uint64_t a0, uint64_t a1, int nc, int lane) {
  const int i = lane & 15;
  const uint64_t l0 = __shfl_sync(kFull, a0, 2 * i), r0 = __shfl_sync(kFull, a0, 2 * i + 1);
  const uint64_t l1 = __shfl_sync(kFull, a1, 2 * i), r1 = __shfl_sync(kFull, a1, 2 * i + 1);
  uint64_t v = lane < 16 ? comb(l0, r0) : comb(l1, r1);
  const int levels = nc == 2 ? 5 : 4;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    if (k < levels) {
      const uint64_t l = __shfl_sync(kFull, v, (2 * lane) & 31);
      const uint64_t r = __shfl_sync(kFull, v, (2 * lane + 1) & 31);
      v = comb(l, r);
    }
  }
  return v;
}

// ---------------------------------------------------------------------------
// Memory helpers
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint4 ld_stream(const uint8_t* p) {
  return __ldcs(reinterpret_cast<const uint4*>(p));
}

__device__ __forceinline__ void st_stream(uint8_t* p, uint4 v) {
  __stcs(reinterpret_cast<uint4*>(p), v);
}

// Bytes [0, n) of a segment (n <= 16) at an address that may not be 16-byte
// aligned; whole 32-bit words when `a4` (4-byte aligned).  The rest read as 0.
__device__ __forceinline__ uint4 ld_small(const uint8_t* p, int n, bool a4) {
  uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (a4 && 4 * j + 4 <= n) {
      w[j] = *reinterpret_cast<const uint32_t*>(p + 4 * j);
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (4 * j + b < n) w[j] |= static_cast<uint32_t>(p[4 * j + b]) << (8 * b);
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Bytes [s, s + 16) of the 32 bytes lo : hi (s in [0, 16)): two word selects
// and four funnel shifts, no branch on s.
__device__ __forceinline__ uint4 align_bytes(uint4 lo, uint4 hi, uint32_t s) {
  const bool w2 = s & 8u, w1 = s & 4u;
  const uint32_t bits = (s & 3u) * 8u;
  const uint32_t u0 = w2 ? lo.z : lo.x, u1 = w2 ? lo.w : lo.y, u2 = w2 ? hi.x : lo.z,
                 u3 = w2 ? hi.y : lo.w, u4 = w2 ? hi.z : hi.x, u5 = w2 ? hi.w : hi.y;
  const uint32_t t0 = w1 ? u1 : u0, t1 = w1 ? u2 : u1, t2 = w1 ? u3 : u2, t3 = w1 ? u4 : u3,
                 t4 = w1 ? u5 : u4;
  return make_uint4(__funnelshift_r(t0, t1, bits), __funnelshift_r(t1, t2, bits),
                    __funnelshift_r(t2, t3, bits), __funnelshift_r(t3, t4, bits));
}

// Zero the bytes of a segment at or past `n` (n in [1, 16)).
__device__ __forceinline__ uint4 mask_tail(uint4 v, int n) {
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int keep = n - 4 * j;  // bytes of word j to keep
    if (keep <= 0) w[j] = 0;
    else if (keep < 4) w[j] &= (1u << (8 * keep)) - 1u;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ uint64_t div_rows(uint64_t x, uint64_t d, int shift) {
  return shift >= 0 ? (x >> shift) : (x / d);
}

// Address of row r of a ROWS / RING stream (null if its id is out of range).
__device__ __forceinline__ uint8_t* row_ptr(const SecDesc& s, uint64_t r, uint32_t* err) {
  uint64_t id, row;
  if (s.layout == kRows) {
    id = static_cast<uint32_t>(__ldg(s.index + r));
    row = id;
  } else {
    // RING: logical row r sits in ring slot (start + r) mod window.
    uint64_t slot = s.ring_start + r;
    if (slot >= s.window) slot -= s.window;
    const uint64_t pg = div_rows(slot, s.page_rows, s.pr_shift);
    id = static_cast<uint32_t>(__ldg(s.index + pg));
    row = id * s.page_rows + (slot - pg * s.page_rows);
  }
  if (id >= s.base_rows) {
    atomicOr(err, kDevErrIndex);
    return nullptr;
  }
  return s.lbase + row * s.row_bytes;
}

// Address of logical byte `off` (a multiple of 16) on the layout side of a
// ROWS / RING stream, or null if its row / page id is out of range.
__device__ __forceinline__ uint8_t* row_addr(const SecDesc& s, uint64_t off, uint32_t* err) {
  const uint64_t y = off + s.row_shift;
  const uint64_t r = div_rows(y, s.row_bytes, s.rb_shift);
  uint8_t* p = row_ptr(s, r, err);
  return p ? p + (y - r * s.row_bytes) : nullptr;
}

// ---------------------------------------------------------------------------
// Streaming kernel
// ---------------------------------------------------------------------------

constexpr int kSegs = 8;  // 16-byte segments per lane per chunk

template <int MODE>
struct ModeTraits {
  static constexpr bool kHash = MODE == kModeHash || MODE == kModePack || MODE == kModeRestoreV;
  static constexpr bool kLoadLayout = MODE == kModeHash || MODE == kModePack;
  static constexpr bool kStore = MODE != kModeHash;
};

// Bytes of the aligned 16-byte vector at `p` that lie in logical bytes [0, L)
// when its first byte is logical byte `off` (negative before the buffer); the
// rest 0.  Words wholly inside are loaded as words.
__device__ __forceinline__ uint4 ld_edge(const uint8_t* p, int64_t off, int64_t L) {
  const int from = off < 0 ? static_cast<int>(-off) : 0;                  // bytes [from, to)
  const int to = L - off < 16 ? static_cast<int>(L - off) : 16;
  uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (4 * j >= from && 4 * j + 4 <= to) {
      w[j] = *reinterpret_cast<const uint32_t*>(p + 4 * j);
    } else if (4 * j + 4 > from && 4 * j < to) {
#pragma unroll
      for (int b = 4 * j; b < 4 * j + 4; ++b)
        if (b >= from && b < to) w[j] |= static_cast<uint32_t>(p[b]) << (8 * (b & 3));
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Store the bytes of `v` that lie in logical bytes [0, L).
__device__ __forceinline__ void st_edge(uint8_t* p, uint4 v, int64_t off, int64_t L) {
  const int from = off < 0 ? static_cast<int>(-off) : 0;
  const int to = L - off < 16 ? static_cast<int>(L - off) : 16;
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (4 * j >= from && 4 * j + 4 <= to) {
      *reinterpret_cast<uint32_t*>(p + 4 * j) = w[j];
    } else if (4 * j + 4 > from && 4 * j < to) {
#pragma unroll
      for (int b = 4 * j; b < 4 * j + 4; ++b)
        if (b >= from && b < to) p[b] = static_cast<uint8_t>(w[j] >> (8 * (b & 3)));
    }
  }
}

// The value of the next (prev) lane; lane 31 (0) gets lane 0's (31's) `wrap`.
__device__ __forceinline__ uint4 from_next_lane(uint4 v, uint4 wrap, int lane) {
  const uint4 x = lane == 0 ? wrap : v;
  const int src = (lane + 1) & 31;
  return make_uint4(__shfl_sync(kFull, x.x, src), __shfl_sync(kFull, x.y, src),
                    __shfl_sync(kFull, x.z, src), __shfl_sync(kFull, x.w, src));
}
__device__ __forceinline__ uint4 from_prev_lane(uint4 v, uint4 wrap, int lane) {
  const uint4 x = lane == 31 ? wrap : v;
  const int src = (lane + 31) & 31;
  return make_uint4(__shfl_sync(kFull, x.x, src), __shfl_sync(kFull, x.y, src),
                    __shfl_sync(kFull, x.z, src), __shfl_sync(kFull, x.w, src));
}

// Segments of chunks [c, c + NC) of a stream, from its read side: v[k] = bytes
// [16 (lane + 32 k), + 16) from c * 4096, zero past the end.  A contiguous
// buffer off a 16-byte boundary is read in the aligned vectors it touches,
// each once: a segment straddles two of them, the second being the next
// lane's.  INSIDE: every byte the chunks and their two neighbouring vectors
// cover lies inside the stream; otherwise the vectors that reach outside the
// buffer, its first and its last, are read by words and bytes.  Called by a
// whole warp.
template <int MODE, int NC, bool INSIDE>
__device__ __forceinline__ void load_chunks(const SecDesc& s, uint64_t c, int lane,
                                            uint4 (&v)[NC * kSegs], uint32_t* err) {
  constexpr int NK = NC * kSegs;
  const uint4 z = make_uint4(0, 0, 0, 0);
  const uint64_t base = c * kChunkBytes;
  if (ModeTraits<MODE>::kLoadLayout && s.layout != kContig) {
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const uint64_t off = base + 512u * k + 16u * lane;
      v[k] = z;
      if (INSIDE || off < s.bytes) {
        const uint8_t* p = row_addr(s, off, err);
        if (p) v[k] = ld_stream(p);
      }
    }
    return;
  }
  // A record's payload is 256-byte aligned and padded to 256 bytes: whole
  // segments are readable, the bytes past the end are masked below.
  const uint8_t* src = ModeTraits<MODE>::kLoadLayout ? s.lbase : s.payload;
  const int64_t L = static_cast<int64_t>(
      ModeTraits<MODE>::kLoadLayout ? s.bytes : (s.bytes + 15) & ~15ull);
  const uint32_t sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src) & 15u);
  const uint8_t* p = src - sh + base + 16u * lane;                   // this lane's vector 0
  const int64_t off = static_cast<int64_t>(base + 16u * lane) - sh;  // and its logical byte
  uint4 extra = z;  // lane 0: the vector after the last one (off a boundary only)
  auto whole = [&](int k) { return INSIDE || (off + 512 * k >= 0 && off + 512 * k + 16 <= L); };
#pragma unroll
  for (int k = 0; k < NK; ++k) v[k] = whole(k) ? ld_stream(p + 512u * k) : z;
  if (ModeTraits<MODE>::kLoadLayout) {
    if (sh != 0 && lane == 0 && whole(NK)) extra = ld_stream(p + 512u * NK);
    if (!INSIDE) {
      // The vector the buffer's end lies in: `last`, of lane last mod 32.
      const int64_t last = ((L + sh) >> 4) - static_cast<int64_t>(base >> 4);
      if (((L + sh) & 15) && last >= 0 && last <= 32 * NK && lane == (last & 31)) {
        const uint4 x = ld_edge(p + 16 * (last - lane), off + 16 * (last - lane), L);
        const int kl = static_cast<int>(last >> 5);
#pragma unroll
        for (int k = 0; k < NK; ++k)
          if (k == kl) v[k] = x;
        if (kl == NK) extra = x;
      }
      if (off < 0 && off > -16) v[0] = ld_edge(p, off, L);
    }
    if (sh != 0) {
      // Segments past the end are zero (the vector there may hold the
      // buffer's last bytes, which belong to the segment before).
      const int64_t used = INSIDE ? NK : (L - static_cast<int64_t>(base) + 511) >> 9;
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        if (INSIDE || k < used)
          v[k] = align_bytes(
              v[k], from_next_lane(v[k], k + 1 < NK ? v[k + 1 < NK ? k + 1 : k] : extra, lane), sh);
        else
          v[k] = z;
      }
    }
  } else if (!INSIDE && (s.bytes & 15u)) {
    // Payload bytes past the logical end read as zero.
    const uint64_t tail = s.bytes & ~15ull;
#pragma unroll
    for (int k = 0; k < NK; ++k)
      if (base + 512u * k + 16u * lane == tail)
        v[k] = mask_tail(v[k], static_cast<int>(s.bytes & 15u));
  }
}

// Store the segments of chunks [c, c + NC) to the stream's write side.  A
// contiguous target off a 16-byte boundary is written in its aligned vectors:
// each takes the end of one segment, the previous lane's, and the beginning
// of the next; the segment before the chunks is read again from the payload.
// INSIDE as above.  Called by a whole warp.
template <int MODE, int NC, bool INSIDE>
__device__ __forceinline__ void store_chunks(const SecDesc& s, uint64_t c, int lane,
                                             const uint4 (&v)[NC * kSegs], uint32_t* err) {
  constexpr int NK = NC * kSegs;
  const uint64_t base = c * kChunkBytes;
  if (MODE == kModePack) {
    // Record payload: write through the 256-byte padding (zeros past the end).
    const uint64_t padded = (s.bytes + kRecordAlign - 1) / kRecordAlign * kRecordAlign;
#pragma unroll
    for (int k = 0; k < NK; ++k)
      if (INSIDE || base + 512u * k + 16u * lane < padded)
        st_stream(s.payload + base + 512u * k + 16u * lane, v[k]);
    return;
  }
  if (s.layout != kContig) {
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const uint64_t off = base + 512u * k + 16u * lane;
      if (INSIDE || off < s.bytes) {
        uint8_t* p = row_addr(s, off, err);
        if (p) st_stream(p, v[k]);
      }
    }
    return;
  }
  const uint32_t sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(s.lbase) & 15u);
  const int64_t L = static_cast<int64_t>(s.bytes);
  uint8_t* p = s.lbase - sh + base + 16u * lane;
  const int64_t off = static_cast<int64_t>(base + 16u * lane) - sh;
  // The target's vector that its end lies in: `last`, of lane last mod 32.
  const int64_t last = ((L + sh) >> 4) - static_cast<int64_t>(base >> 4);
  uint4 first_x = make_uint4(0, 0, 0, 0), last_x = first_x;
  auto put = [&](int k, uint4 x) {
    if (INSIDE || (off + 512 * k >= 0 && off + 512 * k + 16 <= L)) st_stream(p + 512u * k, x);
    if (!INSIDE && k == 0) first_x = x;
    if (!INSIDE && k == (last >> 5)) last_x = x;
  };
  if (sh == 0) {
#pragma unroll
    for (int k = 0; k < NK; ++k) put(k, v[k]);
  } else {
    uint4 before = make_uint4(0, 0, 0, 0);  // lane 31: the segment before the chunks
    if (lane == 31 && c > 0) before = ld_stream(s.payload + base - 16);
    const int64_t used = INSIDE ? NK : (L + sh - static_cast<int64_t>(base) + 511) >> 9;
#pragma unroll
    for (int k = 0; k < NK; ++k)
      if (INSIDE || k < used)
        put(k, align_bytes(from_prev_lane(v[k], k > 0 ? v[k > 0 ? k - 1 : 0] : before, lane), v[k],
                           16 - sh));
  }
  if (!INSIDE && ((L + sh) & 15) && last >= 0) {
    // The vector holding the end: one of these, or (of the last chunk only)
    // the one after them, which takes the end of the last segment.
    const int64_t o = 16 * (last - lane);
    if (last < 32 * NK) {
      if (lane == (last & 31) && off + o >= 0) st_edge(p + o, last_x, off + o, L);
    } else if (last == 32 * NK && lane == 31 && c + NC == s.n_chunks) {
      st_edge(p + o, align_bytes(v[NK - 1], make_uint4(0, 0, 0, 0), 16 - sh), off + o, L);
    }
  }
  if (!INSIDE && off < 0) st_edge(p, first_x, off, L);
}

// Move chunks [c, c + NC) and return their node: one chunk's hash, or the
// pair's (0 in the modes that do not hash).
template <int MODE, int NC, bool INSIDE>
__device__ __forceinline__ uint64_t move_chunks(const SecDesc& s, uint64_t c, int lane,
                                                uint32_t* err) {
  using T = ModeTraits<MODE>;
  uint4 v[NC * kSegs];
  load_chunks<MODE, NC, INSIDE>(s, c, lane, v, err);
  if (T::kStore) store_chunks<MODE, NC, INSIDE>(s, c, lane, v, err);
  if (!T::kHash) return 0;
  uint64_t h[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) h[q] = fmix(kSeed ^ ((c + q) * 32u + lane));
#pragma unroll
  for (int k = 0; k < kSegs; ++k)
#pragma unroll
    for (int q = 0; q < NC; ++q) h[q] = absorb(h[q], v[q * kSegs + k]);
  const uint64_t x = NC == 2 ? tile_tree2(fmix(h[0]), fmix(h[NC - 1]), 2, lane)
                             : warp_tree(fmix(h[0]), 32, lane);
  return __shfl_sync(kFull, x, 0);
}

// Section of warp task `task` in a work list: the last j with begin[j] <=
// task (begin rises), searched from item `lo` on (begin[lo] <= task; lo = 0
// searches the whole list, begin[0] = 0).  Called by a whole warp with a
// warp-uniform task: each round the lanes probe 32 evenly spaced entries of
// the range still open and keep the part after the last probe <= task, so
// that 12,544 items take three dependent loads instead of fourteen.
template <bool GLOBAL = true>
__device__ __forceinline__ int find_item(const uint32_t* begin, int lo, int n_items, uint32_t task,
                                         int lane) {
  int span = n_items - lo;  // the answer lies in [lo, lo + span)
  while (span > 1) {
    const int step = (span + 31) >> 5;
    const int i = lo + lane * step;
    const bool le = i < lo + span && fetch<GLOBAL>(begin + i) <= task;
    const unsigned m = __ballot_sync(kFull, le);  // lane 0 probes lo: never empty
    const int last = 31 - __clz(m);
    lo += last * step;
    span = min(step, span - last * step);
  }
  return lo;
}

// The warp tasks of one streaming pass (body of k_stream and k_small): each
// warp walks a contiguous, balanced range of tasks of 2^glog2 chunks, glog2 =
// 0 or 1, so that the item of a task is searched for once per warp.  After
// each task it calls after_task(its stream, its work list item).
//
// Buffers off a 16-byte boundary are bound by the 16 warps per SM that 128
// registers leave (two chunks of loads each) and by issue: per segment four
// shuffles and a funnel beside the hash.  Measured (byte and word loads of
// each lane's own segment, interleaved tasks -> this): fingerprint of 1 GiB at
// an odd address 1,263 -> 220 us (4.9 TB/s), at a 4-byte one 405 -> 220 us;
// 2,000 observations of 196,613 bytes, three of four off a boundary: pack 693 ->
// 184 us, verified restore 862 -> 211 us.
template <int MODE, bool GLOBAL, typename F>
__device__ __forceinline__ void run_stream_tasks(const SecDesc* secs, const WorkList& wl,
                                                 int glog2, uint64_t* __restrict__ nodes,
                                                 uint32_t* err, SecDesc* sdesc, bool beside,
                                                 F&& after_task) {
  using T = ModeTraits<MODE>;
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const uint64_t gw = static_cast<uint64_t>(blockIdx.x) * kWarps + wib;
  const uint64_t nw = static_cast<uint64_t>(gridDim.x) * kWarps;
  const uint32_t t0 = static_cast<uint32_t>(wl.n_tasks * gw / nw);
  const uint32_t t1 = static_cast<uint32_t>(wl.n_tasks * (gw + 1) / nw);
  // The work list and the descriptors are there before the kernel starts: the
  // first task's are read before waiting for the kernel ahead.
  const SecDesc& s = sdesc[wib];
  auto load_desc = [&](int j) {
    const SecDesc* src = &secs[fetch<GLOBAL>(wl.ids + j)];
    __syncwarp();
    if (lane < static_cast<int>(sizeof(SecDesc) / 16))
      reinterpret_cast<uint4*>(&sdesc[wib])[lane] =
          fetch<GLOBAL>(reinterpret_cast<const uint4*>(src) + lane);
    __syncwarp();
  };
  int j = 0, cur = -1;
  if (t0 < t1) load_desc(cur = j = find_item<GLOBAL>(wl.begin, 0, wl.n_items, t0, lane));
  if (beside) grid_release();
  else grid_dependency();
  for (uint32_t task = t0; task < t1; ++task) {
    while (j + 1 < wl.n_items && fetch<GLOBAL>(wl.begin + j + 1) <= task) ++j;
    if (j != cur) load_desc(cur = j);
    const uint32_t local = task - fetch<GLOBAL>(wl.begin + j);
    const uint64_t c0 = static_cast<uint64_t>(local) << glog2;
    const uint64_t c1 = min(c0 + (1ull << glog2), static_cast<unsigned long long>(s.n_chunks));
    // A pair whose chunks and neighbouring vectors lie inside the stream takes
    // the unchecked path; the ends of a stream go a chunk at a time.
    uint64_t x;
    if (c0 + 1 < c1 && c0 > 0 && (c0 + 2) * kChunkBytes + 16 <= s.bytes) {
      x = move_chunks<MODE, 2, true>(s, c0, lane, err);
    } else {
      x = move_chunks<MODE, 1, false>(s, c0, lane, err);
      if (c0 + 1 < c1) {
        const uint64_t y = move_chunks<MODE, 1, false>(s, c0 + 1, lane, err);
        if (T::kHash) x = comb(x, y);
      }
    }
    if (T::kHash && lane == 0) nodes[s.task_begin + local] = x;
    after_task(s, j);
  }
}

// beside: the kernel ahead on the stream is the TMA (or hash) kernel of the
// same call, which shares nothing with this one, so this one runs beside it
// and waits for it only before it ends (what follows them waits for both so).
// It can start once every block ahead has passed its own wait, so whatever
// came before the call is finished and visible by then.  Measured, whole
// calls: planned checkpoint + restore of 5 odd observations 14.7 -> 11.6 us, of
// 37 29.0 -> 22.4; 36 banks with 64-wide keys, planned, 80.8 -> 75.6; the
// classification of packed buffers 90.3 -> 87.7.
template <int MODE>
__global__ void __launch_bounds__(kThreads, 2)
    k_stream(const SecDesc* __restrict__ secs, WorkList wl, int glog2,
             uint64_t* __restrict__ nodes, uint32_t* err, bool beside) {
  __shared__ SecDesc sdesc[kWarps];
  run_stream_tasks<MODE, true>(secs, wl, glog2, nodes, err, sdesc, beside,
                               [](const SecDesc&, int) {});
  if (beside) grid_wait();
}

// ---------------------------------------------------------------------------
// TMA-staged streaming kernel
//
// Every warp runs its own pipeline over a contiguous range of tiles; a tile
// is 2 chunks (8 KiB) of one stream in payload order.  A warp owns
// kWarpStages shared-memory stages: it stages tile i + kWarpStages while it
// works on tile i.  Staging is one cp.async.bulk copy per run of rows that
// are contiguous in memory (or one copy of the contiguous payload), all
// completing on the stage's mbarrier; working on a tile = hash its chunks
// from shared memory, issue the bulk store of the tile (to the payload, or
// one per row run of the layout side), and wait until the store has read
// the stage.  Warps never wait on each other.  Every wait is bounded; a wait
// that gives up records kDevErrTimeout and the warp stops.
// ---------------------------------------------------------------------------

constexpr int kTileChunks = kBulkTileChunks;
constexpr uint32_t kTileBytes = kTileChunks * kChunkBytes;

// Shape of the TMA kernel (the moving modes: pack, restore, verified
// restore): warps per block and stages per warp, 3 tiles per warp in flight.
// The read-only hash pass has a kernel of its own (k_hash, below).
template <int MODE>
struct BulkShape {
  static_assert(MODE != kModeHash, "the hash-only pass runs in k_hash");
  static constexpr int kWarps = 8;
  static constexpr int kStages = 3;
  static constexpr int kThreads = 32 * kWarps;
};
// Copies one contiguous 8 KiB load of a hashing pass is split into (1 KiB
// each).  Measured, 4,096 and 16,384 Markov sessions of 192 KiB: pack 0.308
// -> 0.276 ms and 1.105 -> 1.001 ms, verified restore 0.304 -> 0.268 ms and
// 1.108 -> 0.993 ms (2, 4 and 16 pieces gained less).  Plain
// restores keep one copy (a fork of 256 KV records lost 1.3 % with pieces),
// and so do loads of a restore into rows (split, the KV step's verified
// restore took twice as long).
constexpr int kContigPieces = 8;
static_assert(kTileBytes / kContigPieces % 16 == 0 && kContigPieces <= 32, "pieces");
// Work sharing of the TMA kernel.  With static ranges alone, warps given
// equal tile counts finish up to 10-25 % apart (a per-warp %globaltimer
// probe: 4,096 Markov sessions 226-263 us, median 236; 64 banks 69-92 us,
// median 79).  A launch of fewer than kDynMaxTilesPerWarp tiles per warp
// runs k_bulk_shared: 1 / kDynShare of its tiles (the last ones) are handed
// out at run time, in chunks of up to kDynChunkMax tiles, about
// kDynGrabsPerWarp per warp.  Measured (alternating builds, one box): the
// 64-bank step 0.273 -> 0.261 ms; at 84 tiles per warp (4,096 Markov
// sessions) no change; at 2,587 (the 256-session KV step) sharing 1/4 or 1/8
// made the step 0.7-1.5 % slower, so large launches keep static ranges.
constexpr uint32_t kDynMaxTilesPerWarp = 64;
constexpr uint32_t kDynShare = 8;
constexpr uint32_t kDynGrabsPerWarp = 8;
constexpr uint32_t kDynChunkMax = 32;
constexpr int kTileRows = 32;  // rows >= 512 bytes touching an 8 KiB tile: at most 17 (18 of a ring)
constexpr long long kWaitCycles = 4000000000ll;  // give up a wait after ~2 s of SM clock
static_assert(kTileBytes / kBulkMinRowBytes + 2 <= kTileRows, "tile rows");

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase of `bar` with the given parity to complete.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}

__device__ __forceinline__ void bulk_g2s(void* sdst, const void* gsrc, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(sdst)),
      "l"(gsrc), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void bulk_s2g(void* gdst, const void* ssrc, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst),
               "r"(smem_u32(ssrc)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// What a stage holds (written by the warp when it stages the tile).
struct WarpStage {
  SecDesc d;                // the tile's stream
  uint32_t sec;             // its index (0xFFFFFFFF: none yet)
  uint64_t p0, p1;          // payload bytes of the tile: [p0, p1)
  uint64_t r0;              // first row touching the tile (ROWS / RING)
  uint32_t node;            // node slot of the tile
  uint32_t n_rows;          // rows touching [p0, min(p1, L))
  uint8_t* rowp[kTileRows]; // layout-side address of each row (null = out of range)
};

template <int W, int S>
struct BulkShared {
  alignas(128) uint8_t buf[W][S][kTileBytes];
  alignas(8) uint64_t bar[W][S];
  WarpStage st[W][S];
};

// End of the bytes of tile [p0, p1) that bulk copies stage: the layout side
// up to its last whole 16-byte segment; the payload (padded to 256 bytes in
// the record) up to its 16-byte-rounded end.
template <int MODE>
__device__ __forceinline__ uint64_t staged_end(const SecDesc& s, uint64_t p1) {
  const uint64_t end =
      ModeTraits<MODE>::kLoadLayout ? (s.bytes & ~15ull) : ((s.bytes + 15) & ~15ull);
  return p1 < end ? p1 : end;
}

// Bytes of [p0, pe) that row i of a stage covers.  SHIFT: some stream of the
// launch begins inside its first row (row_shift), whose own first byte then
// lies before the stream's.  Launches without any keep the unsigned form, in
// kernels of their own: the TMA kernels' timing follows the code of their
// staging (with the signed form for all, 32 KV contexts packed in 990 us
// instead of 979 and came back in 979 instead of 989).
template <bool SHIFT>
__device__ __forceinline__ uint32_t row_share(const WarpStage& m, uint64_t rb, int i, uint64_t pe) {
  if constexpr (SHIFT) {
    const int64_t lo = static_cast<int64_t>((m.r0 + i) * rb) - static_cast<int64_t>(m.d.row_shift);
    const int64_t hi = lo + static_cast<int64_t>(rb);
    const int64_t a = max(lo, static_cast<int64_t>(m.p0)), b = min(hi, static_cast<int64_t>(pe));
    return b > a ? static_cast<uint32_t>(b - a) : 0u;
  } else {
    const uint64_t lo = (m.r0 + i) * rb, hi = lo + rb;
    const uint64_t a = lo > m.p0 ? lo : m.p0, b = hi < pe ? hi : pe;
    return b > a ? static_cast<uint32_t>(b - a) : 0u;
  }
}

// Bulk copies between a stage's buffer and the layout side, one per run of
// rows contiguous in memory, covering payload bytes [m.p0, pe).  Lane i owns
// row i (address rp; null = skipped).  Returns the bytes this lane copied.
template <bool kLoad, bool SHIFT>
__device__ __forceinline__ uint32_t issue_runs(const WarpStage& m, uint8_t* rp, uint64_t pe,
                                               uint8_t* tile, uint64_t* bar, int lane) {
  const uint64_t rb = m.d.row_bytes;
  const int n = static_cast<int>(m.n_rows);
  const uintptr_t u = reinterpret_cast<uintptr_t>(rp);
  const uintptr_t prev = __shfl_up_sync(kFull, u, 1);
  const bool start = lane < n && (lane == 0 || u == 0 || prev == 0 || u != prev + rb);
  const unsigned starts = __ballot_sync(kFull, start);
  if (!start || rp == nullptr) return 0;
  const unsigned later = lane < 31 ? (starts >> (lane + 1)) : 0u;
  const int next = later ? lane + __ffs(later) : n;
  if constexpr (SHIFT) {
    const int64_t sh = static_cast<int64_t>(m.d.row_shift);
    const int64_t row_lo = static_cast<int64_t>((m.r0 + lane) * rb) - sh;
    const int64_t row_hi = static_cast<int64_t>((m.r0 + next) * rb) - sh;
    const int64_t a = max(row_lo, static_cast<int64_t>(m.p0));
    const int64_t b = min(row_hi, static_cast<int64_t>(pe));
    if (a >= b) return 0;
    uint8_t* g = rp + (a - row_lo);
    uint8_t* sp = tile + (a - static_cast<int64_t>(m.p0));
    if (kLoad) bulk_g2s(sp, g, static_cast<uint32_t>(b - a), bar);
    else bulk_s2g(g, sp, static_cast<uint32_t>(b - a));
    return static_cast<uint32_t>(b - a);
  } else {
    const uint64_t row_lo = (m.r0 + lane) * rb, row_hi = (m.r0 + next) * rb;
    const uint64_t a = row_lo > m.p0 ? row_lo : m.p0;
    const uint64_t b = row_hi < pe ? row_hi : pe;
    if (a >= b) return 0;
    uint8_t* g = rp + (a - row_lo);
    uint8_t* sp = tile + (a - m.p0);
    if (kLoad) bulk_g2s(sp, g, static_cast<uint32_t>(b - a), bar);
    else bulk_s2g(g, sp, static_cast<uint32_t>(b - a));
    return static_cast<uint32_t>(b - a);
  }
}

// Copy the descriptor of section `sec` into a stage (a whole warp; nothing
// is read when the stage already holds it).
__device__ __forceinline__ void stage_desc(const SecDesc* __restrict__ secs, uint32_t sec,
                                           WarpStage& st, int lane) {
  if (st.sec != sec) {  // warp-uniform
    __syncwarp();
    if (lane < static_cast<int>(sizeof(SecDesc) / 16))
      reinterpret_cast<uint4*>(&st.d)[lane] = __ldg(reinterpret_cast<const uint4*>(secs + sec) + lane);
    if (lane == 0) st.sec = sec;
  }
  __syncwarp();
}

// Stage tile t (of work list item `item`) into stage `st` / barrier `bar`.
template <int MODE, bool SHIFT>
__device__ __forceinline__ void stage_tile(const SecDesc* __restrict__ secs, const WorkList& wl,
                                           int item, uint32_t t, WarpStage& st, uint8_t* tile,
                                           uint64_t* bar, uint32_t* err, int lane) {
  using T = ModeTraits<MODE>;
  const uint32_t sec = __ldg(wl.ids + item);
  const uint32_t loc = t - __ldg(wl.begin + item);
  stage_desc(secs, sec, st, lane);
  const SecDesc& s = st.d;
  const uint64_t L = s.bytes;
  const uint64_t p0 = static_cast<uint64_t>(loc) * kTileBytes;
  const uint64_t cend = s.n_chunks * kChunkBytes;
  const uint64_t p1 = p0 + kTileBytes < cend ? p0 + kTileBytes : cend;
  const uint64_t pe = staged_end<MODE>(s, p1);
  uint64_t r0 = 0;
  uint32_t n_rows = 0;
  uint8_t* rp = nullptr;
  if (s.layout != kContig) {
    const uint64_t sh = SHIFT ? s.row_shift : 0;  // (0: as if it were not there)
    r0 = div_rows(p0 + sh, s.row_bytes, s.rb_shift);
    const uint64_t lim = L < p1 ? L : p1;
    if (lim > p0)
      n_rows = static_cast<uint32_t>(div_rows(lim - 1 + sh, s.row_bytes, s.rb_shift) + 1 - r0);
    if (lane < static_cast<int>(n_rows)) rp = row_ptr(s, r0 + lane, err);
    st.rowp[lane] = rp;
  }
  if (lane == 0) {
    st.p0 = p0;
    st.p1 = p1;
    st.r0 = r0;
    st.node = s.task_begin + loc;
    st.n_rows = n_rows;
  }
  __syncwarp();
  if (!T::kLoadLayout || s.layout == kContig) {
    // One contiguous piece: the record payload, or a contiguous buffer.  A
    // hashing pass whose layout side is contiguous (a pack from a
    // contiguous buffer, a verified restore into one) loads it as
    // kContigPieces copies issued by as many lanes.
    const uint32_t bytes = pe > p0 ? static_cast<uint32_t>(pe - p0) : 0u;
    const int pieces = (T::kHash && s.layout == kContig) ? kContigPieces : 1;
    if (lane == 0) mbar_arrive_expect_tx(bar, bytes);
    __syncwarp();
    if (lane < pieces && bytes) {
      const uint32_t piece = ((bytes + pieces - 1) / pieces + 15u) & ~15u;
      const uint32_t lo = static_cast<uint32_t>(lane) * piece;
      const uint32_t hi = lo + piece < bytes ? lo + piece : bytes;
      if (hi > lo) bulk_g2s(tile + lo, (T::kLoadLayout ? s.lbase : s.payload) + p0 + lo, hi - lo, bar);
    }
    return;
  }
  // Rows: zero the share of rows whose id was out of range, arm the barrier
  // with the bytes the copies will bring, then one bulk copy per run.
  uint32_t mine = 0;
  if (lane < static_cast<int>(n_rows)) {
    const uint32_t share = row_share<SHIFT>(st, s.row_bytes, lane, pe);
    if (rp == nullptr) {
      uint64_t a;
      if constexpr (SHIFT) {
        const int64_t lo = static_cast<int64_t>((r0 + lane) * s.row_bytes) -
                           static_cast<int64_t>(s.row_shift);
        a = static_cast<uint64_t>(max(lo, static_cast<int64_t>(p0)));
      } else {
        const uint64_t lo = (r0 + lane) * s.row_bytes;
        a = lo > p0 ? lo : p0;
      }
      for (uint32_t o = 0; o < share; o += 16)
        *reinterpret_cast<uint4*>(tile + (a - p0) + o) = make_uint4(0, 0, 0, 0);
      fence_async_smem();
    } else {
      mine = share;
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) mine += __shfl_xor_sync(kFull, mine, d);
  if (lane == 0) mbar_arrive_expect_tx(bar, mine);
  __syncwarp();
  issue_runs<true, SHIFT>(st, rp, pe, tile, bar, lane);
}

// One staged tile whose loads have landed: complete it, issue its stores
// (one bulk group), fold its chunks into the fingerprint and write its node.
// Returns whether stores were issued.  Called by a whole warp.
template <int MODE, bool SHIFT>
__device__ __forceinline__ bool bulk_tile(const WarpStage& m, uint8_t* tile,
                                          uint64_t* __restrict__ nodes, int lane) {
  using T = ModeTraits<MODE>;
  const uint4 zero = make_uint4(0, 0, 0, 0);
  const SecDesc& s = m.d;
  const uint64_t L = s.bytes, p0 = m.p0, p1 = m.p1;
  const uint64_t pe = staged_end<MODE>(s, p1);
  // Complete the tile: [pe, p1) holds the stream's unaligned tail (layout
  // side) and zeros past its end.
  for (uint64_t o = pe + 16u * lane; o < p1; o += 512u) {
    uint4 v = zero;
    if (T::kLoadLayout && o < L) {
      const uint64_t left = L - o;
      v = ld_small(s.lbase + o, left < 16 ? static_cast<int>(left) : 16, true);
    }
    *reinterpret_cast<uint4*>(tile + (o - p0)) = v;
  }
  if (!T::kLoadLayout && (L & 15u) && L >= p0 && L < p1 && lane == 0) {
    // Restore: payload bytes past the logical end read as zero.
    const uint64_t o = L & ~15ull;
    uint4* q = reinterpret_cast<uint4*>(tile + (o - p0));
    *q = mask_tail(*q, static_cast<int>(L - o));
  }
  fence_async_smem();
  __syncwarp();
  bool issued = false;
  if (MODE == kModePack) {
    // Contiguous payload, through the record's 256-byte padding.
    const uint64_t padded = (L + kRecordAlign - 1) / kRecordAlign * kRecordAlign;
    const uint64_t se = p1 < padded ? p1 : padded;
    if (lane == 0 && se > p0) {
      bulk_s2g(s.payload + p0, tile, static_cast<uint32_t>(se - p0));
      bulk_commit();
      issued = true;
    }
  } else if (MODE == kModeRestore || MODE == kModeRestoreV) {
    const uint64_t lim = L < p1 ? L : p1;
    if (s.layout == kContig) {
      const uint64_t vend = lim & ~15ull;  // whole segments by bulk copy
      if (lane == 0 && vend > p0) {
        bulk_s2g(s.lbase + p0, tile, static_cast<uint32_t>(vend - p0));
        bulk_commit();
        issued = true;
      }
      for (uint64_t o = (vend > p0 ? vend : p0) + lane; o < lim; o += 32) s.lbase[o] = tile[o - p0];
    } else {
      uint8_t* rp = m.rowp[lane];
      if (issue_runs<false, SHIFT>(m, rp, lim, tile, nullptr, lane)) {
        bulk_commit();
        issued = true;
      }
    }
  }
  if (T::kHash) {
    // The tile's chunks, interleaved lane chains, read from shared memory.
    const uint64_t c0 = p0 / kChunkBytes;
    const int nc = static_cast<int>((p1 - p0) / kChunkBytes);
    uint64_t h[kTileChunks];
#pragma unroll
    for (int q = 0; q < kTileChunks; ++q) h[q] = fmix(kSeed ^ ((c0 + q) * 32u + lane));
#pragma unroll
    for (int k = 0; k < kSegs; ++k) {
#pragma unroll
      for (int q = 0; q < kTileChunks; ++q) {
        const uint4 v = q < nc ? *reinterpret_cast<const uint4*>(tile + q * kChunkBytes + 512 * k + 16 * lane)
                               : zero;
        h[q] = absorb(h[q], v);
      }
    }
    // Moving passes are bound by DRAM; one tree per chunk paces the warps
    // so that loads and stores interleave best (measured: the shared tree
    // of tile_tree2 makes pack and restore slower).
    uint64_t mine = 0;
#pragma unroll
    for (int q = 0; q < kTileChunks; ++q) {
      const uint64_t x = __shfl_sync(kFull, warp_tree(fmix(h[q]), 32, lane), 0);
      if (lane == q) mine = x;
    }
    const uint64_t root = warp_tree(mine, nc, lane);
    if (lane == 0) nodes[m.node] = root;
  }
  return issued;
}

// The TMA kernel with static work: each warp moves a contiguous, balanced
// range of the launch's tiles, kWarpStages in flight.
template <int MODE, bool SHIFT>
__global__ void __launch_bounds__(BulkShape<MODE>::kThreads, 1)
    k_bulk(const SecDesc* __restrict__ secs, WorkList wl, uint64_t* __restrict__ nodes,
           uint32_t* err) {
  constexpr int kBulkWarps = BulkShape<MODE>::kWarps;
  constexpr int kWarpStages = BulkShape<MODE>::kStages;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  auto& sh = *reinterpret_cast<BulkShared<kBulkWarps, kWarpStages>*>(smem_raw);
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  if (lane < kWarpStages) {
    mbar_init(&sh.bar[warp][lane], 1);
    sh.st[warp][lane].sec = 0xFFFFFFFFu;
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncwarp();

  // This warp's tiles: a contiguous, balanced range [t0, t1).
  const uint64_t T_all = wl.n_tasks;
  const uint64_t gw = static_cast<uint64_t>(blockIdx.x) * kBulkWarps + warp;
  const uint64_t nw = static_cast<uint64_t>(gridDim.x) * kBulkWarps;
  const uint32_t t0 = static_cast<uint32_t>(T_all * gw / nw);
  const uint32_t t1 = static_cast<uint32_t>(T_all * (gw + 1) / nw);
  if (t0 >= t1) return;
  // The work list and the descriptors are there before the kernel starts: the
  // first tile's item and section are found while the kernel ahead on the
  // stream drains.
  int item = find_item(wl.begin, 0, wl.n_items, t0, lane);  // item of the next tile to stage
  stage_desc(secs, __ldg(wl.ids + item), sh.st[warp][0], lane);
  grid_dependency();
  auto item_of = [&](uint32_t t) {
    while (item + 1 < wl.n_items && __ldg(wl.begin + item + 1) <= t) ++item;
    return item;
  };
  const int pre = static_cast<int>(t1 - t0 < static_cast<uint32_t>(kWarpStages) ? t1 - t0 : kWarpStages);
  for (int k = 0; k < pre; ++k)
    stage_tile<MODE, SHIFT>(secs, wl, item_of(t0 + k), t0 + k, sh.st[warp][k], sh.buf[warp][k],
                     &sh.bar[warp][k], err, lane);
  bool any_issued = false;
  for (uint32_t i = 0; t0 + i < t1; ++i) {
    const int sidx = static_cast<int>(i % kWarpStages);
    const uint32_t use = i / kWarpStages;
    uint64_t* bar = &sh.bar[warp][sidx];
    uint8_t* tile = sh.buf[warp][sidx];
    WarpStage& m = sh.st[warp][sidx];
    bool ok = true;
    if (lane == 0) ok = mbar_wait(bar, use & 1);
    ok = __shfl_sync(kFull, ok, 0);
    if (!ok) {
      if (lane == 0) atomicOr(err, kDevErrTimeout);
      break;
    }
    if (bulk_tile<MODE, SHIFT>(m, tile, nodes, lane)) {
      bulk_wait_read();
      any_issued = true;
    }
    __syncwarp();
    // Reuse the stage for tile i + kWarpStages.
    const uint32_t tn = t0 + i + kWarpStages;
    if (tn < t1) stage_tile<MODE, SHIFT>(secs, wl, item_of(tn), tn, m, tile, bar, err, lane);
  }
  if (any_issued) bulk_wait_all();
}

// The TMA kernel with shared work, for launches of fewer than
// kDynMaxTilesPerWarp tiles per warp: each warp first moves a contiguous,
// balanced range of the first T_static tiles, then chunks of the rest
// [T_static, T_all) handed out by an atomic counter (sched[0]) to whichever
// warp asks first, so that warps that drew slower memory do not hold up the
// end of the launch.  sched[0..1] are zero on entry; the last warp to finish
// sets them back to zero.
template <int MODE, bool SHIFT>
__global__ void __launch_bounds__(BulkShape<MODE>::kThreads, 1)
    k_bulk_shared(const SecDesc* __restrict__ secs, WorkList wl, uint64_t* __restrict__ nodes,
                  uint32_t* err, uint32_t* sched) {
  constexpr int kBulkWarps = BulkShape<MODE>::kWarps;
  constexpr int kWarpStages = BulkShape<MODE>::kStages;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  auto& sh = *reinterpret_cast<BulkShared<kBulkWarps, kWarpStages>*>(smem_raw);
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  if (lane < kWarpStages) {
    mbar_init(&sh.bar[warp][lane], 1);
    sh.st[warp][lane].sec = 0xFFFFFFFFu;
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncwarp();

  const uint32_t T_all = wl.n_tasks;
  const uint64_t gw = static_cast<uint64_t>(blockIdx.x) * kBulkWarps + warp;
  const uint64_t nw = static_cast<uint64_t>(gridDim.x) * kBulkWarps;
  const uint32_t T_dyn = T_all / kDynShare;
  const uint32_t T_static = T_all - T_dyn;
  const uint64_t per = T_dyn / (nw * kDynGrabsPerWarp);
  const uint32_t chunk = static_cast<uint32_t>(per < 1 ? 1 : (per > kDynChunkMax ? kDynChunkMax : per));
  const uint32_t t0 = static_cast<uint32_t>(T_static * gw / nw);
  const uint32_t t1 = static_cast<uint32_t>(T_static * (gw + 1) / nw);
  uint32_t next = t0, chunk_end = t1;  // tiles [next, chunk_end) are this warp's
  int item = find_item(wl.begin, 0, wl.n_items, t0, lane);  // item of the last tile taken
  // The work list and the descriptors are there before the kernel starts: the
  // first static tile's section is read before waiting for the kernel ahead.  The
  // counters in `sched` are touched only after the wait.
  if (t0 < t1) stage_desc(secs, __ldg(wl.ids + item), sh.st[warp][0], lane);
  grid_dependency();
  // The next chunk, reserved ahead of need (where the warp would wait on a
  // stage anyway) so that neither the atomic nor the search of its item
  // delays a refill.
  bool reserved = false, drained = false;
  uint32_t res_next = 0, res_end = 0;
  int res_item = 0;
  auto reserve = [&]() {
    if (reserved || drained) return;
    uint32_t g = 0;
    if (lane == 0) g = atomicAdd(sched, chunk);
    g = __shfl_sync(kFull, g, 0);
    if (g >= T_dyn) {
      drained = true;
      return;
    }
    res_next = T_static + g;
    res_end = T_static + (g + chunk < T_dyn ? g + chunk : T_dyn);
    res_item = item + 1 < wl.n_items && __ldg(wl.begin + item + 1) <= res_next
                   ? find_item(wl.begin, item, wl.n_items, res_next, lane)
                   : item;
    reserved = true;
  };
  // The next tile of this warp (and `item`, its item); false once none is left.
  auto take = [&](uint32_t* t) -> bool {
    if (next >= chunk_end) {
      reserve();
      if (!reserved) return false;
      next = res_next;
      chunk_end = res_end;
      item = res_item;
      reserved = false;
    }
    *t = next++;
    while (item + 1 < wl.n_items && __ldg(wl.begin + item + 1) <= *t) ++item;
    return true;
  };
  int staged = 0;
  for (int k = 0; k < kWarpStages; ++k) {
    uint32_t t;
    if (!take(&t)) break;
    stage_tile<MODE, SHIFT>(secs, wl, item, t, sh.st[warp][k], sh.buf[warp][k], &sh.bar[warp][k], err,
                     lane);
    ++staged;
  }
  bool any_issued = false;
  for (int i = 0; i < staged; ++i) {
    const int sidx = i % kWarpStages;
    const uint32_t use = static_cast<uint32_t>(i) / kWarpStages;
    uint64_t* bar = &sh.bar[warp][sidx];
    uint8_t* tile = sh.buf[warp][sidx];
    WarpStage& m = sh.st[warp][sidx];
    if (next + 1 >= chunk_end) reserve();  // the refill after next needs a new chunk
    bool ok = true;
    if (lane == 0) ok = mbar_wait(bar, use & 1);
    ok = __shfl_sync(kFull, ok, 0);
    if (!ok) {
      if (lane == 0) atomicOr(err, kDevErrTimeout);
      break;
    }
    if (bulk_tile<MODE, SHIFT>(m, tile, nodes, lane)) {
      bulk_wait_read();
      any_issued = true;
    }
    __syncwarp();
    // Reuse the stage for this warp's next tile.
    uint32_t tn;
    if (take(&tn)) {
      stage_tile<MODE, SHIFT>(secs, wl, item, tn, m, tile, bar, err, lane);
      ++staged;
    }
  }
  if (any_issued) bulk_wait_all();
  // The last warp out leaves the counters at zero for the next launch.
  if (lane == 0) {
    __threadfence();
    if (atomicAdd(sched + 1, 1u) == static_cast<uint32_t>(nw) - 1) {
      atomicExch(sched, 0u);
      atomicExch(sched + 1, 0u);
    }
  }
}

// ---------------------------------------------------------------------------
// Read-only fingerprint pass (hash mode of the streams the TMA kernel would
// take: 16-byte aligned contiguous device buffers)
//
// Every warp walks a contiguous range of 8 KiB tiles; per tile each lane
// issues its sixteen 16-byte loads (segments lane + 32k of both chunks) into
// registers, then runs the two lane chains interleaved and one shared tree
// (tile_tree2).  No shared memory: 20 warps per SM fit in the register file
// (88 registers), and their loads hide each other's hashing.  Measured on
// the 200-buffer classify sweep: 6.68 TB/s, against 6.27 TB/s for the TMA
// pipeline with two 8 KiB stages per warp (which shared memory capped at 12
// warps) and 6.99 TB/s for a plain-load byte compare of the same pairs;
// 16 warps 6.49, 24 warps (spilling) 6.08, two tiles in flight per warp
// (166 registers, 12 warps) 5.42.
// ---------------------------------------------------------------------------

constexpr int kHashWarps = 20;
constexpr int kHashThreads = 32 * kHashWarps;

__global__ void __launch_bounds__(kHashThreads, 1)
    k_hash(const SecDesc* __restrict__ secs, WorkList wl, uint64_t* __restrict__ nodes) {
  grid_dependency();
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  // This warp's tiles: a contiguous, balanced range [t0, t1).
  const uint64_t T_all = wl.n_tasks;
  const uint64_t gw = static_cast<uint64_t>(blockIdx.x) * kHashWarps + warp;
  const uint64_t nw = static_cast<uint64_t>(gridDim.x) * kHashWarps;
  const uint32_t t0 = static_cast<uint32_t>(T_all * gw / nw);
  const uint32_t t1 = static_cast<uint32_t>(T_all * (gw + 1) / nw);
  if (t0 >= t1) return;
  int item = find_item(wl.begin, 0, wl.n_items, t0, lane);
  for (uint32_t t = t0; t < t1; ++t) {
    while (item + 1 < wl.n_items && __ldg(wl.begin + item + 1) <= t) ++item;
    const SecDesc* s = secs + __ldg(wl.ids + item);
    const uint8_t* base = reinterpret_cast<const uint8_t*>(
        __ldg(reinterpret_cast<const unsigned long long*>(&s->lbase)));
    const uint64_t L = __ldg(reinterpret_cast<const unsigned long long*>(&s->bytes));
    const uint64_t nch = __ldg(reinterpret_cast<const unsigned long long*>(&s->n_chunks));
    const uint32_t loc = t - __ldg(wl.begin + item);
    const uint64_t p0 = static_cast<uint64_t>(loc) * kTileBytes;
    const uint64_t c0 = p0 / kChunkBytes;
    // Bytes at or past L read as zero (the chunk's padding).
    uint4 v[2 * kSegs];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
      for (int k = 0; k < kSegs; ++k) {
        const uint64_t off = p0 + q * kChunkBytes + 512u * k + 16u * lane;
        uint4 x = make_uint4(0, 0, 0, 0);
        if (off + 16 <= L) x = ld_stream(base + off);
        else if (off < L) x = ld_small(base + off, static_cast<int>(L - off), true);
        v[q * kSegs + k] = x;
      }
    }
    uint64_t ha = fmix(kSeed ^ (c0 * 32u + lane));
    uint64_t hb = fmix(kSeed ^ ((c0 + 1) * 32u + lane));
#pragma unroll
    for (int k = 0; k < kSegs; ++k) {
      ha = absorb(ha, v[k]);
      hb = absorb(hb, v[kSegs + k]);
    }
    static_assert(kTileChunks == 2, "tile_tree2 reduces two chunks");
    const uint64_t root = tile_tree2(fmix(ha), fmix(hb), nch - c0 >= 2 ? 2 : 1, lane);
    if (lane == 0) nodes[__ldg(&s->task_begin) + loc] = root;
  }
}

// ---------------------------------------------------------------------------
// Finalisation: stream fps, record headers, verification
// ---------------------------------------------------------------------------

template <bool L2 = false>
__device__ __forceinline__ uint64_t stream_fp(const SecDesc& s, uint64_t* nodes, int lane) {
  const uint64_t root = s.fin_count <= kFinRegNodes ? warp_tree_regs<L2>(nodes + s.fin_begin, s.fin_count, lane)
                                             : warp_tree_inplace(nodes + s.fin_begin, s.fin_count, lane);
  return fmix(root ^ (s.bytes * kP));
}

// One warp per aligned group of 32 nodes of one stream (one reduction level).
__global__ void __launch_bounds__(kThreads)
    k_reduce_nodes(const NodeLevel* __restrict__ lv, int n_secs, uint64_t* nodes, uint32_t base,
                   uint32_t n_groups) {
  grid_dependency();
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * kWarps;
  for (uint32_t g = blockIdx.x * kWarps + (threadIdx.x >> 5); g < n_groups; g += nw) {
    int lo = 0, hi = n_secs - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(&lv[mid].dst) - base <= g) lo = mid;
      else hi = mid - 1;
    }
    const NodeLevel L = lv[lo];
    const uint32_t local = g - (L.dst - base);
    const uint32_t n = min(32u, L.count - 32u * local);
    const uint64_t v = lane < static_cast<int>(n) ? nodes[L.src + 32u * local + lane] : 0;
    const uint64_t r = warp_tree(v, static_cast<int>(n), lane);
    if (lane == 0) nodes[L.dst + local] = r;
  }
}

// Fingerprints of independent buffers (pcs_fingerprint / pcs_classify):
// warps w0, w0 + nw, ... take buffer after buffer.
__device__ __forceinline__ void finalize_hash_warps(const SecDesc* __restrict__ secs, int n_secs,
                                                    uint64_t* nodes, uint64_t* fp_out,
                                                    const uint64_t* fp_before, uint8_t* flags,
                                                    int w0, int nw) {
  const int lane = threadIdx.x & 31;
  for (int i = w0; i < n_secs; i += nw) {
    const SecDesc s = secs[i];
    const uint64_t fp = stream_fp(s, nodes, lane);
    if (lane == 0) {
      if (fp_out) fp_out[i] = fp;
      if (fp_before) flags[i] = fp != fp_before[i] ? 1 : 0;
    }
  }
}

__global__ void __launch_bounds__(kThreads)
    k_finalize_hash(const SecDesc* __restrict__ secs, int n_secs, uint64_t* nodes,
                    uint64_t* fp_out, const uint64_t* fp_before, uint8_t* flags) {
  grid_dependency();
  finalize_hash_warps(secs, n_secs, nodes, fp_out, fp_before, flags,
                      blockIdx.x * kWarps + (threadIdx.x >> 5), gridDim.x * kWarps);
}

constexpr uint32_t kMaxSmemFps = 2048;  // level-1 nodes of up to 65535 fps

// Session fp = fmix(tree(fps) ^ n): fps read with a stride of `stride`
// u64 words (the fp field of consecutive 64-byte entries).  Warp-wide.
__device__ uint64_t session_fp(const uint64_t* fps, uint32_t stride, uint32_t n, uint64_t* smem,
                               int lane) {
  const uint32_t groups = (n + 31) / 32;
  for (uint32_t g = 0; g < groups; ++g) {
    const uint32_t i = 32 * g + lane;
    const uint64_t v = i < n ? fps[static_cast<uint64_t>(i) * stride] : 0;
    const uint64_t r = warp_tree(v, static_cast<int>(min(32u, n - 32 * g)), lane);
    if (lane == 0) smem[g] = r;
  }
  __syncwarp();
  const uint64_t root = warp_tree_inplace(smem, groups, lane);
  return fmix(root ^ static_cast<uint64_t>(n));
}

// Checkpoint: fps into the section table, then header and session fp.
// Restore with verification: compare recomputed fps with the record.
// The whole block handles sessions b0, b0 + stride, ...
template <int MODE>
__device__ void finalize_sessions_block(const SecDesc* secs, const SessDesc* sess, int n_sess,
                                        const Entry* entries, uint64_t* nodes,
                                        uint8_t* corrupt, uint32_t* bad, int b0, int stride,
                                        uint64_t* smem, uint32_t* s_bad) {
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const uint32_t nwarps = blockDim.x >> 5;
  for (int b = b0; b < n_sess; b += stride) {
    const SessDesc S = sess[b];
    Entry* table = reinterpret_cast<Entry*>(S.record + kHeaderBytes);
    if (threadIdx.x == 0) *s_bad = 0;
    __syncthreads();
    for (uint32_t j = wib; j < S.n_sections; j += nwarps) {
      const SecDesc s = secs[S.sec_begin + j];
      uint4 ew = make_uint4(0, 0, 0, 0);  // lanes 0..3: the entry, read before the tree
      if (MODE == kModePack && lane < 4)
        ew = reinterpret_cast<const uint4*>(&entries[S.sec_begin + j])[lane];
      const uint64_t fp = stream_fp(s, nodes, lane);
      if (MODE == kModePack) {
        // Lanes 0..3 write the 64-byte entry as four 16-byte words; the fp
        // (bytes 32..39) is the first half of lane 2's word.
        if (lane == 2) {
          ew.x = static_cast<uint32_t>(fp);
          ew.y = static_cast<uint32_t>(fp >> 32);
        }
        if (lane < 4) reinterpret_cast<uint4*>(&table[j])[lane] = ew;
      } else {
        if (lane == 0 && table[j].fp != fp) atomicOr(s_bad, 1u);
      }
    }
    __syncthreads();
    if (wib == 0) {
      const uint64_t* fps = &table[0].fp;
      const uint64_t sfp = session_fp(fps, kEntryBytes / 8, S.n_sections, smem, lane);
      if (lane == 0) {
        if (MODE == kModePack) {
          uint4* h = reinterpret_cast<uint4*>(S.record);
          h[0] = make_uint4(kMagic, kVersion | (S.n_sections << 16), S.session_id, S.kind);
          h[1] = make_uint4(static_cast<uint32_t>(S.total_bytes),
                            static_cast<uint32_t>(S.total_bytes >> 32), static_cast<uint32_t>(sfp),
                            static_cast<uint32_t>(sfp >> 32));
          h[2] = make_uint4(0, 0, 0, 0);
          h[3] = make_uint4(0, 0, 0, 0);
        } else {
          const uint64_t stored = *reinterpret_cast<const uint64_t*>(S.record + 24);
          const bool broken = *s_bad != 0 || stored != sfp;
          if (corrupt) corrupt[b] = broken ? 1 : 0;
          if (broken) atomicAdd(bad, 1u);
        }
      }
    }
    if (MODE == kModePack) {
      // Zero the gap between the end of the table and the first payload.
      const uint64_t from = kHeaderBytes + static_cast<uint64_t>(kEntryBytes) * S.n_sections;
      for (uint64_t o = from + 16u * threadIdx.x; o < S.payload_start; o += 16u * blockDim.x)
        *reinterpret_cast<uint4*>(S.record + o) = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
  }
}

// Any block size up to 512 threads (a warp per section in turn).
template <int MODE>
__global__ void __launch_bounds__(512)
    k_finalize_sessions(const SecDesc* __restrict__ secs, const SessDesc* __restrict__ sess,
                        int n_sess, const Entry* __restrict__ entries, uint64_t* nodes,
                        uint8_t* corrupt, uint32_t* bad) {
  __shared__ uint64_t smem[kMaxSmemFps];
  __shared__ uint32_t s_bad;
  // The host's descriptors of the block's first session (each warp's first
  // section and, for a checkpoint, its table entry) are brought into L1
  // while the kernel ahead on the stream drains.
  if (static_cast<int>(blockIdx.x) < n_sess) {
    const SessDesc* S0 = sess + blockIdx.x;
    const uint32_t j = threadIdx.x >> 5;
    if (j < __ldg(&S0->n_sections) && (threadIdx.x & 31) == 0) {
      const uint32_t i = __ldg(&S0->sec_begin) + j;
      prefetch_l1(secs + i);
      prefetch_l1(reinterpret_cast<const uint8_t*>(secs + i) + sizeof(SecDesc) - 1);
      if (MODE == kModePack) prefetch_l1(entries + i);
    }
  }
  grid_dependency();
  finalize_sessions_block<MODE>(secs, sess, n_sess, entries, nodes, corrupt, bad, blockIdx.x,
                                gridDim.x, smem, &s_bad);
}

// A session of at most 32 sections, finalised by one warp (lane j keeps
// section j's fp): the same outputs as finalize_sessions_block.  Lane j's part
// of the session's descriptors:
struct SessLane {
  uint32_t fin_begin, fin_count;  // section j's nodes
  uint64_t bytes;                 // and its length
};

template <bool GLOBAL = true>
__device__ __forceinline__ SessLane session_lane(const SessDesc& S, const SecDesc* secs, int lane) {
  SessLane l{0, 0, 0};
  if (lane < static_cast<int>(S.n_sections)) {
    const SecDesc* sj = secs + S.sec_begin + lane;
    l.fin_begin = fetch<GLOBAL>(&sj->fin_begin);
    l.fin_count = fetch<GLOBAL>(&sj->fin_count);
    l.bytes = fetch<GLOBAL>(reinterpret_cast<const unsigned long long*>(&sj->bytes));
  }
  return l;
}

template <int MODE, bool L2>
__device__ __forceinline__ void finalize_session_warp(const SessDesc& S, const SessLane& l, int b,
                                                      const Entry* entries, uint64_t* nodes,
                                                      uint8_t* corrupt, uint32_t* bad, int lane) {
  Entry* table = reinterpret_cast<Entry*>(S.record + kHeaderBytes);
  const int ns = static_cast<int>(S.n_sections);
  // A restore's stored fps (lane j: section j's), read once; each section's
  // tree then starts from its node loads, and a checkpoint's entry is read
  // before the tree.
  uint64_t stored = 0;
  if (MODE != kModePack && lane < ns) stored = table[lane].fp;
  uint64_t mine = 0;
  bool bad_sec = false;
  for (int j = 0; j < ns; ++j) {
    uint4 ew = make_uint4(0, 0, 0, 0);  // pack: lanes 0..3 hold the entry, read before the tree
    if (MODE == kModePack && lane < 4)
      ew = reinterpret_cast<const uint4*>(&entries[S.sec_begin + j])[lane];
    const uint32_t nb = __shfl_sync(kFull, l.fin_begin, j);
    const uint32_t nc = __shfl_sync(kFull, l.fin_count, j);
    const uint64_t by = __shfl_sync(kFull, l.bytes, j);
    const uint64_t root = nc <= kFinRegNodes ? warp_tree_regs<L2>(nodes + nb, nc, lane)
                                             : warp_tree_inplace(nodes + nb, nc, lane);
    const uint64_t fp = fmix(root ^ (by * kP));
    if (MODE == kModePack) {
      // The fp (bytes 32..39 of the entry) is the first half of lane 2's word.
      if (lane == 2) {
        ew.x = static_cast<uint32_t>(fp);
        ew.y = static_cast<uint32_t>(fp >> 32);
      }
      if (lane < 4) reinterpret_cast<uint4*>(&table[j])[lane] = ew;
      if (lane == j) mine = fp;
    } else {
      if (lane == j) {
        mine = stored;
        bad_sec = stored != fp;
      }
    }
  }
  // Session fp = fmix(tree(fps) ^ n), the fps being the table's.
  const uint64_t sfp = fmix(warp_tree(mine, ns, lane) ^ static_cast<uint64_t>(ns));
  const bool any_bad = __any_sync(kFull, bad_sec);
  if (lane == 0) {
    if (MODE == kModePack) {
      uint4* h = reinterpret_cast<uint4*>(S.record);
      h[0] = make_uint4(kMagic, kVersion | (S.n_sections << 16), S.session_id, S.kind);
      h[1] = make_uint4(static_cast<uint32_t>(S.total_bytes),
                        static_cast<uint32_t>(S.total_bytes >> 32), static_cast<uint32_t>(sfp),
                        static_cast<uint32_t>(sfp >> 32));
      h[2] = make_uint4(0, 0, 0, 0);
      h[3] = make_uint4(0, 0, 0, 0);
    } else {
      const uint64_t stored_sfp = *reinterpret_cast<const uint64_t*>(S.record + 24);
      const bool broken = any_bad || stored_sfp != sfp;
      if (corrupt) corrupt[b] = broken ? 1 : 0;
      if (broken) atomicAdd(bad, 1u);
    }
  }
  if (MODE == kModePack) {
    // Zero the gap between the end of the table and the first payload.
    const uint64_t from = kHeaderBytes + static_cast<uint64_t>(kEntryBytes) * S.n_sections;
    for (uint64_t o = from + 16u * lane; o < S.payload_start; o += 16u * 32)
      *reinterpret_cast<uint4*>(S.record + o) = make_uint4(0, 0, 0, 0);
  }
}

// Many sessions of at most 32 sections: a warp per session.
template <int MODE>
__global__ void __launch_bounds__(kThreads)
    k_finalize_sessions_warp(const SecDesc* __restrict__ secs, const SessDesc* __restrict__ sess,
                             int n_sess, const Entry* __restrict__ entries, uint64_t* nodes,
                             uint8_t* corrupt, uint32_t* bad) {
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * kWarps;
  // The warp's first session's descriptors are read while the kernel ahead on
  // the stream drains.
  SessDesc S;
  SessLane l;
  const int b_first = blockIdx.x * kWarps + (threadIdx.x >> 5);
  if (b_first < n_sess) {
    S = sess[b_first];
    l = session_lane(S, secs, lane);
  }
  grid_dependency();
  for (int b = b_first; b < n_sess; b += nw) {
    if (b != b_first) {
      S = sess[b];
      l = session_lane(S, secs, lane);
    }
    finalize_session_warp<MODE, false>(S, l, b, entries, nodes, corrupt, bad, lane);
  }
}

// Small calls in one launch: the streaming pass, then the finalisation.  A
// buffer, and a session of at most 32 sections, is finalised by the warp that
// completes its last task: `done[i]` counts the tasks completed of item i
// (zero on entry; that warp sets it back), so the items' trees run side by
// side, on the warps that are free.  Calls with a session of more sections
// leave all of them to the last block to finish (an atomic ticket, zero on
// entry and reset), a warp per section.  No block or warp waits for another.
// Bound by latency: 49 tasks of one Markov session are one chunk per warp.
// Measured, planned calls (the last block finalising every item, a session at
// a time -> this): 34 sessions of 14,280 bytes pack 50.6 -> 6.0 us, verified
// restore 56.7 -> 6.8 us; 64 of 10,000 bytes 89.4 -> 5.5 and 99.8 -> 5.6 us; one
// of 196,608 bytes 6.2 and 6.3 us either way.
//
// BYTES > 0: the call's descriptors travel as a kernel parameter of that size
// (`blob`; launch_small picks the smallest that holds them), else they are at
// a.plan in the workspace: a plain call whose descriptors are too many for a
// parameter sends them there ahead of the launch (then not an early one), a
// prepared call keeps them there.  Sending them ahead, and the hand-over to
// the kernel, cost a call more than its kernel.  Measured (sent by a copy
// engine -> as a parameter), checkpoint + verified restore + delete of
// one session of 196,608 bytes 31.4 -> 20.1 us, of 34 small ones 31.7 -> 25.8,
// of 64 (27 KB of descriptors) 36.2 -> 31.5; fingerprints of 8 buffers 11.1 -> 5.8.
template <int BYTES>
struct PlanBlob {
  alignas(16) uint8_t b[BYTES > 0 ? BYTES : 16];
};

template <int MODE, int BYTES>
__global__ void __launch_bounds__(kThreads, 2)
    k_small(const __grid_constant__ PlanBlob<BYTES> blob, const SmallArgs a) {
  constexpr bool GLOBAL = BYTES == 0;
  const uint8_t* plan = GLOBAL ? a.plan : blob.b;
  const SecDesc* secs = reinterpret_cast<const SecDesc*>(plan + a.o_secs);
  const SessDesc* sess = reinterpret_cast<const SessDesc*>(plan + a.o_sess);
  const Entry* entries = reinterpret_cast<const Entry*>(plan + a.o_entries);
  const WorkList wl{reinterpret_cast<const uint32_t*>(plan + a.o_ids),
                    reinterpret_cast<const uint32_t*>(plan + a.o_begin), a.n_list, a.n_tasks};
  uint64_t* nodes = a.nodes;
  __shared__ SecDesc sdesc[kWarps];
  const int lane = threadIdx.x & 31;
  if (MODE == kModeHash || a.max_secs <= 32) {
    run_stream_tasks<MODE, GLOBAL>(secs, wl, a.glog2, nodes, a.err, sdesc, false,
                                   [&](const SecDesc& s, int j) {
      const uint32_t i = MODE == kModeHash ? fetch<GLOBAL>(wl.ids + j) : s.sess;
      SessDesc S{};
      SessLane l{};
      if (MODE != kModeHash) {
        S = sess[i];
        l = session_lane<GLOBAL>(S, secs, lane);
      }
      const uint32_t total = MODE == kModeHash ? s.n_tasks : S.n_tasks;
      uint32_t before = 0;
      if (lane == 0) {
        __threadfence();  // the task's node, before it counts as done
        before = atomicAdd(a.done + i, 1u);
      }
      if (__shfl_sync(kFull, before, 0) + 1 != total) return;
      __threadfence();
      if (lane == 0) a.done[i] = 0;
      if (MODE == kModeHash) {
        const uint64_t fp = stream_fp<true>(s, nodes, lane);
        if (lane == 0) {
          if (a.fp_out) a.fp_out[i] = fp;
          if (a.fp_before) a.flags[i] = fp != a.fp_before[i] ? 1 : 0;
        }
      } else {
        finalize_session_warp<MODE == kModeHash ? kModePack : MODE, true>(
            S, l, static_cast<int>(i), entries, nodes, nullptr, a.bad, lane);
      }
    });
    return;
  }
  __shared__ uint64_t smem[64];  // up to 2048 sections per session
  __shared__ uint32_t s_bad;
  __shared__ bool s_last;
  run_stream_tasks<MODE, GLOBAL>(secs, wl, a.glog2, nodes, a.err, sdesc, false,
                                 [](const SecDesc&, int) {});
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (MODE != kModeHash)
    finalize_sessions_block<MODE>(secs, sess, a.n_items, entries, nodes, nullptr, a.bad, 0, 1, smem,
                                  &s_bad);
  if (threadIdx.x == 0) *a.ticket = 0;
}

// ---------------------------------------------------------------------------
// Relevance score and top-k
// ---------------------------------------------------------------------------

// Where a kernel's bank descriptors are: in the workspace (p), or, for a call
// of few banks (BLOB), in the parameter itself: they travel with each of the
// call's launches, as a small call's descriptors do.  Measured, whole calls: a
// global threshold of few entries 22.7 -> 18.1 us, a prune of few 12.5 -> 10.3.
template <bool BLOB>
struct BankArg;
template <>
struct BankArg<false> {
  const BankDesc* p;
  __device__ const BankDesc* get() const { return p; }
};
template <>
struct BankArg<true> {
  BankDesc b[kBankBlob];
  __device__ const BankDesc* get() const { return b; }
};

// Order-preserving map float -> uint32 (-0 ranks as +0, NaN lowest).
__device__ __forceinline__ uint32_t ord32(float s) {
  if (isnan(s)) return 0u;
  if (s == 0.f) s = 0.f;
  const uint32_t u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Digits of the 64-bit ranking key of the global threshold, most significant
// first: 11, 11 and 10 bits of ord32(score), then the same of the position.
__device__ __forceinline__ int gdigit_bits(int pass) { return pass % 3 == 2 ? 10 : 11; }
__device__ __forceinline__ int gdigit_shift(int pass) {
  return pass == 0 ? 53 : pass == 1 ? 42 : pass == 2 ? 32 : pass == 3 ? 21 : pass == 4 ? 10 : 0;
}

constexpr uint32_t kGList = 512;  // keys k_gfinish gathers for its last choice at most
static_assert(2 * kGList * 8 <= kGBins * 4, "the gathered keys fit the bins' shared memory");

// One block's copy of the select state.
struct GLocal {
  uint64_t prefix, mask, remaining, threshold;
  uint32_t done, n_cand;  // n_cand: keys inside the prefix
};

// Add to a 64-bit sum in shared memory as two 32-bit atomics with the carry
// between them: a 64-bit one is a compare-and-swap loop, which the few hot
// digits of a histogram make slow.
__device__ __forceinline__ void add64_shared(unsigned long long* p, uint64_t v) {
  uint32_t* w = reinterpret_cast<uint32_t*>(p);
  const uint32_t lo = static_cast<uint32_t>(v);
  const uint32_t old = atomicAdd(w, lo);
  const uint32_t hi = static_cast<uint32_t>(v >> 32) + (old + lo < lo ? 1u : 0u);
  if (hi) atomicAdd(w + 1, hi);
}

// Inclusive block scan of one uint64 per thread.
__device__ __forceinline__ uint64_t block_incl_scan64(uint64_t v, uint64_t* warp_sum) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint64_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) warp_sum[wib] = incl;
  __syncthreads();
  uint64_t before = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w)
    if (w < wib) before += warp_sum[w];
  __syncthreads();
  return before + incl;
}

// The digit choice of a pass from the summed bins, by the whole block:
// thread t holds the bins top - per*t - j (j < per), highest digits first;
// the first thread whose running bytes overrun the budget left finds the
// digit, which is fixed into the prefix; if it holds a single key, or it was
// the last digit, that key is the first that does not fit and the threshold is
// set.
template <bool UNIFORM>
__device__ void gpick_block(GLocal* s, int pass, uint64_t ubytes, const uint32_t* gc,
                            const unsigned long long* gw, uint64_t* scan64) {
  const int bits = gdigit_bits(pass), shift = gdigit_shift(pass);
  const int nb = 1 << bits, top = nb - 1, per = nb / kThreads;
  uint32_t cn[kGBins / kThreads];
  uint64_t wt[kGBins / kThreads];
  uint64_t local = 0;
#pragma unroll
  for (int j = 0; j < kGBins / kThreads; ++j) {
    cn[j] = 0;
    wt[j] = 0;
    if (j < per) {
      const int bin = top - per * static_cast<int>(threadIdx.x) - j;
      cn[j] = __ldcg(gc + bin);
      wt[j] = UNIFORM ? static_cast<uint64_t>(cn[j]) * ubytes
                      : static_cast<uint64_t>(__ldcg(gw + bin));
      local += wt[j];
    }
  }
  const uint64_t incl = block_incl_scan64(local, scan64);
  const uint64_t R = s->remaining;
  const int fit = __syncthreads_count(incl <= R);
  if (fit == kThreads) {  // every candidate fits (only when the whole population does)
    if (threadIdx.x == 0) {
      s->threshold = 0;
      s->done = 1;
    }
  } else if (static_cast<int>(threadIdx.x) == fit) {
    uint64_t cum = incl - local;
#pragma unroll
    for (int j = 0; j < kGBins / kThreads; ++j) {
      if (j < per && cum + wt[j] > R) {
        const int bin = top - per * static_cast<int>(threadIdx.x) - j;
        const uint64_t np = s->prefix | (static_cast<uint64_t>(bin) << shift);
        const uint64_t nm = s->mask | (static_cast<uint64_t>(top) << shift);
        s->prefix = np;
        s->mask = nm;
        s->remaining = R - cum;
        s->n_cand = cn[j];
        if (cn[j] == 1u || shift == 0) {
          s->threshold = np | ~nm;
          s->done = 1;
        }
        break;
      }
      cum += wt[j];
    }
  }
  __syncthreads();
}

__device__ __forceinline__ void gstate_load(const GState* st, GLocal* s) {
  s->prefix = __ldcg(&st->prefix);
  s->mask = __ldcg(&st->mask);
  s->remaining = __ldcg(&st->remaining);
  s->threshold = __ldcg(&st->threshold);
  s->done = __ldcg(&st->done);
  s->n_cand = __ldcg(&st->n_cand);
}
__device__ __forceinline__ void gstate_store(GState* st, const GLocal& s) {
  st->prefix = s.prefix;
  st->mask = s.mask;
  st->remaining = s.remaining;
  st->threshold = s.threshold;
  st->done = s.done;
  st->n_cand = s.n_cand;
}

// End of a histogram pass, by every block: add the block's bins (ch, wh in
// shared memory) to the global ones; the last block to finish (atomic
// ticket) picks the digit and clears the global bins for the next pass.
template <bool UNIFORM>
__device__ void gpass_finish(GState* st, int pass, uint64_t ubytes, uint32_t* ch,
                             unsigned long long* wh, bool* s_last, bool pick = true) {
  const int nb = 1 << gdigit_bits(pass);
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    if (ch[i]) atomicAdd(&st->chist[i], ch[i]);
    if (!UNIFORM && wh[i]) atomicAdd(reinterpret_cast<unsigned long long*>(&st->whist[i]), wh[i]);
  }
  if (!pick) return;  // a part of a split population: the host sums and picks
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *s_last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  __shared__ GLocal s;
  __shared__ uint64_t scan64[kWarps];
  if (threadIdx.x == 0) gstate_load(st, &s);
  __syncthreads();
  gpick_block<UNIFORM>(&s, pass, ubytes, st->chist,
                       reinterpret_cast<const unsigned long long*>(st->whist), scan64);
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    st->chist[i] = 0;
    st->whist[i] = 0;
  }
  if (threadIdx.x == 0) {
    gstate_store(st, s);
    st->ticket = 0;
  }
}

__device__ __forceinline__ float elem(uint32_t bits16, bool bf16) {
  return bf16 ? __uint_as_float(bits16 << 16)
              : __half2float(__ushort_as_half(static_cast<unsigned short>(bits16)));
}

// Accumulate the key terms (q.k and k.k) of the 8 elements of one 16-byte
// segment, ascending element order, with separately rounded products and
// sums.  (q.q is the same for every key of a bank: accum8_query.)
__device__ __forceinline__ void accum8_key(uint4 q, uint4 k, bool bf16, float& sd, float& sk) {
  const uint32_t qw[4] = {q.x, q.y, q.z, q.w};
  const uint32_t kw[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t qb = (qw[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
    const uint32_t kb = (kw[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
    const float qe = elem(qb, bf16), ke = elem(kb, bf16);
    sd = __fadd_rn(sd, __fmul_rn(qe, ke));
    sk = __fadd_rn(sk, __fmul_rn(ke, ke));
  }
}

// The query's own term, accumulated in the same lane order.
__device__ __forceinline__ void accum8_query(uint4 q, bool bf16, float& sq) {
  const uint32_t qw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float qe = elem((qw[i >> 1] >> (16 * (i & 1))) & 0xFFFFu, bf16);
    sq = __fadd_rn(sq, __fmul_rn(qe, qe));
  }
}

__device__ __forceinline__ float lane_tree_sum(float v) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) v = __fadd_rn(v, __shfl_down_sync(kFull, v, d));
  return v;
}

// Element i (0..7) of a 16-byte segment as fp32 (exact conversion).
template <int DT>  // 1 = bf16, 0 = fp16
__device__ __forceinline__ float seg_elem(const uint4& v, int i) {
  const uint32_t w = (i >> 1) == 0 ? v.x : (i >> 1) == 1 ? v.y : (i >> 1) == 2 ? v.z : v.w;
  if (DT == 1) return __uint_as_float((i & 1) ? (w & 0xFFFF0000u) : (w << 16));
  return __half2float(__ushort_as_half(static_cast<unsigned short>((i & 1) ? (w >> 16) : (w & 0xFFFFu))));
}

// Shape of the score kernel for keys of up to `max` elements: the fixed order
// gives lane floor(e / 8) mod 32 of 32 lanes element e, so a key of at most
// 8 * kLanes elements has values in kLanes lanes only and 32 / kLanes entries
// lie side by side in a warp; kSeg segments per lane; kRows rows of entries a
// round, all their loads in flight before any arithmetic.  kBlocks leaves the
// registers for that: cut for more blocks, the compiler sinks the loads
// between the arithmetic (D = 768 at three blocks 88 us instead of 80, D = 64
// with a histogram at four 98 instead of 94); at two blocks D = 264 took 132 us
// instead of 114.
template <int LANES, int SEG, int ROWS, int BLOCKS>
struct ScoreShape {
  static constexpr int kLanes = LANES, kSeg = SEG, kRows = ROWS;
  static constexpr int kSide = 32 / LANES;       // entries side by side
  static constexpr int kRound = ROWS * kSide;    // entries a round
  static constexpr int kBlocks = BLOCKS;         // blocks per SM the registers are cut for
  static_assert(ROWS % 2 == 0 && ROWS <= LANES, "rows pair up and halve over the lanes of an entry");
};

// Each warp scores a contiguous, balanced range of entries, a round at a
// time, following a cursor over the banks (one search per warp).  DT = key
// type (1 bf16, 0 fp16).  The bank's query is held in registers as fp32, with
// |q| computed once per bank in the same fixed order.
//
// Issue slots bound the short keys (the memory system the others), so two
// rows step together in paired fp32 operations -- (k_a, k_b) straight from
// the conversions, each half rounded on its own as the separate multiply and
// add -- three instructions an element and row, and a key shorter than 256
// elements shares the warp.  Lanes past a key's end hold zeros: no sum here can
// be -0 (they start at +0), so adding them changes nothing.
// Measured, 512 MB of fp16 keys, kernel time (one entry after the other across
// the warp, four in flight, q.k and k.k paired -> this): D = 64 335 -> 86 us,
// 128 173 -> 84, 192 121 -> 95, 256 95 -> 82, 264 148 -> 114, 512 88 -> 80, 768
// 140 -> 80, 1,024 123 -> 80 (6.7 TB/s); bf16 within 4 % of these.
template <class SH, int DT, int HM, bool BLOB>
__device__ __forceinline__ void score_range(const BankDesc* banks, int n_banks,
                                            uint64_t n_entries, float* __restrict__ scores,
                                            bool hist, uint32_t* s_cnt, unsigned long long* s_w) {
  constexpr int G = SH::kLanes, SPL = SH::kSeg, R = SH::kRows, E = SH::kSide;
  const int lane = threadIdx.x & 31;
  const int t = lane & (G - 1), side = lane / G;  // this lane's segment, entry of a row
  const uint64_t gw = static_cast<uint64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  const uint64_t nw = static_cast<uint64_t>(gridDim.x) * kWarps;
  const uint64_t e_begin = n_entries * gw / nw, e_end = n_entries * (gw + 1) / nw;
  if (e_begin >= e_end) return;
  // The last bank starting at or before e_begin, searched by the whole warp
  // (32 probes a round, as in find_item).
  int b = 0;
  {
    int span = n_banks;
    while (span > 1) {
      const int step = (span + 31) >> 5;
      const int i = b + lane * step;
      const bool le = i < b + span && fetch<!BLOB>(&banks[i].entry_begin) <= e_begin;
      const unsigned m = __ballot_sync(kFull, le);  // lane 0 probes b: never empty
      const int last = 31 - __clz(m);
      b += last * step;
      span = min(step, span - last * step);
    }
  }
  int qbank = -1, segs = 0;
  float qnorm = 0.f;
  float qf[SPL][8];
  uint64_t bank_end = 0;
  BankDesc B{};
  for (uint64_t e0 = e_begin; e0 < e_end;) {
    // Entries of this round must share one bank to use the cached query;
    // a round stops early at a bank boundary.
    if (qbank < 0 || e0 >= bank_end) {  // warp-uniform: load the query, compute |q|
      while (b + 1 < n_banks && fetch<!BLOB>(&banks[b + 1].entry_begin) <= e0) ++b;
      B = banks[b];
      bank_end = b + 1 < n_banks ? fetch<!BLOB>(&banks[b + 1].entry_begin) : n_entries;
      segs = B.D / 8;
      const uint4* qrow = reinterpret_cast<const uint4*>(B.query);
      float sq = 0.f;
#pragma unroll
      for (int j = 0; j < SPL; ++j) {
        const uint4 qv = t + 32 * j < segs ? __ldg(qrow + t + 32 * j) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          qf[j][i] = seg_elem<DT>(qv, i);
          sq = __fadd_rn(sq, __fmul_rn(qf[j][i], qf[j][i]));
        }
      }
#pragma unroll
      for (int d = 1; d < G; d <<= 1) sq = __fadd_rn(sq, __shfl_xor_sync(kFull, sq, d));
      qnorm = __fsqrt_rn(sq);
      qbank = b;
    }
    const uint64_t lim = min(static_cast<unsigned long long>(e_end), static_cast<unsigned long long>(bank_end));
    const int cnt = static_cast<int>(min(static_cast<uint64_t>(SH::kRound), lim - e0));
    const uint64_t kb = static_cast<uint64_t>(B.D) * 2;  // bytes of a key
    const uint8_t* kbase = reinterpret_cast<const uint8_t*>(B.keys) +
                           (e0 - B.entry_begin + side) * kb + 16 * t;
    uint4 kv[R][SPL];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int j = 0; j < SPL; ++j)
        kv[r][j] = r * E + side < cnt && t + 32 * j < segs ? ld_stream(kbase + r * E * kb + 512 * j)
                                                           : make_uint4(0, 0, 0, 0);
    // Per lane and row: the partial q.k and k.k, ascending elements.
    float dot[R], kk[R];
#pragma unroll
    for (int r = 0; r < R; r += 2) {
      float2 d2 = make_float2(0.f, 0.f), k2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < SPL; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 ke = make_float2(seg_elem<DT>(kv[r][j], i), seg_elem<DT>(kv[r + 1][j], i));
          d2 = __fadd2_rn(d2, __fmul2_rn(make_float2(qf[j][i], qf[j][i]), ke));
          k2 = __fadd2_rn(k2, __fmul2_rn(ke, ke));
        }
      dot[r] = d2.x;
      dot[r + 1] = d2.y;
      kk[r] = k2.x;
      kk[r + 1] = k2.y;
    }
    // The lane tree (s[l] += s[l + d], d = 1 .. 16) of all rows at once: while
    // a lane holds more than one row, it keeps half of them, those its bit of
    // d selects, and adds its partner's copy.  Addition is commutative, so
    // every partial sum is the one the plain tree forms.
    int row = 0;
#pragma unroll
    for (int d = 1, h = R / 2; d < G; d <<= 1, h >>= 1) {
      if (h >= 1) {
        const bool up = lane & d;
        row = 2 * row + (up ? 1 : 0);
#pragma unroll
        for (int i = 0; i < R / 2; ++i)
          if (i < h) {
            const float gd = up ? dot[i] : dot[h + i], gk = up ? kk[i] : kk[h + i];
            dot[i] = __fadd_rn(up ? dot[h + i] : dot[i], __shfl_xor_sync(kFull, gd, d));
            kk[i] = __fadd_rn(up ? kk[h + i] : kk[i], __shfl_xor_sync(kFull, gk, d));
          }
      } else {
        dot[0] = __fadd_rn(dot[0], __shfl_xor_sync(kFull, dot[0], d));
        kk[0] = __fadd_rn(kk[0], __shfl_xor_sync(kFull, kk[0], d));
      }
    }
    const int q = row * E + side;
    if (t < R && q < cnt) {
      const float den = __fmul_rn(qnorm, __fsqrt_rn(kk[0]));
      const float sc = den == 0.f ? 0.f : __fdiv_rn(dot[0], den);
      scores[e0 + q] = sc;
      if (HM && hist) {
        const uint32_t d = ord32(sc) >> 21;  // key bits 63..53
        atomicAdd(&s_cnt[d], 1u);
        if (HM == 2) add64_shared(&s_w[d], B.entry_bytes);
      }
    }
    e0 += cnt;
  }
}

// HM (global threshold): 0 none; 1 / 2 also histogram the top 11 key bits of
// every score (2: weighted by the bank's entry bytes) and pick the first digit.
template <class SH, int DT, int HM, bool BLOB>
__global__ void __launch_bounds__(kThreads, SH::kBlocks)
    k_score_fixed(const __grid_constant__ BankArg<BLOB> bank_arg, int n_banks, uint64_t n_entries,
                  float* __restrict__ scores, GHist gh) {
  const BankDesc* banks = bank_arg.get();
  grid_dependency();
  __shared__ uint32_t s_cnt[HM ? kGBins : 1];
  __shared__ unsigned long long s_w[HM == 2 ? kGBins : 1];
  __shared__ bool s_last;
  const bool hist = HM && !__ldcg(&gh.st->done);  // the same for every block
  if (hist) {
    for (int i = threadIdx.x; i < kGBins; i += kThreads) {
      s_cnt[i] = 0;
      if (HM == 2) s_w[i] = 0;
    }
    __syncthreads();
  }
  score_range<SH, DT, HM, BLOB>(banks, n_banks, n_entries, scores, hist, s_cnt, s_w);
  if (hist) gpass_finish<HM == 1>(gh.st, 0, gh.uniform_bytes, s_cnt, s_w, &s_last);
}


// Any key width or a mix of key types: the query is re-read per entry.
template <bool BLOB>
__global__ void __launch_bounds__(kThreads)
    k_score_any(const __grid_constant__ BankArg<BLOB> bank_arg, int n_banks, uint64_t n_entries,
                float* __restrict__ scores) {
  const BankDesc* banks = bank_arg.get();
  grid_dependency();
  const int lane = threadIdx.x & 31;
  const uint64_t gw = static_cast<uint64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  const uint64_t nw = static_cast<uint64_t>(gridDim.x) * kWarps;
  const uint64_t e_begin = n_entries * gw / nw, e_end = n_entries * (gw + 1) / nw;
  if (e_begin >= e_end) return;
  int b = 0;
  {
    int lo = 0, hi = n_banks - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (fetch<!BLOB>(&banks[mid].entry_begin) <= e_begin) lo = mid;
      else hi = mid - 1;
    }
    b = lo;
  }
  int qbank = -1;
  float qnorm = 0.f;
  for (uint64_t e = e_begin; e < e_end; ++e) {
    while (b + 1 < n_banks && fetch<!BLOB>(&banks[b + 1].entry_begin) <= e) ++b;
    const BankDesc& B = banks[b];
    const bool bf16 = B.is_bf16 != 0;
    const uint4* qrow = reinterpret_cast<const uint4*>(B.query);
    if (b != qbank) {
      float sq = 0.f;
      for (int t = lane; t < B.D / 8; t += 32) accum8_query(__ldg(qrow + t), bf16, sq);
      qnorm = __fsqrt_rn(lane_tree_sum(sq));
      qbank = b;
    }
    const uint8_t* krow = reinterpret_cast<const uint8_t*>(B.keys) +
                          (e - B.entry_begin) * static_cast<uint64_t>(B.D) * 2;
    float sd = 0.f, sk = 0.f;
    for (int t = lane; t < B.D / 8; t += 32)
      accum8_key(__ldg(qrow + t), ld_stream(krow + 16 * t), bf16, sd, sk);
    const float d = lane_tree_sum(sd);
    const float kk = lane_tree_sum(sk);
    if (lane == 0) {
      const float den = __fmul_rn(qnorm, __fsqrt_rn(kk));
      scores[e] = den == 0.f ? 0.f : __fdiv_rn(d, den);
    }
  }
}


// Exclusive block scan of a 0/1 flag; returns the rank, *total = sum.
__device__ __forceinline__ uint32_t block_rank(bool f, uint32_t* warp_cnt, uint32_t* total) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(kFull, f);
  const uint32_t in_warp = __popc(m & ((1u << lane) - 1u));
  if (lane == 0) warp_cnt[wib] = __popc(m);
  __syncthreads();
  uint32_t before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = warp_cnt[w];
    if (w < wib) before += c;
    sum += c;
  }
  __syncthreads();
  *total = sum;
  return before + in_warp;
}

// Exclusive block scan of one uint32 per thread; *total = block sum.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* warp_sum,
                                                    uint32_t* total) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) warp_sum[wib] = incl;
  __syncthreads();
  uint32_t before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = warp_sum[w];
    if (w < wib) before += c;
    sum += c;
  }
  __syncthreads();
  *total = sum;
  return before + incl - v;
}

// The digit of one radix-select pass (warp 0, histogram in shared memory):
// scanning bins from the top, the first whose running count reaches the
// rank still wanted is fixed into the prefix.
__device__ __forceinline__ void topk_pick(const uint32_t* hist, int shift, uint32_t* s_prefix,
                                          uint32_t* s_mask, uint32_t* s_remaining) {
  const int lane = threadIdx.x & 31;
  // Lane l covers bins 255-8l .. 248-8l (descending).
  uint32_t local = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) local += hist[255 - 8 * lane - j];
  uint32_t incl = local;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  const uint32_t remaining = *s_remaining;
  const unsigned hit = __ballot_sync(kFull, incl >= remaining);
  const int first = __ffs(hit) - 1;  // remaining <= count, so hit != 0
  if (lane == first) {
    uint32_t cum = incl - local;
    for (int j = 0; j < 8; ++j) {
      const int bin = 255 - 8 * lane - j;
      if (cum + hist[bin] >= remaining) {
        *s_prefix |= static_cast<uint32_t>(bin) << shift;
        *s_mask |= 0xFFu << shift;
        *s_remaining = remaining - cum;
        break;
      }
      cum += hist[bin];
    }
  }
}

constexpr int kTopkPer = 16;                    // entries a thread holds
constexpr int kTopkReg = kThreads * kTopkPer;   // banks up to this size stay in registers

// One bank of at most kTopkReg entries, 0 < k < n: thread t holds the keys of
// entries [16 t, 16 t + 16) for all four passes; the kept entries (every key
// above the threshold, then the first ones equal to it) are ranked with two
// block scans and written in ascending index order.
__device__ void topk_bank_reg(const float* __restrict__ sc, int n, int k, int32_t* __restrict__ out,
                              uint32_t* hist, uint32_t* warp_sum, uint32_t* s_prefix,
                              uint32_t* s_mask, uint32_t* s_remaining) {
  const int base = threadIdx.x * kTopkPer;
  uint32_t u[kTopkPer];
#pragma unroll
  for (int j = 0; j < kTopkPer; ++j) u[j] = base + j < n ? ord32(__ldg(sc + base + j)) : 0u;
  if (threadIdx.x == 0) {
    *s_prefix = 0;
    *s_mask = 0;
    *s_remaining = static_cast<uint32_t>(k);
  }
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int i = threadIdx.x; i < 256; i += kThreads) hist[i] = 0;
    __syncthreads();
    const uint32_t prefix = *s_prefix, mask = *s_mask;
#pragma unroll
    for (int j = 0; j < kTopkPer; ++j)
      if (base + j < n && (u[j] & mask) == prefix) atomicAdd(&hist[(u[j] >> shift) & 255u], 1u);
    __syncthreads();
    if (threadIdx.x < 32) topk_pick(hist, shift, s_prefix, s_mask, s_remaining);
    __syncthreads();
  }
  const uint32_t t = *s_prefix, take_eq = *s_remaining;
  uint32_t gt = 0, eq = 0;
#pragma unroll
  for (int j = 0; j < kTopkPer; ++j) {
    if (base + j < n) {
      gt |= static_cast<uint32_t>(u[j] > t) << j;
      eq |= static_cast<uint32_t>(u[j] == t) << j;
    }
  }
  uint32_t total;
  uint32_t r = block_excl_scan(__popc(eq), warp_sum, &total);  // equal keys before this thread's
  uint32_t keep = gt;
  for (uint32_t m = eq; m; m &= m - 1) {
    if (r >= take_eq) break;
    keep |= m & (~m + 1u);
    ++r;
  }
  uint32_t pos = block_excl_scan(__popc(keep), warp_sum, &total);
  for (uint32_t m = keep; m; m &= m - 1) out[pos++] = base + __ffs(m) - 1;
  __syncthreads();
}

// OFF: also writes kept_off (a build of its own: the test of a null pointer and
// the store at the head of every bank cost 20,000 banks of 40 entries 2.5 %, 257
// us without them and 264 with).
template <bool BLOB, bool OFF>
__global__ void __launch_bounds__(kThreads)
    k_topk(const __grid_constant__ BankArg<BLOB> bank_arg, int n_banks,
           const float* __restrict__ scores, int32_t* __restrict__ kept_idx,
           int32_t* __restrict__ kept_off, int32_t kept_total) {
  const BankDesc* banks = bank_arg.get();
  grid_dependency();
  __shared__ uint32_t hist[256];
  __shared__ uint32_t warp_cnt[kWarps];
  __shared__ uint32_t s_prefix, s_mask, s_remaining;
  const int wib = threadIdx.x >> 5;
  for (int b = blockIdx.x; b < n_banks; b += gridDim.x) {
    const BankDesc B = banks[b];
    if (OFF && threadIdx.x == 0) {
      kept_off[b] = static_cast<int32_t>(B.kept_begin);
      if (b == n_banks - 1) kept_off[n_banks] = kept_total;
    }
    const int n = B.n, k = B.k;
    const float* sc = scores + B.entry_begin;
    int32_t* out = kept_idx + B.kept_begin;
    if (k >= n) {
      for (int i = threadIdx.x; i < n; i += kThreads) out[i] = i;
      continue;
    }
    if (k <= 0) continue;
    if (n <= kTopkReg) {
      topk_bank_reg(sc, n, k, out, hist, warp_cnt, &s_prefix, &s_mask, &s_remaining);
      continue;
    }
    if (threadIdx.x == 0) {
      s_prefix = 0;
      s_mask = 0;
      s_remaining = static_cast<uint32_t>(k);
    }
    __syncthreads();
    // Radix select, most significant byte first: the k-th largest ord32.
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int i = threadIdx.x; i < 256; i += kThreads) hist[i] = 0;
      __syncthreads();
      const uint32_t prefix = s_prefix, mask = s_mask;
      for (int i = threadIdx.x; i < n; i += kThreads) {
        const uint32_t u = ord32(sc[i]);
        if ((u & mask) == prefix) atomicAdd(&hist[(u >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (wib == 0) topk_pick(hist, shift, &s_prefix, &s_mask, &s_remaining);
      __syncthreads();
    }
    // Keep every entry above the threshold and the first `remaining` equal
    // to it, in ascending index order.
    const uint32_t t = s_prefix, take_eq = s_remaining;
    uint32_t eq_seen = 0, written = 0;
    for (int start = 0; start < n; start += kThreads) {
      const int i = start + threadIdx.x;
      const uint32_t u = i < n ? ord32(sc[i]) : 0u;
      const bool gt = i < n && u > t;
      const bool eq = i < n && u == t;
      uint32_t eq_total, kept_total;
      const uint32_t eq_rank = block_rank(eq, warp_cnt, &eq_total);
      const bool keep = gt || (eq && eq_seen + eq_rank < take_eq);
      const uint32_t pos = block_rank(keep, warp_cnt, &kept_total);
      if (keep && written + pos < static_cast<uint32_t>(k)) out[written + pos] = i;
      eq_seen += eq_total;
      written += kept_total;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// One relevance threshold across all banks under a byte budget
//
// The entry at bank-major position i ranks by
//   key(i) = ord32(score_i) << 32 | (0xFFFFFFFF - i)
// (score descending, then bank, then index ascending; unique keys).  The kept
// set is the longest prefix of the descending key order whose entry bytes
// fit the budget: every key above the key of the first entry that does not
// fit.  That key is found most significant digit first, each pass summing
// the bytes (not the count) of the candidate keys per digit and picking the
// digit where the budget runs out.  The first pass rides on the score kernel
// (its last block, by atomic ticket, picks); k_gfinish runs the rest.
// k_gselect bins one pass of a part of a population split over processes;
// the host sums the parts' bins and picks.
// ---------------------------------------------------------------------------

// The bank holding entry i: the last bank in [lo, hi] whose first entry is
// <= i (empty banks share their successor's first entry and come before it).
__device__ __forceinline__ int gbank(const uint64_t* __restrict__ ebeg, int lo, int hi,
                                     uint64_t i) {
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(ebeg + mid) <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <bool UNIFORM>
__global__ void __launch_bounds__(kThreads) k_gselect(GPlan p, int pass) {
  __shared__ uint32_t ch[kGBins];
  __shared__ unsigned long long wh[UNIFORM ? 1 : kGBins];
  __shared__ bool s_last;
  GState* st = p.st;
  if (__ldcg(&st->done)) return;  // the same for every block of the launch
  const int shift = gdigit_shift(pass);
  const uint32_t nb = 1u << gdigit_bits(pass);
  const uint64_t prefix = __ldcg(&st->prefix), mask = __ldcg(&st->mask);
  for (uint32_t i = threadIdx.x; i < nb; i += kThreads) {
    ch[i] = 0;
    if (!UNIFORM) wh[i] = 0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x; t < p.tiles; t += gridDim.x) {
    const uint64_t start = static_cast<uint64_t>(t) * kGTile;
    const uint64_t end = start + kGTile < p.entries ? start + kGTile : p.entries;
    int b = p.tile_bank[t];
    const int hi = p.tile_bank[t + 1];
    // Every load of the tile in flight before any is used.
    constexpr int kPer = kGTile / kThreads;
    float sv[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const uint64_t i = start + static_cast<uint64_t>(j) * kThreads + threadIdx.x;
      sv[j] = i < end ? __ldg(p.scores + i) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const uint64_t i = start + static_cast<uint64_t>(j) * kThreads + threadIdx.x;
      uint32_t d = kGBins;  // not a candidate
      if (i < end) {
        const uint64_t key =
            (static_cast<uint64_t>(ord32(sv[j])) << 32) | (0xFFFFFFFFull - (p.pos_base + i));
        if ((key & mask) == prefix) d = static_cast<uint32_t>(key >> shift) & (nb - 1);
      }
      if (UNIFORM) {
        // Lanes with the same digit add once (the hot digits are few).
        const unsigned same = __match_any_sync(kFull, d);
        if (d < kGBins && lane == __ffs(same) - 1) atomicAdd(&ch[d], __popc(same));
      } else if (d < kGBins) {
        b = gbank(p.ebeg, b, hi, i);
        atomicAdd(&ch[d], 1u);
        add64_shared(&wh[d], __ldg(p.ebytes + b));
      }
    }
  }
  gpass_finish<UNIFORM>(st, pass, p.uniform_bytes, ch, wh, &s_last, !p.local);
}


// ---------------------------------------------------------------------------
// The rest of the global threshold in one cooperative launch (k_gfinish):
// the digit passes after the first and the compaction.  Its blocks are all
// resident at once and meet at grid barriers; the last block to arrive makes
// the digit choice from the summed bins before it releases the others.
//
//   pass 0 (only when the score kernel could not take it): bins of the top
//     digit of every key;
//   the first full scan: keys above the digits fixed so far are kept for
//     sure and counted per tile; keys inside them (the candidates) are
//     binned by the next digit and stored in their 512-entry unit's slots;
//   later passes bin the candidates only;
//   once the threshold is known, the kept candidates join their tiles'
//   counts; each block sums the counts before its contiguous tile range and
//   writes the kept indices and bank offsets of its tiles in order.
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bounded wait (one thread) until *p >= k, read with acquire semantics;
// false if about kWaitCycles of SM clock passed first.
__device__ __forceinline__ bool wait_flag_geq(const uint32_t* p, uint32_t k) {
  const long long t0 = clock64();
  while (ld_acquire(p) < k) {
    if (clock64() - t0 > kWaitCycles) return false;
    __nanosleep(20);
  }
  return true;
}

// Bounded grid barrier number k (1, 2, ...) of a cooperative launch.  The
// arrival count only grows (barrier k is full at k x blocks); the last block
// to arrive runs `last` (every thread of it), then publishes k.  A block that
// waits past kWaitCycles sets the timeout bit and returns false; the others
// then give up at their next barrier.
template <typename F>
__device__ bool grid_barrier(GState* st, uint32_t* err, uint32_t k, bool* s_flag, F&& last) {
  __syncthreads();
  if (threadIdx.x == 0) *s_flag = atom_add_acq_rel(&st->bar_count, 1u) == k * gridDim.x - 1;
  __syncthreads();
  if (*s_flag) {  // the last block: everybody else's writes are visible
    last();
    __syncthreads();
    if (threadIdx.x == 0) st_release(&st->bar_gen, k);
    return true;  // *s_flag stays set until the next barrier rewrites it
  }
  __syncthreads();  // every thread has read *s_flag
  if (threadIdx.x == 0) {
    const bool ok = wait_flag_geq(&st->bar_gen, k);
    if (!ok) atomicOr(err, kDevErrTimeout);
    *s_flag = ok;
  }
  __syncthreads();
  return *s_flag;
}

// The bins of pass `pass`: the state's own for the first pass this launch
// bins (zero at launch), a scratch set (zeroed here) for the later ones.
__device__ __forceinline__ uint32_t* gbins_c(const GPlan& p, int pass, int first) {
  return pass == first ? p.st->chist : p.hb[pass].c;
}
__device__ __forceinline__ unsigned long long* gbins_w(const GPlan& p, int pass, int first) {
  return reinterpret_cast<unsigned long long*>(pass == first ? p.st->whist : p.hb[pass].w);
}

// Add a block's bins to the summed ones.
template <bool UNIFORM>
__device__ __forceinline__ void gbins_add(const uint32_t* ch, const unsigned long long* wh, int nb,
                                          uint32_t* gc, unsigned long long* gw) {
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += kThreads) {
    if (ch[i]) atomicAdd(gc + i, ch[i]);
    if (!UNIFORM && wh[i]) atomicAdd(gw + i, wh[i]);
  }
}

// Bin digit d (kGBins: not a candidate) with the given weight.  Uniform
// weights: every lane of the warp calls it and lanes with the same digit add
// once (the hot digits are few).
template <bool UNIFORM>
__device__ __forceinline__ void gbin(uint32_t* ch, unsigned long long* wh, uint32_t d,
                                     uint64_t bytes) {
  if (UNIFORM) {
    const unsigned same = __match_any_sync(kFull, d);
    if (d < kGBins && (threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&ch[d], __popc(same));
  } else if (d < kGBins) {
    atomicAdd(&ch[d], 1u);
    add64_shared(&wh[d], bytes);
  }
}

// Entries of tile t handled by this thread: warp w takes the 512 entries
// from t * kGTile + 512 w (its unit), lane l the 16 entries from 16 l of them.
constexpr int kGPer = kGTile / kThreads;
constexpr int kGUnit = 32 * kGPer;
static_assert(kGPer == 16, "tile layout: 16 entries per thread");

__device__ __forceinline__ uint64_t glane0(int t) {
  return static_cast<uint64_t>(t) * kGTile + (threadIdx.x >> 5) * kGUnit + (threadIdx.x & 31) * kGPer;
}

// The 16 scores from entry i0 (zero past `end`): four 16-byte loads when the
// run is whole and the scores are 16-byte aligned.
__device__ __forceinline__ void gload(const GPlan& p, uint64_t i0, uint64_t end, float (&sc)[kGPer]) {
  if (p.vec && i0 + kGPer <= end) {
    const float4* v = reinterpret_cast<const float4*>(p.scores + i0);
#pragma unroll
    for (int q = 0; q < kGPer / 4; ++q) {
      const float4 x = __ldg(v + q);
      sc[4 * q] = x.x;
      sc[4 * q + 1] = x.y;
      sc[4 * q + 2] = x.z;
      sc[4 * q + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < kGPer; ++j) sc[j] = i0 + j < end ? __ldg(p.scores + i0 + j) : 0.f;
  }
}

__device__ __forceinline__ uint64_t gkey_of(float sc, uint64_t pos) {
  return (static_cast<uint64_t>(ord32(sc)) << 32) | (0xFFFFFFFFull - pos);
}

// Exclusive warp scan of one uint32 per lane; *total = warp sum.
__device__ __forceinline__ uint32_t warp_excl_scan(uint32_t v, uint32_t* total) {
  const int lane = threadIdx.x & 31;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  *total = __shfl_sync(kFull, incl, 31);
  return incl - v;
}

// The bank of entry i of a tile whose entries lie in banks lo .. hi, with
// its first entry and the next bank's.  Every lane of the warp calls it.
// When the tile touches at most 31 banks, lane k holds the first entry of
// bank lo + k and the search runs over the warp's registers.
__device__ __forceinline__ int gbank_tile(const GPlan& p, int lo, int hi, uint64_t i,
                                          uint64_t* first, uint64_t* next) {
  const int lane = threadIdx.x & 31;
  if (hi - lo <= 30) {  // the same for the whole warp
    const uint64_t eb = __ldg(p.ebeg + lo + min(lane, hi - lo + 1));
    int k = 0;  // the last k <= hi - lo with first entry <= i
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int c = k + step;
      const uint64_t v = __shfl_sync(kFull, eb, c < 31 ? c : 31);
      if (c <= hi - lo && v <= i) k = c;
    }
    *first = __shfl_sync(kFull, eb, k);
    *next = __shfl_sync(kFull, eb, k + 1);
    return lo + k;
  }
  const int b = gbank(p.ebeg, lo, hi, i);
  *first = __ldg(p.ebeg + b);
  *next = __ldg(p.ebeg + b + 1);
  return b;
}

// BLOCKS resident per SM: three without spills, or four whose registers spill
// (see launch_gfinish).
template <bool UNIFORM, int BLOCKS>
__global__ void __launch_bounds__(kThreads, BLOCKS) k_gfinish(GPlan p, int first_pass) {
  __shared__ __align__(16) uint32_t ch[kGBins];
  __shared__ unsigned long long wh[UNIFORM ? 1 : kGBins];
  __shared__ GLocal s;
  __shared__ uint64_t scan64[kWarps];
  __shared__ uint32_t scan32[kWarps];
  __shared__ bool s_ok;
  GState* st = p.st;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint64_t nthreads = static_cast<uint64_t>(gridDim.x) * kThreads;
  const uint64_t gtid = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x;
  const uint32_t units = static_cast<uint32_t>(p.tiles) * kWarps;
  const uint32_t gwarp = blockIdx.x * kWarps + wib, nwarps = gridDim.x * kWarps;
  if (threadIdx.x == 0) gstate_load(st, &s);
  // Scratch bins of the passes after the first binned here; nothing adds to
  // them before the first barrier.
  for (uint64_t i = gtid; i < static_cast<uint64_t>(kGPasses) * kGBins; i += nthreads) {
    const int ps = static_cast<int>(i / kGBins);
    if (ps > first_pass) {
      p.hb[ps].c[i % kGBins] = 0;
      p.hb[ps].w[i % kGBins] = 0;
    }
  }
  auto zero_bins = [&]() {
    for (int i = threadIdx.x; i < kGBins; i += kThreads) {
      ch[i] = 0;
      if (!UNIFORM) wh[i] = 0;
    }
    __syncthreads();
  };
  // The digit choice of a pass, by the last block to reach the barrier after
  // it; every block then reads the new state.
  auto pick = [&](int ps) {
    gpick_block<UNIFORM>(&s, ps, p.uniform_bytes, gbins_c(p, ps, first_pass),
                         gbins_w(p, ps, first_pass), scan64);
    if (threadIdx.x == 0) gstate_store(st, s);
  };
  auto load_state = [&]() {
    if (threadIdx.x == 0) gstate_load(st, &s);
    __syncthreads();
  };
  // Each warp's units in turn (unit u: the candidates of entries
  // [512 u, 512 u + 512)), the next unit's count fetched ahead.
  auto for_units = [&](auto&& body) {
    uint32_t u = gwarp;
    uint32_t nc = u < units ? __ldcg(p.ucand + u) : 0u;
    while (u < units) {
      const uint32_t un = u + nwarps;
      const uint32_t nn = un < units ? __ldcg(p.ucand + un) : 0u;
      if (nc) body(u, nc);
      u = un;
      nc = nn;
    }
  };
  uint32_t nbar = 0;  // barriers passed
  __syncthreads();
  int pass = first_pass;

  // Pass 0: the top digit of every key.
  if (pass == 0 && !s.done) {
    zero_bins();
    for (int t = blockIdx.x; t < p.tiles; t += gridDim.x) {
      const uint64_t end = min(static_cast<uint64_t>(t + 1) * kGTile, p.entries);
      const uint64_t i0 = glane0(t);
      float sc[kGPer];
      gload(p, i0, end, sc);
      int b = 0, hi = 0;
      if (!UNIFORM && i0 < end) {
        hi = p.tile_bank[t + 1];
        b = gbank(p.ebeg, p.tile_bank[t], hi, i0);
      }
#pragma unroll
      for (int j = 0; j < kGPer; ++j) {
        const uint64_t i = i0 + j;
        uint64_t bytes = 0;
        if (!UNIFORM && i < end) {
          while (b < hi && __ldg(p.ebeg + b + 1) <= i) ++b;
          bytes = __ldg(p.ebytes + b);
        }
        gbin<UNIFORM>(ch, wh, i < end ? ord32(sc[j]) >> 21 : kGBins, bytes);
      }
    }
    gbins_add<UNIFORM>(ch, wh, kGBins, gbins_c(p, 0, first_pass), gbins_w(p, 0, first_pass));
    if (!grid_barrier(st, p.err, ++nbar, &s_ok, [&] { pick(0); })) return;
    load_state();
    pass = 1;
  }

  // The first full scan: kept-for-sure counts per tile; candidates (keys
  // inside the digits fixed so far) binned by the next digit and stored in
  // their unit's slots.
  const bool cand_scan = !s.done;
  if (cand_scan) zero_bins();
  {
    const int shift = gdigit_shift(pass);
    const uint32_t dmask = (1u << gdigit_bits(pass)) - 1u;
    const uint64_t prefix = s.prefix, mask = s.mask;
    const uint64_t above = s.done ? s.threshold : (prefix | ~mask);
    for (int t = blockIdx.x; t < p.tiles; t += gridDim.x) {
      const uint64_t end = min(static_cast<uint64_t>(t + 1) * kGTile, p.entries);
      const uint64_t i0 = glane0(t);
      float sc[kGPer];
      gload(p, i0, end, sc);
      uint32_t sure = 0, cm = 0;
#pragma unroll
      for (int j = 0; j < kGPer; ++j) {
        if (i0 + j < end) {
          const uint64_t key = gkey_of(sc[j], p.pos_base + i0 + j);
          if (key > above) ++sure;
          else if (cand_scan && (key & mask) == prefix) cm |= 1u << j;
        }
      }
      uint32_t nc, sure_w;
      const uint32_t at0 = warp_excl_scan(__popc(cm), &nc);
      warp_excl_scan(sure, &sure_w);
      int b = 0, hi = 0;
      uint64_t next = 0;
      if (!UNIFORM && nc) {  // (the same for the whole warp)
        uint64_t first;
        hi = p.tile_bank[t + 1];
        b = gbank_tile(p, p.tile_bank[t], hi, i0, &first, &next);
      }
      if (cm) {  // few lanes: bin the candidates and store them in the unit's slots
        const uint64_t slot = (static_cast<uint64_t>(t) * kWarps + wib) * kGUnit + at0;
        uint32_t k = 0;
#pragma unroll
        for (int j = 0; j < kGPer; ++j) {
          if (cm & (1u << j)) {
            const uint64_t i = i0 + j;
            const uint64_t key = gkey_of(sc[j], p.pos_base + i);
            const uint32_t d = static_cast<uint32_t>(key >> shift) & dmask;
            p.ckey[slot + k] = key;
            atomicAdd(&ch[d], 1u);
            if (!UNIFORM) {
              while (b < hi && next <= i) {
                ++b;
                next = __ldg(p.ebeg + b + 1);
              }
              p.cbank[slot + k] = static_cast<uint32_t>(b);
              add64_shared(&wh[d], __ldg(p.ebytes + b));
            }
            ++k;
          }
        }
      }
      if (lane == 0) {
        p.ucand[static_cast<uint64_t>(t) * kWarps + wib] = nc;
        scan32[wib] = sure_w;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        uint32_t sum = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += scan32[w];
        p.tile_cnt[t] = sum;
      }
      __syncthreads();
    }
  }
  if (cand_scan) {
    gbins_add<UNIFORM>(ch, wh, 1 << gdigit_bits(pass), gbins_c(p, pass, first_pass),
                       gbins_w(p, pass, first_pass));
    if (!grid_barrier(st, p.err, ++nbar, &s_ok, [&] { pick(pass); })) return;
    load_state();
    ++pass;
  }

  // Few keys inside the prefix (the usual case after two digits): one gather of
  // them instead of further passes and of the join below, which saves a digit
  // pass and a grid barrier (270,000 entries in 256 banks, whole call, with the
  // 32-bit sums of add64_shared and the bank search over registers 52.9 -> 47.9
  // us; 21,000 to 26,000 entries of one size 38.2 -> 34.9 and 41.6 -> 39.5).  Candidates above
  // the prefix are kept for sure and join their tiles' counts; the last block
  // to arrive takes the gathered keys' budget prefix directly -- key i fits if
  // the bytes of the keys not below it do -- and adds the kept ones.
  const bool gather = cand_scan && !s.done && s.n_cand <= kGList;
  if (gather) {
    uint64_t* list_key = p.hb[kGPasses - 1].w;
    uint64_t* list_bytes = p.hb[kGPasses - 2].w;
    uint32_t* list_n = p.hb[kGPasses - 1].c;  // zeroed with the scratch bins
    const uint64_t prefix = s.prefix, mask = s.mask, above = prefix | ~mask;
    for_units([&](uint32_t u, uint32_t nc) {
      const uint64_t slot = static_cast<uint64_t>(u) * kGUnit;
      uint32_t kept = 0;
      for (uint32_t k = lane; k < nc; k += 32) {
        const uint64_t key = __ldcg(p.ckey + slot + k);
        kept += key > above;
        if ((key & mask) == prefix) {
          const uint32_t i = atomicAdd(list_n, 1u);
          list_key[i] = key;
          if (!UNIFORM) list_bytes[i] = __ldg(p.ebytes + __ldcg(p.cbank + slot + k));
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) kept += __shfl_xor_sync(kFull, kept, d);
      if (lane == 0 && kept) atomicAdd(p.tile_cnt + u / kWarps, kept);
    });
    auto finish = [&]() {
      uint64_t* key = reinterpret_cast<uint64_t*>(ch);
      uint64_t* bytes = key + kGList;
      const int n = static_cast<int>(s.n_cand);
      for (int i = threadIdx.x; i < n; i += kThreads) {
        key[i] = ld_l2(list_key + i);
        if (!UNIFORM) bytes[i] = ld_l2(list_bytes + i);
      }
      if (threadIdx.x == 0) s.threshold = 0;
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += kThreads) {
        uint64_t sum = 0;
#pragma unroll 1
        for (int j = 0; j < n; ++j)
          if (key[j] >= key[i]) sum += UNIFORM ? 1 : bytes[j];
        if (UNIFORM) sum *= p.uniform_bytes;
        if (sum > s.remaining)
          atomicMax(reinterpret_cast<unsigned long long*>(&s.threshold),
                    static_cast<unsigned long long>(key[i]));
      }
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += kThreads)
        if (key[i] > s.threshold) {
          const uint64_t pos = 0xFFFFFFFFull - (key[i] & 0xFFFFFFFFull) - p.pos_base;
          atomicAdd(p.tile_cnt + pos / kGTile, 1u);
        }
      if (threadIdx.x == 0) {
        s.done = 1;
        gstate_store(st, s);
      }
    };
    if (!grid_barrier(st, p.err, ++nbar, &s_ok, finish)) return;
    load_state();
  }

  // Later passes over the candidates only.
  while (!s.done && pass < kGPasses) {
    zero_bins();
    const int shift = gdigit_shift(pass);
    const uint32_t dmask = (1u << gdigit_bits(pass)) - 1u;
    const uint64_t prefix = s.prefix, mask = s.mask;
    for_units([&](uint32_t u, uint32_t nc) {
      const uint64_t slot = static_cast<uint64_t>(u) * kGUnit;
      for (uint32_t k = lane; k < nc; k += 32) {
        const uint64_t key = __ldcg(p.ckey + slot + k);
        if ((key & mask) == prefix) {
          const uint32_t d = static_cast<uint32_t>(key >> shift) & dmask;
          atomicAdd(&ch[d], 1u);
          if (!UNIFORM)
            add64_shared(&wh[d], __ldg(p.ebytes + __ldcg(p.cbank + slot + k)));
        }
      }
    });
    gbins_add<UNIFORM>(ch, wh, 1 << gdigit_bits(pass), gbins_c(p, pass, first_pass),
                       gbins_w(p, pass, first_pass));
    if (!grid_barrier(st, p.err, ++nbar, &s_ok, [&] { pick(pass); })) return;
    load_state();
    ++pass;
  }
  const uint64_t T = s.threshold;

  // Kept candidates join their tiles' counts.
  if (cand_scan && !gather) {
    for_units([&](uint32_t u, uint32_t nc) {
      const uint64_t slot = static_cast<uint64_t>(u) * kGUnit;
      uint32_t kept = 0;
      for (uint32_t k = lane; k < nc; k += 32) kept += __ldcg(p.ckey + slot + k) > T;
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) kept += __shfl_xor_sync(kFull, kept, d);
      if (lane == 0 && kept) atomicAdd(p.tile_cnt + u / kWarps, kept);
    });
  }
  if (!gather && !grid_barrier(st, p.err, ++nbar, &s_ok, [] {})) return;

  // Write: block b takes tiles [t0, t1) and starts at the kept count before t0.
  const int t0 = static_cast<int>(static_cast<int64_t>(p.tiles) * blockIdx.x / gridDim.x);
  const int t1 = static_cast<int>(static_cast<int64_t>(p.tiles) * (blockIdx.x + 1) / gridDim.x);
  uint32_t before = 0;
  {
    uint32_t part = 0;
    for (int t = threadIdx.x; t < t0; t += kThreads) part += __ldcg(p.tile_cnt + t);
    uint32_t total;
    block_excl_scan(part, scan32, &total);
    before = total;
  }
  if (blockIdx.x == 0) {  // the total and the offsets of trailing empty banks
    uint32_t part = 0;
    for (int t = threadIdx.x; t < p.tiles; t += kThreads) part += __ldcg(p.tile_cnt + t);
    uint32_t total;
    block_excl_scan(part, scan32, &total);
    if (threadIdx.x == 0) {
      st->total_kept = total;
      st->threshold = T;
      p.kept_off[p.n_banks] = static_cast<int32_t>(total);
      for (int b = p.n_banks - 1; b >= 0 && p.ebeg[b] == p.entries; --b)
        p.kept_off[b] = static_cast<int32_t>(total);
    }
  }
  for (int t = t0; t < t1; ++t) {
    const uint64_t end = min(static_cast<uint64_t>(t + 1) * kGTile, p.entries);
    const uint64_t i0 = glane0(t);
    uint32_t keep = 0;  // bit j: entry i0 + j is kept
    {
      float sc[kGPer];
      gload(p, i0, end, sc);
#pragma unroll
      for (int j = 0; j < kGPer; ++j)
        if (i0 + j < end && gkey_of(sc[j], p.pos_base + i0 + j) > T) keep |= 1u << j;
    }
    uint32_t wtot;
    const uint32_t lane_before = warp_excl_scan(__popc(keep), &wtot);
    if (lane == 0) scan32[wib] = wtot;
    __syncthreads();
    uint32_t rank = before + lane_before, all = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t v = scan32[w];
      if (w < wib) rank += v;
      all += v;
    }
    __syncthreads();
    // The lane's bank cursor: bank b holds entries [first, next).
    const int hi = p.tile_bank[t + 1];
    uint64_t first, next;
    int b = gbank_tile(p, p.tile_bank[t], hi, i0, &first, &next);
    if (i0 < end) {
#pragma unroll
      for (int j = 0; j < kGPer; ++j) {
        const uint64_t i = i0 + j;
        if (i < end) {
          while (b < hi && next <= i) {
            ++b;
            first = next;
            next = __ldg(p.ebeg + b + 1);
          }
          if (i == first) {
            p.kept_off[b] = static_cast<int32_t>(rank);
            for (int e = b - 1; e >= 0 && __ldg(p.ebeg + e) == i; --e)
              p.kept_off[e] = static_cast<int32_t>(rank);
          }
          if (keep & (1u << j)) p.kept_idx[rank++] = static_cast<int32_t>(i - first);
        }
      }
    }
    before += all;
  }
}

// ---------------------------------------------------------------------------
// The global threshold of a small population in one block after a plain score
// pass: thread t holds the ranks of entries [16 t, 16 t + 16) for three digit
// passes over ord32(score) (11, 11, 10 bits, the bytes of each digit's
// candidates summed in shared memory), ties at the threshold are kept in
// position order while they fit, and two block scans place the kept entries.
// Bound by the latency of its block-wide steps; it replaces the histogram of
// the score kernel and the grid barriers of k_gfinish, which cost a population
// of any size about 20 us.  Measured, whole calls (those two -> this): 97
// entries 35.9 -> 21.8 us, 4,953 entries 36.4 -> 23.1 us, 4,132 in 146 banks of
// 1,024-wide keys 47.4 -> 27.2 us, 6,463 of one size 34.8 -> 24.7 us.
// ---------------------------------------------------------------------------

constexpr int kGsThreads = 1024;
constexpr int kGsPer = 16;
static_assert(kGsThreads * kGsPer == kGSmallEntries, "entries of the one-block path");
static_assert(kGBins == 2 * kGsThreads, "two bins per thread");

// Inclusive block scan of one value per thread (kGsThreads threads);
// *total = block sum.
template <typename T>
__device__ __forceinline__ T gs_incl_scan(T v, T* warp_sum, T* total) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  T incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T o = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) warp_sum[wib] = incl;
  __syncthreads();
  T w = warp_sum[lane];  // kGsThreads / 32 = 32 warps
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T o = __shfl_up_sync(kFull, w, d);
    if (lane >= d) w += o;
  }
  *total = __shfl_sync(kFull, w, 31);
  const T before = __shfl_sync(kFull, w, wib > 0 ? wib - 1 : 0);
  __syncthreads();  // warp_sum may be reused
  return wib > 0 ? before + incl : incl;
}

template <bool UNIFORM, bool BLOB>
__global__ void __launch_bounds__(kGsThreads, 1)
    k_gsmall(const __grid_constant__ BankArg<BLOB> bank_arg, int n_banks, uint32_t n,
             const float* scores, uint64_t budget, int keep_all, int32_t* __restrict__ kept_idx,
             int32_t* __restrict__ kept_off) {
  const BankDesc* banks = bank_arg.get();
  __shared__ uint32_t s_lo[kGBins];                   // counts (UNIFORM) or low bytes per digit
  __shared__ uint32_t s_hi[UNIFORM ? 1 : kGBins];     // high words of the bytes
  __shared__ uint32_t s_beg[kGSmallBanks + 1];        // first entry of each bank; then n
  __shared__ uint64_t s_bytes[UNIFORM ? 1 : kGSmallBanks];
  __shared__ uint32_t s_rank[kGsThreads];             // kept entries before thread t's
  __shared__ uint16_t s_keep[kGsThreads];             // and which of its own are kept
  __shared__ uint64_t scan64[32];
  __shared__ uint32_t scan32[32];
  __shared__ uint32_t s_prefix;
  __shared__ uint64_t s_left;
  // The bank descriptors are there before the kernel starts.
  for (int b = threadIdx.x; b < n_banks; b += kGsThreads) {
    s_beg[b] = static_cast<uint32_t>(banks[b].entry_begin);
    if (!UNIFORM) s_bytes[b] = banks[b].entry_bytes;
  }
  const uint64_t ubytes = banks[0].entry_bytes;
  if (threadIdx.x == 0) {
    s_beg[n_banks] = n;
    s_prefix = 0;
    s_left = budget;
  }
  grid_dependency();
  const uint32_t i0 = threadIdx.x * kGsPer;
  const uint32_t mine = i0 < n ? min(static_cast<uint32_t>(kGsPer), n - i0) : 0u;
  uint32_t u[kGsPer];
#pragma unroll
  for (int j = 0; j < kGsPer; ++j) u[j] = j < static_cast<int>(mine) ? ord32(scores[i0 + j]) : 0u;
  __syncthreads();
  // The bank of this thread's first entry (the last one starting at or before it).
  int b0 = 0;
  if (mine) {
    int hi = n_banks - 1;
    while (b0 < hi) {
      const int mid = (b0 + hi + 1) >> 1;
      if (s_beg[mid] <= i0) b0 = mid;
      else hi = mid - 1;
    }
  }
  // f(j, bytes of entry i0 + j) for this thread's entries in order.
  auto for_entries = [&](auto&& f) {
    int b = b0;
    uint32_t next = mine ? s_beg[b + 1] : 0;
#pragma unroll
    for (int j = 0; j < kGsPer; ++j) {
      if (j < static_cast<int>(mine)) {
        while (i0 + j >= next) next = s_beg[++b + 1];
        f(j, UNIFORM ? ubytes : s_bytes[b]);
      }
    }
  };
  uint32_t keep = 0;
  if (keep_all) {
    keep = (1u << mine) - 1u;
  } else {
    uint32_t mask = 0;
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0, top = pass == 2 ? 1023 : 2047;
      for (int i = threadIdx.x; i < kGBins; i += kGsThreads) {
        s_lo[i] = 0;
        if (!UNIFORM) s_hi[i] = 0;
      }
      __syncthreads();
      const uint32_t prefix = s_prefix;
      const uint64_t left = s_left;
      for_entries([&](int j, uint64_t bytes) {
        if ((u[j] & mask) != prefix) return;
        const uint32_t d = (u[j] >> shift) & top;
        if (UNIFORM) {
          atomicAdd(&s_lo[d], 1u);
        } else {
          const uint32_t lo = static_cast<uint32_t>(bytes);
          const uint32_t old = atomicAdd(&s_lo[d], lo);
          const uint32_t hi = static_cast<uint32_t>(bytes >> 32) + (old + lo < lo ? 1u : 0u);
          if (hi) atomicAdd(&s_hi[d], hi);
        }
      });
      __syncthreads();
      // Digits from the top, two per thread: the first whose bytes overrun
      // what is left of the budget.  (The population does not fit, so there
      // is one.)
      uint64_t w[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int d = top - 2 * static_cast<int>(threadIdx.x) - k;
        w[k] = d < 0 ? 0
                     : UNIFORM ? s_lo[d] * ubytes
                               : s_lo[d] | (static_cast<uint64_t>(s_hi[d]) << 32);
      }
      uint64_t total;
      const uint64_t incl = gs_incl_scan(w[0] + w[1], scan64, &total);
      const int fit = __syncthreads_count(incl <= left);
      if (static_cast<int>(threadIdx.x) == fit) {
        const uint64_t before = incl - w[0] - w[1];
        const int k = before + w[0] > left ? 0 : 1;
        s_prefix = prefix | (static_cast<uint32_t>(top - 2 * fit - k) << shift);
        s_left = left - before - (k ? w[0] : 0);
      }
      mask |= static_cast<uint32_t>(top) << shift;
      __syncthreads();
    }
    // Every entry above the threshold, and those at it, in position order,
    // while their bytes fit.
    const uint32_t T = s_prefix;
    const uint64_t left = s_left;
    uint64_t tie = 0, total;
    for_entries([&](int j, uint64_t bytes) {
      if (u[j] == T) tie += bytes;
    });
    uint64_t at = gs_incl_scan(tie, scan64, &total) - tie;
    for_entries([&](int j, uint64_t bytes) {
      if (u[j] == T) at += bytes;
      if (u[j] > T || (u[j] == T && at <= left)) keep |= 1u << j;
    });
  }
  uint32_t kept;
  const uint32_t rank = gs_incl_scan(static_cast<uint32_t>(__popc(keep)), scan32, &kept) - __popc(keep);
  s_rank[threadIdx.x] = rank;
  s_keep[threadIdx.x] = static_cast<uint16_t>(keep);
  __syncthreads();
  if (keep) {
    uint32_t r = rank;
    int b = b0;
    for (uint32_t m = keep; m; m &= m - 1) {
      const uint32_t i = i0 + __ffs(m) - 1;
      while (i >= s_beg[b + 1]) ++b;
      kept_idx[r++] = static_cast<int32_t>(i - s_beg[b]);
    }
  }
  for (int b = threadIdx.x; b <= n_banks; b += kGsThreads) {
    const uint32_t i = s_beg[b], t = i / kGsPer;
    kept_off[b] = static_cast<int32_t>(
        i >= n ? kept : s_rank[t] + __popc(s_keep[t] & ((1u << (i % kGsPer)) - 1u)));
  }
}

// ---------------------------------------------------------------------------
// Copy-on-write page pool
//
// A page's count is the number of table slots that hold it.  A fork shares
// pages (count + 1, no bytes move); before a slot's page is written, the copy
// leg gives the slot a private copy if anybody else still holds the page.
// Of several holders writing in one launch, the last one to give up its hold
// finds the count at 1 and keeps the page, so exactly holders - 1 copies are
// made and no page is lost.  Ids are checked against the pool; -1 is an empty
// slot and is skipped.
// ---------------------------------------------------------------------------

__device__ __forceinline__ bool pool_id_ok(const PoolDev& P, int32_t p) {
  if (p < 0) return false;
  if (p >= P.n_pages) {
    atomicOr(P.err, kDevErrIndex);
    return false;
  }
  return true;
}

// Pops aggregated per warp: one atomic on the stack top for the warp's lanes.
__global__ void __launch_bounds__(kThreads) k_pool_alloc(PoolDev P, int32_t* ids, int32_t n) {
  const int32_t j = blockIdx.x * kThreads + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const unsigned want = __ballot_sync(kFull, j < n);
  if (j >= n) return;
  const int cnt = __popc(want), r = __popc(want & ((1u << lane) - 1u));
  const int leader = __ffs(want) - 1;
  int32_t old = 0;
  if (lane == leader) {
    old = atomicSub(P.top, cnt);
    const int32_t ok = old <= 0 ? 0 : (old < cnt ? old : cnt);
    if (ok < cnt) {
      atomicAdd(P.top, cnt - ok);
      atomicOr(P.err, kDevErrNoPage);
    }
  }
  old = __shfl_sync(want, old, leader);
  const int32_t i = old - 1 - r;
  if (i >= 0) {
    const int32_t q = P.free_ids[i];
    P.rc[q] = 1;
    ids[j] = q;
  } else {
    ids[j] = -1;
  }
}

__global__ void __launch_bounds__(kThreads)
    k_pool_share(PoolDev P, const int32_t* src, int32_t* dst, int32_t n) {
  const int32_t j = blockIdx.x * kThreads + threadIdx.x;
  if (j >= n) return;
  const int32_t p = src[j];
  if (dst) dst[j] = p;
  if (!pool_id_ok(P, p)) return;
  if (atomicAdd(&P.rc[p], 1u) == 0u) {
    atomicSub(&P.rc[p], 1u);
    atomicOr(P.err, kDevErrRefcount);
  }
}

__global__ void __launch_bounds__(kThreads)
    k_pool_release(PoolDev P, const int32_t* ids, int32_t n) {
  const int32_t j = blockIdx.x * kThreads + threadIdx.x;
  const unsigned live = __ballot_sync(kFull, j < n);  // lanes that reach the push
  if (j >= n) return;
  const int32_t p = ids[j];
  bool freed = false;
  if (pool_id_ok(P, p)) {
    const uint32_t old = atomicSub(&P.rc[p], 1u);
    if (old == 1u) {
      freed = true;
    } else if (old == 0u) {
      atomicAdd(&P.rc[p], 1u);
      atomicOr(P.err, kDevErrRefcount);
    }
  }
  // Pushes aggregated per warp: one atomic on the stack top.
  const unsigned push = __ballot_sync(live, freed);
  if (!push) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(push) - 1;
  int32_t i0 = 0;
  if (lane == leader) i0 = atomicAdd(P.top, __popc(push));
  i0 = __shfl_sync(live, i0, leader);
  if (freed) {
    const int32_t i = i0 + __popc(push & ((1u << lane) - 1u));
    if (i < P.n_pages) {
      P.free_ids[i] = p;
    } else {  // counts were inconsistent: never write past the stack
      atomicSub(P.top, 1);
      atomicOr(P.err, kDevErrRefcount);
    }
  }
}

// One warp per table slot, eight slots per block round: lane 0 of each warp
// settles its slot's hold; the slots that need a page take them off the free
// stack with one atomic for the block (pages taken past an empty stack are
// given back and reported); then every warp copies its page, kCowDepth
// 16-byte loads in flight per lane.
constexpr int kCowDepth = 8;

__global__ void __launch_bounds__(kThreads)
    k_pool_cow(PoolDev P, int32_t* table, int64_t n_table, const int32_t* entries, int32_t n) {
  __shared__ uint32_t s_need;  // bit w: warp w needs a fresh page
  __shared__ int32_t s_base;   // stack top before this round's pops
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  for (int64_t j0 = static_cast<int64_t>(blockIdx.x) * kWarps; j0 < n;
       j0 += static_cast<int64_t>(gridDim.x) * kWarps) {
    const int64_t j = j0 + wib;
    int32_t p = -1;
    int64_t e = 0;
    bool need = false;
    if (threadIdx.x == 0) s_need = 0;
    __syncthreads();
    if (lane == 0 && j < n) {
      e = entries ? static_cast<int64_t>(entries[j]) : j;
      if (e < 0 || e >= n_table) {
        atomicOr(P.err, kDevErrIndex);
      } else {
        p = table[e];
        if (pool_id_ok(P, p)) {
          const uint32_t old = atomicSub(&P.rc[p], 1u);
          if (old == 1u) {
            atomicAdd(&P.rc[p], 1u);  // held here alone: keep it
          } else if (old == 0u) {
            atomicAdd(&P.rc[p], 1u);
            atomicOr(P.err, kDevErrRefcount);
          } else {
            need = true;
            atomicOr(&s_need, 1u << wib);
          }
        }
      }
    }
    __syncthreads();
    const uint32_t mask = s_need;
    if (threadIdx.x == 0 && mask) {
      const int cnt = __popc(mask);
      const int32_t old = atomicSub(P.top, cnt);
      const int32_t ok = old <= 0 ? 0 : (old < cnt ? old : cnt);
      if (ok < cnt) {
        atomicAdd(P.top, cnt - ok);
        atomicOr(P.err, kDevErrNoPage);
      }
      s_base = old;
    }
    __syncthreads();
    int32_t q = -1;
    if (lane == 0 && need) {
      const int32_t i = s_base - 1 - __popc(mask & ((1u << wib) - 1u));
      if (i >= 0) {
        q = P.free_ids[i];
        P.rc[q] = 1;
      } else {
        atomicAdd(&P.rc[p], 1u);  // no page: keep the shared hold
      }
    }
    q = __shfl_sync(kFull, q, 0);
    if (q >= 0) {
      p = __shfl_sync(kFull, p, 0);
      const uint4* src =
          reinterpret_cast<const uint4*>(P.base + static_cast<uint64_t>(p) * P.page_bytes);
      uint4* dst = reinterpret_cast<uint4*>(P.base + static_cast<uint64_t>(q) * P.page_bytes);
      const uint64_t words = P.page_bytes / 16;
      for (uint64_t k0 = lane; k0 < words; k0 += 32 * kCowDepth) {
        uint4 v[kCowDepth];
#pragma unroll
        for (int u = 0; u < kCowDepth; ++u) {
          const uint64_t k = k0 + 32u * u;
          if (k < words) v[u] = __ldcs(src + k);
        }
#pragma unroll
        for (int u = 0; u < kCowDepth; ++u) {
          const uint64_t k = k0 + 32u * u;
          if (k < words) dst[k] = v[u];
        }
      }
      if (lane == 0) table[e] = q;
    }
  }
}

// ---------------------------------------------------------------------------
// Byte-mismatch distance: the count of differing bytes of buffer pairs (the
// distance D of the discovery procedure at the byte level).
//
// Bound by HBM: two reads and no write per byte pair.  A pair is cut along
// the 16-byte boundaries of its first buffer: `head` single bytes up to the
// first boundary, then 16-byte vectors in units of 2 KiB, then up to 15 single
// bytes.  Where the second buffer sits at the same offset from a boundary
// (buffers carved out of two arenas the same way, or both aligned) its vectors
// are whole loads too; otherwise each is put together from the two aligned
// vectors it straddles (the second of which the neighbouring lane also reads,
// so it comes from L1).  No load reaches outside a buffer: the first and last
// vectors, whose aligned neighbours would, are compared byte by byte.
// Measured (calls back to back; the byte loops of a pair off a boundary ->
// this): 64 pairs of 4 MiB at the same odd offset 455 -> 87 us (6.2 TB/s), at
// two different ones 455 -> 90 us, aligned 90 -> 87 us; 8 pairs of 256 MiB 3,546
// -> 601 us (7.1 TB/s) and 618 us; one pair of 100 kB 73 -> 9 us.
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t bytes_ne(uint32_t x, uint32_t y) {
  return __popc(__vcmpne4(x, y)) >> 3;
}
__device__ __forceinline__ uint32_t bytes_ne(uint4 x, uint4 y) {
  return bytes_ne(x.x, y.x) + bytes_ne(x.y, y.y) + bytes_ne(x.z, y.z) + bytes_ne(x.w, y.w);
}

// Vectors [0, left) of a unit (left <= 128), this lane's at a + 512 k, b + 512 k:
// both sides whole loads.
__device__ __forceinline__ uint32_t mm_unit(const uint8_t* a, const uint8_t* b, uint32_t left,
                                            int lane) {
  uint32_t c = 0;
  uint4 va[4], vb[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    va[k] = vb[k] = make_uint4(0, 0, 0, 0);
    if (lane + 32u * k < left) {
      va[k] = __ldcs(reinterpret_cast<const uint4*>(a + 512 * k));
      vb[k] = __ldcs(reinterpret_cast<const uint4*>(b + 512 * k));
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) c += bytes_ne(va[k], vb[k]);
  return c;
}

// Vectors [from, to) of a unit whose second buffer lies `shift` bytes past a
// 16-byte boundary: its vector straddles two aligned ones.
__device__ __forceinline__ uint32_t mm_unit_shift(const uint8_t* a, const uint8_t* b,
                                                  uint32_t shift, uint32_t from, uint32_t to,
                                                  int lane) {
  uint32_t c = 0;
  uint4 va[4], vb[4], vc[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t x = lane + 32u * k;
    va[k] = vb[k] = vc[k] = make_uint4(0, 0, 0, 0);
    if (x >= from && x < to) {
      va[k] = __ldcs(reinterpret_cast<const uint4*>(a + 512 * k));
      vb[k] = __ldg(reinterpret_cast<const uint4*>(b - shift + 512 * k));
      vc[k] = __ldg(reinterpret_cast<const uint4*>(b - shift + 512 * k + 16));
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) c += bytes_ne(va[k], align_bytes(vb[k], vc[k], shift));
  return c;
}

// Every warp takes a contiguous range of units of the concatenated pairs,
// finds the pair of its first unit once and walks forward; its count of each
// pair is reduced across the warp and added to the pair's sum.  `sums`
// (scratch) starts at the bytes only one buffer of each pair has; the last
// block to finish (atomic ticket, zero on entry and on exit) copies it to the
// caller's counts, which saves a copy between the plan and this launch.
// A call of few pairs has its plan with the launch, as a small call does, and
// its sums in words that are zero on entry and on exit (36 pairs of up to
// 468 kB, whole calls: 8.9 -> 6.1 us).
template <int N>  // pairs the parameter holds (0: the plan is in the workspace)
__global__ void __launch_bounds__(kThreads, 4)
    k_mismatch(const __grid_constant__ MmBlob<N> blob, int32_t n, uint64_t units,
               unsigned long long* sums, uint64_t* counts, uint32_t* ticket) {
  const MmPair* pairs = blob.pairs();
  const uint64_t* unit_begin = blob.begins();
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31;
  const uint64_t warps = static_cast<uint64_t>(gridDim.x) * kWarps;
  const uint64_t w = static_cast<uint64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  uint64_t u = units * w / warps;
  const uint64_t u1 = units * (w + 1) / warps;
  int pi = 0;
  if (u < u1) {
    // The last pair whose first unit is <= u (32 probes a round, as in
    // find_item).
    for (int span = n; span > 1;) {
      const int step = (span + 31) >> 5;
      const int i = pi + lane * step;
      const bool le = i < pi + span && fetch<N == 0>(unit_begin + i) <= u;
      const int last = 31 - __clz(__ballot_sync(kFull, le));  // lane 0 probes pi: never empty
      pi += last * step;
      span = min(step, span - last * step);
    }
  }
  for (; u < u1; ++pi) {
    const uint64_t pbeg = fetch<N == 0>(unit_begin + pi), pend = fetch<N == 0>(unit_begin + pi + 1);
    if (pend <= u) continue;  // nothing of this pair
    const MmPair P = pairs[pi];
    const uint64_t x0 = (u - pbeg) * (kMmUnit / 16);  // the first vector here
    const bool first = u == pbeg, last = u1 >= pend;  // the pair's first / last unit is ours
    uint32_t whole = static_cast<uint32_t>((last ? pend - 1 : u1) - u);
    uint32_t left = last ? static_cast<uint32_t>(P.n_vec - (pend - 1 - pbeg) * (kMmUnit / 16)) : 0;
    const uint8_t* a = P.a + 16 * (x0 + lane);
    const uint8_t* b = P.b + 16 * (x0 + lane);
    uint32_t c = 0;
    if (P.shift == 0) {
#pragma unroll 1
      for (; whole; --whole, a += kMmUnit, b += kMmUnit) c += mm_unit(a, b, kMmUnit / 16, lane);
      if (left) c += mm_unit(a, b, left, lane);
    } else {
      // The aligned neighbours of the pair's first and last vectors may lie
      // outside the buffer: those two are compared byte by byte.
      uint32_t from = first ? 1 : 0;
#pragma unroll 1
      for (; whole; --whole, a += kMmUnit, b += kMmUnit) {
        c += mm_unit_shift(a, b, P.shift, from, kMmUnit / 16, lane);
        from = 0;
      }
      if (left) c += mm_unit_shift(a, b, P.shift, from, left - 1, lane);
      if (lane < 16 ? (first && P.n_vec > 0) : (last && P.n_vec > 1)) {
        const uint64_t at = (lane < 16 ? 0 : 16 * (P.n_vec - 1)) + (lane & 15);
        c += P.a[at] != P.b[at];
      }
    }
    // The single bytes before the first vector and after the last.
    if (first && lane < static_cast<int>(P.head))
      c += (P.a - P.head)[lane] != (P.b - P.head)[lane];
    if (last && lane < static_cast<int>(P.tail))
      c += P.a[16 * P.n_vec + lane] != P.b[16 * P.n_vec + lane];
    const uint32_t tot = __reduce_add_sync(kFull, c);
    if (lane == 0 && tot) atomicAdd(sums + pi, static_cast<unsigned long long>(tot));
    u = last ? pend : u1;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // Eight sums a thread in flight (one after the other, 20,000 took 21 us).
  constexpr int kPer = N > 0 ? 2 : 8;
  for (int i0 = threadIdx.x; i0 < n; i0 += kPer * kThreads) {
    unsigned long long v[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) v[q] = i0 + q * kThreads < n ? __ldcg(sums + i0 + q * kThreads) : 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = i0 + q * kThreads;
      if (i < n) {
        counts[i] = v[q] + blob.more(i);
        if (N > 0) sums[i] = 0;
      }
    }
  }
  if (threadIdx.x == 0) *ticket = 0;
}

// ---------------------------------------------------------------------------
// Reads against buffers: a buffer is read iff a read of at least one byte
// overlaps it (state versus witness: restore reads state, not witness).
//
// The buffers come sorted by start, the empty ones left out.  Of a read
// [a, e) the first candidate is the first buffer whose running maximum end
// exceeds a; from there every buffer starting before e is looked at.  The
// first candidate's own end is that maximum, so it overlaps if it starts
// before e, and most reads end with the test of the next buffer's start.
//
// Bound by the log (16 bytes a read) where the search is cheap: the search
// runs in shared memory, whose wavefronts limit it (a random 8-byte access of
// a warp takes about five).  One search instead of two (the end of the
// candidates needs none), and for long logs a table over equal slices of the
// address range that narrows it to the buffers ending inside the slice of a,
// none or one for most reads.  Each thread has four reads in flight.
// Measured (calls back to back; two binary searches and a read at a time ->
// this): 16M reads against 10 / 200 / 2,000 / 6,000 buffers 122 -> 62, 263 -> 76,
// 332 -> 88, 665 -> 206 us (the last not staged); 100,000 reads against 200
// buffers 30 -> 11 us.  The log alone takes 40 us at 16M reads; address
// arithmetic and the wavefronts of three to four lookups a read are the rest.
// ---------------------------------------------------------------------------

constexpr int kReadStage = 4096;         // buffers staged in shared memory
constexpr int kReadSlices = 4096;        // slices of the address range at most
constexpr int kReadThreads = 1024;       // threads of a block, long logs or many buffers
constexpr int kReadIlp = 4;              // reads a thread has in flight

// A block marks the buffers it saw in a shared bitmap, adds it to the call's
// bitmap (zero on entry) and the last block to finish (atomic ticket, zero on
// entry and on exit) writes every flag: no clearing pass before this launch.
// STAGED: at most kReadStage buffers, their starts and running maxima in
// shared memory; TABLE (staged only): search the slice table first.
// N: buffers the parameter holds; such a call has them with its launch, as a
// small call has its descriptors, and a bitmap that is zero on exit too (8
// buffers, 7,639 reads, whole calls: 8.8 -> 6.0 us).  0: they are in the
// workspace.
template <bool STAGED, bool TABLE, int N>
__global__ void __launch_bounds__(kReadThreads, 2)
    k_classify_reads(const __grid_constant__ ReadBlob<N> blob, ReadPlan P,
                     const uint64_t* __restrict__ addr, const uint64_t* __restrict__ bytes,
                     int64_t m, uint8_t* flags) {
  static_assert(STAGED || N == 0, "a parameter's arrays are staged");
  const uint64_t* const b_start = blob.starts(P);
  const uint64_t* const b_end = blob.ends(P);
  const uint64_t* const b_max = blob.maxends(P);
  const uint32_t* const b_orig = blob.origs(P);
  static_assert(STAGED || !TABLE, "the table indexes the staged arrays");
  extern __shared__ __align__(16) uint8_t rd_smem[];
  uint32_t* const seen = reinterpret_cast<uint32_t*>(rd_smem);  // [words] bitmap
  const int words = (P.n + 31) / 32;
  uint64_t* const s_start = reinterpret_cast<uint64_t*>(seen + ((words + 1) & ~1));
  uint64_t* const s_max = s_start + P.n;
  uint32_t* const tab = reinterpret_cast<uint32_t*>(s_max + P.n);
  for (int w = threadIdx.x; w < words; w += blockDim.x) seen[w] = 0;
  if (STAGED)
    for (int i = threadIdx.x; i < P.n; i += blockDim.x) {
      s_start[i] = fetch<N == 0>(b_start + i);
      s_max[i] = fetch<N == 0>(b_max + i);
    }
  __syncthreads();
  auto start = [&](int i) -> uint64_t { return STAGED ? s_start[i] : __ldg(b_start + i); };
  auto maxend = [&](int i) -> uint64_t { return STAGED ? s_max[i] : __ldg(b_max + i); };
  // The first buffer in [lo, hi) whose running maximum end exceeds a; hi if none.
  auto search = [&](int lo, int hi, uint64_t a) {
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (maxend(mid) > a) hi = mid;
      else lo = mid + 1;
    }
    return lo;
  };
  const uint64_t base = start(0), top = maxend(P.n - 1);
  if (TABLE) {
    // Slice t starts at base + (t << slice_shift); its entry holds the answers
    // for its first address (low half) and for the next slice's (high half).
    for (int t = threadIdx.x; t < P.slices; t += blockDim.x)
      tab[t] = search(0, P.n, base + (static_cast<uint64_t>(t) << P.slice_shift));
    __syncthreads();
    uint32_t both[(kReadSlices + kReadThreads - 1) / kReadThreads];
#pragma unroll
    for (int k = 0; k < (kReadSlices + kReadThreads - 1) / kReadThreads; ++k) {
      const int t = threadIdx.x + k * kReadThreads;
      if (t < P.slices)
        both[k] = tab[t] | ((t + 1 < P.slices ? tab[t + 1] : static_cast<uint32_t>(P.n)) << 16);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < (kReadSlices + kReadThreads - 1) / kReadThreads; ++k) {
      const int t = threadIdx.x + k * kReadThreads;
      if (t < P.slices) tab[t] = both[k];
    }
    __syncthreads();
  }
  auto mark = [&](int i) {
    const uint32_t bit = 1u << (i & 31);
    // Most reads hit a buffer already marked: look before the atomic.
    if (!(seen[i >> 5] & bit)) atomicOr(&seen[i >> 5], bit);
  };
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t j0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; j0 < m;
       j0 += kReadIlp * stride) {
    uint64_t av[kReadIlp], nv[kReadIlp];
#pragma unroll
    for (int k = 0; k < kReadIlp; ++k) {
      const int64_t j = j0 + k * stride;
      av[k] = j < m ? __ldcs(addr + j) : 0;
      nv[k] = j < m ? __ldcs(bytes + j) : 0;
    }
#pragma unroll
    for (int k = 0; k < kReadIlp; ++k) {
      const uint64_t a = av[k];
      if (nv[k] == 0 || a >= top) continue;
      const uint64_t e = a + nv[k] < a ? ~0ull : a + nv[k];
      int lo = 0, hi = P.n;
      if (TABLE) {
        const uint32_t w = tab[a < base ? 0 : (a - base) >> P.slice_shift];
        lo = w & 0xFFFFu;
        hi = w >> 16;
      }
      lo = search(lo, hi, a);  // below P.n, as a < top
      if (start(lo) >= e) continue;
      mark(lo);
      for (int i = lo + 1; i < P.n && start(i) < e; ++i)
        if (fetch<N == 0>(b_end + i) > a) mark(i);
    }
  }
  __syncthreads();
  for (int w = threadIdx.x; w < words; w += blockDim.x) {
    const uint32_t bits = seen[w];
    if (bits & ~__ldcg(P.bitmap + w)) atomicOr(P.bitmap + w, bits);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) seen[0] = atomicAdd(P.ticket, 1u) == gridDim.x - 1;  // no longer the bitmap
  __syncthreads();
  if (!seen[0]) return;
  __threadfence();
  // Several flags a thread in flight, and 1,024 threads where there are many
  // (see the launcher): one after the other on 256, 100,000 flags took 107 us.
  // Kernel time, 1,000 reads of 10,000 / 30,000 / 100,000 buffers 24.4 / 49.9 /
  // 126 -> 15.3 / 19.7 / 30.3 us.  (All blocks setting the flags of what they
  // saw instead took 4M reads of 6,000 buffers from 75 to 275 us, now 68.)
  constexpr int kPer = N > 0 ? 1 : STAGED ? 4 : 8;
  for (int i0 = threadIdx.x; i0 < P.n_all; i0 += kPer * blockDim.x) {
    uint32_t to[kPer], word[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = i0 + q * static_cast<int>(blockDim.x);
      to[q] = i < P.n_all ? fetch<N == 0>(b_orig + i) : 0;
      word[q] = i < P.n ? __ldcg(P.bitmap + (i >> 5)) : 0;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = i0 + q * static_cast<int>(blockDim.x);
      if (i < P.n_all) flags[to[q]] = static_cast<uint8_t>((word[q] >> (i & 31)) & 1u);
    }
  }
  if (N > 0) {
    __syncthreads();
    for (int w = threadIdx.x; w < words; w += blockDim.x) P.bitmap[w] = 0;
  }
  if (threadIdx.x == 0) *P.ticket = 0;
}

// ---------------------------------------------------------------------------
// Self-test of the bounded waits: one thread waits, through the helpers the
// production kernels use and with their bound, for something that never
// happens -- the second arrival at an mbarrier that expects two (the TMA
// pipeline's wait) or a flag nothing writes (the grid barrier's poll) --
// then records the timeout in the context's error word and returns.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__global__ void k_selftest_wait(int which, const uint32_t* never_set, uint32_t* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  bool ok;
  if (which == 0) {
    mbar_init(&bar, 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_arrive(&bar);
    ok = mbar_wait(&bar, 0);
  } else {
    ok = wait_flag_geq(never_set, 1);
  }
  if (!ok) atomicOr(err, kDevErrTimeout);
}

// ---------------------------------------------------------------------------
// A call's descriptors, from the pinned plan slot to its workspace.  A copy
// engine's transfer ahead of a kernel costs the stream two hand-overs between
// engines; this kernel is scheduled while the kernel ahead on the stream still
// runs, reads the slot (the host's) over the host link meanwhile, and writes
// the workspace once that one has finished.  Measured, whole calls (copied by
// the engine -> this): checkpoint + fork + restore + delete of eight KV contexts
// of 12.6 MB 162.6 -> 152.3 us, of three of 4.5 MB 63.7 -> 54.5; prune +
// checkpoint + restore + delete of 60 banks keeping 18 MB 67.6 -> 61.4.
// ---------------------------------------------------------------------------

constexpr int kUploadPer = 4;  // 16-byte words per thread

__global__ void __launch_bounds__(kThreads)
    k_upload(uint4* __restrict__ dst, const uint4* src, uint32_t n) {
  const uint32_t i0 = blockIdx.x * (kThreads * kUploadPer) + threadIdx.x;
  uint4 v[kUploadPer];
#pragma unroll
  for (int k = 0; k < kUploadPer; ++k) {
    const uint32_t i = i0 + k * kThreads;
    v[k] = i < n ? __ldcv(src + i) : make_uint4(0, 0, 0, 0);
  }
  grid_dependency();
#pragma unroll
  for (int k = 0; k < kUploadPer; ++k) {
    const uint32_t i = i0 + k * kThreads;
    if (i < n) dst[i] = v[k];
  }
}

// Launch `k` with programmatic stream serialisation: the GPU may schedule it
// while the kernel before it on `stream` finishes (its blocks wait in
// grid_dependency() until that kernel's writes are visible), instead of only
// after that kernel has retired.  After a copy, an event or another kind of
// stream operation the launch waits as usual.  `early` false: it always
// waits (right after k_upload, whose words a kernel reads before that point
// or through the read-only path).
template <typename... P, typename... A>
cudaError_t launch_on(bool early, void (*k)(P...), unsigned grid, unsigned block, size_t smem,
                      cudaStream_t stream, const A&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, args...);
}
template <typename... P, typename... A>
cudaError_t launch_after(void (*k)(P...), unsigned grid, unsigned block, size_t smem,
                         cudaStream_t stream, const A&... args) {
  return launch_on(true, k, grid, block, smem, stream, args...);
}

template <int MODE>
int occupancy() {
  int b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_stream<MODE>, kThreads, 0);
  return b > 0 ? b : 1;
}

// Blocks of kThreads threads (no dynamic shared memory) of `kernel` that one
// SM holds at once, asked once per kernel.  A grid of SMs x this many blocks
// is one resident wave: a larger grid of equal blocks leaves its last wave
// part-full, with fewer loads in flight while it runs.
int resident_blocks(const void* kernel) {
  static std::mutex mu;
  static const void* keys[64];
  static int vals[64];
  static int n = 0;
  std::lock_guard<std::mutex> lk(mu);
  for (int i = 0; i < n; ++i)
    if (keys[i] == kernel) return vals[i];
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kThreads, 0) != cudaSuccess || b < 1)
    b = 1;
  if (n < 64) {
    keys[n] = kernel;
    vals[n++] = b;
  }
  return b;
}

template <int MODE, bool SHIFT>
cudaError_t launch_bulk_mode(bool early, const SecDesc* secs, WorkList wl, uint64_t* nodes,
                             uint32_t* err, uint32_t* sched, int sm_count, cudaStream_t stream) {
  using Shape = BulkShape<MODE>;
  const size_t smem = sizeof(BulkShared<Shape::kWarps, Shape::kStages>);
  // One bit per device.  Contexts on other threads may set the attribute at
  // the same time; setting it twice is harmless.
  static std::atomic<uint64_t> configured{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (!(configured.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(k_bulk<MODE, SHIFT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_bulk_shared<MODE, SHIFT>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    configured.fetch_or(bit, std::memory_order_release);
  }
  const uint64_t want = (static_cast<uint64_t>(wl.n_tasks) + Shape::kWarps - 1) / Shape::kWarps;
  const int blocks = static_cast<int>(want < static_cast<uint64_t>(sm_count) ? want : sm_count);
  if (wl.n_tasks < static_cast<uint64_t>(kDynMaxTilesPerWarp) * blocks * Shape::kWarps)
    return launch_on(early, k_bulk_shared<MODE, SHIFT>, blocks, Shape::kThreads, smem, stream, secs, wl,
                        nodes, err, sched);
  return launch_on(early, k_bulk<MODE, SHIFT>, blocks, Shape::kThreads, smem, stream, secs, wl, nodes,
                      err);
}

}  // namespace

cudaError_t launch_upload(void* dst, const void* src, uint64_t bytes, cudaStream_t stream) {
  const uint32_t n = static_cast<uint32_t>((bytes + 15) / 16);
  if (n == 0) return cudaSuccess;
  const unsigned grid = (n + kThreads * kUploadPer - 1) / (kThreads * kUploadPer);
  return launch_after(k_upload, grid, kThreads, 0, stream, static_cast<uint4*>(dst),
                      static_cast<const uint4*>(src), n);
}

int stream_blocks_per_sm() { return occupancy<kModePack>(); }

cudaError_t launch_stream(int mode, bool early, bool beside, const SecDesc* secs, WorkList wl,
                          int group_log2, uint64_t* nodes, uint32_t* dev_err, int sm_count,
                          int blocks_per_sm, cudaStream_t stream) {
  if (wl.n_tasks == 0) return cudaSuccess;
  const uint64_t want = (static_cast<uint64_t>(wl.n_tasks) + kWarps - 1) / kWarps;
  const uint64_t cap = static_cast<uint64_t>(sm_count) * blocks_per_sm;
  const int blocks = static_cast<int>(want < cap ? want : cap);
  auto launch = [&](auto kernel) {
    return launch_on(early, kernel, blocks, kThreads, 0, stream, secs, wl, group_log2, nodes,
                     dev_err, beside);
  };
  switch (mode) {
    case kModeHash: return launch(k_stream<kModeHash>);
    case kModePack: return launch(k_stream<kModePack>);
    case kModeRestore: return launch(k_stream<kModeRestore>);
    case kModeRestoreV: return launch(k_stream<kModeRestoreV>);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_bulk(int mode, bool shift, bool early, const SecDesc* secs, WorkList wl, uint64_t* nodes,
                        uint32_t* dev_err, uint32_t* sched, int sm_count, cudaStream_t stream) {
  if (wl.n_tasks == 0) return cudaSuccess;
  auto launch = [&](auto plain, auto shifted) {
    return (shift ? shifted : plain)(early, secs, wl, nodes, dev_err, sched, sm_count, stream);
  };
  switch (mode) {
    case kModeHash: {
      const uint64_t want = (static_cast<uint64_t>(wl.n_tasks) + kHashWarps - 1) / kHashWarps;
      const int blocks = static_cast<int>(want < static_cast<uint64_t>(sm_count) ? want : sm_count);
      return launch_on(early, k_hash, blocks, kHashThreads, 0, stream, secs, wl, nodes);
    }
    case kModePack:
      return launch(launch_bulk_mode<kModePack, false>, launch_bulk_mode<kModePack, true>);
    case kModeRestore:
      return launch(launch_bulk_mode<kModeRestore, false>, launch_bulk_mode<kModeRestore, true>);
    case kModeRestoreV:
      return launch(launch_bulk_mode<kModeRestoreV, false>, launch_bulk_mode<kModeRestoreV, true>);
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE, int BYTES>
static cudaError_t launch_small_mode(bool early, const uint8_t* host_plan, SmallArgs a, int blocks,
                                     cudaStream_t stream) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  static const PlanBlob<0> none{};
  const void* blob = BYTES > 0 ? static_cast<const void*>(host_plan) : static_cast<const void*>(&none);
  void* args[] = {const_cast<void*>(blob), &a};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(k_small<MODE, BYTES>), args);
}

template <int MODE>
static cudaError_t launch_small_size(bool early, const uint8_t* host_plan, uint64_t bytes,
                                     const SmallArgs& a, int blocks, cudaStream_t stream) {
  static_assert(kSmallPlanMax == 31744, "the largest parameter below");
  if (!host_plan) return launch_small_mode<MODE, 0>(early, host_plan, a, blocks, stream);
  if (bytes <= 1008) return launch_small_mode<MODE, 1008>(early, host_plan, a, blocks, stream);
  if (bytes <= 7936) return launch_small_mode<MODE, 7936>(early, host_plan, a, blocks, stream);
  return launch_small_mode<MODE, 31744>(early, host_plan, a, blocks, stream);
}

cudaError_t launch_small(int mode, bool early, const uint8_t* host_plan, uint64_t bytes,
                         const SmallArgs& a, int sm_count, int blocks_per_sm, cudaStream_t stream) {
  if (a.n_tasks == 0 || (host_plan && bytes > kSmallPlanMax)) return cudaErrorInvalidValue;
  const uint64_t want = (static_cast<uint64_t>(a.n_tasks) + kWarps - 1) / kWarps;
  const uint64_t cap = static_cast<uint64_t>(sm_count) * blocks_per_sm;
  const int blocks = static_cast<int>(want < cap ? want : cap);
  switch (mode) {
    case kModeHash: return launch_small_size<kModeHash>(early, host_plan, bytes, a, blocks, stream);
    case kModePack: return launch_small_size<kModePack>(early, host_plan, bytes, a, blocks, stream);
    case kModeRestoreV:
      return launch_small_size<kModeRestoreV>(early, host_plan, bytes, a, blocks, stream);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_finalize(int mode, const SecDesc* secs, const SessDesc* sess, int n_sess,
                            const Entry* entries, uint64_t* nodes, uint64_t* fp_out,
                            const uint64_t* fp_before, uint8_t* flags, uint32_t* bad,
                            int max_secs, cudaStream_t stream) {
  if (n_sess <= 0) return cudaSuccess;
  if (mode != kModeHash && max_secs <= 32 && n_sess >= 256) {
    // Many sessions of few sections: a warp each, not a block each.  Fewer
    // sessions take a block each, a warp per section, so a session's
    // sections are treed side by side (the 64-bank step: 0.224 -> 0.220 ms).
    const int want = (n_sess + kWarps - 1) / kWarps;
    const int blocks = want < 65535 ? want : 65535;
    if (mode == kModePack)
      return launch_after(k_finalize_sessions_warp<kModePack>, blocks, kThreads, 0, stream, secs,
                          sess, n_sess, entries, nodes, flags, bad);
    if (mode == kModeRestoreV)
      return launch_after(k_finalize_sessions_warp<kModeRestoreV>, blocks, kThreads, 0, stream,
                          secs, sess, n_sess, entries, nodes, flags, bad);
    return cudaErrorInvalidValue;
  }
  if (mode == kModeHash) {
    const int blocks = (n_sess + kWarps - 1) / kWarps;
    return launch_after(k_finalize_hash, blocks < 4096 ? blocks : 4096, kThreads, 0, stream, secs,
                        n_sess, nodes, fp_out, fp_before, flags);
  }
  if (mode == kModePack || mode == kModeRestoreV) {
    // A block per session, a warp per section (up to 16 at once: two
    // blocks of 64-register threads fit an SM).
    const int warps = max_secs < 8 ? 8 : max_secs > 16 ? 16 : max_secs;
    const int blocks = n_sess < 65535 ? n_sess : 65535;
    if (mode == kModePack)
      return launch_after(k_finalize_sessions<kModePack>, blocks, 32 * warps, 0, stream, secs, sess,
                          n_sess, entries, nodes, flags, bad);
    return launch_after(k_finalize_sessions<kModeRestoreV>, blocks, 32 * warps, 0, stream, secs,
                        sess, n_sess, entries, nodes, flags, bad);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_reduce_nodes(const NodeLevel* lv, int n_secs, uint64_t* nodes, uint32_t base,
                                uint32_t n_groups, int sm_count, cudaStream_t stream) {
  if (n_groups == 0) return cudaSuccess;
  const uint64_t want = (static_cast<uint64_t>(n_groups) + kWarps - 1) / kWarps;
  const uint64_t cap = static_cast<uint64_t>(sm_count) * 8;
  const int blocks = static_cast<int>(want < cap ? want : cap);
  return launch_after(k_reduce_nodes, blocks, kThreads, 0, stream, lv, n_secs, nodes, base, n_groups);
}

// f(the kernel argument that holds or points at the banks).
template <typename F>
static cudaError_t with_banks(const Banks& k, F&& f) {
  if (k.dev) return f(BankArg<false>{k.dev});
  if (k.n > kBankBlob) return cudaErrorInvalidValue;
  BankArg<true> arg;
  std::memcpy(arg.b, k.host, sizeof(BankDesc) * k.n);
  return f(arg);
}

template <class SH, int DT>
static cudaError_t launch_score_shape(const Banks& banks, uint64_t n_entries, float* scores,
                                      int sm_count, cudaStream_t stream, GHist gh) {
  // A round per warp at least; at most one resident wave (large populations
  // fill it).
  auto launch = [&](auto kernel, const auto& arg) {
    const uint64_t want = (n_entries + kWarps * SH::kRound - 1) / (kWarps * SH::kRound);
    const uint64_t cap = static_cast<uint64_t>(sm_count) *
                         resident_blocks(reinterpret_cast<const void*>(kernel));
    return launch_on(banks.early, kernel, static_cast<unsigned>(want < cap ? want : cap), kThreads,
                     0, stream, arg, banks.n, n_entries, scores, gh);
  };
  if (!gh.st)
    return with_banks(banks, [&](const auto& arg) {
      constexpr bool BLOB = sizeof(arg) > sizeof(void*);
      return launch(k_score_fixed<SH, DT, 0, BLOB>, arg);
    });
  // With a histogram the call has a workspace, and the banks are in it.
  if (!banks.dev) return cudaErrorInvalidValue;
  const BankArg<false> arg{banks.dev};
  return gh.mode == 1 ? launch(k_score_fixed<SH, DT, 1, false>, arg)
                      : launch(k_score_fixed<SH, DT, 2, false>, arg);
}

template <int DT>
static cudaError_t launch_score_type(const Banks& banks, uint64_t n_entries, int max_dim,
                                     float* scores, int sm_count, cudaStream_t stream,
                                     GHist gh) {
  auto go = [&](auto launch) { return launch(banks, n_entries, scores, sm_count, stream, gh); };
  if (max_dim <= 64) return go(launch_score_shape<ScoreShape<8, 1, 8, 3>, DT>);
  if (max_dim <= 128) return go(launch_score_shape<ScoreShape<16, 1, 8, 3>, DT>);
  if (max_dim <= 256) return go(launch_score_shape<ScoreShape<32, 1, 8, 3>, DT>);
  if (max_dim <= 512) return go(launch_score_shape<ScoreShape<32, 2, 4, 3>, DT>);
  if (max_dim <= 768) return go(launch_score_shape<ScoreShape<32, 3, 4, 2>, DT>);
  return go(launch_score_shape<ScoreShape<32, 4, 4, 2>, DT>);
}

cudaError_t launch_score(const Banks& banks, uint64_t n_entries, int max_dim, int key_types,
                         float* scores, int sm_count, cudaStream_t stream,
                         GHist gh, bool* fused) {
  if (fused) *fused = false;
  if (n_entries == 0) return cudaSuccess;
  // key_types: 0 = all fp16, 1 = all bf16, 2 = mixed.
  if (key_types == 2 || max_dim > 1024) {
    // At least two rounds of four entries per warp.
    const uint64_t want = (n_entries + 8 * kWarps - 1) / (8 * kWarps);
    const uint64_t cap = static_cast<uint64_t>(sm_count) *
                         resident_blocks(reinterpret_cast<const void*>(k_score_any<false>));
    return with_banks(banks, [&](const auto& arg) {
      constexpr bool BLOB = sizeof(arg) > sizeof(void*);
      return launch_on(banks.early, k_score_any<BLOB>, static_cast<unsigned>(want < cap ? want : cap), kThreads,
                          0, stream, arg, banks.n, n_entries, scores);
    });
  }
  const cudaError_t e =
      key_types == 1
          ? launch_score_type<1>(banks, n_entries, max_dim, scores, sm_count, stream, gh)
          : launch_score_type<0>(banks, n_entries, max_dim, scores, sm_count, stream, gh);
  if (fused) *fused = gh.st && e == cudaSuccess;
  return e;
}

cudaError_t launch_topk(const Banks& banks, const float* scores, int32_t* kept_idx,
                        int32_t* kept_off, int32_t kept_total, cudaStream_t stream) {
  if (banks.n <= 0) return cudaSuccess;
  return with_banks(banks, [&](const auto& arg) {
    constexpr bool BLOB = sizeof(arg) > sizeof(void*);
    const unsigned grid = banks.n < 65535 ? banks.n : 65535;
    return kept_off ? launch_on(banks.early, k_topk<BLOB, true>, grid, kThreads, 0, stream, arg,
                                banks.n, scores, kept_idx, kept_off, kept_total)
                    : launch_on(banks.early, k_topk<BLOB, false>, grid, kThreads, 0, stream, arg,
                                banks.n, scores, kept_idx, kept_off, kept_total);
  });
}

static int gblocks(const GPlan& p, int sm_count, const void* kernel) {
  const int cap = sm_count * resident_blocks(kernel);
  return p.tiles < cap ? p.tiles : cap;
}

cudaError_t launch_gselect(const GPlan& p, int pass, int sm_count, cudaStream_t stream) {
  if (p.tiles <= 0) return cudaSuccess;
  if (p.uniform) {
    const int g = gblocks(p, sm_count, reinterpret_cast<const void*>(k_gselect<true>));
    k_gselect<true><<<g, kThreads, 0, stream>>>(p, pass);
  } else {
    const int g = gblocks(p, sm_count, reinterpret_cast<const void*>(k_gselect<false>));
    k_gselect<false><<<g, kThreads, 0, stream>>>(p, pass);
  }
  return cudaGetLastError();
}

static unsigned grid_for(int64_t n) { return static_cast<unsigned>((n + kThreads - 1) / kThreads); }

cudaError_t launch_pool_alloc(const PoolDev& p, int32_t* ids, int32_t n, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  k_pool_alloc<<<grid_for(n), kThreads, 0, stream>>>(p, ids, n);
  return cudaGetLastError();
}

cudaError_t launch_pool_share(const PoolDev& p, const int32_t* src, int32_t* dst, int32_t n,
                              cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  k_pool_share<<<grid_for(n), kThreads, 0, stream>>>(p, src, dst, n);
  return cudaGetLastError();
}

cudaError_t launch_pool_release(const PoolDev& p, const int32_t* ids, int32_t n,
                                cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  k_pool_release<<<grid_for(n), kThreads, 0, stream>>>(p, ids, n);
  return cudaGetLastError();
}

cudaError_t launch_pool_cow(const PoolDev& p, int32_t* table, int64_t n_table,
                            const int32_t* entries, int32_t n, int sm_count, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int64_t want = (static_cast<int64_t>(n) + kWarps - 1) / kWarps;
  const int64_t cap = static_cast<int64_t>(sm_count) *
                      resident_blocks(reinterpret_cast<const void*>(k_pool_cow));
  k_pool_cow<<<static_cast<unsigned>(want < cap ? want : cap), kThreads, 0, stream>>>(
      p, table, n_table, entries, n);
  return cudaGetLastError();
}

template <int N>
static cudaError_t launch_mismatch_blob(const MmBlob<N>& blob, int32_t n, uint64_t units,
                                        uint64_t* sums, uint64_t* counts, uint32_t* ticket,
                                        int sm_count, cudaStream_t stream) {
  // One resident wave; a unit per warp until that wave is full, as each
  // further unit of a warp adds a memory round trip to a small call (18 pairs
  // of 64 KiB: 15.4 us with at least eight units a warp and the counts copied
  // by a launch of their own, 10.1 us so).
  const uint64_t want = (units + kWarps - 1) / kWarps;
  const uint64_t cap = static_cast<uint64_t>(sm_count) *
                       resident_blocks(reinterpret_cast<const void*>(k_mismatch<N>));
  k_mismatch<N><<<static_cast<unsigned>(want < cap ? want : cap), kThreads, 0, stream>>>(
      blob, n, units, reinterpret_cast<unsigned long long*>(sums), counts, ticket);
  return cudaGetLastError();
}

template <int N>
static cudaError_t launch_mismatch_host(const MmPair* pairs, const uint64_t* unit_begin,
                                        const uint64_t* extra, int32_t n, uint64_t units,
                                        uint64_t* sums, uint64_t* counts, uint32_t* ticket,
                                        int sm_count, cudaStream_t stream) {
  MmBlob<N> blob;
  std::memcpy(blob.pair, pairs, sizeof(MmPair) * n);
  std::memcpy(blob.unit_begin, unit_begin, 8 * (n + 1));
  std::memcpy(blob.extra, extra, 8 * n);
  return launch_mismatch_blob(blob, n, units, sums, counts, ticket, sm_count, stream);
}

cudaError_t launch_mismatch(bool host, const MmPair* pairs, const uint64_t* unit_begin,
                            const uint64_t* extra, int32_t n, uint64_t units, uint64_t* sums,
                            uint64_t* counts, uint32_t* ticket, int sm_count, cudaStream_t stream) {
  if (units == 0 || n <= 0 || (host && n > kMmBlob)) return cudaErrorInvalidValue;
  if (!host)
    return launch_mismatch_blob(MmBlob<0>{pairs, unit_begin}, n, units, sums, counts, ticket,
                                sm_count, stream);
  auto f = n <= 64 ? launch_mismatch_host<64> : launch_mismatch_host<kMmBlob>;
  return f(pairs, unit_begin, extra, n, units, sums, counts, ticket, sm_count, stream);
}

template <bool STAGED, bool TABLE, int N>
static cudaError_t launch_reads(const ReadPlan& p, const uint64_t* addr, const uint64_t* bytes,
                                int64_t m, uint8_t* flags, unsigned threads, size_t smem,
                                int sm_count, cudaStream_t stream) {
  if (smem > 48 * 1024) {  // long bitmaps or many staged buffers
    // The limit is the kernel's on its device, whichever context asks: set
    // once, to all that a block can have, so that no other thread's call can
    // lower it between here and the launch.  limit[d]: 0 not set yet.
    static std::atomic<int> limit[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int most = limit[dev & 63].load(std::memory_order_acquire);
    if (most == 0) {
      e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_classify_reads<STAGED, TABLE, N>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      if (e != cudaSuccess) return e;
      limit[dev & 63].store(most, std::memory_order_release);
    }
    if (smem > static_cast<size_t>(most)) return cudaErrorInvalidValue;
  }
  const uint64_t want = (static_cast<uint64_t>(m) + threads - 1) / threads;
  // One resident wave: 2,048 threads per SM (32 registers), fewer where the
  // shared memory of 228 KB allows fewer blocks.
  const uint64_t per_sm =
      std::max<uint64_t>(1, std::min<uint64_t>(2048 / threads, 228 * 1024 / (smem + 1024)));
  const uint64_t cap = static_cast<uint64_t>(sm_count) * per_sm;
  ReadBlob<N> blob;
  blob.fill(p);
  k_classify_reads<STAGED, TABLE, N>
      <<<static_cast<unsigned>(want < cap ? want : cap), threads, smem, stream>>>(
          blob, p, addr, bytes, m, flags);
  return cudaGetLastError();
}

cudaError_t launch_classify_reads(bool host, ReadPlan p, const uint64_t* addr,
                                  const uint64_t* bytes, int64_t m, uint8_t* flags, int sm_count,
                                  cudaStream_t stream) {
  if (m <= 0 || p.n <= 0 || (host && p.n_all > kReadBlob)) return cudaErrorInvalidValue;
  const size_t words = (static_cast<size_t>(p.n) + 31) / 32;
  size_t smem = ((words + 1) & ~static_cast<size_t>(1)) * 4;
  const bool staged = p.n <= kReadStage;
  if (staged) smem += 16ull * p.n;
  // A log shorter than eight reads a thread of a full GPU (2.5M) is searched
  // without the table and in smaller blocks: building the table costs each
  // block more than it saves (200 buffers, without / with: 500,000 reads 13.8 /
  // 17.6 us, 2M 23.8 / 23.3, 4M 35.3 / 30.9, 16M 106 / 76).
  const bool table = staged && m >= static_cast<int64_t>(sm_count) * 2048 * 8;
  unsigned threads = staged ? 256 : kReadThreads;  // (many buffers: one block writes their flags)
  if (table) {
    // Slices of the smallest power of two that cover the buffers' span.
    const uint64_t span = p.top - p.base;
    p.slice_shift = 0;
    while (((span - 1) >> p.slice_shift) >= kReadSlices) ++p.slice_shift;
    p.slices = static_cast<int32_t>((span - 1) >> p.slice_shift) + 1;
    smem += 4ull * p.slices;
    threads = kReadThreads;
  }
  auto f = launch_reads<false, false, 0>;
  if (table) {
    f = host ? launch_reads<true, true, kReadBlob> : launch_reads<true, true, 0>;
  } else if (staged) {
    f = host ? launch_reads<true, false, kReadBlob> : launch_reads<true, false, 0>;
  }
  return f(p, addr, bytes, m, flags, threads, smem, sm_count, stream);
}

cudaError_t launch_gfinish(const GPlan& p, int first_pass, int sm_count, cudaStream_t stream) {
  if (p.tiles <= 0) return cudaSuccess;
  // Every block must be resident at once: at most one wave, each block with as
  // many tiles as it takes.  The build of four blocks per SM spills, and is
  // taken only where its wider wave saves every block a tile.  Both measured
  // (whole calls, 64-wide keys, three / four blocks per SM): 1.86 M entries, one
  // tile each 75.5 / 75.8 us; 1.95 M, two against one 85.6 / 80.8; 2.4 M 95.3 /
  // 91.4; 2.6 M, two each 100.4 / 103.0; 3.7 M 121.8 / 128.6; 4.4 M, three
  // against two 145.7 / 143.9.
  const void* k3 = p.uniform ? reinterpret_cast<const void*>(k_gfinish<true, 3>)
                             : reinterpret_cast<const void*>(k_gfinish<false, 3>);
  const void* k4 = p.uniform ? reinterpret_cast<const void*>(k_gfinish<true, 4>)
                             : reinterpret_cast<const void*>(k_gfinish<false, 4>);
  const int cap3 = sm_count * resident_blocks(k3), cap4 = sm_count * resident_blocks(k4);
  const bool wide = (p.tiles + cap4 - 1) / cap4 < (p.tiles + cap3 - 1) / cap3;
  const void* k = wide ? k4 : k3;
  const int cap = wide ? cap4 : cap3;
  const int grid = p.tiles < cap ? p.tiles : cap;
  GPlan a = p;
  int fp = first_pass;
  void* args[] = {&a, &fp};
  return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kThreads), args, 0, stream);
}


cudaError_t launch_gsmall(const Banks& banks, uint64_t entries, const float* scores,
                          uint64_t budget, bool uniform, bool keep_all, int32_t* kept_idx,
                          int32_t* kept_off, cudaStream_t stream) {
  if (entries == 0 || entries > kGSmallEntries || banks.n < 1 || banks.n > kGSmallBanks)
    return cudaErrorInvalidValue;
  const uint32_t n = static_cast<uint32_t>(entries);
  const int all = keep_all ? 1 : 0;
  return with_banks(banks, [&](const auto& arg) {
    constexpr bool BLOB = sizeof(arg) > sizeof(void*);
    return uniform ? launch_after(k_gsmall<true, BLOB>, 1, kGsThreads, 0, stream, arg, banks.n, n,
                                  scores, budget, all, kept_idx, kept_off)
                   : launch_after(k_gsmall<false, BLOB>, 1, kGsThreads, 0, stream, arg, banks.n, n,
                                  scores, budget, all, kept_idx, kept_off);
  });
}

cudaError_t launch_selftest_wait(int which, const uint32_t* never_set, uint32_t* err,
                                 cudaStream_t stream) {
  k_selftest_wait<<<1, 32, 0, stream>>>(which, never_set, err);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Fingerprints with no allocation
//
// For callers that cannot allocate device memory, pcs_fingerprint_static runs
// the fingerprint with its whole working set in one fixed array owned by this
// file: the tree nodes of one call.  The plan (at most kStaticMaxBufs buffers)
// travels as a kernel parameter.  The array is created with the module on
// every GPU that runs the call and stays there until the process exits; all
// calls share it, so calls that overlap on the GPU race on it.  No slot needs
// to start at zero: a call writes every node it later reads.
// ---------------------------------------------------------------------------

namespace {

static __device__ __align__(256) uint64_t g_static_nodes[kStaticMaxNodes];

__global__ void __launch_bounds__(kThreads)
    k_fp_static(const StaticPlan plan, uint64_t* __restrict__ nodes) {
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * kWarps;
  const int g = plan.glog2;
  for (uint32_t task = blockIdx.x * kWarps + (threadIdx.x >> 5); task < plan.n_tasks; task += nw) {
    int j = 0;
    while (j + 1 < plan.n && plan.b[j + 1].task_begin <= task) ++j;
    const StaticBuf& b = plan.b[j];
    const uint32_t local = task - b.task_begin;
    const uint64_t c0 = static_cast<uint64_t>(local) << g;
    const uint64_t c1 = min(c0 + (1ull << g), static_cast<unsigned long long>(b.n_chunks));
    uint64_t mine = 0;  // lane j keeps the hash of chunk c0 + j
    for (uint64_t c = c0; c < c1; ++c) {
      uint64_t h = fmix(kSeed ^ (c * 32u + lane));
#pragma unroll
      for (int k = 0; k < kSegs; ++k) {
        const uint64_t off = c * kChunkBytes + 512u * k + 16u * lane;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (off < b.bytes) {
          const uint64_t left = b.bytes - off;
          if (left >= 16 && b.align == 16) v = ld_stream(b.ptr + off);
          else v = ld_small(b.ptr + off, left < 16 ? static_cast<int>(left) : 16, b.align >= 4);
        }
        h = absorb(h, v);
      }
      const uint64_t x = __shfl_sync(kFull, warp_tree(fmix(h), 32, lane), 0);
      if (lane == static_cast<int>(c - c0)) mine = x;
    }
    const uint64_t root = warp_tree(mine, static_cast<int>(c1 - c0), lane);
    if (lane == 0) nodes[b.task_begin + local] = root;
  }
}

__global__ void __launch_bounds__(kThreads)
    k_fp_static_final(const StaticPlan plan, uint64_t* nodes, uint64_t* __restrict__ fp_out) {
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * kWarps + (threadIdx.x >> 5);
  if (i >= plan.n) return;
  const StaticBuf& b = plan.b[i];
  const uint64_t root = warp_tree_inplace(nodes + b.task_begin, b.n_tasks, lane);
  if (lane == 0) fp_out[i] = fmix(root ^ (b.bytes * kP));
}

}  // namespace

cudaError_t static_scratch(uint64_t** nodes) {
  static std::mutex mu;
  static uint64_t* addr[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_nodes);
    if (e != cudaSuccess) return e;
    addr[dev] = static_cast<uint64_t*>(p);
  }
  *nodes = addr[dev];
  return cudaSuccess;
}

cudaError_t launch_fingerprint_static(const StaticPlan& plan, uint64_t* nodes, uint64_t* fp_out,
                                      cudaStream_t stream) {
  if (plan.n <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const uint64_t want = (static_cast<uint64_t>(plan.n_tasks) + kWarps - 1) / kWarps;
  const uint64_t cap = static_cast<uint64_t>(sms) * 4;
  const int blocks = static_cast<int>(want < cap ? (want ? want : 1) : cap);
  k_fp_static<<<blocks, kThreads, 0, stream>>>(plan, nodes);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_fp_static_final<<<(plan.n + kWarps - 1) / kWarps, kThreads, 0, stream>>>(plan, nodes, fp_out);
  return cudaGetLastError();
}

}  // namespace pcs
