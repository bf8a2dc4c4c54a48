// GPU library of the two-layer codec: block index, fused two-layer decode
// (whole archive and unified seek), closure search, verification, and the
// C ABI declared in include/ace.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "ace.h"
#include "ace_device.cuh"
#include "ace_format.h"

using namespace ace;

namespace {

constexpr uint64_t kDefaultTimeoutNs = 2000000000ull;
constexpr uint32_t kMaxLevelLaunches = 32;  // whole decodes with more levels wait on flags instead
// A seek's closure marks its blocks' ready flags with the call's epoch and
// this bit; publishing a decoded block clears it.  A source block whose flag
// shows neither is outside the closure: the archive is corrupt.  (Epochs
// count calls on one scratch buffer and stay below 2^31.)
constexpr uint32_t kPendingFlag = 0x80000000u;

inline uint64_t align256(uint64_t v) { return (v + 255) & ~255ull; }

__host__ __device__ inline uint32_t esc_cap(uint32_t log2B) { return 2 * ((1u << log2B) / 255) + 2; }

// ------------------------------------------------------------ index kernels

struct IndexArgs {
  uint64_t* match_ptr;  // n_blocks + 1 entries: first match record of each block
  const uint8_t* arc;
  const ace_block_dir* dir;
  const uint32_t* dep_ptr;
  const uint32_t* dep_iv;
  IndexHdr* ih;
  uint32_t* level;
  uint32_t* order;
  uint32_t* lv_count;  // n_blocks + 1 entries
  uint32_t* lv_cursor; // n_blocks + 1 entries
  uint64_t nb, total, payload_off, arc_bytes, deps_off;
  uint64_t max_iv;  // intervals that fit between the pointer table and the payload
  uint32_t log2B, w;
};

// Checks every directory entry and dependency record so the decoder may trust
// stream bounds and token counts (Section 2 block layout, Section 3 streams).
__global__ void validate_kernel(IndexArgs a) {
  uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (b == 0) {  // the interval table must end before the payload
    const uint32_t niv = a.dep_ptr[a.nb];
    a.ih->n_iv = niv;
    if (a.deps_off + 4 * (a.nb + 1) + 8ull * niv > a.payload_off)
      record_error(&a.ih->status, &a.ih->err_block, &a.ih->err_where, ACE_E_CORRUPT, 0, 12);
  }
  if (b >= a.nb) return;
  const ace_block_dir d = a.dir[b];
  uint64_t B = (uint64_t)1 << a.log2B, bstart = b << a.log2B;
  uint64_t blen = min(B, a.total - bstart);
  uint32_t where = 0;
  for (int k = 0; k < 3 && !where; k++) {
    if (d.mode[k] > 1) where = 1;  // 0: rANS, 1: stored
    else if (d.nsym[k] == 0 && d.stream_bytes[k] != 0) where = 2;
    else if (d.nsym[k] != 0) {
      if (d.mode[k] == 1 ? d.stream_bytes[k] != d.nsym[k] : d.stream_bytes[k] < ACE_STREAM_HEAD) where = 3;
      else if (d.stream_off[k] & 15) where = 3;
      else if (a.payload_off + d.stream_off[k] + d.stream_bytes[k] > a.arc_bytes ||
               d.stream_off[k] > a.arc_bytes)
        where = 4;
    }
  }
  if (!where) {
    if (d.ntok == 0 || d.ntok > blen + 1) where = 5;
    else if (d.nsym[ACE_S_LIT] > blen) where = 6;
    else if ((uint64_t)d.nsym[ACE_S_LEN] != 2ull * d.nesc + 2ull * d.ntok) where = 7;
    else if ((uint64_t)d.nsym[ACE_S_OFF] != (uint64_t)a.w * (d.ntok - 1)) where = 8;
    else if (d.nesc > esc_cap(a.log2B)) where = 9;
  }
  if (!where) {
    uint32_t lo = a.dep_ptr[b], hi = a.dep_ptr[b + 1], niv = a.dep_ptr[a.nb];
    if (lo > hi || hi > niv || hi > a.max_iv) where = 10;  // intervals read below stay before the payload
    else
      for (uint32_t i = lo; i < hi && !where; i++) {
        uint32_t f = a.dep_iv[2 * i], l = a.dep_iv[2 * i + 1];
        if (f > l || l >= b) where = 11;
      }
  }
  if (where) record_error(&a.ih->status, &a.ih->err_block, &a.ih->err_where, ACE_E_CORRUPT, (uint32_t)b, where);
  else atomicMax(&a.ih->max_ntok, d.ntok);
  a.match_ptr[b + 1] = d.ntok ? d.ntok - 1 : 0;  // this block's matches; scanned below
}

// Inclusive scan of the per-block match counts into record offsets (one CTA).
__global__ void match_scan_kernel(IndexArgs a) {
  __shared__ unsigned long long carry;
  __shared__ unsigned long long wsum[32];
  if (threadIdx.x == 0) {
    carry = 0;
    a.match_ptr[0] = 0;
  }
  __syncthreads();
  uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (uint64_t c0 = 1; c0 <= a.nb; c0 += blockDim.x) {
    uint64_t i = c0 + threadIdx.x;
    unsigned long long v = i <= a.nb ? a.match_ptr[i] : 0, incl = v;
    for (int d = 1; d < 32; d <<= 1) {
      unsigned long long u = __shfl_up_sync(kFull, incl, d);
      if (lane >= (uint32_t)d) incl += u;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      unsigned long long x = lane < nw ? wsum[lane] : 0, xi = x;
      for (int d = 1; d < 32; d <<= 1) {
        unsigned long long u = __shfl_up_sync(kFull, xi, d);
        if (lane >= (uint32_t)d) xi += u;
      }
      if (lane < nw) wsum[lane] = xi - x;
    }
    __syncthreads();
    unsigned long long out = carry + wsum[wid] + incl;
    if (i <= a.nb) a.match_ptr[i] = out;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = out;
    __syncthreads();
  }
  if (threadIdx.x == 0) a.ih->n_matches = carry;
}

// Dependency levels: level[b] = 0 without sources in other blocks, else
// 1 + the deepest block it reads (Section 2).  Sources always precede, so
// one CTA walks the blocks in chunks and relaxes each chunk to its fixed point.
// One sweep of the dependency levels (Section 2: a block decodes once the
// blocks it reads are present), a warp per block with its lanes over the
// block's dependency intervals: level[b] <- max(level[b], 1 + the largest
// level of a block it reads).  Levels only grow toward each block's depth in
// the dependency graph, and reach it after as many sweeps as there are
// levels; a sweep that changes a level sets its flag.
constexpr uint32_t kLevelSweeps = 8;

__global__ void levels_sweep_kernel(IndexArgs a, uint32_t sweep) {
  __shared__ uint32_t changed;
  if (*(volatile uint32_t*)&a.ih->status) return;
  if (sweep > 0 && !*(volatile uint32_t*)&a.ih->relax[sweep - 1]) return;  // settled already
  if (threadIdx.x == 0) changed = 0;
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t nw = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t b = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; b < a.nb; b += nw) {
    uint32_t lv = 0;
    const uint32_t e1 = a.dep_ptr[b + 1];
    for (uint32_t e = a.dep_ptr[b] + lane; e < e1; e += 32)
      for (uint32_t k = a.dep_iv[2 * e]; k <= a.dep_iv[2 * e + 1]; k++) lv = max(lv, a.level[k] + 1);
#pragma unroll
    for (int d = 16; d; d >>= 1) lv = max(lv, __shfl_xor_sync(kFull, lv, d));
    if (lane == 0 && lv > a.level[b]) {
      a.level[b] = lv;
      changed = 1;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && changed) a.ih->relax[sweep] = 1;  // one store per CTA, not per block
}

// The levels in one CTA, block chunk by block chunk, for archives whose
// levels did not settle within the sweeps (deep dependency chains).
__global__ void levels_kernel(IndexArgs a) {
  __shared__ int changed;
  if (*(volatile uint32_t*)&a.ih->status || !*(volatile uint32_t*)&a.ih->relax[kLevelSweeps - 1]) return;
  for (uint64_t c0 = 0; c0 < a.nb; c0 += blockDim.x) {
    uint64_t b = c0 + threadIdx.x;
    if (b < a.nb) a.level[b] = 0;
    __syncthreads();
    while (true) {
      if (threadIdx.x == 0) changed = 0;
      __syncthreads();
      if (b < a.nb) {
        uint32_t lv = 0;
        for (uint32_t i = a.dep_ptr[b]; i < a.dep_ptr[b + 1]; i++)
          for (uint32_t k = a.dep_iv[2 * i]; k <= a.dep_iv[2 * i + 1]; k++) lv = max(lv, a.level[k] + 1);
        if (lv != a.level[b]) {
          a.level[b] = lv;
          changed = 1;
        }
      }
      __syncthreads();
      if (!changed) break;
      __syncthreads();
    }
  }
}

__global__ void level_hist_kernel(IndexArgs a) {
  if (*(volatile uint32_t*)&a.ih->status) return;
  uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (b < a.nb) {
    const uint32_t lv = a.level[b];
    atomicAdd(&a.lv_count[lv], 1u);
    atomicMax(&a.ih->n_levels, lv + 1);
  }
}

// Exclusive scan of the level histogram into level start offsets (one CTA).
__global__ void level_scan_kernel(IndexArgs a) {
  __shared__ uint32_t carry;
  __shared__ uint32_t wsum[32];
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (uint64_t c0 = 0; c0 < a.nb + 1; c0 += blockDim.x) {
    uint64_t i = c0 + threadIdx.x;
    uint32_t v = i < a.nb + 1 ? a.lv_count[i] : 0;
    uint32_t incl = warp_incl_sum(v, lane);
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      uint32_t s = lane < nw ? wsum[lane] : 0;
      uint32_t si = warp_incl_sum(s, lane);
      if (lane < nw) wsum[lane] = si - s;
    }
    __syncthreads();
    uint32_t ex = carry + wsum[wid] + incl - v;
    if (i < a.nb + 1) a.lv_cursor[i] = ex;
    if (i < 33) a.ih->lvc[i] = v;  // the host reads the first levels' sizes with the header
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = ex + v;
    __syncthreads();
  }
}

__global__ void level_scatter_kernel(IndexArgs a) {
  if (*(volatile uint32_t*)&a.ih->status) return;
  uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (b < a.nb) a.order[atomicAdd(&a.lv_cursor[a.level[b]], 1u)] = (uint32_t)b;
}

// An index read back from storage, checked against its archive instead of
// rebuilt.  Each block's level must be the fixed point of the level rule
// (0 without dependencies, else 1 + the deepest block it reads): one sweep
// verifies what the build reaches by iterating.  A warp per block.
__global__ void level_verify_kernel(IndexArgs a) {
  if (*(volatile uint32_t*)&a.ih->status) return;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t nw = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t b = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; b < a.nb; b += nw) {
    uint32_t lv = 0;
    const uint32_t e1 = a.dep_ptr[b + 1];
    for (uint32_t e = a.dep_ptr[b] + lane; e < e1; e += 32)
      for (uint32_t k = a.dep_iv[2 * e]; k <= a.dep_iv[2 * e + 1]; k++) lv = max(lv, a.level[k] + 1);
#pragma unroll
    for (int d = 16; d; d >>= 1) lv = max(lv, __shfl_xor_sync(kFull, lv, d));
    if (lane == 0 && (lv != a.level[b] || lv >= a.ih->n_levels))
      record_error(&a.ih->status, &a.ih->err_block, &a.ih->err_where, ACE_E_CORRUPT, (uint32_t)b, 60);
  }
}

// The decode order of a stored index: a permutation of the blocks (seen
// marks each once), in non-decreasing level, position i inside its level's
// range of the order (the level's end in lv_cursor, its size in lv_count).
__global__ void order_verify_kernel(IndexArgs a, uint32_t* seen) {
  if (*(volatile uint32_t*)&a.ih->status) return;
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  // the first levels' sizes in the header (the host's level ranges) match
  if (i < 33 && i < a.ih->n_levels && i <= a.nb && a.ih->lvc[i] != a.lv_count[i])
    record_error(&a.ih->status, &a.ih->err_block, &a.ih->err_where, ACE_E_CORRUPT, (uint32_t)i, 62);
  if (i >= a.nb) return;
  const uint32_t b = a.order[i];
  bool bad = b >= a.nb;
  if (!bad) {
    bad = atomicExch(seen + b, 1u) != 0;
    const uint32_t L = a.level[b];
    bad |= L >= a.ih->n_levels || L > a.nb;
    if (!bad) {
      const uint32_t end = a.lv_cursor[L], cnt = a.lv_count[L];
      bad |= i >= end || end < cnt || i < end - cnt;
    }
  }
  if (bad) record_error(&a.ih->status, &a.ih->err_block, &a.ih->err_where, ACE_E_CORRUPT, (uint32_t)i, 61);
}

// ----------------------------------------------------------- decode kernel

struct DecodeArgs {
  const uint8_t* arc;
  const ace_block_dir* dir;
  uint64_t payload_off;
  uint64_t total;
  uint64_t nb;
  uint32_t log2B, w;
  uint32_t window;         // tokens whose positions sit in shared memory at a time (multiple of 32)
  uint32_t esc_cap;        // escape values a block may hold
  uint32_t warp_smem;      // bytes of shared memory per warp
  uint32_t max_ntok;       // most tokens in any block
  uint32_t n_items;        // whole decode: work items; seek: read from the scratch header
  const uint32_t* items;   // whole decode: blocks in (level, block) order; seek: the closure
  uint8_t* out;            // whole decode: output (absolute positions); seek: block slots
  ScratchHdr* sh;
  uint32_t* ready;         // per block: the epoch once the block is decoded
  const uint32_t* slot_of; // seek: block -> slot
  uint32_t n_slots;        // seek: slots in the call's scratch (every slot_of entry read is checked against it)
  uint8_t* slice;          // seek: caller's output
  uint64_t coord, len;     // seek: requested range
  uint64_t timeout_ns;
  MatchRec* recs;          // match records, from the token pass to the literal and match passes
  const uint64_t* match_ptr;  // whole decode: block -> first record; null: max_ntok records per slot
  const uint32_t* level;   // each block's dependency level
  uint32_t cur_level;      // whole decode by levels: the level this launch resolves
  bool closure_flags;      // seek: the closure marked its blocks' ready flags (kPendingFlag)
  // fused schedule: per level the blocks whose matches are resolved, and
  // (whole decodes) the blocks the level holds (seeks read them from the
  // scratch header)
  uint32_t* lv_done;
  const uint32_t* lv_count;
  // seek batches: match records per work item rather than per slot
  const uint32_t* rec_index;
  uint32_t n_rec_slots;
  uint32_t long_min;       // matches at least this long (not overlapping) copy in 16-byte pieces
};

// Shared memory of one warp in the token pass: one stream's tables at a
// time, the length and offset streams' renormalisation rings, and the block's
// escape values.
struct TokMem {
  Lut* lut;
  uint8_t* ring;   // [2][kRing]: lengths, offsets
  uint16_t* esc;   // [esc_cap]
};

// Shared memory of one warp in the literal pass: the literal stream's tables
// and ring, and where the literals of the current step go: a bit per literal
// that starts a run (at most 32 literals per token of the window), and each
// run's shift (its place in the block less its first literal's index), after
// the shift of the run the step starts in (at most two runs per token).
struct LitMem {
  Lut* lut;
  uint8_t* ring;    // [kRing]
  uint32_t* start;  // [window]
  uint16_t* shift;  // [2 window + 1]
};

constexpr uint32_t kMatchGroup = 32;  // matches resolved together, one per lane
// Groups of match records in flight to shared memory (a ring after the
// group's own arrays).
constexpr uint32_t kRecDepth = 4;
constexpr uint32_t kRowMax = 64;  // longest match of a group resolved in rows
constexpr uint32_t kRecRingOff = 16 * kMatchGroup + kMatchGroup * kRowMax / 8;
static_assert(kRecRingOff >= 20 * kMatchGroup + 16, "room for the rounds' arrays too");
// The match pass keeps only its match-record area in shared memory.
constexpr uint32_t kMatchSmem = kRecRingOff + 16 * kMatchGroup * kRecDepth;

__host__ __device__ inline uint32_t tok_smem_bytes(uint32_t escn) {
  return (sizeof(Lut) + 2 * kRing + 2 * escn + 15) & ~15u;
}

// A plain seek's literal pass runs a handful of warps, each on its own
// critical path: a deeper ring keeps its renormalisation bytes ahead of it.
constexpr uint32_t kSeekRing = 2048;

__host__ __device__ inline uint32_t lit_smem_bytes(uint32_t window, uint32_t ring) {
  return (sizeof(Lut) + ring + 4 * window + 2 * (2 * window + 1) + 15) & ~15u;
}

__device__ inline TokMem carve_tok(uint8_t* base) {
  TokMem m;
  m.lut = reinterpret_cast<Lut*>(base);
  m.ring = base + sizeof(Lut);
  m.esc = reinterpret_cast<uint16_t*>(m.ring + 2 * kRing);
  return m;
}

__device__ inline LitMem carve_lit(uint8_t* base, uint32_t window, uint32_t ring) {
  LitMem m;
  m.lut = reinterpret_cast<Lut*>(base);
  m.ring = base + sizeof(Lut);
  m.start = reinterpret_cast<uint32_t*>(m.ring + ring);
  m.shift = reinterpret_cast<uint16_t*>(m.start + window);
  return m;
}

// Slot of block k in a seek's scratch.  The entry is read back from scratch
// that earlier calls may have left in another state, so it is clamped to the
// call's slots: whatever it holds, the address stays inside the scratch (a
// block outside the call's closure is rejected before its bytes are used).
__device__ __forceinline__ uint32_t slot_index(const DecodeArgs& a, uint64_t k) {
  const uint32_t s = __ldg(a.slot_of + k);
  return s < a.n_slots ? s : 0u;
}
__device__ __forceinline__ uint64_t slot_base(const DecodeArgs& a, uint64_t k) {
  return (uint64_t)slot_index(a, k) << a.log2B;
}

template <bool SEEK>
struct Addr {
  // device address of absolute output position p
  __device__ __forceinline__ static const uint8_t* at(const DecodeArgs& a, uint64_t p) {
    if (SEEK) return a.out + slot_base(a, p >> a.log2B) + (p & ((1ull << a.log2B) - 1));
    return a.out + p;
  }
  // the same, with block b's own bytes at obase without a slot lookup
  __device__ __forceinline__ static const uint8_t* at(const DecodeArgs& a, uint64_t p, uint64_t b, const uint8_t* obase) {
    if (SEEK) {
      uint64_t k = p >> a.log2B;
      const uint64_t off = p & ((1ull << a.log2B) - 1);
      if (k == b) return obase + off;
      return a.out + slot_base(a, k) + off;
    }
    return a.out + p;
  }
};

__device__ __forceinline__ void fail(const DecodeArgs& a, bool& ok, ace_status code, uint32_t b, uint32_t where,
                                     uint32_t lane) {
  if (ok && lane == 0) record_error(&a.sh->status, &a.sh->err_block, &a.sh->err_where, code, b, where);
  ok = false;
}

// Source byte i of a match (sequential LZ77 semantics): with distance
// d = D - S, byte i of the destination equals byte S + (i mod d) when the
// source overlaps the destination (d < len), and S + i otherwise; either way
// every byte read precedes D and is final when the copy starts.
__device__ __forceinline__ uint64_t src_index(uint64_t S, uint64_t d, uint32_t len, uint32_t i) {
  return d >= len ? S + i : S + (i % (uint32_t)d);
}

// A record's source: five bytes.  Stream jobs keep the literals before the match
// in the three above them, where a later call's match pass still finds them.
__device__ __forceinline__ uint64_t record_source(uint4 r) {
  return (uint64_t)r.x | (uint64_t)(r.y & 0xffu) << 32;
}

// The records of block b: whole decodes by the index's prefix count of
// matches; seeks max_ntok per slot; seek batches max_ntok per work item
// (rec_index: block -> its place in the batch's work list).
template <bool SEEK>
__device__ __forceinline__ MatchRec* recs_of(const DecodeArgs& a, uint32_t b) {
  if (!SEEK) return a.recs + __ldg(a.match_ptr + b);
  if (a.rec_index) {
    uint32_t w = __ldg(a.rec_index + b);
    if (w >= a.n_rec_slots) w = 0;  // the closure wrote it this batch; clamped all the same
    return a.recs + (uint64_t)w * a.max_ntok;
  }
  return a.recs + (uint64_t)slot_index(a, b) * a.max_ntok;
}

// Bytes r .. r + 15 of B:A (r < 16, the same on every lane).
__device__ __forceinline__ uint4 funnel128(uint4 A, uint4 B, uint32_t r) {
  const uint32_t t = 8 * (r & 3);
  uint32_t y0, y1, y2, y3, y4;
  switch (r >> 2) {
    case 0: y0 = A.x; y1 = A.y; y2 = A.z; y3 = A.w; y4 = B.x; break;
    case 1: y0 = A.y; y1 = A.z; y2 = A.w; y3 = B.x; y4 = B.y; break;
    case 2: y0 = A.z; y1 = A.w; y2 = B.x; y3 = B.y; y4 = B.z; break;
    default: y0 = A.w; y1 = B.x; y2 = B.y; y3 = B.z; y4 = B.w; break;
  }
  return make_uint4(__funnelshift_r(y0, y1, t), __funnelshift_r(y1, y2, t), __funnelshift_r(y2, y3, t),
                    __funnelshift_r(y3, y4, t));
}

// n bytes from src to dst by one warp, any alignment: 16-byte stores to dst,
// each from the one or two aligned 16-byte vectors of the source that hold its
// bytes (a vector is read only if it holds one), four in flight per lane; the
// ends of dst bytewise.  The source's vectors must be whole (slots of a block
// cache or a seek's scratch are).  Copied bytewise where the two differ modulo
// 16, as nearly every request's range does, the block cache's copies of 15 MB
// took 0.162 ms, by a CTA per request; with these and more CTAs for long
// requests 0.026 ms (0.6 TB/s written).
__device__ __forceinline__ void warp_copy(uint8_t* dst, const uint8_t* src, uint64_t n, uint32_t lane) {
  const uint32_t head = (uint32_t)min((uint64_t)(-reinterpret_cast<uintptr_t>(dst) & 15), n);
  if (lane < head) dst[lane] = __ldcg(src + lane);
  dst += head;
  src += head;
  n -= head;
  const uint64_t nv = n >> 4;
  const uint32_t r = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15);
  const uint4* s4 = reinterpret_cast<const uint4*>(src - r);
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  for (uint64_t v0 = 0; v0 < nv; v0 += 128) {
    uint4 t[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; u++) {
      const uint64_t v = v0 + 32 * u + lane;
      if (v < nv) {
        t[u] = __ldcg(s4 + v);
        if (r) t[u] = funnel128(t[u], __ldcg(s4 + v + 1), r);
      }
    }
#pragma unroll
    for (uint32_t u = 0; u < 4; u++) {
      const uint64_t v = v0 + 32 * u + lane;
      if (v < nv) d4[v] = t[u];
    }
  }
  const uint32_t tail = (uint32_t)(n & 15);
  if (lane < tail) dst[16 * nv + lane] = __ldcg(src + 16 * nv + lane);
}

// A block's directory entry, a word per lane, and what follows from it.
struct BlockHead {
  uint32_t dv, blen, ntok, nesc, nlit;
  __device__ BlockHead(const DecodeArgs& a, uint32_t b, uint32_t lane) {
    const uint32_t* dw = reinterpret_cast<const uint32_t*>(a.dir + b);
    dv = lane < 16 ? __ldg(dw + lane) : 0u;
    blen = (uint32_t)min((uint64_t)1 << a.log2B, a.total - ((uint64_t)b << a.log2B));
    ntok = __shfl_sync(kFull, dv, 12);
    nesc = __shfl_sync(kFull, dv, 13);
    nlit = __shfl_sync(kFull, dv, 9 + ACE_S_LIT);
  }
  // opens stream k: entry states, first renormalisation bytes
  template <uint32_t RING>
  __device__ bool open(const DecodeArgs& a, uint32_t k, uint8_t* ring, Stream& st, uint32_t lane) const {
    const uint64_t soff =
        (uint64_t)__shfl_sync(kFull, dv, 2 * k) | ((uint64_t)__shfl_sync(kFull, dv, 2 * k + 1) << 32);
    const uint32_t sbytes = __shfl_sync(kFull, dv, 6 + k), nsym = __shfl_sync(kFull, dv, 9 + k);
    const uint32_t mode = (__shfl_sync(kFull, dv, 14) >> (8 * k)) & 0xffu;  // mode[k] in byte k
    return stream_open<RING>(a.arc + a.payload_off + soff, sbytes, nsym, ring, st, lane, mode);
  }
};

// A block's opened length stream: the escape values, then two codes per token,
// into the destination and length of every match's record.  Match t ends
// token t (t < ntok - 1); its destination is the token's start plus its run.
// SPLIT: the offset stream is decoded by another warp, which fills the
// source's w bytes, and the rest of the source's eight are set here: above the
// fifth, the literals before the match.  Returns false if
// the stream is corrupt (recorded).
template <bool SEEK, uint32_t RING, bool SPLIT>
__device__ bool length_stream(const DecodeArgs& a, const BlockHead& h, Stream& sn, Lut& lut, uint8_t* ring,
                              uint16_t* esc, uint32_t b, uint32_t lane) {
  bool ok = true;
  const uint32_t lt = lanemask_lt(), ntok = h.ntok, nesc = h.nesc;
  if (!lut_build(sn, lut, lane, SPLIT ? kSplitSearch : kSearchMaxSymbols)) fail(a, ok, ACE_E_CORRUPT, b, 30, lane);
  uint8_t* escb = reinterpret_cast<uint8_t*>(esc);
  if (ok)
    rans_run<RING>(sn, ring, lut, 2 * nesc, lane, lt, [&](bool act, uint32_t i, uint32_t s) {
      if (act) escb[i] = (uint8_t)s;
    });
  __syncwarp();
  uint32_t out_pos = 0, lit_pos = 0, esc_rank = 0;
  bool bad = false;
  const uint32_t cbase = 2 * nesc, cend = cbase + 2 * ntok;
  uint4* const rec4 = reinterpret_cast<uint4*>(recs_of<SEEK>(a, b));
  if (ok) rans_run<RING>(sn, ring, lut, cend, lane, lt, [&](bool act, uint32_t i, uint32_t s) {
    bool e = act && s == 255;
    uint32_t eb = __ballot_sync(kFull, e);
    uint32_t r = esc_rank + __popc(eb & lt);
    uint32_t v = s;
    if (e) {
      if (r < nesc) v = 255u + esc[r];
      else bad = true;
    }
    esc_rank += __popc(eb);
    uint32_t lr = __shfl_sync(kFull, v, lane & ~1u), ml = __shfl_sync(kFull, v, lane | 1u);
    bool own = act && !(lane & 1);  // codes start at an even index: pairs never straddle rounds
    uint32_t to = own ? lr + ml : 0u, tl = own ? lr : 0u;
    uint32_t io = warp_incl_sum(to, lane), il = warp_incl_sum(tl, lane);
    if (own) {
      uint32_t t = (i - cbase) >> 1;
      const uint32_t D = out_pos + io - to + lr;
      if (t + 1 >= ntok) {
        if (ml) bad = true;  // the block's last token carries no match
      } else if (SPLIT) {
        uint8_t* const r8 = reinterpret_cast<uint8_t*>(rec4 + t);
        const uint32_t lits = lit_pos + il;
        if (a.w == 4) {
          *reinterpret_cast<uint32_t*>(r8 + 4) = lits << 8;
        } else {
          r8[5] = (uint8_t)lits;
          *reinterpret_cast<uint16_t*>(r8 + 6) = (uint16_t)(lits >> 8);
        }
        *reinterpret_cast<uint2*>(r8 + 8) = make_uint2(D, ml);
      } else {
        rec4[t] = make_uint4(0u, 0u, D, ml);
      }
    }
    out_pos += __shfl_sync(kFull, io, 31);
    lit_pos += __shfl_sync(kFull, il, 31);
    if (out_pos > h.blen) bad = true;
  });
  bad |= out_pos != h.blen || lit_pos != h.nlit || esc_rank != nesc;
  if (__any_sync(kFull, bad)) fail(a, ok, ACE_E_CORRUPT, b, 32, lane);
  if (ok && !stream_finished(sn)) fail(a, ok, ACE_E_CORRUPT, b, 40, lane);
  return ok;
}

// A block's opened offset stream: off_width bytes for every token but the
// last, the match's absolute source (little endian), written straight into
// its record.  A source at or after its destination is caught where sources
// are read: match_block and match_cta check every record.
template <bool SEEK, uint32_t RING>
__device__ bool offset_stream(const DecodeArgs& a, const BlockHead& h, Stream& so, Lut& lut, uint8_t* ring, uint32_t b,
                              uint32_t lane, uint32_t search) {
  bool ok = true;
  const uint32_t lt = lanemask_lt(), w = a.w, nm = h.ntok - 1;
  if (nm) {
    if (!lut_build(so, lut, lane, search)) fail(a, ok, ACE_E_CORRUPT, b, 33, lane);
    const uint32_t oend = w * nm;
    // offset byte i is byte i mod w of match i / w's source
    uint8_t* const rb = reinterpret_cast<uint8_t*>(recs_of<SEEK>(a, b));
    auto at = [&](uint32_t i) -> uint8_t* {
      const uint32_t t = w == 4 ? i >> 2 : __umulhi(i, 0xCCCCCCCDu) >> 2;  // floor(i / 5) for every 32-bit i
      return rb + 16 * (size_t)t + (i - w * t);
    };
    auto put = [&](bool act, uint32_t i, uint32_t s) {
      if (act) *at(i) = (uint8_t)s;
    };
    if (ok && !so.stored && so.k == 0 && oend >= 64) {  // slot-table streams: full rounds in the fast loop
      uint32_t i = lane;
      table_full_rounds<RING>(so, ring, lut, oend >> 5, lane, lt, [](uint32_t) {}, [&](uint32_t s, uint32_t) {
        *at(i) = (uint8_t)s;
        i += 32;
      });
    }
    if (ok) rans_run<RING>(so, ring, lut, oend, lane, lt, put);
  }
  if (ok && !stream_finished(so)) fail(a, ok, ACE_E_CORRUPT, b, 40, lane);
  return ok;
}

// Token pass of one block (Section 3: the block boundary is the entry point
// of the entropy layer): the length stream parsed into token positions, the
// offset stream, and one record per match -- absolute source, destination in
// the block, length -- for the match pass; the literal pass rebuilds the
// token positions from these records.  Returns false if the block is corrupt
// (the error is recorded).
template <bool SEEK>
__device__ bool token_block(const DecodeArgs& a, const TokMem& m, uint32_t b, uint32_t lane) {
  bool ok = true;
  const BlockHead h(a, b, lane);
  Stream sn, so;
  if (!h.open<kRing>(a, ACE_S_LEN, m.ring, sn, lane)) fail(a, ok, ACE_E_CORRUPT, b, 21, lane);
  if (!h.open<kRing>(a, ACE_S_OFF, m.ring + kRing, so, lane)) fail(a, ok, ACE_E_CORRUPT, b, 22, lane);
  if (!ok || h.ntok > a.max_ntok) {
    fail(a, ok, ACE_E_CORRUPT, b, 23, lane);
    cp_async_wait<0>();
    __syncwarp();
    return false;
  }
  cp_async_wait<2>();
  __syncwarp();
  ok = length_stream<SEEK, kRing, false>(a, h, sn, *m.lut, m.ring, m.esc, b, lane);
  __syncwarp();  // the records' zero source bytes are written before any lane fills them
  if (ok) ok = offset_stream<SEEK, kRing>(a, h, so, *m.lut, m.ring + kRing, b, lane, kSearchMaxSymbols);
  cp_async_wait<0>();  // no ring fill may land after the next block reuses the rings
  __syncwarp();
  return ok;
}

// One stream of a block by a warp of its own, for calls of few blocks
// (entropy_kernel): lengths and offsets into the match records as the token
// pass does, literals in order to the end of the block's place in the output,
// from where match_cta places them (a literal's final position is never after
// this one, so placing in ascending windows never overwrites one still to be
// read).
template <bool SEEK, uint32_t RING>
__device__ void stream_job(const DecodeArgs& a, uint8_t* smem, uint32_t b, uint32_t k, uint32_t lane) {
  bool ok = true;
  Lut& lut = *reinterpret_cast<Lut*>(smem);
  uint8_t* ring = smem + sizeof(Lut);
  uint16_t* esc = reinterpret_cast<uint16_t*>(ring + RING);
  const BlockHead h(a, b, lane);
  Stream st;
  if (!h.open<RING>(a, k, ring, st, lane)) fail(a, ok, ACE_E_CORRUPT, b, 20 + k, lane);
  if (h.ntok > a.max_ntok) fail(a, ok, ACE_E_CORRUPT, b, 23, lane);
  cp_async_wait<RING / kSeg - 2>();
  __syncwarp();
  if (ok && k == ACE_S_LEN) length_stream<SEEK, RING, true>(a, h, st, lut, ring, esc, b, lane);
  if (ok && k == ACE_S_OFF) offset_stream<SEEK, RING>(a, h, st, lut, ring, b, lane, kSplitSearch);
  if (ok && k == ACE_S_LIT && st.nsym) {
    if (!lut_build(st, lut, lane, kSplitSearch)) fail(a, ok, ACE_E_CORRUPT, b, 35, lane);
    const uint32_t lt = lanemask_lt();
    uint8_t* const to =
        (SEEK ? a.out + slot_base(a, b) : a.out + ((uint64_t)b << a.log2B)) + (h.blen - h.nlit);  // nlit <= blen: the index
    if (ok && !st.stored && st.k == 0 && st.nsym >= 64) {
      uint8_t* op = to + lane;
      table_full_rounds<RING, 4>(st, ring, lut, st.nsym >> 5, lane, lt, [](uint32_t) {}, [&](uint32_t s, uint32_t) {
        *op = (uint8_t)s;
        op += 32;
      });
    }
    if (ok)
      rans_run<RING>(st, ring, lut, st.nsym, lane, lt, [&](bool act, uint32_t i, uint32_t s) {
        if (act) to[i] = (uint8_t)s;
      });
    if (ok && !stream_finished(st)) fail(a, ok, ACE_E_CORRUPT, b, 41, lane);
  }
  cp_async_wait<0>();
  __syncwarp();
}

__host__ __device__ inline uint32_t job_smem_bytes(uint32_t escn, uint32_t ring) {
  return (sizeof(Lut) + ring + 2 * escn + 15) & ~15u;
}

// Literal pass of one block, after the token pass of every block succeeded:
// literal i lands at i plus the shift of its run.  Token t's run starts where
// the previous match ended and ends at its own match's destination (the last
// token's at the block end), so the match records give every run; 32 tokens at
// a time, a lane each, they mark the runs' first literals in a bit map of the
// step and list the shifts.  A round of 32 literals then finds its runs from
// one word of the map (a lane's run is the number of bits up to its own), with
// no walk from token to token: with a lane following the tokens one by one,
// 128 MiB of text (nine runs a round) took 0.244 ms, 1 MiB of mixed data 0.105
// and 256 MiB of FASTQ (a run per five rounds) 0.433; this takes 0.144, 0.061
// and 0.395.  Bound by issue: the rANS chain and the ring alone are 43 warp
// instructions a round.
// Returns false if the literal stream is corrupt.
template <bool SEEK, uint32_t RING>
__device__ bool literal_block(const DecodeArgs& a, const LitMem& m, uint32_t b, uint32_t lane) {
  bool ok = true;
  const BlockHead h(a, b, lane);
  const uint32_t blen = h.blen, ntok = h.ntok, nm = ntok ? ntok - 1 : 0;
  uint8_t* obase = SEEK ? a.out + slot_base(a, b) : a.out + ((uint64_t)b << a.log2B);
  const uint32_t lt = lanemask_lt();
  Stream sl;
  if (!h.open<RING>(a, ACE_S_LIT, m.ring, sl, lane)) fail(a, ok, ACE_E_CORRUPT, b, 20, lane);
  cp_async_wait<RING / kSeg - 2>();
  __syncwarp();
  if (ok && sl.nsym) {
    if (!lut_build(sl, *m.lut, lane)) fail(a, ok, ACE_E_CORRUPT, b, 35, lane);
    const uint4* rec = reinterpret_cast<const uint4*>(recs_of<SEEK>(a, b));
    // the loaded group of 32 tokens: this lane's run (first literal, shift),
    // and where the runs after the group start
    uint32_t tok = 0, gat = 0, gshift = 0, glit = 0, gdst = 0;
    bool grun = false;
    uint2 nxt = make_uint2(blen, 0u);  // the next group's destination and length
    auto fetch = [&](uint32_t t0) {
      nxt = make_uint2(blen, 0u);  // the last token's run ends at the block end
      if (t0 + lane < nm) nxt = __ldcg(reinterpret_cast<const uint2*>(rec + t0 + lane) + 1);
    };
    auto group = [&]() {
      const uint32_t D = nxt.x, end = D + nxt.y;  // end: where the next token's run starts
      fetch(tok + 32);
      const uint32_t prev = __shfl_up_sync(kFull, end, 1);
      const uint32_t st0 = lane ? prev : gdst;
      const uint32_t lr = tok + lane < ntok ? D - st0 : 0u;
      const uint32_t incl = warp_incl_sum(lr, lane);
      gat = glit + incl - lr;
      gshift = st0 - gat;
      grun = lr != 0;
      gdst = __shfl_sync(kFull, end, min(31u, ntok - 1 - tok));
      glit += __shfl_sync(kFull, incl, 31);
    };
    fetch(0);
    group();
    // Steps [c0, c1), c1 a multiple of 32 but at the end.  Runs are listed up
    // to hi; those at or after c1 (their bits left, their shifts a lane each)
    // pass on to the next step.
    uint32_t carry = 0, hi = 0, left = 0, lshift = 0, c1;  // carry: shift of the run a step starts in
    for (uint32_t c0 = 0; ok && c0 < sl.nsym; c0 = c1) {
      const uint32_t cmax = min(c0 + 32 * a.window, sl.nsym);
      for (uint32_t k = 4 * lane; k < a.window; k += 128)
        *reinterpret_cast<uint4*>(m.start + k) = make_uint4(k ? 0u : left, 0u, 0u, 0u);
      uint32_t n = __popc(left);
      if (lane == 0) m.shift[0] = (uint16_t)carry;
      if (lane < n) m.shift[1 + lane] = (uint16_t)lshift;
      uint32_t sh = carry;
      __syncwarp();
      while (true) {
        const bool in = grun && gat >= hi && gat < cmax;
        const uint32_t have = __ballot_sync(kFull, in);
        if (in) {
          m.shift[1 + n + __popc(have & lt)] = (uint16_t)gshift;
          atomicOr(m.start + ((gat - c0) >> 5), 1u << (gat & 31));
        }
        n += __popc(have);
        if (glit >= cmax || tok + 32 >= ntok || n > 2 * a.window - 32) break;
        tok += 32;
        group();
      }
      hi = min(glit, cmax);
      c1 = hi == sl.nsym ? hi : hi & ~31u;
      if ((hi < cmax && tok + 32 >= ntok) || c1 <= c0) {  // the token pass checked these counts: only a changed
        fail(a, ok, ACE_E_CORRUPT, b, 36, lane);          // archive gets here
        break;
      }
      __syncwarp();
      left = c1 < hi ? m.start[(c1 - c0) >> 5] : 0u;
      lshift = m.shift[min(n - __popc(left) + 1 + lane, 2 * a.window)];
      carry = m.shift[n - __popc(left)];
      // rounds of 32 from a multiple of 32 on; rank: runs started before the
      // round.  A round without a start keeps every lane's shift, unless the
      // round before had one.
      const uint32_t le = lt | 1u << lane;
      uint32_t rank = 0, before = 0;
      const uint32_t* word = m.start;
      uint8_t* op = obase + c0 + lane + sh;  // where this lane's literal of the round goes
      auto place = [&](uint32_t s, uint32_t bits, uint32_t i, bool act) {
        if (bits | before) {
          sh = m.shift[rank + __popc(bits & le)];
          rank += __popc(bits);
          before = bits;
          op = obase + (i + sh);
        }
        if (act) *op = (uint8_t)s;
        op += 32;
      };
      const uint32_t nfull = (c1 - c0) >> 5;
      if (!sl.stored && sl.k == 0 && nfull >= 2) {  // slot-table streams: full rounds in the fast loop
        uint32_t i = c0 + lane;
        uint4 bits;
        table_full_rounds<RING, 4>(
            sl, m.ring, *m.lut, nfull, lane, lt,
            [&](uint32_t group) {
              if (group == 4) bits = *reinterpret_cast<const uint4*>(word);  // groups start 16-byte aligned
              else bits.x = *word;
              word += group;
            },
            [&](uint32_t s, uint32_t u) {
              place(s, u == 0 ? bits.x : u == 1 ? bits.y : u == 2 ? bits.z : bits.w, i, true);
              i += 32;
            });
      }
      auto sink = [&](bool act, uint32_t i, uint32_t s) { place(s, *word++, i, act); };
      rans_run<RING>(sl, m.ring, *m.lut, c1, lane, lt, sink);
      __syncwarp();
    }
  }
  if (ok) {
    bool fin = stream_finished(sl);
    if (!__all_sync(kFull, fin)) fail(a, ok, ACE_E_CORRUPT, b, 41, lane);
  }
  cp_async_wait<0>();
  __syncwarp();
  return ok;
}

// Rows of 32 bytes in flight in the copy of a group by rows.
constexpr uint32_t kRowUnroll = 8;
// Bytes in flight per lane in the bytewise copy of a round's matches.
constexpr uint32_t kCopyUnroll = 8;
// Copy classes of a group resolved in rounds: a non-overlapping match of at
// least the call's long_min bytes is copied by the whole warp in aligned
// 16-byte pieces, one of at most kShortMax bytes (WAY_LANES) by one lane in
// aligned 8-byte words, every other one bytewise with the round's other such
// matches.  long_min is the copy-width knob: kLongMinWide (16-byte pieces for
// everything above 32 bytes) or kLongMinNarrow (bytewise up to 511 bytes).
constexpr uint32_t kShortMax = 32;
constexpr uint32_t kLongMinNarrow = 512;
constexpr uint32_t kLongMinWide = kShortMax + 1;

// The ways a warp takes through a group of matches (match_block).
enum { WAY_ROUNDS = 0, WAY_LANES = 1, WAY_ROWS = 2 };

// A load of match source bytes.  L1: through the SM's L1 cache, for a pass
// whose sources were all written by earlier launches or by this warp (one
// launch per dependency level); else at L2 only, which every SM sees
// coherently (source blocks published by other warps of the same launch).
template <bool L1, class T>
__device__ __forceinline__ T ld_src(const T* p) {
  return L1 ? __ldca(p) : __ldcg(p);
}

// Source of a short match: the aligned 8-byte words covering [S, S + len).
template <bool SEEK, bool L1>
__device__ __forceinline__ void short_load(const DecodeArgs& a, uint64_t S, uint32_t len, uint64_t (&w)[5], uint64_t b,
                                           const uint8_t* obase) {
  const uint64_t a0 = S & ~7ull;
  const uint32_t off = (uint32_t)(S & 7);
#pragma unroll
  for (uint32_t k = 0; k < 5; k++) {
    const uint64_t q = a0 + 8ull * k;
    w[k] = 0;
    if (8 * k < off + len) {
      if (q + 8 <= a.total) {
        w[k] = ld_src<L1>(reinterpret_cast<const unsigned long long*>(Addr<SEEK>::at(a, q, b, obase)));
      } else {
        for (uint32_t t = 0; t < 8 && q + t < a.total; t++)
          w[k] |= (uint64_t)ld_src<L1>(Addr<SEEK>::at(a, q + t, b, obase)) << (8 * t);
      }
    }
  }
}

// Bytes sh .. sh + 7 of hi:lo (sh < 8).
__device__ __forceinline__ uint64_t funnel64(uint64_t lo, uint64_t hi, uint32_t sh) {
  return sh ? (lo >> (8 * sh)) | (hi << (64 - 8 * sh)) : lo;
}

// Bytes [lo, hi) of w to the 8-byte aligned p, in the widest aligned stores
// that fit.  The lanes of a round store to different lines, so every store
// a lane saves is an L1 and L2 transaction saved.
__device__ __forceinline__ void store_bytes8(uint8_t* p, uint64_t w, uint32_t lo, uint32_t hi) {
  uint32_t k = lo;
  while (k < hi) {
    if (!(k & 3) && k + 4 <= hi) {
      *reinterpret_cast<uint32_t*>(p + k) = (uint32_t)(w >> (8 * k));
      k += 4;
    } else if (!(k & 1) && k + 2 <= hi) {
      *reinterpret_cast<uint16_t*>(p + k) = (uint16_t)(w >> (8 * k));
      k += 2;
    } else {
      p[k] = (uint8_t)(w >> (8 * k));
      k++;
    }
  }
}

// Destination of a short match: aligned 8-byte words where the match covers
// them, the widest aligned stores that fit at its two ends.  Source byte off + i (off = S mod 8,
// counted from the first source word) lands at dp[i].
__device__ __forceinline__ void short_store(uint8_t* dp, uint32_t off, uint32_t len, const uint64_t (&w)[5]) {
  const uint32_t hd = (uint32_t)(reinterpret_cast<uintptr_t>(dp) & 7);
  uint8_t* dal = dp - hd;
  const bool same = off >= hd;  // destination word i starts in source word i, else in word i - 1
  const uint32_t sh = (off - hd) & 7;
#pragma unroll
  for (uint32_t i = 0; i < 5; i++) {
    const int first = 8 * (int)i - (int)hd;  // match byte held by the word's first byte
    if (first >= (int)len) break;
    const uint64_t lo = same ? w[i] : (i ? w[i - 1] : 0ull);
    const uint64_t hi = same ? (i + 1 < 5 ? w[i + 1] : 0ull) : w[i];
    const uint64_t word = funnel64(lo, hi, sh);
    if (first >= 0 && first + 8 <= (int)len) {
      *reinterpret_cast<uint64_t*>(dal + 8 * i) = word;
    } else {
      store_bytes8(dal + 8 * i, word, (uint32_t)max(0, -first), (uint32_t)min(8, (int)len - first));
    }
  }
}

// First index i in [0, n) with key(i) > x, for keys that never decrease.
template <class Key>
__device__ __forceinline__ uint32_t upper_bound(uint32_t n, uint32_t x, Key key) {
  uint32_t lo = 0, len = n;
  while (len) {
    const uint32_t h = len >> 1;
    if (key(lo + h) <= x) {
      lo += h + 1;
      len -= h + 1;
    } else {
      len = h;
    }
  }
  return lo;
}

// Match pass of one block (Section 2: a block decodes once the blocks holding
// its sources are present).  Groups of 32 matches, a lane each: their records
// are loaded together; with WAIT the source blocks before this one are checked
// with overlapping relaxed loads (a bounded wait only for one not yet
// published); without it (one launch per dependency level) each source
// block's level must be below this launch's level, else the archive's
// dependency lists disagree with its matches.  Returns false if a record is
// corrupt or a wait gave up.
//
// WAY_ROWS: a group whose matches are all short (at most kRowMax bytes) and do
// not overlap their sources -- text, FASTQ and mixed data are almost only such --
// is copied in rows: its match bytes laid end to end, 32 consecutive ones per
// row, a lane's match found by counting start bits in a bit map of the group,
// so that loads and stores of a row touch the few lines its two or three
// matches lie in.  Rows go in output order, so a source byte is final unless
// it lies at or after the first byte of the rows in flight; such bytes wait
// until those before them are stored.  Any other group, and every one of the
// other ways, is copied in rounds of matches none of which reads bytes another
// pending one of the group writes (literal bytes are final after the literal
// pass; the first pending match is always ready, so every round makes progress).
//
// Short matches by lanes (WAY_LANES) touch 32 lines with every load and store:
// FASTQ 256 MiB, a launch per level, 0.145 ms, by rows 0.106.  But a group is then
// two trips to memory where its rows are four, and where waits have already cost
// one and few warps are resident that decides: 115 MB of FASTQ objects in 64 KiB
// blocks 411 us by lanes, 447 by rows; in 1 KiB blocks 908 and 909.  Bound by the
// latency of a group after another.
template <bool SEEK, bool WAIT, bool L1, int WAY>
__device__ bool match_block(const DecodeArgs& a, MatchRec* gm, uint32_t b, uint32_t lane, uint32_t epoch,
                            uint32_t nm, uint32_t lvl = 0) {
  // L1: every source was written before the launch or by this warp (one
  // launch per level), so source loads may go through L1; otherwise other
  // SMs wrote them during the launch and loads go to L2.  Without WAIT, lvl
  // is the block's level: its sources must lie in lower ones.
  constexpr bool kL1 = L1;
  static_assert(kMatchGroup == 32, "one match per lane");
  bool ok = true, bad = false;
  const uint64_t B = (uint64_t)1 << a.log2B, bstart = (uint64_t)b << a.log2B;
  const uint32_t blen = (uint32_t)min(B, a.total - bstart);
  const uint32_t lt = lanemask_lt(), le = lt | 1u << lane;
  uint8_t* obase = SEEK ? a.out + slot_base(a, b) : a.out + bstart;
  const uint4* rec = reinterpret_cast<const uint4*>(recs_of<SEEK>(a, b));
  // records reach a ring of kRecDepth groups by cp.async, kRecDepth - 1
  // groups ahead of the one resolving; lane j copies and later reads record
  // j of each group, so no lane reads another's copy
  uint4* const rring = reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(gm) + kRecRingOff);
  auto issue = [&](uint32_t g) {  // one commit group per call, empty past the last record
    const uint32_t t = g * kMatchGroup + lane;
    if (t < nm) cp_async16(rring + (g % kRecDepth) * kMatchGroup + lane, rec + t);
    cp_async_commit();
  };
#pragma unroll
  for (uint32_t g = 0; g + 1 < kRecDepth; g++) issue(g);
  for (uint32_t t0 = 0, g = 0; ok && t0 < nm; t0 += kMatchGroup, g++) {
    issue(g + kRecDepth - 1);
    cp_async_wait<kRecDepth - 1>();  // group g has landed
    uint4 r = make_uint4(0, 0, 0, 0);
    if (t0 + lane < nm) r = rring[(g % kRecDepth) * kMatchGroup + lane];
    const uint64_t S = record_source(r);
    const uint32_t D = r.z;
    uint32_t L = r.w;
    if (L && (S >= bstart + D || (uint64_t)D + L > blen)) {  // checked again: the token pass may have failed
      bad = true;
      L = 0;
    }
    if (__any_sync(kFull, bad)) fail(a, ok, ACE_E_CORRUPT, b, 37, lane);
    if (!ok) break;

    // source blocks before this one: all flags loaded, then compared
    const uint64_t dist = bstart + D - S, rend = S + min((uint64_t)L, dist), k0 = S >> a.log2B;
    const uint64_t k1 = min((rend - 1) >> a.log2B, (uint64_t)b - 1);  // blocks k0 .. k1 hold the bytes before this block
    const bool ext = L && k0 < b;
    uint32_t f0 = epoch, f1 = epoch;
    if (ext) {
      if (WAIT) {  // flags that other warps publish during the launch
        f0 = ld_relaxed(a.ready + k0);
        f1 = k1 != k0 ? ld_relaxed(a.ready + k1) : f0;
      } else {  // levels, fixed for the launch: through the read-only cache
        f0 = __ldg(a.level + k0);
        f1 = k1 != k0 ? __ldg(a.level + k1) : f0;
      }
    }
    if (WAIT) {
      bool timeout = false;
      // a source block must sit at a lower dependency level (work lists are
      // in level order, so it was handed out before this block and the wait
      // ends)
      if (ext) {
        bool low = true;
        const uint32_t my_level = __ldg(a.level + b);
        for (uint64_t k = k0; k <= k1; k++) low &= __ldg(a.level + k) < my_level;
        if (SEEK && a.closure_flags) {
          // every source block must be a member of this seek's closure: its
          // flag carries the call's epoch (pending or published).  Anything
          // else means the dependency table disagrees with the matches.
          low &= (f0 & ~kPendingFlag) == epoch && (f1 & ~kPendingFlag) == epoch;
          for (uint64_t k = k0 + 1; low && k < k1; k++) low = (ld_relaxed(a.ready + k) & ~kPendingFlag) == epoch;
        }
        if (!low) bad = true;  // the dependency table disagrees with the matches
        else if (f0 != epoch || f1 != epoch || k1 > k0 + 1)  // blocks between them: the bounded wait
          for (uint64_t k = k0; k <= k1 && !timeout; k++)
            if (!wait_flag(a.ready + k, epoch, a.timeout_ns, &a.sh->status)) timeout = true;
      }
      if (__any_sync(kFull, bad)) fail(a, ok, ACE_E_CORRUPT, b, 39, lane);
      if (__any_sync(kFull, timeout)) fail(a, ok, ACE_E_TIMEOUT, b, 38, lane);
      if (!ok) break;
      if (__any_sync(kFull, ext)) fence_acquire();
      __syncwarp();  // any lane may copy a match whose flags another lane checked
    }
    // without WAIT the level check below need not hold up the copies: a
    // corrupt archive fails the call whatever bytes they wrote

    if (WAY == WAY_ROWS && __all_sync(kFull, L <= kRowMax && (!L || (dist >= L && (!SEEK || k0 == (S + L - 1) >> a.log2B))))) {
      // rows.  Per match: where byte c of the group's bytes comes from (address
      // of the source less the match's start among them) and goes to, and the
      // source's place in the block (below 0: an earlier block, always final).
      uint4* const row = reinterpret_cast<uint4*>(gm);
      uint32_t* const bits = reinterpret_cast<uint32_t*>(row + kMatchGroup);
#pragma unroll
      for (uint32_t k = 0; k < kRowMax / 32; k++) bits[32 * k + lane] = 0;
      const uint32_t incl = warp_incl_sum(L, lane), X = incl - L, T = __shfl_sync(kFull, incl, 31);
      const uint32_t have = __ballot_sync(kFull, L != 0);
      if (L) {
        const uint64_t from = reinterpret_cast<uintptr_t>(Addr<SEEK>::at(a, S, b, obase)) - X;
        const int32_t rel = (int32_t)max((int64_t)(S - bstart), -(int64_t)(1 << 30));
        row[__popc(have & lt)] = make_uint4((uint32_t)from, (uint32_t)(from >> 32), D - X, (uint32_t)(rel - (int32_t)X));
      }
      __syncwarp();
      if (L) atomicOr(bits + (X >> 5), 1u << (X & 31));
      __syncwarp();
      uint32_t rank = ~0u;  // the match before the row's first start
      for (uint32_t c0 = 0; c0 < T; c0 += 32 * kRowUnroll) {
        uint32_t v[kRowUnroll], dst[kRowUnroll], pend = 0;
        const uint32_t rank0 = rank;
        // bytes at or after F are written by the rows in flight
        const int32_t F = (int32_t)(row[rank + (bits[c0 >> 5] & 1)].z + c0);
#pragma unroll
        for (uint32_t u = 0; u < kRowUnroll; u++) {
          if (c0 + 32 * u >= T) break;
          const uint32_t c = c0 + 32 * u + lane, w = bits[(c0 >> 5) + u];
          const uint4 m = row[rank + __popc(w & le)];
          rank += __popc(w);
          dst[u] = m.z + c;
          if (c < T) {
            if ((int32_t)(m.w + c) < F)
              v[u] = ld_src<kL1>(reinterpret_cast<const uint8_t*>(((uint64_t)m.y << 32 | m.x) + c));
            else
              pend |= 1u << u;
          }
        }
#pragma unroll
        for (uint32_t u = 0; u < kRowUnroll; u++)
          if (c0 + 32 * u + lane < T && !(pend >> u & 1)) obase[dst[u]] = (uint8_t)v[u];
        __syncwarp();
        const uint32_t rows = __reduce_or_sync(kFull, pend);
        if (!rows) continue;
        uint32_t k = rank0;  // the rows that wait, one after another
        for (uint32_t u = 0; rows >> u; u++) {
          const uint32_t c = c0 + 32 * u + lane, w = bits[(c0 >> 5) + u];
          if (rows >> u & 1) {
            const uint4 m = row[k + __popc(w & le)];
            bool p = pend >> u & 1;
            while (__any_sync(kFull, p)) {
              const uint32_t first = __reduce_min_sync(kFull, p ? m.z + c : ~0u);  // not yet written
              if (p && (int32_t)(m.w + c) < (int32_t)first) {
                obase[m.z + c] = ld_src<kL1>(reinterpret_cast<const uint8_t*>(((uint64_t)m.y << 32 | m.x) + c));
                p = false;
              }
              __syncwarp();
            }
          }
          k += __popc(w);
        }
      }
    } else {
      uint64_t* gS = reinterpret_cast<uint64_t*>(gm);                 // sources
      uint32_t* gD = reinterpret_cast<uint32_t*>(gS + kMatchGroup);   // destinations in the block
      uint32_t* gL = gD + kMatchGroup;                                // lengths
      uint32_t* gX = gL + kMatchGroup;                                // [kMatchGroup + 1] starts in a round's copy
      gS[lane] = S;
      gD[lane] = D;
      gL[lane] = L;
      __syncwarp();
      uint32_t feeds = 0;  // the group's matches that write bytes this one's source reads
      if (L && rend > bstart) {
        const uint32_t s_rel = S > bstart ? (uint32_t)(S - bstart) : 0u, e_rel = (uint32_t)(rend - bstart);
        const uint32_t lo = upper_bound(lane, s_rel, [&](uint32_t i) { return gD[i] + gL[i]; });
        const uint32_t hi = upper_bound(lane, e_rel - 1, [&](uint32_t i) { return gD[i]; });  // first with gD >= e_rel
        if (hi > lo) feeds = ((1u << hi) - 1) & ~((1u << lo) - 1);  // hi <= lane <= 31
      }
      uint32_t pend = __ballot_sync(kFull, L != 0);
      while (pend) {
        const bool go = (pend >> lane & 1) && !(pend & feeds);
        const bool lgo = go && L >= a.long_min && dist >= L;
        const bool sgo = WAY == WAY_LANES && go && L <= kShortMax && dist >= L;
        if (sgo) {
          uint64_t w[5];
          short_load<SEEK, kL1>(a, S, L, w, b, obase);
          short_store(obase + D, (uint32_t)(S & 7), L, w);
        }
        // long: one match after another by the whole warp, in aligned 16-byte
        // stores, each from the two aligned vectors of the source that hold its
        // bytes (which end before the match does: it does not overlap its
        // source); the ragged ends a byte per lane
        for (uint32_t todo = __ballot_sync(kFull, lgo); todo; todo &= todo - 1) {
          const uint32_t j = __ffs(todo) - 1, Dj = __shfl_sync(kFull, D, j), Lj = __shfl_sync(kFull, L, j);
          const uint64_t Sj = (uint64_t)__shfl_sync(kFull, (uint32_t)S, j) | (uint64_t)__shfl_sync(kFull, (uint32_t)(S >> 32), j) << 32;
          const uint32_t head = (0u - Dj) & 15, tail = (Dj + Lj) & 15, n = (Lj - head) >> 4;
          const bool ragged = lane < 16 ? lane < head : lane - 16 < tail;
          const uint32_t i = lane < 16 ? lane : Lj - tail + (lane - 16);
          uint8_t end = 0;
          if (ragged) end = ld_src<kL1>(Addr<SEEK>::at(a, Sj + i, b, obase));
          const uint32_t off = (uint32_t)(Sj + head) & 15;
          const uint64_t q0 = Sj + head - off;
          uint4* const dp = reinterpret_cast<uint4*>(obase + Dj + head);
          for (uint32_t c = lane; c < n; c += 32) {
            const uint64_t q = q0 + 16ull * c;
            uint4 v = ld_src<kL1>(reinterpret_cast<const uint4*>(Addr<SEEK>::at(a, q, b, obase)));
            if (off) v = funnel128(v, ld_src<kL1>(reinterpret_cast<const uint4*>(Addr<SEEK>::at(a, q + 16, b, obase))), off);
            dp[c] = v;
          }
          if (ragged) obase[Dj + i] = end;
        }
        // the rest laid end to end in group order: gX[j] is where match j
        // starts, gX[kMatchGroup] the total
        const bool bgo = go && !lgo && !sgo;
        if (__any_sync(kFull, bgo)) {
          const uint32_t len = bgo ? L : 0u;
          const uint32_t incl = warp_incl_sum(len, lane), total = __shfl_sync(kFull, incl, 31);
          gX[lane] = incl - len;
          if (lane == 0) gX[kMatchGroup] = total;
          __syncwarp();
          // lane l copies bytes c + 32 u + l: consecutive lanes read and write
          // consecutive bytes of a match, kCopyUnroll loads in flight before
          // their stores (a round's ready matches read no byte it writes); the
          // lane's match index only moves forward
          uint32_t jc = 0;
          for (uint32_t c = 0; c < total; c += 32 * kCopyUnroll) {
            uint8_t v[kCopyUnroll];
            uint32_t dp[kCopyUnroll];
#pragma unroll
            for (uint32_t u = 0; u < kCopyUnroll; u++) {
              const uint32_t p = c + 32 * u + lane;
              dp[u] = ~0u;
              if (p < total) {
                while (gX[jc + 1] <= p) jc++;
                const uint32_t i = p - gX[jc], ml = gL[jc];
                const uint64_t Sj = gS[jc], d = bstart + gD[jc] - Sj;
                v[u] = ld_src<kL1>(Addr<SEEK>::at(a, src_index(Sj, d, ml, i), b, obase));
                dp[u] = gD[jc] + i;
              }
            }
#pragma unroll
            for (uint32_t u = 0; u < kCopyUnroll; u++)
              if (dp[u] != ~0u) obase[dp[u]] = v[u];
          }
        }
        pend &= ~__ballot_sync(kFull, go);
        __syncwarp();  // the round's copies are seen by the next round's loads
      }
    }
    if (!WAIT) {
      if (ext) {
        if (f0 >= lvl || f1 >= lvl) bad = true;
        for (uint64_t k = k0 + 1; k < k1; k++)  // a source spanning more than two earlier blocks
          if (__ldg(a.level + k) >= lvl) bad = true;
      }
      if (__any_sync(kFull, bad)) fail(a, ok, ACE_E_CORRUPT, b, 39, lane);
    }
    __syncwarp();  // the next group reuses the arrays
  }
  cp_async_wait<0>();  // no record copy may land after the caller reuses the area
  __syncwarp();
  return ok;
}

// Sixteen known bytes as entries of match_cta.
__device__ __forceinline__ void known16(uint4* e, uint4 v) {
  e[0] = make_uint4(__byte_perm(v.x, 0x80u, 0x4140), __byte_perm(v.x, 0x80u, 0x4342), __byte_perm(v.y, 0x80u, 0x4140),
                    __byte_perm(v.y, 0x80u, 0x4342));
  e[1] = make_uint4(__byte_perm(v.z, 0x80u, 0x4140), __byte_perm(v.z, 0x80u, 0x4342), __byte_perm(v.w, 0x80u, 0x4140),
                    __byte_perm(v.w, 0x80u, 0x4342));
}

// The match pass of one block by a CTA, in windows of kCtaWindow bytes (one for
// blocks of at most that).  Every byte of the window gets a 16-bit entry in
// shared memory: 0x8000 | its value where that is known (a literal, or a match
// byte whose source lies before the window, which is final), else the address
// of the entry of the byte it copies (twice its place in the window).  A match
// byte equals the byte one distance before it (Section 2, the sequential LZ77
// copy; overlapping matches too), so entries form chains that end at known ones.  The warps set the entries a
// group of 32 matches each, in rows of 32 match bytes (as match_block, but in
// any order: an entry waits for nothing), then every thread follows the chains
// of its 16 bytes and stores them.  Chains longer than kHops (matches of one
// match after another, runs) are shortened by pointer jumping first: every
// entry takes its target's, which ends all of them in log2 of the length.
//
// No match waits for another, so a block is a few thousand cycles of
// independent loads over 8 or 16 warps where the warp-per-block pass is a
// chain of its groups, and whole sectors are written.  It pays for blocks of
// many short matches (text 128 MiB: 0.25 ms, 0.38 by warps in rounds, 0.33 in
// rows; bound by issue, about 26,000 warp instructions a 16 KiB block) and
// wherever blocks are few: levels of 64 blocks 6 to 18 us (9 to 25 by 512
// threads a block with a sweep of pointer jumping per step), a FASTQ seek's
// match pass 0.040 ms (0.094 by a warp per block), 1900 blocks of a cached
// batch 0.11 (0.21), 192 uneven objects 0.49 (0.79).
// With WAIT a source block before this one may not be published yet: a bounded
// wait; without it its level must be below lvl.  Returns false, for the whole
// CTA, if a record is corrupt or a wait gave up (recorded).
//
// LITS: after stream jobs.  The literals are still in order at the end of the
// block's place (a record's source holds above its five bytes the literals
// before the match), so literal runs are laid in rows too, the last one as
// token nm, and every byte of the window gets its entry from a row.
constexpr uint32_t kCtaWindow = 16384;
constexpr uint32_t kCtaThreads = 512;                       // at most
constexpr uint32_t kCtaRowBytes = 2048;                     // match bytes whose starts the bit map holds
constexpr uint32_t kCtaWarpSmem = 16 * 32 + kCtaRowBytes / 8;
constexpr uint32_t kCtaUnroll = 4;                          // rows in flight per warp (a vector of the map's words)
constexpr uint32_t kHops = 6;
constexpr uint32_t kCtaLong = 256;                          // shortest run of known bytes set 16 at a time

// Threads of a CTA: 256, or 512 where blocks are few and each one's time
// counts; less for small blocks.
__host__ __device__ inline uint32_t cta_threads(uint32_t log2B, bool few) {
  return log2B >= 12 ? few ? 512 : 256 : log2B >= 10 ? 128 : 64;
}
// ... where they are many and dense: a thread to 64 bytes.  48 MiB of text (with
// no match below 12 bytes), match pass, us by 32, 64, 128, 256 threads: 1 KiB
// blocks 142, 167, 225 (110, 137, 205); 2 KiB 144, 157, 173 (115, 117, 146); 4 KiB
// 186, 155, 156, 178 (148, 124, 123, 156); 8 KiB 318, 193, 155, 160; 16 KiB 589,
// 329, 202, 162.  256 threads had been 178 (156) where a warp per block took 176
// (125).
__host__ __device__ inline uint32_t dense_threads(uint32_t log2B) {
  return log2B >= 14 ? 256 : log2B > 11 ? 1u << (log2B - 6) : 32;
}
// (enough for smaller blocks of the same launch too)
__host__ __device__ inline uint32_t cta_smem_bytes(uint32_t log2B, uint32_t threads) {
  return 2 * (log2B >= 14 ? kCtaWindow : 1u << log2B) + threads / 32 * kCtaWarpSmem;
}

template <bool SEEK, bool WAIT, bool LITS>
__device__ bool match_cta(const DecodeArgs& a, uint8_t* smem, uint32_t b, uint32_t nm, uint32_t epoch, uint32_t lvl) {
  __shared__ uint32_t s_group;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const uint32_t lt = lanemask_lt(), le = lt | 1u << lane;
  const uint64_t B = 1ull << a.log2B, bstart = (uint64_t)b << a.log2B;
  const uint32_t blen = (uint32_t)min(B, a.total - bstart);
  uint8_t* obase = SEEK ? a.out + slot_base(a, b) : a.out + bstart;
  const uint4* rec = reinterpret_cast<const uint4*>(recs_of<SEEK>(a, b));
  uint16_t* e = reinterpret_cast<uint16_t*>(smem);
  const uint32_t ebase = (uint32_t)__cvta_generic_to_shared(e);
  // groups of 32 matches, a warp each; with fewer groups than warps, several
  // warps each, sharing the group's bytes
  const uint32_t nt32 = nm + (LITS ? 1 : 0), ng = (nt32 + 31) / 32, split = ng ? max(1u, nw / ng) : 1u;
  uint32_t nlit = 0;
  if (LITS) {  // the block's literals: those before its last match, and what follows it
    const uint4 r = nm ? __ldcg(rec + nm - 1) : make_uint4(0, 0, 0, 0);
    nlit = (r.y >> 8) + blen - r.z - r.w;
  }
  const uint32_t part = wid % split, step = nw / split;
  uint4* row = reinterpret_cast<uint4*>(smem + 2 * min((uint32_t)B, kCtaWindow) + wid * kCtaWarpSmem);
  uint32_t* bits = reinterpret_cast<uint32_t*>(row + 32);
  uint32_t first = 0;  // the group that reaches the window
  for (uint32_t w0 = 0; w0 < blen; w0 += kCtaWindow) {
    const uint32_t wn = min(kCtaWindow, blen - w0);
    uint32_t g = first + wid / split;
    if (wid >= step * split) g = ng;  // a warp left over
    uint4 rn;  // records one group ahead
    auto fetch = [&](uint32_t q) {
      return 32 * q + lane < nm ? __ldcg(rec + 32 * q + lane) : make_uint4(0, 0, 0, 0);
    };
    rn = fetch(g);
    // every byte known as the literal pass left it; match bytes are set next
    const uint8_t* wbase = obase + w0;
    for (uint32_t j0 = 16 * tid; !LITS && j0 < wn; j0 += 16 * nt * 4) {
      uint4 v[4];
#pragma unroll
      for (uint32_t u = 0; u < 4; u++) {
        const uint32_t j = j0 + 16 * nt * u;
        v[u] = make_uint4(0, 0, 0, 0);
        if (j + 16 <= wn) {
          v[u] = __ldcg(reinterpret_cast<const uint4*>(wbase + j));
        } else if (j < wn) {
          uint32_t x[4] = {0, 0, 0, 0};
#pragma unroll
          for (uint32_t k = 0; k < 16; k++)
            if (j + k < wn) x[k >> 2] |= (uint32_t)__ldcg(wbase + j + k) << (8 * (k & 3));
          v[u] = make_uint4(x[0], x[1], x[2], x[3]);
        }
      }
#pragma unroll
      for (uint32_t u = 0; u < 4; u++) {
        const uint32_t j = j0 + 16 * nt * u;
        if (j >= wn) continue;
        known16(reinterpret_cast<uint4*>(e + j), v[u]);
      }
    }
    if (LITS && tid < 16 && wn + tid < ((wn + 15) & ~15u)) e[wn + tid] = 0x8000;  // the last vector's rest
    if (tid == 0) s_group = first;
    __syncthreads();

    bool bad = false, timeout = false;
    uint32_t last = first;
    // with waits, the literals of every group first: they wait for nothing
    constexpr uint32_t kPhases = LITS && WAIT ? 2 : 1;
#pragma unroll
    for (uint32_t phase = 0; phase < kPhases; phase++) {
      const bool place = LITS && phase == 0, copy = phase + 1 == kPhases;
      if (phase) {
        g = wid >= step * split ? ng : first + wid / split;
        rn = fetch(g);
      }
      for (; g < ng; g += step) {
        const uint4 r = rn;
        rn = fetch(g + step);
        const uint64_t S = record_source(r);
        uint32_t D = r.z, lits = 0, lr = 0;
        uint32_t L = r.w;
        if (LITS) {  // lits: literals before the match; lr: those of its token's run
          lits = r.y >> 8;
          if (32 * g + lane >= nm) {
            D = blen;
            lits = nlit;
          }
          uint32_t before = __shfl_up_sync(kFull, lits, 1);
          if (lane == 0) before = g ? __ldcg(&rec[32 * g - 1].y) >> 8 : 0u;
          lr = lits - before;  // (0 past token nm)
        }
        if (L && (S >= bstart + D || (uint64_t)D + L > blen)) {  // a source precedes its match, which stays in the block
          bad = true;
          L = 0;
        }
        if (lr > D) bad = true, lr = 0;  // the length stream's own checks hold: only a changed archive gets here
        if (__shfl_sync(kFull, D - lr, 0) >= w0 + wn) break;  // (destinations ascend) past the window
        last = g;
        const uint64_t dist = bstart + D - S;
        if (copy && L && S < bstart) {  // the blocks before this one that it reads
          const uint32_t k0 = (uint32_t)(S >> a.log2B);
          const uint32_t k1 = (uint32_t)((min(S + min((uint64_t)L, dist), bstart) - 1) >> a.log2B);
          for (uint32_t k = k0; k <= k1; k++) {
            if (!WAIT) {
              bad |= __ldg(a.level + k) >= lvl;
              continue;
            }
            // at a lower level (work lists are in level order, so the wait ends;
            // the block cache keeps no levels), and a member of a seek's closure
            // (its flag carries the call's epoch, pending or published)
            if (a.level && __ldg(a.level + k) >= __ldg(a.level + b)) bad = true;
            const uint32_t f = ld_relaxed(a.ready + k);
            if (SEEK && a.closure_flags && (f & ~kPendingFlag) != epoch) bad = true;
            if (!bad && !timeout && f != epoch && !wait_flag(a.ready + k, epoch, a.timeout_ns, &a.sh->status)) timeout = true;
          }
          if (bad || timeout) L = 0;
        }
        if (WAIT && copy && __any_sync(kFull, L && S < bstart)) {
          fence_acquire();
          __syncwarp();  // any lane may read a source whose flags another lane checked
        }
        // Long runs of bytes from before the window (big, per lane), one after
        // another by the whole warp (the group's warps in turn): 16 entries per
        // lane from the one or two aligned vectors that hold them, the ragged
        // ends a byte per lane.
        auto copy_long = [&](bool big, uint32_t n, uint32_t dst, uint64_t from) {
          uint32_t todo = __ballot_sync(kFull, big);
          for (uint32_t q = 0; todo; todo &= todo - 1, q++) {
            if (q % split != part) continue;
            const uint32_t j = __ffs(todo) - 1, nj = __shfl_sync(kFull, n, j), dj = __shfl_sync(kFull, dst, j);
            const uint8_t* const src = reinterpret_cast<const uint8_t*>(
                (uint64_t)__shfl_sync(kFull, (uint32_t)from, j) | (uint64_t)__shfl_sync(kFull, (uint32_t)(from >> 32), j) << 32);
            const uint32_t head = (0u - dj) & 15, tail = (dj + nj) & 15, nv = (nj - head) >> 4;
            const uint32_t i = lane < 16 ? lane : nj - tail + (lane - 16);
            if (lane < 16 ? lane < head : lane - 16 < tail) e[dj + i] = (uint16_t)(0x8000u | ld_src<!WAIT>(src + i));
            const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(src + head) & 15);
            const uint4* const sv = reinterpret_cast<const uint4*>(src + head - off);
            uint4* const ev = reinterpret_cast<uint4*>(e + dj + head);
            for (uint32_t c = lane; c < nv; c += 32) {
              uint4 v = ld_src<!WAIT>(sv + c);
              if (off) v = funnel128(v, ld_src<!WAIT>(sv + c + 1), off);
              known16(ev + 2 * c, v);
            }
          }
        };
        // The warp's share of n bytes per lane laid end to end, in rows.  Byte c
        // of them: its entry's address, twice its source's place in the window
        // (below 0: before it, or marked) and its source's address, each less
        // c's share.  Marked in the address's top bits: a seek's source in more
        // than one slot (the position instead), and a match overlapping its
        // source (distance and start instead: its bytes repeat the first
        // distance's, not one another down a long chain).
        auto lay = [&](uint32_t n, uint32_t dst, int32_t rel, uint64_t from, bool marked) {
          const uint32_t incl = warp_incl_sum(n, lane), X = incl - n, T = __shfl_sync(kFull, incl, 31);
          const uint32_t have = __ballot_sync(kFull, n != 0);
          if (n)
            row[__popc(have & lt)] =
                marked && (from >> 62 & 1)
                    ? make_uint4((uint32_t)from, (uint32_t)(from >> 32), ebase + 2 * (dst - X), 0xC0000000u)
                    : make_uint4((uint32_t)(from - X), (uint32_t)((from - X) >> 32) | (marked ? 0x80000000u : 0u),
                                 ebase + 2 * (dst - X), (uint32_t)(2 * (rel - (int32_t)X)));
          const bool odd = __any_sync(kFull, marked);
          constexpr uint32_t kBatch = 32 * kCtaUnroll;
          const uint32_t share = ((T + split - 1) / split + kBatch - 1) & ~(kBatch - 1);
          const uint32_t te = min(T, (part + 1) * share);
          for (uint32_t cb = part * share; cb < te; cb += kCtaRowBytes) {  // one turn but for long matches
  #pragma unroll
            for (uint32_t k = 0; k < kCtaRowBytes / 32; k += 32) bits[k + lane] = 0;
            __syncwarp();
            if (n && X - cb < kCtaRowBytes) atomicOr(bits + ((X - cb) >> 5), 1u << (X & 31));
            uint32_t rank = __popc(__ballot_sync(kFull, n && X < cb)) - 1;  // the one before the row's first start
            __syncwarp();
            const uint32_t ce = min(te, cb + kCtaRowBytes);
            auto rows = [&](auto kind) {
              constexpr bool special = decltype(kind)::value;
              const uint4* words = reinterpret_cast<const uint4*>(bits);
              for (uint32_t c = cb + lane; c < ce + lane; c += kBatch) {
                const uint4 w4 = *words++;
                const uint32_t w[kCtaUnroll] = {w4.x, w4.y, w4.z, w4.w};
                uint32_t v[kCtaUnroll], at[kCtaUnroll];
  #pragma unroll
                for (uint32_t u = 0; u < kCtaUnroll; u++) {
                  const uint4 m = row[rank + __popc(w[u] & le)];
                  rank += __popc(w[u]);
                  const uint32_t q = c + 32 * u;
                  at[u] = m.z + 2 * q;
                  v[u] = m.w + 2 * q;
                  if ((int32_t)v[u] < 0 && q < ce) {
                    const uint64_t src = ((uint64_t)m.y << 32 | m.x) + q;
                    if (special && m.y >> 30 == 1) {  // overlapping: byte (place - start) mod distance of the source
                      const int32_t start = (int32_t)(m.y & 0x3ffffu) - 0x10000;
                      const int32_t s = start - (int32_t)m.x + (int32_t)(((at[u] - ebase) / 2 - (uint32_t)start) % m.x);
                      v[u] = s >= 0 ? 2 * (uint32_t)s
                                    : 0x8000u | ld_src<!WAIT>(Addr<SEEK>::at(a, bstart + w0 + (int64_t)s, b, obase));
                    } else if (special && SEEK && m.y >> 31) {
                      v[u] = 0x8000u | ld_src<!WAIT>(Addr<SEEK>::at(a, src & ~(1ull << 63), b, obase));
                    } else {
                      v[u] = 0x8000u | ld_src<!WAIT>(reinterpret_cast<const uint8_t*>(src));
                    }
                  }
                }
  #pragma unroll
                for (uint32_t u = 0; u < kCtaUnroll; u++)
                  if (c + 32 * u < ce) asm volatile("st.shared.u16 [%0], %1;" ::"r"(at[u]), "h"((uint16_t)v[u]) : "memory");
              }
            };
            if (odd) rows(std::true_type());
            else rows(std::false_type());
            __syncwarp();  // the next bytes reuse the map
          }
          __syncwarp();
        };
        if (place) {  // the literal run before the match, as far as it lies in the window
          const uint32_t d0 = max(D - lr, w0), d1 = min(D, w0 + wn), n = d0 < d1 && lr ? d1 - d0 : 0u;
          const uint8_t* from = obase + (blen - nlit) + (lits - (D - d0));
          lay(n, d0 - w0, -(1 << 29), reinterpret_cast<uintptr_t>(from), false);
        }
        if (!copy) continue;
        // the match, as far as it lies in the window
        const uint32_t d0 = max(D, w0), d1 = min(D + L, w0 + wn), n = L && d0 < d1 ? d1 - d0 : 0u;
        const uint64_t s0 = bstart + d0 - dist;
        const int32_t rel = n ? (int32_t)max((int64_t)(s0 - bstart) - (int64_t)w0, -(int64_t)(1 << 29)) : 0;
        uint64_t from = 0;
        bool marked = false;
        if (n) {
          if (dist < L) {
            from = (uint64_t)(0x40000000u | (D + 0x10000u - w0)) << 32 | dist;
            marked = true;
          } else if (SEEK && rel < 0 && s0 >> a.log2B != min(s0 + n - 1, bstart + w0 - 1) >> a.log2B) {
            from = s0;
            marked = true;
          } else {
            from = reinterpret_cast<uintptr_t>(Addr<SEEK>::at(a, s0, b, obase));
          }
        }
        const bool big = n >= kCtaLong && !marked && rel + (int32_t)n <= 0;
        copy_long(big, n, d0 - w0, from);
        lay(big ? 0u : n, d0 - w0, rel, from, marked);
      }
    }
    if (lane == 0) atomicMax(&s_group, last);
    const bool any_bad = __syncthreads_or(bad), any_late = __syncthreads_or(timeout);
    if (any_bad || any_late) {
      if (tid == 0)
        record_error(&a.sh->status, &a.sh->err_block, &a.sh->err_where, any_bad ? ACE_E_CORRUPT : ACE_E_TIMEOUT, b,
                     any_bad ? 39 : 38);
      return false;
    }
    first = s_group;

    // each thread's bytes: their chains followed to known entries
    bool deep = false;
    auto settle = [&]() {
      for (uint32_t j = 16 * tid; j < wn; j += 16 * nt) {
        const uint4 lo = *reinterpret_cast<const uint4*>(e + j), hi = *reinterpret_cast<const uint4*>(e + j + 8);
        const uint32_t q[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        uint32_t x[16], all = ~0u;
#pragma unroll
        for (uint32_t k = 0; k < 16; k++) x[k] = k & 1 ? q[k >> 1] >> 16 : q[k >> 1] & 0xffffu;
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) all &= q[k];
        bool open = (all & 0x80008000u) != 0x80008000u;
        for (uint32_t h = 0; open && h < kHops; h++) {
          all = ~0u;
#pragma unroll
          for (uint32_t k = 0; k < 16; k++) {
            asm volatile(
                "{\n.reg .pred p;\n.reg .u32 t, c;\nand.b32 t, %0, 0x8000;\nsetp.eq.u32 p, t, 0;\nadd.u32 c, %0, %1;\n"
                "@p ld.shared.u16 %0, [c];\n}"
                : "+r"(x[k])
                : "r"(ebase)
                : "memory");
            all &= x[k];
          }
          open = !(all & 0x8000u);
        }
        deep |= open;
        uint4 v;
        uint32_t* const y = &v.x;
#pragma unroll
        for (uint32_t k = 0; k < 4; k++)
          y[k] = __byte_perm(__byte_perm(x[4 * k], x[4 * k + 1], 0x0040), __byte_perm(x[4 * k + 2], x[4 * k + 3], 0x0040),
                             0x5410);
        if (j + 16 <= wn) {
          *reinterpret_cast<uint4*>(obase + w0 + j) = v;
        } else {
          for (uint32_t k = 0; j + k < wn; k++) {
            const uint32_t z = k < 4 ? v.x : k < 8 ? v.y : k < 12 ? v.z : v.w;
            obase[w0 + j + k] = (uint8_t)(z >> (8 * (k & 3)));
          }
        }
      }
    };
    settle();
    if (__syncthreads_or(deep)) {
      // Entries change while others read them: each read sees an entry of the
      // same chain, old or new, and 16-bit shared stores do not tear.
      volatile uint16_t* ev = e;
      while (true) {
        int pending = 0;
        for (uint32_t j = tid; j < wn; j += nt) {
          const uint32_t x = ev[j];
          if (!(x & 0x8000u)) {
            const uint32_t y = ev[x >> 1];
            ev[j] = (uint16_t)y;
            pending |= !(y & 0x8000u);
          }
        }
        if (!__syncthreads_or(pending)) break;  // every target precedes its entry: at most log2(kCtaWindow) + 1 turns
      }
      settle();
      __syncthreads();
    }
  }
  return true;
}

// The three passes of a decode, each a persistent launch over the blocks:
// tokens (lengths, offsets, match records), literals, and matches.
// PASS_MATCH resolves blocks in (level, block) order with bounded waits on
// their source blocks (match_level_kernel resolves one level of a whole
// decode without them).
// PASS_FUSED runs all three for one block in one warp, block after block:
// tokens, then literals, then matches with bounded waits on the source
// blocks' flags, then the block's publication.  One launch covers the whole
// decode, so the issue-bound entropy decode of some warps overlaps the
// latency-bound match copies of others on the same SM.
// PASS_PLACE is PASS_MATCH after stream jobs, which leave the literals to it.
// PASS_WARP is PASS_MATCH with a warp per block instead of a CTA: for many
// blocks of few matches, where a CTA's sweep over all of the block's bytes
// costs more than the matches do.
enum { PASS_TOKENS = 0, PASS_LITERALS = 1, PASS_MATCH = 2, PASS_FUSED = 3, PASS_PLACE = 4, PASS_WARP = 5 };

// A pass is held to 64 registers a thread: 256 threads, or the match pass's
// CTAs of up to 512; the match pass by warps and the fused pass to 80.  (Fused, us
// at 80, at 64 with its spills: FASTQ 256 MiB 766, 806, text 64 MiB 831, 826,
// mixed data in 4 KiB blocks 264, 297; with rows of match bytes instead of lanes
// 811, 795, 308 at 80 and 926, 1080, 390 at 64.)
#define ACE_PASS_CTA(P) ((P) == PASS_MATCH || (P) == PASS_PLACE)
#define ACE_PASS_BOUNDS(P) \
  __launch_bounds__(ACE_PASS_CTA(P) ? kCtaThreads : 256, ACE_PASS_CTA(P) ? 2 : (P) == PASS_WARP || (P) == PASS_FUSED ? 3 : 4)

// Publishes block b (its writes visible device-wide before the flag).
__device__ __forceinline__ void publish(uint32_t* ready, uint32_t b, uint32_t epoch, uint32_t lane) {
  __threadfence();
  __syncwarp();
  if (lane == 0) st_release(ready + b, epoch);
}

// Publishes a block that the CTA wrote together.
__device__ __forceinline__ void publish_cta(uint32_t* ready, uint32_t b, uint32_t epoch) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) st_release(ready + b, epoch);
}

// Work items one after another from a ticket, each for the whole CTA.
template <class F>
__device__ __forceinline__ void cta_blocks(uint32_t n_items, uint32_t* ticket, F&& block) {
  __shared__ uint32_t drawn;
  while (true) {
    __syncthreads();  // every thread is done with the block before, and has read its number
    if (threadIdx.x == 0) drawn = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t it = drawn;
    if (it >= n_items) return;
    block(it);
  }
}

// Whether the call recorded an error before this pass: the same answer for a
// whole CTA in the match pass, whose threads meet at barriers (other CTAs may
// be recording one now).
template <int PASS>
__device__ __forceinline__ bool stop_early(const uint32_t* status) {
  const bool set = *(const volatile uint32_t*)status != 0;
  return ACE_PASS_CTA(PASS) ? __syncthreads_or(set) : set;
}

// Blocks level l of a fused call holds (whole decode: the index's level
// histogram; seek: the closure's level ranges in the scratch header).
template <bool SEEK>
__device__ __forceinline__ uint32_t level_size(const DecodeArgs& a, uint32_t l) {
  if (SEEK) return *(volatile uint32_t*)&a.sh->lv_start[l + 1] - *(volatile uint32_t*)&a.sh->lv_start[l];
  return __ldg(a.lv_count + l);
}

// The part of a seek's block inside [coord, coord + len) to the caller, by a warp.
__device__ __forceinline__ void slice_part(const DecodeArgs& a, uint32_t b, uint32_t lane) {
  const uint64_t bs = (uint64_t)b << a.log2B, be = min(bs + ((uint64_t)1 << a.log2B), a.total);
  const uint64_t lo = max(bs, a.coord), hi = min(be, a.coord + a.len);
  const uint8_t* src = a.out + slot_base(a, b) - bs;
  if (hi > lo) warp_copy(a.slice + (lo - a.coord), src + lo, hi - lo, lane);
}

// The work of one archive (whole decode or seek): its list, in level order.
template <bool SEEK>
struct ArchiveJobs {
  const DecodeArgs& a;
  __device__ const DecodeArgs& job(uint32_t v, uint32_t& b) const {
    b = __ldg(a.items + v);
    return a;
  }
  __device__ uint32_t below(const DecodeArgs& x, uint32_t L) const { return level_size<SEEK>(x, L - 1); }
};

// Deferred match jobs a warp holds at most; warps per CTA at most.
constexpr uint32_t kDeferred = 4;
constexpr uint32_t kMaxWarps = 8;

// The fused schedule (Section 2's rule, a block decodes once the blocks its
// matches read are present, applied inside one launch).  Warps take blocks
// from the level-ordered list.  For each one a warp first decodes the
// entropy layer (length, offset and literal streams; literals placed at
// their output positions), then defers the block's match job until every
// block of the lower levels has its matches resolved (the level counters).
// A warp resolves its oldest deferred block as soon as that holds, and takes
// a new block while it waits, up to kDeferred held; so issue-bound entropy
// decode and latency-bound match copies of different warps share each SM
// and no warp idles while there is entropy work left.  With kDeferred held,
// or no blocks left, it waits (bounded, giving up on any recorded error).
// This always ends: the earliest unresolved block of the list has every
// lower level resolved (they come before it), and it is the oldest block of
// the warp holding it.
template <bool SEEK, class Jobs>
__device__ void fused_loop(const Jobs& jobs, ScratchHdr* sh, uint32_t n_items, uint64_t timeout_ns, uint8_t* wsm,
                           uint32_t lane, uint32_t epoch, uint32_t window) {
  uint32_t* const ticket = &sh->ticket;
  constexpr uint32_t ring = SEEK ? kSeekRing : kRing;
  // list positions of the warp's deferred blocks, a ring in shared memory
  // (registers are the scarce resource here): q[(q0 + k) % kDeferred]
  __shared__ uint32_t qs[kMaxWarps][kDeferred];
  uint32_t* const q = qs[threadIdx.x >> 5];
  uint32_t q0 = 0, nq = 0;
  bool more = true;  // blocks may remain in the list
  while (true) {
    if (*(volatile uint32_t*)&sh->status) break;
    if (nq) {
      uint32_t b;
      auto&& a = jobs.job(q[q0], b);
      const uint32_t L = __ldg(a.level + b);
      const uint32_t need = L ? jobs.below(a, L) : 0u;
      bool rdy = true;
      if (lane == 0 && L) rdy = ld_acquire(a.lv_done + L - 1) == need;
      rdy = __shfl_sync(kFull, rdy, 0);
      if (rdy || nq == kDeferred || !more) {
        if (!rdy) {  // nothing else to do: wait, bounded
          uint32_t ok = 1;
          if (lane == 0) {
            const uint64_t t0 = globaltimer();
            uint32_t ns = 32;
            while (ld_acquire(a.lv_done + L - 1) != need) {
              if (*(volatile uint32_t*)&sh->status) {
                ok = 0;
                break;
              }
              if (globaltimer() - t0 > timeout_ns) {
                record_error(&sh->status, &sh->err_block, &sh->err_where, ACE_E_TIMEOUT, b, 38);
                ok = 0;
                break;
              }
              __nanosleep(ns);
              if (ns < 1024) ns <<= 1;
            }
          }
          if (!__shfl_sync(kFull, ok, 0)) break;
        }
        // The bytes of the blocks below were written by other SMs.  Source
        // loads may still go through L1: a block's bytes are written by the
        // one warp that holds it, and read by other warps only after the
        // acquire below has seen its level complete, so no SM can hold an
        // older copy of them.
        fence_acquire();
        const uint32_t ntok = __ldg(reinterpret_cast<const uint32_t*>(a.dir + b) + 12);
        bool ok;
        if (SEEK) {
          // source blocks must be members of the closure; published ones
          // carry the epoch without the pending bit, so the flag checks do
          // not wait
          ok = match_block<true, true, true, WAY_LANES>(a, reinterpret_cast<MatchRec*>(wsm), b, lane, epoch,
                                             ntok ? ntok - 1 : 0);
          if (ok && a.slice) slice_part(a, b, lane);
          if (ok) publish(a.ready, b, epoch, lane);
        } else {
          ok = match_block<false, false, true, WAY_LANES>(a, reinterpret_cast<MatchRec*>(wsm), b, lane, epoch,
                                               ntok ? ntok - 1 : 0, L);
        }
        if (!ok) break;  // the error is recorded; every warp stops
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(a.lv_done + L, 1u);
        q0 = (q0 + 1) % kDeferred;
        nq--;
        continue;
      }
    }
    if (!more) {
      if (!nq) break;
      continue;
    }
    uint32_t u = 0;
    if (lane == 0) u = atomicAdd(ticket, 1u);
    u = __shfl_sync(kFull, u, 0);
    if (u >= n_items) {
      more = false;
      continue;
    }
    uint32_t b;
    auto&& a = jobs.job(u, b);
    bool ok = token_block<SEEK>(a, carve_tok(wsm), b, lane);
    if (ok) ok = literal_block<SEEK, ring>(a, carve_lit(wsm, window, ring), b, lane);
    if (!ok) break;
    if (lane == 0) q[(q0 + nq) % kDeferred] = u;
    __syncwarp();
    nq++;
  }
}

// One pass over a work list by persistent warps: the token pass decodes every
// block's length and offset streams into match records; the literal pass
// decodes every block's literal stream straight to its output positions; the
// match pass, launched after them, resolves every block's matches in (level,
// block) order, waiting on source blocks' flags, and publishes the block.
template <bool SEEK, int PASS>
__global__ void ACE_PASS_BOUNDS(PASS) decode_kernel(DecodeArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t epoch = *(volatile uint32_t*)&a.sh->epoch;
  const uint32_t n_items = SEEK ? *(volatile uint32_t*)&a.sh->n_work : a.n_items;
  // the literal and match passes run only after every block's tokens decoded
  if (PASS != PASS_TOKENS && stop_early<PASS>(&a.sh->status)) return;
  uint8_t* wsm = smem + (size_t)wid * a.warp_smem;
  if (PASS == PASS_FUSED) {
    fused_loop<SEEK>(ArchiveJobs<SEEK>{a}, a.sh, n_items, a.timeout_ns, wsm, lane, epoch, a.window);
    return;
  }
  if (ACE_PASS_CTA(PASS)) {
    cta_blocks(n_items, &a.sh->ticket3, [&](uint32_t it) {
      const uint32_t b = __ldg(a.items + it);
      const uint32_t ntok = __ldg(reinterpret_cast<const uint32_t*>(a.dir + b) + 12);
      const bool ok = match_cta<SEEK, true, PASS == PASS_PLACE>(a, smem, b, ntok ? ntok - 1 : 0, epoch, 0);
      publish_cta(a.ready, b, epoch);
      if (SEEK && ok && a.slice) {
        // the part of this block inside [coord, coord + len) to the caller, a share per warp
        uint64_t bs = (uint64_t)b << a.log2B, be = min(bs + ((uint64_t)1 << a.log2B), a.total);
        uint64_t lo = max(bs, a.coord), hi = min(be, a.coord + a.len);
        if (hi > lo) {
          const uint32_t nw = blockDim.x >> 5;
          const uint64_t part = ((hi - lo + nw - 1) / nw + 15) & ~15ull;
          const uint8_t* src = a.out + slot_base(a, b) - bs;
          lo += wid * part;
          hi = min(hi, lo + part);
          if (hi > lo) warp_copy(a.slice + (lo - a.coord), src + lo, hi - lo, lane);
        }
      }
    });
    return;
  }
  uint32_t* ticket = PASS == PASS_TOKENS ? &a.sh->ticket : PASS == PASS_LITERALS ? &a.sh->ticket2 : &a.sh->ticket3;
  while (true) {
    uint32_t it = 0;
    if (lane == 0) it = atomicAdd(ticket, 1u);
    it = __shfl_sync(kFull, it, 0);
    if (it >= n_items) break;
    uint32_t b = __ldg(a.items + it);
    if (PASS == PASS_TOKENS) {
      token_block<SEEK>(a, carve_tok(wsm), b, lane);
      continue;
    }
    if (PASS == PASS_WARP) {
      const uint32_t ntok = __ldg(reinterpret_cast<const uint32_t*>(a.dir + b) + 12);
      const bool ok = match_block<SEEK, true, false, WAY_ROWS>(a, reinterpret_cast<MatchRec*>(wsm), b, lane, epoch,
                                                               ntok ? ntok - 1 : 0);
      if (SEEK && ok && a.slice) slice_part(a, b, lane);
      publish(a.ready, b, epoch, lane);
      continue;
    }
    constexpr uint32_t ring = SEEK ? kSeekRing : kRing;
    literal_block<SEEK, ring>(a, carve_lit(wsm, a.window, ring), b, lane);
  }
}

// The entropy layer of few blocks: a warp per stream (a block's three streams
// are independent entry points, Section 3), each a CTA of its own so that they
// spread over the SMs.  A block's time is then its longest stream's, where the
// token and literal passes add the three up.
template <bool SEEK>
__global__ void __launch_bounds__(32) entropy_kernel(DecodeArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x;
  const uint32_t n_jobs = 3 * (SEEK ? *(volatile uint32_t*)&a.sh->n_work : a.n_items);
  for (uint32_t j = blockIdx.x; j < n_jobs; j += gridDim.x) stream_job<SEEK, kSeekRing>(a, smem, __ldg(a.items + j / 3), j % 3, lane);
}

// The match pass of one dependency level of a whole decode: every lower
// level was finished by the launches before, so blocks need no flags or
// waits.  Blocks are dealt out statically (block k of the level to warp
// k mod the warps in the grid), and each warp fetches its next block's
// number and record range while it resolves the current one.
// WAY_ROWS for matches mostly short, WAY_ROUNDS, in fewer registers, for few long
// ones (genome 1 GiB, the match pass: 342 us at 56 registers, 360 at 72; the rows
// spill below 72: FASTQ 129 us, 147 at 56).  A long match by the whole warp, not the round's long matches laid end
// to end in pieces with the next lane's vector shuffled in, took the genome's
// from 518 us.
template <int WAY>
__global__ void __maxnreg__(WAY == WAY_ROUNDS ? 56 : 72) match_level_kernel(DecodeArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  if (*(volatile uint32_t*)&a.sh->status) return;
  MatchRec* gm = reinterpret_cast<MatchRec*>(smem + (size_t)wid * kMatchSmem);
  uint32_t it = blockIdx.x * (blockDim.x >> 5) + wid;
  if (it >= a.n_items) return;
  auto n_matches = [&](uint32_t b) -> uint32_t {
    return (uint32_t)(__ldg(a.match_ptr + b + 1) - __ldg(a.match_ptr + b));
  };
  uint32_t b = __ldg(a.items + it);
  uint32_t nm = n_matches(b);
  while (true) {
    const uint32_t nx = it + nw;
    uint32_t bn = 0, nmn = 0;
    if (nx < a.n_items) {
      bn = __ldg(a.items + nx);
      nmn = n_matches(bn);
    }
    match_block<false, false, true, WAY>(a, gm, b, lane, 0, nm, a.cur_level);
    if (nx >= a.n_items) break;
    it = nx;
    b = bn;
    nm = nmn;
  }
}

// The same with a CTA per block.
template <uint32_t THREADS, bool LITS>
__global__ void __launch_bounds__(THREADS, THREADS == 512 ? 2 : 4) match_cta_kernel(DecodeArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  if (__syncthreads_or(*(volatile uint32_t*)&a.sh->status != 0)) return;  // the same answer for the whole CTA
  for (uint32_t it = blockIdx.x; it < a.n_items; it += gridDim.x) {
    const uint32_t b = __ldg(a.items + it);
    const uint64_t m0 = __ldg(a.match_ptr + b);
    if (!match_cta<false, false, LITS>(a, smem, b, (uint32_t)(__ldg(a.match_ptr + b + 1) - m0), 0, a.cur_level)) return;
  }
}

// ----------------------------------------------------------- batch decode

// One independent archive of a batch, as the batch kernel sees it.
struct ObjDesc {
  const uint8_t* arc;
  const ace_block_dir* dir;
  uint64_t payload_off;
  uint64_t total;
  uint8_t* out;
  uint32_t* ready;
  const uint32_t* order;  // the archive's blocks in (level, block) order
  const uint32_t* level;  // each block's dependency level
  MatchRec* recs;         // the archive's match records
  const uint64_t* match_ptr;
  uint32_t* lv_done;         // fused schedule: blocks of each level with matches resolved
  const uint32_t* lv_count;  // blocks per level
  uint32_t log2B, w, nb, pad;
};

// Consecutive work items of a batch: blocks of one archive, from a place in
// its order on.
struct BatchSeg {
  uint32_t start;  // first work item
  uint32_t obj, first, pad;
};

// Two lists of the same items.  The token and literal passes take the archives
// of the largest blocks first: a 64 KiB block is a warp's chain of 0.2 ms, and
// one begun last would be the pass's tail.  The match pass (and the fused
// schedule) takes the lowest level of every archive first, so that hardly a
// block waits for its sources: archive by archive, each one's first levels
// waited for one another while nothing else had been handed out.  192 objects
// of 4 KiB to 4 MiB: match pass 536 to 252 us.
struct BatchArgs {
  const ObjDesc* objs;
  const BatchSeg* by_size;   // [n_size]
  const BatchSeg* by_level;  // [n_level]
  uint32_t n_size, n_level, n_items;
  uint32_t window, warp_smem, esc_cap, max_ntok;
  ScratchHdr* sh;
  uint64_t timeout_ns;
  uint32_t long_min;
};

// The work of a batch: (archive, block) items in one of the two orders, each
// archive's blocks in its own level order in both.
struct BatchJobs {
  const BatchArgs& ba;
  const BatchSeg* segs;
  uint32_t n_segs;
  __device__ DecodeArgs job(uint32_t v, uint32_t& b) const;
  __device__ uint32_t below(const DecodeArgs& x, uint32_t L) const { return __ldg(x.lv_count + L - 1); }
};

// Thousands of independent archives in one persistent launch per pass: warps
// (match pass: CTAs) take (archive, block) items from one ticket; each
// archive's items are in its own (level, block) order, so in the match pass a
// block only ever waits on blocks of its archive handed out before it.
__device__ DecodeArgs batch_args(const BatchArgs& ba, const ObjDesc& od) {
  DecodeArgs a{};
  a.arc = od.arc;
  a.dir = od.dir;
  a.payload_off = od.payload_off;
  a.total = od.total;
  a.nb = od.nb;
  a.log2B = od.log2B;
  a.w = od.w;
  a.window = ba.window;
  a.esc_cap = ba.esc_cap;
  a.warp_smem = ba.warp_smem;
  a.max_ntok = ba.max_ntok;
  a.out = od.out;
  a.sh = ba.sh;
  a.ready = od.ready;
  a.timeout_ns = ba.timeout_ns;
  a.recs = od.recs;
  a.match_ptr = od.match_ptr;
  a.level = od.level;
  a.lv_done = od.lv_done;
  a.lv_count = od.lv_count;
  a.long_min = ba.long_min;
  return a;
}

__device__ DecodeArgs BatchJobs::job(uint32_t v, uint32_t& b) const {
  uint32_t lo = 0, hi = n_segs;  // the last segment that starts at or before item v
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(&segs[mid].start) <= v) lo = mid;
    else hi = mid;
  }
  const uint4 sg = __ldg(reinterpret_cast<const uint4*>(segs + lo));
  const ObjDesc od = ba.objs[sg.y];
  b = __ldg(od.order + sg.z + (v - sg.x));
  return batch_args(ba, od);
}

template <int PASS>
__global__ void ACE_PASS_BOUNDS(PASS) batch_decode_kernel(BatchArgs ba) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (PASS != PASS_TOKENS && PASS != PASS_FUSED && stop_early<PASS>(&ba.sh->status)) return;
  uint8_t* wsm = smem + (size_t)wid * ba.warp_smem;
  const uint32_t epoch = *(volatile uint32_t*)&ba.sh->epoch;
  if (PASS == PASS_FUSED) {
    fused_loop<false>(BatchJobs{ba, ba.by_level, ba.n_level}, ba.sh, ba.n_items, ba.timeout_ns, wsm, lane, epoch, ba.window);
    return;
  }
  const BatchJobs jobs = ACE_PASS_CTA(PASS) || PASS == PASS_WARP ? BatchJobs{ba, ba.by_level, ba.n_level}
                                                                  : BatchJobs{ba, ba.by_size, ba.n_size};
  if (ACE_PASS_CTA(PASS)) {
    cta_blocks(ba.n_items, &ba.sh->ticket3, [&](uint32_t it) {
      uint32_t b;
      const DecodeArgs a = jobs.job(it, b);
      const uint32_t ntok = __ldg(reinterpret_cast<const uint32_t*>(a.dir + b) + 12);
      match_cta<false, true, PASS == PASS_PLACE>(a, smem, b, ntok ? ntok - 1 : 0, epoch, 0);
      publish_cta(a.ready, b, epoch);
    });
    return;
  }
  uint32_t* ticket =
      PASS == PASS_TOKENS ? &ba.sh->ticket : PASS == PASS_LITERALS ? &ba.sh->ticket2 : &ba.sh->ticket3;
  while (true) {
    uint32_t it = 0;
    if (lane == 0) it = atomicAdd(ticket, 1u);
    it = __shfl_sync(kFull, it, 0);
    if (it >= ba.n_items) break;
    uint32_t b;
    const DecodeArgs a = jobs.job(it, b);
    if (PASS == PASS_TOKENS) {
      token_block<false>(a, carve_tok(wsm), b, lane);
    } else if (PASS == PASS_WARP) {
      const uint32_t ntok = __ldg(reinterpret_cast<const uint32_t*>(a.dir + b) + 12);
      match_block<false, true, false, WAY_LANES>(a, reinterpret_cast<MatchRec*>(wsm), b, lane, epoch, ntok ? ntok - 1 : 0);
      publish(a.ready, b, epoch, lane);
    } else {
      literal_block<false, kRing>(a, carve_lit(wsm, ba.window, kRing), b, lane);
    }
  }
}

// The entropy layer of a batch, a warp per stream, largest blocks first: one
// launch whose time is its longest stream's, where the token and literal
// passes each had that tail.
constexpr uint32_t kBatchEntropyWarps = 4;
__global__ void __launch_bounds__(32 * kBatchEntropyWarps, 8) batch_entropy_kernel(BatchArgs ba) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const BatchJobs jobs{ba, ba.by_size, ba.n_size};
  uint8_t* wsm = smem + wid * job_smem_bytes(ba.esc_cap, kRing);
  while (true) {
    uint32_t it = 0;
    if (lane == 0) it = atomicAdd(&ba.sh->ticket, 1u);
    it = __shfl_sync(kFull, it, 0);
    if (it / 3 >= ba.n_items) break;
    uint32_t b;
    const DecodeArgs a = jobs.job(it / 3, b);
    stream_job<false, kRing>(a, wsm, b, it % 3, lane);
  }
}

// ---------------------------------------------------------- seek closure

struct ClosureArgs {
  const uint32_t* dep_ptr;
  const uint32_t* dep_iv;
  ScratchHdr* sh;
  uint32_t* marks;   // one bit per block, all clear between calls
  uint32_t* front0;
  uint32_t* front1;
  uint32_t* work;
  uint32_t* slot_of;
  uint64_t nb;
  uint64_t first, last;  // target blocks
  uint64_t cap;          // slots available
  const uint32_t* level; // by levels: each block's dependency level (else null)
  uint32_t n_levels;
  uint32_t* ready;       // closure blocks get the call's epoch with kPendingFlag set
  uint32_t* lv_done;     // fused seeks: per-level counters, cleared here (null otherwise)
};

// CTAs of a closure search, one cluster (the largest portable size).
constexpr uint32_t kClosureCtas = 8;

// The blocks a seek must decode: its target blocks and, transitively, every
// block their matches read (Section 2).  Breadth first from the targets, a
// warp per frontier block with its lanes over the block's dependency
// intervals; then an ordered compaction of the marked blocks gives each its
// slot, and the work list is ordered by dependency level (blocks of a level
// in ascending order) with the level ranges in the scratch header -- a valid
// decode order either way, since sources always precede.
//
// A frontier block is four or five loads that wait for one another, so the
// search is bound by their latency times the blocks a warp takes in turn: the
// frontier is spread over the 256 warps of a cluster, with a cluster barrier
// per step; the rest, short, is the first CTA's.  By one CTA the closure of a
// 16 MiB range of a genome took 35 to 49 us; this takes 20.
__global__ void __cluster_dims__(kClosureCtas, 1, 1) __launch_bounds__(1024, 1) closure_kernel(ClosureArgs a) {
  __shared__ uint32_t wsum[32];
  __shared__ uint32_t carry;
  __shared__ uint32_t lcnt[kMaxLevelLaunches + 1];
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  const uint32_t rank = cluster_rank();
  const uint32_t ntar = (uint32_t)(a.last - a.first + 1);
  if (rank == 0 && tid == 0) {
    const uint32_t e = (a.sh->epoch + 1) & ~kPendingFlag;  // never 0, never with the pending bit
    a.sh->epoch = e ? e : 1u;
    a.sh->ticket = 0;
    a.sh->ticket2 = 0;
    a.sh->ticket3 = 0;
    a.sh->min_block = (uint32_t)a.first;
    a.sh->front[0] = ntar;
    a.sh->front[1] = 0;
  }
  if (rank == 0 && tid <= kMaxLevelLaunches && a.lv_done) a.lv_done[tid] = 0;
  for (uint32_t i = rank * blockDim.x + tid; i < ntar; i += kClosureCtas * blockDim.x) {
    const uint32_t b = (uint32_t)a.first + i;
    atomicOr(&a.marks[b >> 5], 1u << (b & 31));
    a.front0[i] = b;
  }
  cluster_sync();
  // step k: the frontier's blocks in front0/front1 in turn, their count in
  // front[k mod 3]; the next step's counted in front[k + 1 mod 3], the one
  // after cleared
  uint32_t* cur = a.front0;
  uint32_t* nxt = a.front1;
  for (uint32_t k = 0;; k++) {
    const uint32_t n_front = __ldcg(&a.sh->front[k % 3]);
    if (!n_front) break;  // the same for every CTA: counted before the last barrier
    uint32_t* n_next = &a.sh->front[(k + 1) % 3];
    if (rank == 0 && tid == 0) a.sh->front[(k + 2) % 3] = 0;
    for (uint32_t f = rank * nw + wid; f < n_front; f += kClosureCtas * nw) {
      const uint32_t b = __ldcg(cur + f);
      const uint32_t e1 = __ldg(a.dep_ptr + b + 1);
      for (uint32_t e = __ldg(a.dep_ptr + b) + lane; e < e1; e += 32) {
        const uint32_t k0 = __ldg(a.dep_iv + 2 * e), k1 = __ldg(a.dep_iv + 2 * e + 1);
        for (uint32_t q = k0; q <= k1; q++) {
          const uint32_t old = atomicOr(&a.marks[q >> 5], 1u << (q & 31));
          if (!(old & (1u << (q & 31)))) {
            nxt[atomicAdd(n_next, 1u)] = q;
            atomicMin(&a.sh->min_block, q);
          }
        }
      }
    }
    cluster_sync();
    uint32_t* const t = cur;
    cur = nxt;
    nxt = t;
  }
  if (rank) return;
  if (tid <= kMaxLevelLaunches) lcnt[tid] = 0;
  // ordered compaction of the marked blocks into front0, clearing the marks
  // behind it; a block's slot is its place in ascending order
  if (tid == 0) carry = 0;
  __syncthreads();
  uint32_t w0 = __ldcg(&a.sh->min_block) >> 5, w1 = (uint32_t)(a.last >> 5);
  for (uint32_t c0 = w0; c0 <= w1; c0 += blockDim.x) {
    uint32_t wi = c0 + tid;
    uint32_t bits = wi <= w1 ? __ldcg(a.marks + wi) : 0u;
    uint32_t cnt = __popc(bits);
    uint32_t incl = warp_incl_sum(cnt, lane);
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      uint32_t s = lane < nw ? wsum[lane] : 0;
      uint32_t si = warp_incl_sum(s, lane);
      if (lane < nw) wsum[lane] = si - s;
    }
    __syncthreads();
    uint32_t pos = carry + wsum[wid] + incl - cnt;
    while (bits) {
      uint32_t bit = __ffs(bits) - 1;
      bits &= bits - 1;
      uint32_t b = wi * 32 + bit;
      if (pos < a.cap) {
        a.front0[pos] = b;
        a.slot_of[b] = pos;
      }
      pos++;
    }
    if (wi <= w1) a.marks[wi] = 0;
    __syncthreads();
    if (tid == blockDim.x - 1) carry = pos;
    __syncthreads();
  }
  const uint32_t n = carry;
  if (n > a.cap) {
    if (tid == 0) {
      record_error(&a.sh->status, &a.sh->err_block, &a.sh->err_where, ACE_E_NOMEM, n, 50);
      a.sh->n_work = 0;
    }
    return;
  }
  // the work list by level (one level when levels are not used)
  const uint32_t epoch = a.sh->epoch;
  for (uint32_t i = tid; i < n; i += blockDim.x) {
    const uint32_t b = a.front0[i];
    atomicAdd(&lcnt[a.level ? a.level[b] : 0], 1u);
    if (a.ready) a.ready[b] = epoch | kPendingFlag;  // a member of this seek's closure, not yet decoded
  }
  __syncthreads();
  if (tid == 0) {
    const uint32_t nl = a.level ? a.n_levels : 1;
    uint32_t c = 0;
    for (uint32_t l = 0; l < nl; l++) {
      const uint32_t k = lcnt[l];
      lcnt[l] = c;
      a.sh->lv_start[l] = c;
      c += k;
    }
    a.sh->lv_start[nl] = c;
    a.sh->n_work = n;
  }
  __syncthreads();
  for (uint32_t i = tid; i < n; i += blockDim.x) {
    const uint32_t b = a.front0[i];
    // (any order inside a level; without levels the ascending order is the
    // decode order, and blocks must not be handed out before their sources)
    a.work[a.level ? atomicAdd(&lcnt[a.level[b]], 1u) : i] = b;
  }
}

// ------------------------------------------------------ seek batches (cache)

// One archive attached to a decoded-block cache.
struct CacheArc {
  const uint8_t* arc;
  const ace_block_dir* dir;
  uint64_t payload_off;
  uint64_t total;
  const uint32_t* dep_ptr;
  const uint32_t* dep_iv;
  uint32_t* ready;    // == cache epoch: the block sits decoded in its slot
  uint32_t* slot_of;
  uint32_t* marks;    // closure marks, clear between calls
  uint32_t* wpos;     // a block decoded by the current batch: its place in the work list
  uint32_t nb, w;
};

// Header of a cache (first 256 bytes of its memory).
struct CacheHdr {
  uint32_t status, err_block, err_where;
  uint32_t epoch;      // blocks whose ready flag equals it are cached
  uint32_t ticket;
  uint32_t n_work;
  uint32_t n_cached;   // slots holding a decoded block
  uint32_t reserved;
  uint32_t hand;       // clock hand: the next slot the allocation looks at
  uint32_t serial;     // batches run: the slots a batch uses carry its serial
  uint64_t evicted;    // cached blocks evicted to make room, since creation
  uint32_t ticket2;    // next work item of the literal pass
  uint32_t ticket3;    // next work item of the match pass
  uint64_t decoded;    // blocks decoded, since creation
  uint32_t front[3];   // frontier sizes during the closure search
  uint32_t overflow;   // a frontier outgrew its room (serial of the batch)
  uint32_t pad[44];
};
static_assert(sizeof(CacheHdr) == 256, "cache header");
static_assert(offsetof(CacheHdr, ticket2) == offsetof(ScratchHdr, ticket2), "shared header fields");
static_assert(offsetof(CacheHdr, ticket3) == offsetof(ScratchHdr, ticket3), "shared header fields");
static_assert(offsetof(CacheHdr, epoch) == offsetof(ScratchHdr, epoch), "shared header fields");
static_assert(offsetof(CacheHdr, ticket) == offsetof(ScratchHdr, ticket), "shared header fields");
static_assert(offsetof(CacheHdr, n_work) == offsetof(ScratchHdr, n_work), "shared header fields");

struct CacheArgs {
  CacheHdr* h;
  const CacheArc* arcs;
  uint32_t n_arcs;
  uint32_t log2B;
  uint32_t n_slots;
  uint32_t front_cap;    // blocks one batch may decode (work items), and the frontier's capacity
  uint32_t* front0;      // (archive, block) pairs
  uint32_t* front1;
  uint32_t* work;        // (archive, block) pairs in decode order
  uint32_t* taken;       // the slots the allocation took, one per work item
  uint32_t* arc_minmax;  // per archive: smallest, largest block marked
  uint32_t* owner_arc;   // per slot: the archive and block it holds (archive ~0: none)
  uint32_t* owner_blk;
  uint32_t* ref;         // per slot: the clock's reference bit
  uint32_t* use;         // per slot: the serial of the last batch that used it
  uint8_t* slots;
  MatchRec* recs;        // max_ntok match records per work item
  const ace_seek_req* reqs;
  uint32_t n_reqs;
};

// A block the batch needs: a cached one has its slot kept from eviction for
// this batch and its reference bit set (true: nothing to decode); an
// uncached one is marked for decoding (returns whether it was newly marked).
__device__ __forceinline__ bool cache_visit(const CacheArgs& c, uint32_t a, uint32_t b, uint32_t epoch,
                                            uint32_t serial, bool& cached) {
  const CacheArc& ca = c.arcs[a];
  // flags are set by earlier launches on this stream, ordered before this one
  cached = ld_relaxed(ca.ready + b) == epoch;
  if (cached) {
    const uint32_t sl = ca.slot_of[b];
    if (sl < c.n_slots) {
      c.use[sl] = serial;
      c.ref[sl] = 1;
    }
    return false;
  }
  const uint32_t bit = 1u << (b & 31);
  return !(atomicOr(ca.marks + (b >> 5), bit) & bit);
}

// The blocks a batch of seeks must decode: every target block that is not
// cached and, transitively, every uncached block their matches read
// (Section 2), listed archive by archive in ascending block order.  Each
// gets a slot from a clock over the slots: slots this batch uses are passed
// over, a slot whose reference bit is set gets a second chance (the bit is
// cleared), and a slot taken from a cached block evicts it.
//
// Bound by latency like the plain seek's closure, and searched by a cluster
// in the same way (a warp per request for the targets, then per frontier
// block); the listing and the clock are the first CTA's.  By one CTA, with a
// thread per request, 128 requests over 1900 blocks took 0.297 ms; this takes
// 0.069 ms.
__global__ void __cluster_dims__(kClosureCtas, 1, 1) __launch_bounds__(1024, 1) cache_closure_kernel(CacheArgs c) {
  __shared__ uint32_t carry;
  __shared__ uint32_t s_taken, s_hand, s_scanned, s_stop;
  __shared__ uint32_t wsum[32];
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  const uint32_t rank = cluster_rank();
  const uint32_t epoch = c.h->epoch, serial = c.h->serial + 1;
  // front[] and overflow are of no use between batches: cleared here, counted
  // from the first barrier on
  if (rank == 0) {
    if (tid < 3) c.h->front[tid] = 0;
    if (tid == 3) c.h->overflow = 0;
    for (uint32_t a = tid; a < c.n_arcs; a += blockDim.x) {
      c.arc_minmax[2 * a] = 0xffffffffu;
      c.arc_minmax[2 * a + 1] = 0;
    }
  }
  cluster_sync();
  if (rank == 0 && tid == 0) c.h->serial = serial;  // every CTA has read it
  auto push = [&](uint32_t* front, uint32_t* count, uint32_t a, uint32_t b) {
    const uint32_t i = atomicAdd(count, 1u);
    if (i < c.front_cap) {
      front[2 * i] = a;
      front[2 * i + 1] = b;
    } else {
      c.h->overflow = 1;
    }
    atomicMin(&c.arc_minmax[2 * a], b);
  };
  // targets: a warp per request, its lanes over the request's blocks
  const uint32_t gw = rank * nw + wid;
  for (uint32_t r = gw; r < c.n_reqs; r += kClosureCtas * nw) {
    const ace_seek_req q = c.reqs[r];
    const uint64_t first = q.coord >> c.log2B, last = (q.coord + q.len - 1) >> c.log2B;
    for (uint64_t b = first + lane; b <= last; b += 32) {
      bool cached;
      if (cache_visit(c, q.archive, (uint32_t)b, epoch, serial, cached)) {
        push(c.front0, &c.h->front[0], q.archive, (uint32_t)b);
        atomicMax(&c.arc_minmax[2 * q.archive + 1], (uint32_t)b);
      }
    }
  }
  cluster_sync();
  uint32_t* cur = c.front0;
  uint32_t* nxt = c.front1;
  for (uint32_t k = 0;; k++) {  // counts as in the plain seek's closure
    const uint32_t n_front = min(__ldcg(&c.h->front[k % 3]), c.front_cap);
    if (!n_front || __ldcg(&c.h->overflow)) break;  // the same for every CTA: written before the last barrier
    cluster_sync();                                 // ... and this step's overflow after this one
    uint32_t* n_next = &c.h->front[(k + 1) % 3];
    if (rank == 0 && tid == 0) c.h->front[(k + 2) % 3] = 0;
    for (uint32_t i = gw; i < n_front; i += kClosureCtas * nw) {  // a warp per frontier block, lanes over its intervals
      const uint32_t a = __ldcg(cur + 2 * i), b = __ldcg(cur + 2 * i + 1);
      const CacheArc& ca = c.arcs[a];
      const uint32_t e1 = __ldg(ca.dep_ptr + b + 1);
      for (uint32_t e = __ldg(ca.dep_ptr + b) + lane; e < e1; e += 32)
        for (uint32_t q = __ldg(ca.dep_iv + 2 * e); q <= __ldg(ca.dep_iv + 2 * e + 1); q++) {
          bool cached;
          if (cache_visit(c, a, q, epoch, serial, cached)) push(nxt, n_next, a, q);
        }
    }
    cluster_sync();
    uint32_t* const t = cur;
    cur = nxt;
    nxt = t;
  }
  if (rank) return;
  const bool overflow = __ldcg(&c.h->overflow) != 0;
  // ordered compaction into the work list, archive by archive, clearing the
  // marks behind it
  if (tid == 0) carry = 0;
  __syncthreads();
  for (uint32_t a = 0; a < c.n_arcs; a++) {
    uint32_t lo = __ldcg(c.arc_minmax + 2 * a), hi = __ldcg(c.arc_minmax + 2 * a + 1);
    if (lo > hi) continue;
    const CacheArc& ca = c.arcs[a];
    for (uint32_t c0 = lo >> 5; c0 <= (hi >> 5); c0 += blockDim.x) {
      uint32_t wi = c0 + tid;
      uint32_t bits = wi <= (hi >> 5) ? __ldcg(ca.marks + wi) : 0u;
      uint32_t cnt = __popc(bits);
      uint32_t incl = warp_incl_sum(cnt, lane);
      if (lane == 31) wsum[wid] = incl;
      __syncthreads();
      if (wid == 0) {
        uint32_t v = lane < nw ? wsum[lane] : 0;
        uint32_t vi = warp_incl_sum(v, lane);
        if (lane < nw) wsum[lane] = vi - v;
      }
      __syncthreads();
      uint32_t pos = carry + wsum[wid] + incl - cnt;
      while (bits) {
        uint32_t bit = __ffs(bits) - 1;
        bits &= bits - 1;
        uint32_t b = wi * 32 + bit;
        if (pos < c.front_cap) {
          c.work[2 * pos] = a;
          c.work[2 * pos + 1] = b;
        }
        pos++;
      }
      if (wi <= (hi >> 5)) ca.marks[wi] = 0;
      __syncthreads();
      if (tid == blockDim.x - 1) carry = pos;
      __syncthreads();
    }
  }
  const uint32_t n = carry;
  if (tid == 0) {
    s_taken = 0;
    s_hand = c.h->hand;
    s_scanned = 0;
  }
  __syncthreads();
  // the clock: at most two turns over the slots (after one, every bit of a
  // slot this batch does not use is clear)
  const uint64_t limit = overflow || n > c.front_cap ? 0ull : 2ull * c.n_slots;
  while (true) {
    const uint32_t taken = s_taken, hand = s_hand, scanned = s_scanned;
    if (taken >= n || scanned >= limit) break;
    const uint64_t room = limit - scanned;
    const uint32_t win = (uint32_t)min(min((uint64_t)blockDim.x, (uint64_t)c.n_slots), room);
    const uint32_t sl = (uint32_t)(((uint64_t)hand + tid) % c.n_slots);
    bool pinned = false, refd = false, elig = false;
    if (tid < win) {
      pinned = __ldcg(c.use + sl) == serial;
      refd = __ldcg(c.ref + sl) != 0;
      elig = !pinned && !refd;
    }
    const uint32_t e = elig ? 1u : 0u;
    const uint32_t incl = warp_incl_sum(e, lane);
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      uint32_t v = lane < nw ? wsum[lane] : 0;
      uint32_t vi = warp_incl_sum(v, lane);
      if (lane < nw) wsum[lane] = vi - v;
      if (lane == nw - 1) s_stop = vi;  // the window's eligible total, for a moment
    }
    __syncthreads();
    const uint32_t total = s_stop, rank = wsum[wid] + incl - e, rem = n - taken;
    __syncthreads();
    // the hand stops just after the rem-th eligible slot, else at the window's end
    if (total >= rem) {
      if (elig && rank == rem - 1) s_stop = tid;
    } else if (tid == 0) {
      s_stop = win - 1;
    }
    __syncthreads();
    const uint32_t stop = s_stop;
    if (tid <= stop && tid < win) {
      if (!pinned && refd) c.ref[sl] = 0;  // second chance
      if (elig && rank < rem) {
        c.taken[taken + rank] = sl;
        c.use[sl] = serial;  // taken: the next turn of the hand passes it over
      }
    }
    __syncthreads();
    if (tid == 0) {
      s_taken = taken + min(total, rem);
      s_hand = (uint32_t)(((uint64_t)hand + stop + 1) % c.n_slots);
      s_scanned = scanned + stop + 1;
    }
    __syncthreads();
  }
  const bool fits = !overflow && n <= c.front_cap && s_taken >= n;
  // each work item into its slot, evicting the slot's cached block
  if (fits) {
    for (uint32_t i = tid; i < n; i += blockDim.x) {
      const uint32_t sl = c.taken[i], a = c.work[2 * i], b = c.work[2 * i + 1];
      const uint32_t oa = c.owner_arc[sl], ob = c.owner_blk[sl];
      if (oa < c.n_arcs) {
        const CacheArc& o = c.arcs[oa];
        if (o.slot_of[ob] == sl && o.ready[ob] == epoch) {
          o.ready[ob] = 0;
          atomicAdd(reinterpret_cast<unsigned long long*>(&c.h->evicted), 1ull);
        }
      } else {
        atomicAdd(&c.h->n_cached, 1u);
      }
      c.owner_arc[sl] = a;
      c.owner_blk[sl] = b;
      c.use[sl] = serial;
      c.ref[sl] = 1;
      const CacheArc& ca = c.arcs[a];
      ca.slot_of[b] = sl;
      ca.wpos[b] = i;
    }
  }
  __syncthreads();
  if (tid == 0) {
    c.h->hand = s_hand;
    uint32_t nn = n;
    if (!fits) {
      record_error(&c.h->status, &c.h->err_block, &c.h->err_where, ACE_E_NOMEM, n, 51);
      nn = 0;
    } else {
      c.h->decoded += n;
    }
    c.h->n_work = nn;
    c.h->ticket = 0;
    c.h->ticket2 = 0;
    c.h->ticket3 = 0;
  }
}

struct CacheDecodeArgs {
  CacheArgs c;
  uint32_t window, warp_smem, esc_cap, max_ntok;
  uint64_t timeout_ns;
  uint32_t long_min;
};

// The decode arguments of a batch's work item, and its block.
__device__ __forceinline__ DecodeArgs cache_job(const CacheDecodeArgs& ca, uint32_t it, uint32_t& b) {
  const CacheArgs& c = ca.c;
  const uint32_t ai = __ldg(c.work + 2 * it);
  b = __ldg(c.work + 2 * it + 1);
  const CacheArc& arc = c.arcs[ai];
  DecodeArgs a{};
  a.arc = arc.arc;
  a.dir = arc.dir;
  a.payload_off = arc.payload_off;
  a.total = arc.total;
  a.nb = arc.nb;
  a.log2B = c.log2B;
  a.w = arc.w;
  a.window = ca.window;
  a.esc_cap = ca.esc_cap;
  a.warp_smem = ca.warp_smem;
  a.max_ntok = ca.max_ntok;
  a.out = c.slots;
  a.sh = reinterpret_cast<ScratchHdr*>(c.h);
  a.ready = arc.ready;
  a.slot_of = arc.slot_of;
  a.n_slots = c.n_slots;
  a.rec_index = arc.wpos;
  a.n_rec_slots = c.front_cap;
  a.long_min = ca.long_min;
  a.timeout_ns = ca.timeout_ns;
  a.recs = c.recs;
  a.match_ptr = nullptr;
  return a;
}

// Decodes a batch's work list into cache slots: the same three passes as a
// seek, archive by archive.
template <int PASS>
__global__ void ACE_PASS_BOUNDS(PASS) cache_decode_kernel(CacheDecodeArgs ca) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint8_t* wsm = smem + (size_t)wid * ca.warp_smem;
  const CacheArgs& c = ca.c;
  if (PASS != PASS_TOKENS && stop_early<PASS>(&c.h->status)) return;
  const uint32_t epoch = *(volatile uint32_t*)&c.h->epoch;
  const uint32_t n_items = *(volatile uint32_t*)&c.h->n_work;
  if (ACE_PASS_CTA(PASS)) {
    cta_blocks(n_items, &c.h->ticket3, [&](uint32_t it) {
      uint32_t b;
      const DecodeArgs a = cache_job(ca, it, b);
      const uint32_t ntok = __ldg(reinterpret_cast<const uint32_t*>(a.dir + b) + 12);
      match_cta<true, true, PASS == PASS_PLACE>(a, smem, b, ntok ? ntok - 1 : 0, epoch, 0);
      publish_cta(a.ready, b, epoch);
    });
    return;
  }
  uint32_t* ticket = PASS == PASS_TOKENS ? &c.h->ticket : &c.h->ticket2;
  while (true) {
    uint32_t it = 0;
    if (lane == 0) it = atomicAdd(ticket, 1u);
    it = __shfl_sync(kFull, it, 0);
    if (it >= n_items) break;
    uint32_t b;
    const DecodeArgs a = cache_job(ca, it, b);
    if (PASS == PASS_TOKENS) token_block<true>(a, carve_tok(wsm), b, lane);
    else literal_block<true, kSeekRing>(a, carve_lit(wsm, ca.window, kSeekRing), b, lane);
  }
}

// The entropy layer of a batch's work list, a warp per stream (entropy_kernel).
__global__ void __launch_bounds__(32) cache_entropy_kernel(CacheDecodeArgs ca) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x, n_jobs = 3 * *(volatile uint32_t*)&ca.c.h->n_work;
  for (uint32_t j = blockIdx.x; j < n_jobs; j += gridDim.x) {
    uint32_t b;
    const DecodeArgs a = cache_job(ca, j / 3, b);
    stream_job<true, kSeekRing>(a, smem, b, j % 3, lane);
  }
}

// Each request's bytes from the cache slots to its place in the output pool:
// CTAs (., y) take the request's blocks y apart, a warp each.
__global__ void cache_copy_kernel(CacheArgs c, uint8_t* pool) {
  if (*(volatile uint32_t*)&c.h->status) return;  // a failed batch copies nothing
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint64_t B = (uint64_t)1 << c.log2B;
  for (uint32_t r = blockIdx.x; r < c.n_reqs; r += gridDim.x) {
    const ace_seek_req q = c.reqs[r];
    const CacheArc& ca = c.arcs[q.archive];
    if (q.len == 0) continue;
    // a warp per block the request covers: one slot lookup, then a batched copy
    const uint64_t k0 = q.coord >> c.log2B, k1 = (q.coord + q.len - 1) >> c.log2B;
    for (uint64_t k = k0 + blockIdx.y * nw + wid; k <= k1; k += nw * gridDim.y) {
      const uint64_t lo = max(k << c.log2B, q.coord), hi = min((k + 1) << c.log2B, q.coord + q.len);
      const uint32_t slot = __ldg(ca.slot_of + k);
      warp_copy(pool + q.out_off + (lo - q.coord), c.slots + ((uint64_t)slot << c.log2B) + (lo & (B - 1)), hi - lo,
                lane);
    }
  }
}

// New cache epoch: every cached block is forgotten, every slot is free
// (owners left behind no longer match their blocks' flags).
__global__ void cache_reset_kernel(CacheHdr* h) {
  h->epoch += 1;
  h->n_cached = 0;
  h->hand = 0;
  h->ticket = 0;
  h->ticket2 = 0;
  h->ticket3 = 0;
  h->n_work = 0;
}

// ------------------------------------------------------------ verification

__device__ __forceinline__ uint8_t pattern_byte(uint32_t seed, uint64_t i) {
  uint64_t z = (i + 1) * 0x9e3779b97f4a7c15ull ^ ((uint64_t)seed << 32 | seed);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return (uint8_t)(z ^ (z >> 31));
}

__global__ void fill_pattern_kernel(uint8_t* p, uint64_t n, uint32_t seed) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    p[i] = pattern_byte(seed, i);
}

__global__ void count_pattern_mismatch_kernel(const uint8_t* p, uint64_t n, uint32_t seed, uint64_t* bad) {
  uint64_t c = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    c += p[i] != pattern_byte(seed, i);
  if (c) atomicAdd((unsigned long long*)bad, (unsigned long long)c);
}

// New call on a scratch buffer: next epoch, ticket back to zero.
__global__ void begin_call_kernel(ScratchHdr* sh) {
  const uint32_t e = (sh->epoch + 1) & ~kPendingFlag;  // never 0, never with the pending bit
  sh->epoch = e ? e : 1u;
  sh->ticket = 0;
  sh->ticket2 = 0;
  sh->ticket3 = 0;
}

// FNV-1a 64 (Fowler/Noll/Vo): sequential by definition, one thread.  The
// bytes arrive in aligned 16-byte vectors, kFnvBatch at a time, the next
// batch's loads issued before the current batch is hashed, so the hash chain
// rather than the load latency sets the time.  The state is kept as two
// 32-bit halves: with the prime P = 2^40 + 0x1b3, h P mod 2^64 has low word
// (lo 0x1b3) mod 2^32 and high word ((lo 0x1b3) >> 32) + hi 0x1b3 + (lo << 8),
// so the chain from byte to byte runs through the low word alone.
constexpr uint32_t kFnvBatch = 8;
__global__ void fnv_kernel(const uint8_t* p, uint64_t n, uint64_t* out) {
  uint32_t lo = 0x84222325u, hi = 0xcbf29ce4u;  // the 64-bit offset basis
  auto step = [&](uint32_t b) {
    lo ^= b;
    hi = hi * 0x1b3u + __umulhi(lo, 0x1b3u) + (lo << 8);  // beside the low word's chain
    lo *= 0x1b3u;
  };
  uint64_t i = 0;
  for (; i < n && (reinterpret_cast<uintptr_t>(p + i) & 15); i++) step(p[i]);
  const uint4* v = reinterpret_cast<const uint4*>(p + i);
  const uint64_t nb = (n - i) / (16 * kFnvBatch);  // whole batches
  uint4 cur[kFnvBatch], nxt[kFnvBatch];
#pragma unroll
  for (uint32_t k = 0; k < kFnvBatch; k++) cur[k] = nb ? v[k] : make_uint4(0, 0, 0, 0);
  for (uint64_t q = 0; q < nb; q++) {
#pragma unroll
    for (uint32_t k = 0; k < kFnvBatch; k++) nxt[k] = q + 1 < nb ? v[(q + 1) * kFnvBatch + k] : cur[k];
#pragma unroll
    for (uint32_t k = 0; k < kFnvBatch; k++) {
      const uint32_t w[4] = {cur[k].x, cur[k].y, cur[k].z, cur[k].w};
#pragma unroll
      for (uint32_t j = 0; j < 16; j++) step((w[j >> 2] >> (8 * (j & 3))) & 0xffu);
    }
#pragma unroll
    for (uint32_t k = 0; k < kFnvBatch; k++) cur[k] = nxt[k];
  }
  for (i += nb * 16 * kFnvBatch; i < n; i++) step(p[i]);
  *out = ((uint64_t)hi << 32) | lo;
}

}  // namespace

// ---------------------------------------------------------------- host side

struct ace_index {
  const uint8_t* d_arc;
  uint64_t arc_bytes;
  ace_file_header h;
  uint8_t* d_mem;
  uint64_t mem_bytes;
  IndexHdr* d_ih;
  uint32_t* d_level;
  uint32_t* d_order;
  const uint32_t* d_dep_ptr;
  const uint32_t* d_dep_iv;
  uint64_t n_iv;
  uint32_t n_levels;
  uint32_t max_ntok;
  uint64_t n_matches;
  uint64_t* d_match_ptr;
  uint32_t* d_lv_count;  // blocks per level
  int device;
  int num_sms;
  ace_tune tune;
  // occupancy of the decode kernels, per (seek?, pass, warps per CTA, window)
  mutable int occ_cache[2][4][9][9];  // [3]: the fused pass
  mutable int occ_level[9];  // the per-level match kernels: a warp per block by warps per CTA; [0] a CTA per block
  // whole decodes resolve matches with one launch per level when there are
  // at most kMaxLevelLaunches levels: level L's blocks are
  // order[level_start[L] .. level_start[L + 1])
  bool by_levels;
  uint32_t level_start[kMaxLevelLaunches + 1];
};

namespace {

struct IndexLayout {
  uint64_t level, order, lv_count, lv_cursor, match_ptr, seen, total;
};

IndexLayout index_layout(uint64_t nb) {
  IndexLayout L;
  uint64_t o = sizeof(IndexHdr);
  L.level = o;
  o = align256(o + 4 * nb);
  L.order = o;
  o = align256(o + 4 * nb);
  L.lv_count = o;
  o = align256(o + 4 * (nb + 1));
  L.lv_cursor = o;
  o = align256(o + 4 * (nb + 1));
  L.match_ptr = o;
  o = align256(o + 8 * (nb + 1));
  L.seen = o;  // a stored index's order check marks each block here
  o = align256(o + 4 * nb);
  L.total = o;
  return L;
}

struct ScratchLayout {
  uint64_t ready, slot_of, work, marks, front0, front1, lv_done, tail, total;
};

// Bytes one seek slot needs: the decoded block and its match records.
inline uint64_t slot_bytes(uint32_t log2B, uint64_t max_ntok) {
  return (1ull << log2B) + 16 * max_ntok;
}

constexpr uint32_t kMaxWindow = 256;
constexpr uint32_t kMaxWarpsPerCta = 8;  // the decode kernel's launch bounds: 256 threads

// One layout serves every call on a scratch buffer, so whole decodes and
// seeks may share it: header, ready flags, the seek's slot map, work list,
// closure marks and frontiers, the fused schedule's level counters, then a
// tail that a whole decode uses for the archive's match records and a seek
// for its block slots followed by their match records.
ScratchLayout scratch_layout(uint64_t nb, uint32_t log2B, uint64_t max_seek, uint64_t max_ntok,
                             uint64_t n_matches) {
  ScratchLayout L;
  uint64_t o = sizeof(ScratchHdr);
  L.ready = o;
  o = align256(o + 4 * nb);
  L.slot_of = o;
  o = align256(o + 4 * nb);
  L.work = o;
  o = align256(o + 4 * nb);
  L.marks = o;
  o = align256(o + 4 * ((nb + 31) / 32));
  L.front0 = o;
  o = align256(o + 4 * nb);
  L.front1 = o;
  o = align256(o + 4 * nb);
  L.lv_done = o;
  o = align256(o + 4 * (nb + 1));
  L.tail = o;
  o = align256(o + std::max<uint64_t>(16 * n_matches, max_seek * slot_bytes(log2B, max_ntok)));
  L.total = o;
  return L;
}

ace_status parse_header(const void* h_header, uint64_t header_bytes, ace_file_header* h) {
  if (!h_header || header_bytes < sizeof(ace_file_header)) return ACE_E_INVAL;
  std::memcpy(h, h_header, sizeof *h);
  if (h->magic != ACE_MAGIC || h->version != ACE_VERSION || h->n_streams != ACE_NSTREAMS ||
      h->n_states != ACE_NSTATES || h->scale_bits != ACE_SCALE_BITS)
    return ACE_E_CORRUPT;
  if (h->off_width != 4 && h->off_width != 5) return ACE_E_CORRUPT;
  if (h->log2_block < ACE_MIN_LOG2_BLOCK || h->log2_block > ACE_MAX_LOG2_BLOCK) return ACE_E_CORRUPT;
  uint64_t B = 1ull << h->log2_block;
  if (h->n_blocks != (h->total_size + B - 1) / B || h->n_blocks > 0xFFFFFFF0ull) return ACE_E_CORRUPT;
  if (h->dir_off < sizeof(ace_file_header) || h->dir_off + h->n_blocks * sizeof(ace_block_dir) > h->deps_off)
    return ACE_E_CORRUPT;
  if (h->deps_off + 4 * (h->n_blocks + 1) > h->payload_off || h->payload_off > h->archive_bytes)
    return ACE_E_CORRUPT;
  if ((h->dir_off & 7) || (h->deps_off & 3) || (h->payload_off & 15) || (h->archive_bytes & 15))
    return ACE_E_CORRUPT;
  return ACE_OK;
}

inline bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

#define CUDA_TRY(x)                         \
  do {                                      \
    if ((x) != cudaSuccess) return ACE_E_CUDA; \
  } while (0)

// Small device headers (status words, counts) come back to the host through
// pinned, mapped host memory written by a one-warp kernel, not through a
// copy: a copy would queue on the copy engines behind large transfers that
// other streams have in flight.  The library's only allocation, 256 KiB of
// host memory, is made once per process; calls take 256-byte slots in turn
// and hold one only while they wait for their stream.
constexpr uint32_t kMirrorSlots = 1024, kMirrorBytes = 256;

__global__ void mirror_kernel(const uint32_t* src, uint32_t* dst, uint32_t words) {
  for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) dst[i] = *(volatile const uint32_t*)(src + i);
}

std::once_flag g_mirror_once;
uint8_t* g_mirror_host = nullptr;
uint8_t* g_mirror_dev = nullptr;
std::atomic<uint32_t> g_mirror_next{0};

// Reads bytes (a multiple of 4, at most 256) at d_src into h_dst after the
// work already on s; synchronises s.
ace_status read_header(const void* d_src, void* h_dst, uint32_t bytes, cudaStream_t s) {
  std::call_once(g_mirror_once, [] {
    void* h = nullptr;
    void* d = nullptr;
    if (cudaHostAlloc(&h, (size_t)kMirrorSlots * kMirrorBytes, cudaHostAllocMapped | cudaHostAllocPortable) !=
        cudaSuccess)
      return;
    if (cudaHostGetDevicePointer(&d, h, 0) != cudaSuccess) {
      cudaFreeHost(h);
      return;
    }
    g_mirror_host = static_cast<uint8_t*>(h);
    g_mirror_dev = static_cast<uint8_t*>(d);
  });
  if (!g_mirror_host || bytes > kMirrorBytes || (bytes & 3)) return ACE_E_CUDA;
  const uint32_t k = g_mirror_next.fetch_add(1) % kMirrorSlots;
  mirror_kernel<<<1, 64, 0, s>>>(static_cast<const uint32_t*>(d_src),
                                 reinterpret_cast<uint32_t*>(g_mirror_dev + (size_t)k * kMirrorBytes), bytes / 4);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaStreamSynchronize(s));
  std::memcpy(h_dst, (const void*)(g_mirror_host + (size_t)k * kMirrorBytes), bytes);
  return ACE_OK;
}

// Launch shape of one three-pass decode: per pass the shared memory of a warp
// (tokens: tables, two rings and escape values; literals: tables, a ring and
// the token window; matches: the match records) and the grid.
struct Launch {
  uint32_t warps, chunk;
  uint32_t smem[4];  // [PASS_FUSED]: the largest of the three (its phases reuse one area)
  uint32_t grid[4];
  uint64_t timeout;
  uint32_t schedule;
  uint32_t long_min;       // the copy-width knob as the long class's shortest match
  uint32_t match_threads;  // threads of the match pass's CTAs, a block each
  bool warp_match;         // ... or a block per warp (PASS_WARP)
};

// The match pass of a level of many blocks, by the archive's matches per 16 KiB.
// Dense archives, in blocks of at least 512 bytes: a CTA per block.  It costs a
// sweep over the block whatever the matches, a warp's rows cost by the match.
// Match pass of 48 MiB of text with ever fewer matches, us by CTAs (rows): 4 KiB
// blocks 155 (245) at 774, 124 (156) at 512, 110 (108) at 349; 1 KiB 142 (185) at
// 647, 110 (120) at 442, 91 (84) at 293; 512 bytes 147 (180) at 576, 130 (126) at
// 401; 256 bytes 392 (203) at 505.  In larger blocks CTAs are ahead from fewer on
// (128 MiB of spread copies, 16 KiB blocks: 210 (261) at 349, 151 (147) at 190);
// one line for all keeps FASTQ, 100 to 220, with the rows that suit 16 KiB blocks.
constexpr double kCtaMatches = 400;
constexpr uint32_t kCtaLog2B = 9;
// Others go by warps: in rows, unless matches are few and, by the archive's size,
// long.  128 MiB, us by rows (rounds): genome (18 matches per 16 KiB, of 880 bytes)
// 126 (109) in 16 KiB blocks, 79 (74) in 4 KiB; copies of 32 bytes at 41 per 16
// KiB 52 (85) and 36 (48), in 64 KiB blocks 99 (197); of 17 bytes at 20 in 64 KiB
// blocks 62 (81); of 490 at 16 68 (70), 42 (40); FASTQ 128 (177), 82 (100).
constexpr double kRowMatches = 48;
inline bool dense_matches(uint64_t matches, uint64_t bytes) {
  return (double)matches * 16384 >= kCtaMatches * (double)bytes;
}
// Levels of at most this many blocks per SM: a CTA per block whatever the archive.
// Match pass, us by CTAs (warps) at 2, 4, 6 and 12 blocks per SM: genome in 16 KiB
// blocks 52 (74), 60 (62), 68 (60), 101 (102); FASTQ 40 (52), 46 (53), 53 (52), 70
// (54); genome in 64 KiB blocks 122 (124), 126 (124), 144 (140), 267 (148).
constexpr uint32_t kCtaLevel = 4;
// Calls of few blocks decode a stream per warp (entropy_kernel) and leave the
// literals to the match pass, whose CTAs place them.  That shortens a block's
// chain and spreads it wider, and costs more instructions per literal, so the
// limit depends on the literals.  Against the token and literal passes, us:
// FASTQ 2 MiB 99 (109), 4 MiB 132 (128), 16 MiB 161 (150); text 2 MiB 81
// (158), 16 MiB 177 (224), 32 MiB 270 (271); genome 2 MiB 95 (105), 16 MiB 139
// (158), 32 MiB 167 (163).  Word text in 64 KiB blocks: 1 MiB 152 (361), 16
// MiB 304 (496).
constexpr uint32_t kSplitBlocks = 1;       // whole decodes, blocks per SM
constexpr uint32_t kSplitBlocksLight = 8;  // ... of archives with many matches or few compressed bytes (few literals)
// ... in blocks up to this: where literals are many, placing those of a large
// block takes its CTA longer than the shorter chain saves.  FASTQ in 64 KiB
// blocks: 1.5 MiB 339 (308), 9 MiB 528 (386), 600 KB in 10 levels 1117 (464); in
// 32 KiB blocks 1.5 MiB 154 (170), 19 levels 695 (355).
constexpr uint32_t kSplitLog2B = 14;
// ... of at most this many levels, unless dense and in blocks of 4 KiB or more:
// placing the literals is a part of every level's time.  26 blocks written with
// the most recent sources first, us split (passes): FASTQ in 16 KiB blocks, 26
// levels, 392 (273), 4 KiB, 21 levels, 201 (175); mixed data in 1 KiB blocks, 27
// levels, 236 (208), in 4 KiB blocks 249 (279).
constexpr uint32_t kSplitLevels = 8;
// Seeks decode a stream per warp too: dense archives, and others in blocks up to
// kSplitLog2B unless few blocks of few matches are wanted (one long stream each,
// no shorter alone).  Us (in two passes): FASTQ in 64 KiB blocks 1 byte 375 (312),
// 7 MiB 515 (400); genome in 4 KiB blocks 1 block 59 (50), 51 blocks 58 (57), 257
// blocks 76 (79), in 16 KiB blocks 1 block 102 (97), 65 blocks 111 (118), in 1 KiB
// blocks 1 block 48 (48), 17 blocks 46 (49).  By target blocks: FASTQ 1 block 154
// (179), 1024 259 (275), 2048 366 (350); text 239 (326), 402 (476), 591 (639),
// 4096 1048 (986); genome 119 (122), 195 (203), 272 (272).
constexpr uint64_t kSplitSeek = 1024;
constexpr uint64_t kSplitFew = 48;
constexpr uint32_t kSplitFewLog2B = 12;
// Seek batches, by target blocks where the host has the requests, us (in two
// passes): 1900 blocks over four profiles 301 (371); genome, 1152 blocks of 16 KiB
// 204 (226), 1040 of 4 KiB 126 (133), 4224 of them 264 (242), 4112 of 1 KiB 159
// (163), 16512 of them 405 (322); text 361 (428), 185 (218), 400 (395), 215 (213)
// and 538 (462).  Else by their number, which says less: genome, 64 requests of 16
// KiB 162 (180) in 16 KiB blocks, 97 (103) in 4 KiB, 128 of them 172 (190) and 107
// (117), but 128 requests of 128 KiB in 1 KiB blocks 400 (318).
constexpr uint64_t kSplitBatch = 3072;
constexpr uint32_t kSplitReqs = 64;

// Archives of more than 32 levels: the match pass by warps, where a block is
// short or has few matches.  600 KB written with the most recent sources first,
// us by CTAs (warps by rows): text in 256-byte blocks 4811 (3657), 1 KiB 3669
// (6201), 16 KiB 1270 (5749); FASTQ in 1 KiB blocks 239 (202), 4 KiB 469 (390), 8
// KiB 417 (427), 16 KiB 315 (468).
inline bool deep_by_warps(const ace_index* x) {
  const bool dense = x->h.total_size && dense_matches(x->n_matches, x->h.total_size);
  return !x->by_levels && (x->h.log2_block < 9 || (!dense && x->h.log2_block < 13));
}

template <class K>
ace_status occupancy(K kernel, int device, uint32_t warps, size_t smem, int* occ) {
  int optin = 0;
  CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
  cudaFuncAttributes fa;
  CUDA_TRY(cudaFuncGetAttributes(&fa, kernel));
  const size_t dyn_max = (size_t)optin - fa.sharedSizeBytes;  // the kernel's static shared memory counts too
  if (smem > dyn_max) {
    *occ = -1;  // this many warps with this much shared memory do not fit one CTA
    return ACE_OK;
  }
  // allow every configuration up to the opt-in limit, so launches planned
  // earlier with other shapes stay valid
  CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn_max));
  int o = 0;
  CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kernel, 32 * warps, smem));
  *occ = o > 0 ? o : -1;
  return ACE_OK;
}

// occ_cache: 4 x 9 x 9 ints (pass, warps per CTA, window / 32), 0 = unknown;
// k3 is the fused pass
template <class K0, class K1, class K2, class K3>
ace_status plan_launch(const ace_index* idx, const ace_tune* tune, uint32_t log2B, uint64_t max_items,
                       K0 k0, K1 k1, K2 k2, K3 k3, int* occ_cache, Launch* L, uint32_t lit_ring, bool few,
                       bool warp_match) {
  ace_tune t = tune ? *tune : idx->tune;
  L->warps = t.warps_per_cta ? t.warps_per_cta : 4;
  L->chunk = t.chunk_tokens ? t.chunk_tokens : 128;
  if (L->warps > kMaxWarpsPerCta || (L->chunk & 31) || L->chunk > kMaxWindow) return ACE_E_INVAL;
  L->timeout = t.wait_timeout_ns ? t.wait_timeout_ns : kDefaultTimeoutNs;
  L->schedule = t.schedule;
  if (L->schedule > ACE_SCHEDULE_FUSED) return ACE_E_INVAL;
  if (t.copy_width != 0 && t.copy_width != 8 && t.copy_width != 16) return ACE_E_INVAL;
  // the library's choice (0): 16-byte pieces from 33 bytes (genome 1 GiB
  // 1.37 ms against 1.43; FASTQ and text unchanged)
  L->long_min = t.copy_width == 8 ? kLongMinNarrow : kLongMinWide;
  // automatic: the pass schedule, measured faster on every profile (the
  // fused launch's match jobs of the first levels form a serial chain)
  if (L->schedule == ACE_SCHEDULE_AUTO) L->schedule = ACE_SCHEDULE_PASSES;
  L->smem[PASS_TOKENS] = tok_smem_bytes(esc_cap(log2B));
  L->smem[PASS_LITERALS] = lit_smem_bytes(L->chunk, lit_ring);
  L->warp_match = warp_match;
  L->match_threads = warp_match ? 32 * L->warps : cta_threads(log2B, few);
  // per CTA; the other passes': per warp
  L->smem[PASS_MATCH] = warp_match ? L->warps * kMatchSmem : cta_smem_bytes(log2B, L->match_threads);
  L->smem[PASS_FUSED] = std::max(std::max(L->smem[PASS_TOKENS], L->smem[PASS_LITERALS]), kMatchSmem);
  int per[4];
  for (int p = 0; p < 4; p++) {
    int& c = occ_cache[(p * 9 + L->warps) * 9 + L->chunk / 32];
    if (c == 0) {
      const size_t smem = (size_t)L->warps * L->smem[p];
      ace_status rc = p == 0   ? occupancy(k0, idx->device, L->warps, smem, &c)
                      : p == 1 ? occupancy(k1, idx->device, L->warps, smem, &c)
                      : p == 2 ? occupancy(k2, idx->device, L->match_threads / 32, L->smem[PASS_MATCH], &c)
                               : occupancy(k3, idx->device, L->warps, smem, &c);
      if (rc) return rc;
    }
    if (c < 0) return ACE_E_INVAL;
    per[p] = c;
    if (t.ctas_per_sm && (int)t.ctas_per_sm < per[p]) per[p] = (int)t.ctas_per_sm;
  }
  uint64_t need = std::max<uint64_t>(1, (max_items + L->warps - 1) / L->warps);
  for (int p = 0; p < 4; p++) L->grid[p] = (uint32_t)std::min<uint64_t>((uint64_t)idx->num_sms * per[p], need);
  if (!warp_match)
    L->grid[PASS_MATCH] =
        (uint32_t)std::min<uint64_t>((uint64_t)idx->num_sms * per[PASS_MATCH], std::max<uint64_t>(1, max_items));
  return ACE_OK;
}

template <bool SEEK>
ace_status plan_index_launch(const ace_index* idx, const ace_tune* tune, uint64_t max_items, Launch* L) {
  const bool warps = deep_by_warps(idx);
  return plan_launch(idx, tune, idx->h.log2_block, max_items, decode_kernel<SEEK, PASS_TOKENS>,
                     decode_kernel<SEEK, PASS_LITERALS>,
                     warps ? decode_kernel<SEEK, PASS_WARP> : decode_kernel<SEEK, PASS_MATCH>,
                     decode_kernel<SEEK, PASS_FUSED>, &idx->occ_cache[SEEK][0][0][0], L, SEEK ? kSeekRing : kRing, SEEK,
                     warps);
}

// Launches the passes in the mask (bit p: pass p) in order on s, each with
// its own shared memory per warp.
template <class K0, class K1, class K2, class Args>
void launch_passes(const Launch& L, uint32_t passes, K0 k0, K1 k1, K2 k2, Args a, cudaStream_t s) {
  const uint32_t th = 32 * L.warps;
  if (passes & 1) {
    a.warp_smem = L.smem[0];
    k0<<<L.grid[0], th, (size_t)L.warps * L.smem[0], s>>>(a);
  }
  if (passes & 2) {
    a.warp_smem = L.smem[1];
    k1<<<L.grid[1], th, (size_t)L.warps * L.smem[1], s>>>(a);
  }
  if (passes & 4) {
    a.warp_smem = kMatchSmem;  // (a warp per block)
    k2<<<L.grid[2], L.match_threads, L.smem[2], s>>>(a);
  }
}

// The fused pass: one launch for the whole decode.
template <class K3, class Args>
void launch_fused(const Launch& L, K3 k3, Args a, cudaStream_t s) {
  a.warp_smem = L.smem[PASS_FUSED];
  k3<<<L.grid[PASS_FUSED], 32 * L.warps, (size_t)L.warps * L.smem[PASS_FUSED], s>>>(a);
}

// A seek after its closure kernel, over the level-ordered work list: by the pass
// schedule (the automatic choice) the entropy layer a stream per warp or in two
// passes over the list, then one match launch whose blocks wait, bounded, on
// pending members of the closure; or one fused launch that waits the same way.
// (One launch per level, as whole decodes by passes do, is slower for a seek's
// hundred-odd blocks.)
void launch_seek(const ace_index* idx, const Launch& L, const DecodeArgs& a, uint64_t targets, cudaStream_t s) {
  const bool dense = dense_matches(idx->n_matches, idx->h.total_size);
  const bool few = (double)idx->n_matches * 16384 < kRowMatches * (double)idx->h.total_size;
  const bool split = targets <= kSplitSeek && !L.warp_match &&
                     (dense || (idx->h.log2_block <= kSplitLog2B &&
                                (!few || idx->h.log2_block < kSplitFewLog2B || targets > kSplitFew)));
  if (L.schedule == ACE_SCHEDULE_FUSED) {
    launch_fused(L, decode_kernel<true, PASS_FUSED>, a, s);
  } else if (split) {
    const uint32_t grid = (uint32_t)std::min<uint64_t>(3ull * a.n_slots, 16ull * idx->num_sms);
    entropy_kernel<true><<<grid, 32, job_smem_bytes(a.esc_cap, kSeekRing), s>>>(a);
    decode_kernel<true, PASS_PLACE><<<L.grid[PASS_MATCH], L.match_threads, L.smem[PASS_MATCH], s>>>(a);
  } else {
    launch_passes(L, 7, decode_kernel<true, PASS_TOKENS>, decode_kernel<true, PASS_LITERALS>,
                  L.warp_match ? decode_kernel<true, PASS_WARP> : decode_kernel<true, PASS_MATCH>, a, s);
  }
}

}  // namespace

extern "C" {

const char* ace_status_str(ace_status s) {
  switch (s) {
    case ACE_OK: return "ACE_OK";
    case ACE_E_INVAL: return "ACE_E_INVAL";
    case ACE_E_CORRUPT: return "ACE_E_CORRUPT";
    case ACE_E_RANGE: return "ACE_E_RANGE";
    case ACE_E_NOMEM: return "ACE_E_NOMEM";
    case ACE_E_TIMEOUT: return "ACE_E_TIMEOUT";
    case ACE_E_CUDA: return "ACE_E_CUDA";
    default: return "ACE_E_UNKNOWN";
  }
}

ace_status ace_index_size(const void* h_header, uint64_t header_bytes, uint64_t* index_bytes) {
  if (!index_bytes) return ACE_E_INVAL;
  ace_file_header h;
  ace_status rc = parse_header(h_header, header_bytes, &h);
  if (rc) return rc;
  *index_bytes = index_layout(h.n_blocks).total;
  return ACE_OK;
}

}  // extern "C"

namespace {

// A new host handle over the archive and index memory, and the arguments of
// the index kernels.  Returns null with *rc set on failure.
ace_index* index_handle(const void* d_archive, uint64_t archive_bytes, const void* h_header, uint64_t header_bytes,
                        void* d_index_mem, uint64_t index_bytes, IndexArgs* a, ace_status* rc) {
  *rc = ACE_E_INVAL;
  if (!d_index_mem || (!d_archive && archive_bytes)) return nullptr;
  if (!aligned(d_archive, 16) || !aligned(d_index_mem, 256)) return nullptr;
  ace_file_header h;
  *rc = parse_header(h_header, header_bytes, &h);
  if (*rc) return nullptr;
  *rc = ACE_E_CORRUPT;
  if (h.archive_bytes > archive_bytes) return nullptr;
  IndexLayout L = index_layout(h.n_blocks);
  *rc = ACE_E_NOMEM;
  if (index_bytes < L.total) return nullptr;
  ace_index* idx = new (std::nothrow) ace_index();
  if (!idx) return nullptr;
  idx->d_arc = static_cast<const uint8_t*>(d_archive);
  idx->arc_bytes = archive_bytes;
  idx->h = h;
  idx->d_mem = static_cast<uint8_t*>(d_index_mem);
  idx->mem_bytes = index_bytes;
  idx->d_ih = reinterpret_cast<IndexHdr*>(idx->d_mem);
  idx->d_level = reinterpret_cast<uint32_t*>(idx->d_mem + L.level);
  idx->d_order = reinterpret_cast<uint32_t*>(idx->d_mem + L.order);
  idx->d_dep_ptr = reinterpret_cast<const uint32_t*>(idx->d_arc + h.deps_off);
  idx->tune = ace_tune{};
  *rc = ACE_E_CUDA;
  if (cudaGetDevice(&idx->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&idx->num_sms, cudaDevAttrMultiProcessorCount, idx->device) != cudaSuccess) {
    delete idx;
    return nullptr;
  }
  // the interval table's bounds are checked on the device with the rest
  idx->d_dep_iv = reinterpret_cast<const uint32_t*>(idx->d_arc + h.deps_off + 4 * (h.n_blocks + 1));
  a->arc = idx->d_arc;
  a->dir = reinterpret_cast<const ace_block_dir*>(idx->d_arc + h.dir_off);
  a->dep_ptr = idx->d_dep_ptr;
  a->dep_iv = idx->d_dep_iv;
  a->ih = idx->d_ih;
  a->level = idx->d_level;
  a->order = idx->d_order;
  a->lv_count = reinterpret_cast<uint32_t*>(idx->d_mem + L.lv_count);
  a->lv_cursor = reinterpret_cast<uint32_t*>(idx->d_mem + L.lv_cursor);
  a->match_ptr = reinterpret_cast<uint64_t*>(idx->d_mem + L.match_ptr);
  idx->d_match_ptr = a->match_ptr;
  idx->d_lv_count = a->lv_count;
  a->nb = h.n_blocks;
  a->total = h.total_size;
  a->payload_off = h.payload_off;
  a->arc_bytes = h.archive_bytes;
  a->deps_off = h.deps_off;
  a->max_iv = (h.payload_off - h.deps_off - 4 * (h.n_blocks + 1)) / 8;
  a->log2B = h.log2_block;
  a->w = h.off_width;
  *rc = ACE_OK;
  return idx;
}

// The handle's copies of what the index header holds.
ace_status index_adopt(ace_index* idx, const IndexHdr& ih) {
  if (ih.status) return (ace_status)ih.status;
  idx->n_iv = ih.n_iv;
  idx->max_ntok = ih.max_ntok;
  idx->n_levels = ih.n_levels;
  idx->n_matches = ih.n_matches;
  idx->by_levels = ih.n_levels <= kMaxLevelLaunches;
  if (idx->by_levels) {
    idx->level_start[0] = 0;
    for (uint32_t l = 0; l < ih.n_levels; l++) idx->level_start[l + 1] = idx->level_start[l] + ih.lvc[l];
    if (idx->level_start[ih.n_levels] != idx->h.n_blocks) return ACE_E_CORRUPT;
  }
  return ACE_OK;
}

// FNV-1a 64 of host bytes (the stored index's checksum).
uint64_t host_fnv1a64(const uint8_t* p, uint64_t n) {
  uint64_t h = 0xcbf29ce484222325ull;
  for (uint64_t i = 0; i < n; i++) {
    h ^= p[i];
    h *= 0x100000001b3ull;
  }
  return h;
}

// Header of a stored index: the archive header it belongs to, the index
// memory's size and checksum; the index memory follows.
struct IndexBlobHdr {
  uint32_t magic;  // "ACEI"
  uint32_t version;
  ace_file_header arc;
  uint64_t index_bytes;
  uint64_t fnv;
  uint8_t pad[168];
};
static_assert(sizeof(IndexBlobHdr) == 256, "stored index header");
constexpr uint32_t kIndexMagic = 0x49454341u;  // "ACEI"

}  // namespace

extern "C" {

ace_status ace_index_build(const void* d_archive, uint64_t archive_bytes, const void* h_header,
                           uint64_t header_bytes, void* d_index_mem, uint64_t index_bytes, cudaStream_t s,
                           ace_index** out) {
  if (!out) return ACE_E_INVAL;
  IndexArgs a;
  ace_status rc;
  ace_index* idx = index_handle(d_archive, archive_bytes, h_header, header_bytes, d_index_mem, index_bytes, &a, &rc);
  if (!idx) return rc;
  auto bail = [&](ace_status r) {
    delete idx;
    return r;
  };
  const ace_file_header& h = idx->h;
  if (cudaMemsetAsync(idx->d_mem, 0, index_layout(h.n_blocks).total, s) != cudaSuccess) return bail(ACE_E_CUDA);
  if (h.n_blocks) {
    // every step on the device, each skipping once the header holds an
    // error; the host reads the header once at the end
    uint32_t g = (uint32_t)((h.n_blocks + 255) / 256);
    validate_kernel<<<g, 256, 0, s>>>(a);
    match_scan_kernel<<<1, 1024, 0, s>>>(a);
    const uint32_t gs = (uint32_t)std::min<uint64_t>((h.n_blocks + 7) / 8, (uint64_t)idx->num_sms * 8);
    for (uint32_t k = 0; k < kLevelSweeps; k++) levels_sweep_kernel<<<gs, 256, 0, s>>>(a, k);
    levels_kernel<<<1, 1024, 0, s>>>(a);
    level_hist_kernel<<<g, 256, 0, s>>>(a);
    level_scan_kernel<<<1, 1024, 0, s>>>(a);
    level_scatter_kernel<<<g, 256, 0, s>>>(a);
    IndexHdr ih;
    if (read_header(idx->d_ih, &ih, sizeof ih, s) != ACE_OK) return bail(ACE_E_CUDA);
    rc = index_adopt(idx, ih);
    if (rc) return bail(rc);
  }
  *out = idx;
  return ACE_OK;
}

ace_status ace_index_export_size(const ace_index* idx, uint64_t* bytes) {
  if (!idx || !bytes) return ACE_E_INVAL;
  *bytes = sizeof(IndexBlobHdr) + index_layout(idx->h.n_blocks).total;
  return ACE_OK;
}

ace_status ace_index_export(const ace_index* idx, void* h_blob, uint64_t blob_bytes, cudaStream_t s) {
  if (!idx || !h_blob) return ACE_E_INVAL;
  const uint64_t n = index_layout(idx->h.n_blocks).total;
  if (blob_bytes < sizeof(IndexBlobHdr) + n) return ACE_E_NOMEM;
  uint8_t* p = static_cast<uint8_t*>(h_blob);
  CUDA_TRY(cudaMemcpyAsync(p + sizeof(IndexBlobHdr), idx->d_mem, n, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  IndexBlobHdr bh{};
  bh.magic = kIndexMagic;
  bh.version = 1;
  bh.arc = idx->h;
  bh.index_bytes = n;
  bh.fnv = host_fnv1a64(p + sizeof(IndexBlobHdr), n);
  std::memcpy(p, &bh, sizeof bh);
  return ACE_OK;
}

ace_status ace_index_import(const void* d_archive, uint64_t archive_bytes, const void* h_header, uint64_t header_bytes,
                            const void* h_blob, uint64_t blob_bytes, void* d_index_mem, uint64_t index_bytes,
                            cudaStream_t s, ace_index** out) {
  if (!out || !h_blob || blob_bytes < sizeof(IndexBlobHdr)) return ACE_E_INVAL;
  IndexArgs a;
  ace_status rc;
  ace_index* idx = index_handle(d_archive, archive_bytes, h_header, header_bytes, d_index_mem, index_bytes, &a, &rc);
  if (!idx) return rc;
  auto bail = [&](ace_status r) {
    delete idx;
    return r;
  };
  const ace_file_header& h = idx->h;
  const uint64_t n = index_layout(h.n_blocks).total;
  IndexBlobHdr bh;
  std::memcpy(&bh, h_blob, sizeof bh);
  const uint8_t* body = static_cast<const uint8_t*>(h_blob) + sizeof(IndexBlobHdr);
  // the stored index must belong to this archive and arrive whole
  if (bh.magic != kIndexMagic || bh.version != 1 || std::memcmp(&bh.arc, &h, sizeof h) != 0 || bh.index_bytes != n ||
      blob_bytes < sizeof(IndexBlobHdr) + n || host_fnv1a64(body, n) != bh.fnv)
    return bail(ACE_E_CORRUPT);
  if (cudaMemcpyAsync(idx->d_mem, body, n, cudaMemcpyHostToDevice, s) != cudaSuccess) return bail(ACE_E_CUDA);
  if (h.n_blocks) {
    // the archive is checked as at a build (directory, dependency table,
    // match counts, largest token count: recomputed over the stored values),
    // then the stored levels and order against it
    IndexLayout L = index_layout(h.n_blocks);
    if (cudaMemsetAsync(idx->d_mem, 0, 12, s) != cudaSuccess) return bail(ACE_E_CUDA);  // status words
    uint32_t g = (uint32_t)((h.n_blocks + 255) / 256);
    validate_kernel<<<g, 256, 0, s>>>(a);
    match_scan_kernel<<<1, 1024, 0, s>>>(a);
    const uint32_t gs = (uint32_t)std::min<uint64_t>((h.n_blocks + 7) / 8, (uint64_t)idx->num_sms * 8);
    level_verify_kernel<<<gs, 256, 0, s>>>(a);
    uint32_t* seen = reinterpret_cast<uint32_t*>(idx->d_mem + L.seen);
    if (cudaMemsetAsync(seen, 0, 4 * h.n_blocks, s) != cudaSuccess) return bail(ACE_E_CUDA);
    order_verify_kernel<<<g, 256, 0, s>>>(a, seen);
    IndexHdr ih;
    if (read_header(idx->d_ih, &ih, sizeof ih, s) != ACE_OK) return bail(ACE_E_CUDA);
    rc = index_adopt(idx, ih);
    if (rc) return bail(rc);
  }
  *out = idx;
  return ACE_OK;
}

ace_status ace_index_info(const ace_index* idx, ace_info* info) {
  if (!idx || !info) return ACE_E_INVAL;
  info->total_size = idx->h.total_size;
  info->n_blocks = idx->h.n_blocks;
  info->archive_bytes = idx->h.archive_bytes;
  info->n_dep_intervals = idx->n_iv;
  info->block_size = 1u << idx->h.log2_block;
  info->off_width = idx->h.off_width;
  info->n_levels = idx->n_levels;
  info->reserved = 0;
  return ACE_OK;
}

ace_status ace_index_levels(const ace_index* idx, uint32_t* h_counts, uint32_t n, cudaStream_t s) {
  if (!idx || (!h_counts && n)) return ACE_E_INVAL;
  const uint32_t m = std::min(n, idx->n_levels);
  if (!m) return ACE_OK;
  if (idx->by_levels) {
    for (uint32_t l = 0; l < m; l++) h_counts[l] = idx->level_start[l + 1] - idx->level_start[l];
    return ACE_OK;
  }
  const IndexLayout L = index_layout(idx->h.n_blocks);
  CUDA_TRY(cudaMemcpyAsync(h_counts, idx->d_mem + L.lv_count, 4ull * m, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  return ACE_OK;
}

ace_status ace_index_set_tune(ace_index* idx, const ace_tune* tune) {
  if (!idx) return ACE_E_INVAL;
  if (tune && (tune->warps_per_cta > kMaxWarpsPerCta || (tune->chunk_tokens & 31) || tune->chunk_tokens > kMaxWindow ||
               tune->schedule > ACE_SCHEDULE_FUSED ||
               (tune->copy_width != 0 && tune->copy_width != 8 && tune->copy_width != 16)))
    return ACE_E_INVAL;
  idx->tune = tune ? *tune : ace_tune{};
  return ACE_OK;
}

ace_status ace_index_free(ace_index* idx) {
  delete idx;
  return ACE_OK;
}

ace_status ace_scratch_size(const ace_index* idx, uint64_t max_seek_blocks, uint64_t* bytes) {
  if (!idx || !bytes) return ACE_E_INVAL;
  *bytes = scratch_layout(idx->h.n_blocks, idx->h.log2_block, max_seek_blocks, idx->max_ntok, idx->n_matches).total;
  return ACE_OK;
}

ace_status ace_scratch_init(const ace_index* idx, void* d_scratch, uint64_t scratch_bytes, cudaStream_t s) {
  if (!idx || !d_scratch || !aligned(d_scratch, 256)) return ACE_E_INVAL;
  ScratchLayout L0 = scratch_layout(idx->h.n_blocks, idx->h.log2_block, 0, idx->max_ntok, idx->n_matches);
  if (scratch_bytes < L0.total) return ACE_E_NOMEM;
  // header, ready flags, and (when present) slot map, work list and marks
  uint64_t clear = L0.tail;
  CUDA_TRY(cudaMemsetAsync(d_scratch, 0, clear, s));
  return ACE_OK;
}

}  // extern "C"

namespace {

// passes: bit 0 the token pass (with the call's header reset before it),
// bit 1 the literal pass, bit 2 the match pass.
ace_status decode_all_passes(const ace_index* idx, uint32_t passes, void* d_out, uint64_t out_bytes, void* d_scratch,
                             uint64_t scratch_bytes, const ace_tune* tune, cudaStream_t s) {
  if (!idx || !d_scratch || (!d_out && idx->h.total_size)) return ACE_E_INVAL;
  if (!aligned(d_scratch, 256) || !aligned(d_out, 16)) return ACE_E_INVAL;
  if (out_bytes < idx->h.total_size) return ACE_E_NOMEM;
  ScratchLayout SL = scratch_layout(idx->h.n_blocks, idx->h.log2_block, 0, idx->max_ntok, idx->n_matches);
  if (scratch_bytes < SL.total) return ACE_E_NOMEM;
  if (!idx->h.n_blocks) return ACE_OK;
  Launch L;
  ace_status rc = plan_index_launch<false>(idx, tune, idx->h.n_blocks, &L);
  if (rc) return rc;
  ScratchHdr* sh = static_cast<ScratchHdr*>(d_scratch);
  DecodeArgs a{};
  a.arc = idx->d_arc;
  a.dir = reinterpret_cast<const ace_block_dir*>(idx->d_arc + idx->h.dir_off);
  a.payload_off = idx->h.payload_off;
  a.total = idx->h.total_size;
  a.nb = idx->h.n_blocks;
  a.log2B = idx->h.log2_block;
  a.w = idx->h.off_width;
  a.window = L.chunk;
  a.max_ntok = idx->max_ntok;
  a.esc_cap = esc_cap(a.log2B);
  a.warp_smem = L.smem[PASS_TOKENS];
  a.n_items = (uint32_t)idx->h.n_blocks;
  a.items = idx->d_order;
  a.out = static_cast<uint8_t*>(d_out);
  a.sh = sh;
  a.ready = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(d_scratch) + SL.ready);
  a.timeout_ns = L.timeout;
  a.recs = reinterpret_cast<MatchRec*>(static_cast<uint8_t*>(d_scratch) + SL.tail);
  a.match_ptr = idx->d_match_ptr;
  a.level = idx->d_level;
  a.long_min = L.long_min;
  if (passes == 7 && L.schedule == ACE_SCHEDULE_FUSED) {
    // one launch over the (level, block) order; the level counters start at 0
    a.lv_done = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(d_scratch) + SL.lv_done);
    a.lv_count = idx->d_lv_count;
    CUDA_TRY(cudaMemsetAsync(a.lv_done, 0, 4ull * idx->n_levels, s));
    begin_call_kernel<<<1, 1, 0, s>>>(sh);
    launch_fused(L, decode_kernel<false, PASS_FUSED>, a, s);
    CUDA_TRY(cudaGetLastError());
    return ACE_OK;
  }
  // a warp per block by rounds, a warp per block by rows, a CTA per block:
  // by the archive's matches per 16 KiB
  const bool dense = dense_matches(idx->n_matches, idx->h.total_size);
  const bool by_cta = dense && idx->h.log2_block >= kCtaLog2B;
  const bool rows = (double)idx->n_matches * 16384 >= kRowMatches * (double)idx->h.total_size ||
                    idx->h.archive_bytes >= idx->h.total_size / 2;
  const bool light = dense || idx->h.archive_bytes < idx->h.total_size / 4;
  const bool split = passes == 7 && idx->by_levels && (light || idx->h.log2_block <= kSplitLog2B) &&
                     (idx->n_levels <= kSplitLevels || (dense && idx->h.log2_block >= 12)) &&
                     idx->h.n_blocks <= (uint64_t)(light ? kSplitBlocksLight : kSplitBlocks) * idx->num_sms;
  if (split) entropy_kernel<false><<<3 * a.n_items, 32, job_smem_bytes(a.esc_cap, kSeekRing), s>>>(a);  // (needs no ticket or epoch)
  else if (passes & 1) begin_call_kernel<<<1, 1, 0, s>>>(sh);
  launch_passes(L, split ? 0u : passes & (idx->by_levels ? 3u : 7u), decode_kernel<false, PASS_TOKENS>,
                decode_kernel<false, PASS_LITERALS>,
                L.warp_match ? decode_kernel<false, PASS_WARP> : decode_kernel<false, PASS_MATCH>, a, s);
  if ((passes & 4) && idx->by_levels) {
    const ace_tune t = tune ? *tune : idx->tune;
    int &occ = idx->occ_level[L.warps], &occ_cta = idx->occ_level[0];
    const uint32_t log2B = idx->h.log2_block, few = cta_threads(log2B, true), many = dense_threads(log2B);
    const auto level_kernel = rows ? match_level_kernel<WAY_ROWS> : match_level_kernel<WAY_ROUNDS>;
    if (occ == 0) {
      rc = occupancy(level_kernel, idx->device, L.warps, (size_t)L.warps * kMatchSmem, &occ);
      if (rc) return rc;
    }
    if (occ_cta == 0) {
      int o = 0;  // (levels of few blocks need no count: a CTA each)
      rc = occupancy(match_cta_kernel<512, false>, idx->device, few / 32, cta_smem_bytes(log2B, few), &o);
      if (rc == ACE_OK && o > 0)
        rc = occupancy(match_cta_kernel<256, false>, idx->device, many / 32, cta_smem_bytes(log2B, many), &occ_cta);
      if (rc) return rc;
    }
    if (occ < 0 || occ_cta <= 0) return ACE_E_INVAL;
    auto sms = [&](int per) {
      return (uint64_t)idx->num_sms * (t.ctas_per_sm && (int)t.ctas_per_sm < per ? t.ctas_per_sm : (uint32_t)per);
    };
    for (uint32_t l = 0; l < idx->n_levels; l++) {
      const uint32_t n = idx->level_start[l + 1] - idx->level_start[l];
      if (!n) continue;
      a.items = idx->d_order + idx->level_start[l];
      a.n_items = n;
      a.cur_level = l;
      if (split || n <= kCtaLevel * idx->num_sms) {  // (a split decode's levels: every block by a CTA)
        (split ? match_cta_kernel<512, true> : match_cta_kernel<512, false>)<<<n, few, cta_smem_bytes(log2B, few), s>>>(a);
        continue;
      }
      if (by_cta) {
        match_cta_kernel<256, false><<<(uint32_t)std::min<uint64_t>(sms(occ_cta), n), many, cta_smem_bytes(log2B, many), s>>>(a);
        continue;
      }
      const uint32_t grid = (uint32_t)std::min<uint64_t>(sms(occ), (n + L.warps - 1) / L.warps);
      level_kernel<<<grid, 32 * L.warps, (size_t)L.warps * kMatchSmem, s>>>(a);
    }
  }
  CUDA_TRY(cudaGetLastError());
  return ACE_OK;
}

}  // namespace

extern "C" {

ace_status ace_decode_all(const ace_index* idx, void* d_out, uint64_t out_bytes, void* d_scratch,
                          uint64_t scratch_bytes, const ace_tune* tune, cudaStream_t s) {
  return decode_all_passes(idx, 7, d_out, out_bytes, d_scratch, scratch_bytes, tune, s);
}

ace_status ace_decode_pass(const ace_index* idx, int pass, void* d_out, uint64_t out_bytes, void* d_scratch,
                           uint64_t scratch_bytes, const ace_tune* tune, cudaStream_t s) {
  if (pass != ACE_PASS_TOKENS && pass != ACE_PASS_LITERALS && pass != ACE_PASS_MATCH) return ACE_E_INVAL;
  return decode_all_passes(idx, 1u << pass, d_out, out_bytes, d_scratch, scratch_bytes, tune, s);
}

ace_status ace_seek(const ace_index* idx, uint64_t coord, uint64_t len, void* d_out, uint64_t out_bytes,
                    void* d_scratch, uint64_t scratch_bytes, cudaStream_t s) {
  if (!idx || !d_out || !d_scratch || !aligned(d_scratch, 256)) return ACE_E_INVAL;
  if (len == 0 || coord >= idx->h.total_size || len > idx->h.total_size - coord) return ACE_E_RANGE;
  if (out_bytes < len) return ACE_E_NOMEM;
  uint64_t nb = idx->h.n_blocks;
  uint32_t log2B = idx->h.log2_block;
  ScratchLayout S1 = scratch_layout(nb, log2B, 1, idx->max_ntok, 0);
  if (scratch_bytes < S1.total) return ACE_E_NOMEM;
  // the layout before the slots does not depend on the slot count (a seek
  // never decodes more than n_blocks blocks)
  uint64_t cap = std::min<uint64_t>(nb, (scratch_bytes - S1.tail) / slot_bytes(log2B, idx->max_ntok));
  uint64_t first = coord >> log2B, last = (coord + len - 1) >> log2B;
  if (last - first + 1 > cap) return ACE_E_NOMEM;
  uint8_t* base = static_cast<uint8_t*>(d_scratch);
  ScratchHdr* sh = reinterpret_cast<ScratchHdr*>(base);
  ClosureArgs c;
  c.dep_ptr = idx->d_dep_ptr;
  c.dep_iv = idx->d_dep_iv;
  c.sh = sh;
  c.marks = reinterpret_cast<uint32_t*>(base + S1.marks);
  c.front0 = reinterpret_cast<uint32_t*>(base + S1.front0);
  c.front1 = reinterpret_cast<uint32_t*>(base + S1.front1);
  c.work = reinterpret_cast<uint32_t*>(base + S1.work);
  c.slot_of = reinterpret_cast<uint32_t*>(base + S1.slot_of);
  c.nb = nb;
  c.first = first;
  c.last = last;
  c.cap = cap;
  c.level = idx->by_levels ? idx->d_level : nullptr;
  c.n_levels = idx->n_levels;
  c.ready = reinterpret_cast<uint32_t*>(base + S1.ready);
  Launch L;
  ace_status rc = plan_index_launch<true>(idx, nullptr, cap, &L);
  if (rc) return rc;
  // the fused schedule needs the closure's work list in level order
  if (!idx->by_levels) L.schedule = ACE_SCHEDULE_PASSES;
  c.lv_done = L.schedule == ACE_SCHEDULE_FUSED ? reinterpret_cast<uint32_t*>(base + S1.lv_done) : nullptr;
  closure_kernel<<<kClosureCtas, 1024, 0, s>>>(c);
  DecodeArgs a{};
  a.arc = idx->d_arc;
  a.dir = reinterpret_cast<const ace_block_dir*>(idx->d_arc + idx->h.dir_off);
  a.payload_off = idx->h.payload_off;
  a.total = idx->h.total_size;
  a.nb = nb;
  a.log2B = log2B;
  a.w = idx->h.off_width;
  a.window = L.chunk;
  a.max_ntok = idx->max_ntok;
  a.esc_cap = esc_cap(log2B);
  a.warp_smem = L.smem[PASS_TOKENS];
  a.items = c.work;
  a.out = base + S1.tail;
  a.sh = sh;
  a.ready = reinterpret_cast<uint32_t*>(base + S1.ready);
  a.slot_of = c.slot_of;
  a.n_slots = (uint32_t)cap;
  a.slice = static_cast<uint8_t*>(d_out);
  a.coord = coord;
  a.len = len;
  a.timeout_ns = L.timeout;
  a.recs = reinterpret_cast<MatchRec*>(base + S1.tail + (cap << log2B));
  a.match_ptr = nullptr;
  a.level = idx->d_level;
  a.closure_flags = true;
  a.long_min = L.long_min;
  a.lv_done = c.lv_done;
  launch_seek(idx, L, a, last - first + 1, s);
  CUDA_TRY(cudaGetLastError());
  return ACE_OK;
}

ace_status ace_sync(const ace_index* idx, void* d_scratch, cudaStream_t s) {
  if (!idx || !d_scratch) return ACE_E_INVAL;
  ScratchHdr h;
  ace_status rc = read_header(d_scratch, &h, sizeof h, s);
  if (rc) return rc;
  if (h.status) {
    CUDA_TRY(cudaMemsetAsync(d_scratch, 0, 3 * sizeof(uint32_t), s));
    CUDA_TRY(cudaStreamSynchronize(s));
  }
  return (ace_status)h.status;
}

ace_status ace_host_register(void* h_p, uint64_t bytes, uint32_t read_only, void** d_p) {
  if (!h_p || !bytes || !d_p) return ACE_E_INVAL;
  unsigned flags = cudaHostRegisterMapped | cudaHostRegisterPortable;
  int dev = 0, ro = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  // read-only registration where the platform offers it (a hint only)
  if (read_only && cudaDeviceGetAttribute(&ro, cudaDevAttrHostRegisterReadOnlySupported, dev) == cudaSuccess && ro)
    flags |= cudaHostRegisterReadOnly;
  CUDA_TRY(cudaHostRegister(h_p, bytes, flags));
  if (cudaHostGetDevicePointer(d_p, h_p, 0) != cudaSuccess) {
    cudaHostUnregister(h_p);
    return ACE_E_CUDA;
  }
  return ACE_OK;
}

ace_status ace_host_unregister(void* h_p) {
  if (!h_p) return ACE_E_INVAL;
  CUDA_TRY(cudaHostUnregister(h_p));
  return ACE_OK;
}

ace_status ace_fnv1a64(const void* d_p, uint64_t n, uint64_t* d_result, cudaStream_t s) {
  if ((!d_p && n) || !d_result) return ACE_E_INVAL;
  fnv_kernel<<<1, 1, 0, s>>>(static_cast<const uint8_t*>(d_p), n, d_result);
  CUDA_TRY(cudaGetLastError());
  return ACE_OK;
}

ace_status ace_verify(const ace_index* idx, uint64_t coord, uint64_t len, void* d_buf, uint64_t guard_bytes,
                      uint64_t expected, uint32_t canary_seed, void* d_scratch, uint64_t scratch_bytes,
                      ace_verify_report* rep, cudaStream_t s) {
  if (!idx || !d_buf || !d_scratch || !rep) return ACE_E_INVAL;
  if (len == 0 || coord >= idx->h.total_size || len > idx->h.total_size - coord) return ACE_E_RANGE;
  std::memset(rep, 0, sizeof *rep);
  uint8_t* buf = static_cast<uint8_t*>(d_buf);
  uint8_t* slice = buf + guard_bytes;
  ScratchHdr* sh = static_cast<ScratchHdr*>(d_scratch);
  uint32_t poison_seed = canary_seed ^ 0x5bd1e995u;
  auto guards_bad = [&](uint64_t* out_bad) -> ace_status {
    CUDA_TRY(cudaMemsetAsync(&sh->guard_bad, 0, 8, s));
    if (guard_bytes) {
      count_pattern_mismatch_kernel<<<64, 256, 0, s>>>(buf, guard_bytes, canary_seed, &sh->guard_bad);
      count_pattern_mismatch_kernel<<<64, 256, 0, s>>>(slice + len, guard_bytes, canary_seed ^ 0x9e3779b9u,
                                                       &sh->guard_bad);
    }
    CUDA_TRY(cudaMemcpyAsync(out_bad, &sh->guard_bad, 8, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    return ACE_OK;
  };
  // set up: canaries around, poison inside
  if (guard_bytes) {
    fill_pattern_kernel<<<64, 256, 0, s>>>(buf, guard_bytes, canary_seed);
    fill_pattern_kernel<<<64, 256, 0, s>>>(slice + len, guard_bytes, canary_seed ^ 0x9e3779b9u);
  }
  fill_pattern_kernel<<<256, 256, 0, s>>>(slice, len, poison_seed);
  CUDA_TRY(cudaGetLastError());
  // phase 1: the slice holds none of the original
  fnv_kernel<<<1, 1, 0, s>>>(slice, len, &sh->fnv);
  CUDA_TRY(cudaMemcpyAsync(&rep->fnv_before, &sh->fnv, 8, cudaMemcpyDeviceToHost, s));
  ace_status rc = guards_bad(&rep->guard_bad_before);
  if (rc) return rc;
  rep->phase1_ok = rep->fnv_before != expected;
  // the seek through both layers
  rc = ace_seek(idx, coord, len, slice, len, d_scratch, scratch_bytes, s);
  if (rc) return rc;
  rep->seek_status = ace_sync(idx, d_scratch, s);
  // phase 2: the slice equals the original; phase 3: the guards are untouched
  fnv_kernel<<<1, 1, 0, s>>>(slice, len, &sh->fnv);
  CUDA_TRY(cudaMemcpyAsync(&rep->fnv_after, &sh->fnv, 8, cudaMemcpyDeviceToHost, s));
  rc = guards_bad(&rep->guard_bad_after);
  if (rc) return rc;
  rep->phase2_ok = rep->seek_status == ACE_OK && rep->fnv_after == expected;
  rep->phase3_ok = rep->guard_bad_before == 0 && rep->guard_bad_after == 0;
  return ACE_OK;
}

// ------------------------------------------------------------ batch (host)

struct ace_batch {
  int device;
  uint32_t n;
  uint8_t* d_scratch;
  uint64_t scratch_bytes;
  uint64_t lv_done_off, lv_done_bytes;  // the fused schedule's level counters
  BatchArgs args;
  Launch L;
  bool split;             // the entropy layer a stream per warp, literals placed by the match CTAs
  uint32_t entropy_grid;
  int occ[4][9][9];
};

namespace {

struct BatchLayout {
  uint64_t objs, by_size, by_level, ready, lv_done, lv_done_bytes, recs, total, max_ntok, items;
  uint32_t max_log2B;
  bool split, warp_match;  // the way its passes take (batch_route)
};

// A batch's entropy layer goes a block per warp (two passes) or a stream per
// warp (one launch, split), and its match pass a CTA or a warp per block.
//
// Match pass.  A CTA sweeps all of its block's bytes, which pays for dense
// archives alone: 115 MB of text in 16 KiB blocks 0.71 ms by CTAs and 1.02 by
// warps, in 4 KiB blocks 1.05 and 1.00; FASTQ 0.40 and 0.32, 0.74 and 0.45;
// genome 0.35 and 0.31, 0.61 and 0.37.  A 64 KiB text block is 1 ms of a warp
// whatever else there is, so warps take over only where hardly anything is dense
// (by those costs, a sixth of the bytes) and no dense block is large.
//
// Entropy layer.  Split, a block takes as long as its longest stream, where the
// passes add its streams up; but it costs more per block, in the match CTAs above
// all, which then place the literals.  For dense archives both are estimated: the
// longest block's chain (about 8 and 2.3 ns a byte) or the sum of the work (3 us
// a MB, 2 where matches are few), the larger of the two, plus a second launch or
// 17 ns a block (6 where matches are few; less in proportion below 4 KiB, at least
// 2).  Text, us split (passes): 4 MB in 256-byte blocks 179 (158), 1 KiB 109 (104),
// 2 KiB 83 (93), 4 KiB 72 (104), 16 KiB 85 (170), 64 KiB 250 (549); 36 MB 500 (360), 269 (279), 348 (622); 115 MB 1670 (1054), 844 (710),
// 783 (910).  Uneven objects of all profiles: 57 MB 503 (781), 118 MB 804 (900),
// 183 MB 1157 (1122).  Without dense archives only few blocks are worth it: FASTQ,
// 4 MB in 8 KiB blocks 70 (79), 16 KiB 101 (116), 64 KiB 380 (342); genome 70
// (68), 97 (101), 285 (291); 36 MB in 16 KiB blocks 210 (147) and 177 (162).
constexpr uint32_t kSplitBatchSparse = 4;  // blocks per SM
constexpr uint32_t kSplitSparseLog2B = 15;

void batch_route(const ace_index* const* idx, uint32_t n, BatchLayout* B) {
  double bytes = 0, dense_bytes = 0, chain = 0, per_block = 0;
  for (uint32_t i = 0; i < n; i++) {
    const ace_index& x = *idx[i];
    const double total = (double)x.h.total_size, block = std::min(total, (double)(1ull << x.h.log2_block));
    const bool dense = x.h.total_size && dense_matches(x.n_matches, x.h.total_size);
    bytes += total;
    per_block += (double)x.h.n_blocks * std::max(0.12, std::min(1.0, block / 4096)) * (dense ? 17e-3 : 6e-3);
    if (dense) {
      dense_bytes += total;
      chain = std::max(chain, block);
    }
  }
  const double work = (2 * bytes + dense_bytes) * 1e-6;  // us
  B->warp_match = dense_bytes * 6 <= bytes && chain <= 8192;
  if (B->warp_match)
    B->split = B->items <= (uint64_t)kSplitBatchSparse * idx[0]->num_sms && B->max_log2B <= kSplitSparseLog2B;
  else
    B->split = std::max(2.3e-3 * chain, work) + per_block < std::max(8e-3 * chain, work) + 25;
  if (B->split) B->warp_match = false;
}

ace_status batch_layout(const ace_index* const* idx, uint32_t n, BatchLayout* B) {
  if (!idx || n == 0) return ACE_E_INVAL;
  uint64_t ready = 0, items = 0, max_ntok = 0, matches = 0, levels = 0, segs = 0;
  uint32_t max_log2B = 0;
  int dev = idx[0] ? idx[0]->device : -1;
  for (uint32_t i = 0; i < n; i++) {
    if (!idx[i] || idx[i]->device != dev) return ACE_E_INVAL;
    items += idx[i]->h.n_blocks;
    ready += align256(4 * idx[i]->h.n_blocks);
    matches += idx[i]->n_matches;
    levels += idx[i]->n_levels;
    segs += idx[i]->by_levels ? idx[i]->n_levels : 1;
    max_ntok = std::max<uint64_t>(max_ntok, idx[i]->max_ntok);
    max_log2B = std::max<uint32_t>(max_log2B, idx[i]->h.log2_block);
  }
  if (items > 0xFFFFFFF0ull) return ACE_E_INVAL;
  uint64_t o = sizeof(ScratchHdr);
  B->objs = o;
  o = align256(o + n * sizeof(ObjDesc));
  B->by_size = o;
  o = align256(o + n * sizeof(BatchSeg));
  B->by_level = o;
  o = align256(o + segs * sizeof(BatchSeg));
  B->ready = o;
  o += ready;
  B->lv_done = o;
  B->lv_done_bytes = 4 * levels;
  o = align256(o + 4 * levels);
  B->recs = o;
  o = align256(o + 16 * matches);
  B->total = o;
  B->max_ntok = max_ntok;
  B->items = items;
  B->max_log2B = max_log2B;
  batch_route(idx, n, B);
  return ACE_OK;
}

}  // namespace

ace_status ace_batch_scratch_size(const ace_index* const* idx, uint32_t n, uint64_t* bytes) {
  if (!bytes) return ACE_E_INVAL;
  BatchLayout B;
  ace_status rc = batch_layout(idx, n, &B);
  if (rc) return rc;
  *bytes = B.total;
  return ACE_OK;
}

ace_status ace_batch_create(const ace_index* const* idx, uint32_t n, void* const* d_outs, const uint64_t* out_bytes,
                            void* d_scratch, uint64_t scratch_bytes, const ace_tune* tune, cudaStream_t s,
                            ace_batch** out) {
  if (!out || !d_outs || !out_bytes || !d_scratch || !aligned(d_scratch, 256)) return ACE_E_INVAL;
  BatchLayout B;
  ace_status rc = batch_layout(idx, n, &B);
  if (rc) return rc;
  if (scratch_bytes < B.total) return ACE_E_NOMEM;
  uint8_t* base = static_cast<uint8_t*>(d_scratch);
  std::vector<ObjDesc> od(n);
  uint64_t ready = B.ready, recs = B.recs, lvd = B.lv_done;
  for (uint32_t i = 0; i < n; i++) {
    const ace_index* x = idx[i];
    if (out_bytes[i] < x->h.total_size || (!d_outs[i] && x->h.total_size)) return ACE_E_NOMEM;
    if (!aligned(d_outs[i], 16)) return ACE_E_INVAL;
    od[i] = ObjDesc{x->d_arc,
                    reinterpret_cast<const ace_block_dir*>(x->d_arc + x->h.dir_off),
                    x->h.payload_off,
                    x->h.total_size,
                    static_cast<uint8_t*>(d_outs[i]),
                    reinterpret_cast<uint32_t*>(base + ready),
                    x->d_order,
                    x->d_level,
                    reinterpret_cast<MatchRec*>(base + recs),
                    x->d_match_ptr,
                    reinterpret_cast<uint32_t*>(base + lvd),
                    x->d_lv_count,
                    x->h.log2_block,
                    x->h.off_width,
                    (uint32_t)x->h.n_blocks,
                    0};
    ready += align256(4 * x->h.n_blocks);
    recs += 16 * x->n_matches;
    lvd += 4ull * x->n_levels;
  }
  // the work items' two orders
  std::vector<uint32_t> large(n);
  for (uint32_t i = 0; i < n; i++) large[i] = i;
  std::stable_sort(large.begin(), large.end(),
                   [&](uint32_t x, uint32_t y) { return idx[x]->h.log2_block > idx[y]->h.log2_block; });
  std::vector<BatchSeg> by_size, by_level;
  uint32_t at = 0;
  for (uint32_t i : large) {
    if (!idx[i]->h.n_blocks) continue;
    by_size.push_back({at, i, 0, 0});
    at += (uint32_t)idx[i]->h.n_blocks;
  }
  at = 0;
  for (uint32_t l = 0; l < kMaxLevelLaunches; l++)
    for (uint32_t i : large) {
      const ace_index* x = idx[i];
      // (an archive of more levels: all of it, in its own order)
      const uint32_t first = x->by_levels && l < x->n_levels ? x->level_start[l] : 0;
      const uint32_t cnt = x->by_levels ? (l < x->n_levels ? x->level_start[l + 1] - first : 0) : (l ? 0 : (uint32_t)x->h.n_blocks);
      if (!cnt) continue;
      by_level.push_back({at, i, first, 0});
      at += cnt;
    }
  ace_batch* b = new (std::nothrow) ace_batch();
  if (!b) return ACE_E_NOMEM;
  b->device = idx[0]->device;
  b->n = n;
  b->d_scratch = base;
  b->scratch_bytes = scratch_bytes;
  b->lv_done_off = B.lv_done;
  b->lv_done_bytes = B.lv_done_bytes;
  // the launch shape uses the largest block size's escape table
  rc = plan_launch(idx[0], tune, B.max_log2B, B.items, batch_decode_kernel<PASS_TOKENS>,
                   batch_decode_kernel<PASS_LITERALS>,
                   B.warp_match ? batch_decode_kernel<PASS_WARP> : batch_decode_kernel<PASS_MATCH>,
                   batch_decode_kernel<PASS_FUSED>, &b->occ[0][0][0], &b->L, kRing, false, B.warp_match);
  if (rc == ACE_OK &&
      (cudaMemsetAsync(base, 0, B.recs, s) != cudaSuccess ||
       cudaMemcpyAsync(base + B.objs, od.data(), n * sizeof(ObjDesc), cudaMemcpyHostToDevice, s) != cudaSuccess ||
       cudaMemcpyAsync(base + B.by_size, by_size.data(), by_size.size() * sizeof(BatchSeg), cudaMemcpyHostToDevice, s) !=
           cudaSuccess ||
       cudaMemcpyAsync(base + B.by_level, by_level.data(), by_level.size() * sizeof(BatchSeg), cudaMemcpyHostToDevice,
                       s) != cudaSuccess ||
       cudaStreamSynchronize(s) != cudaSuccess))
    rc = ACE_E_CUDA;
  if (rc) {
    delete b;
    return rc;
  }
  BatchArgs& a = b->args;
  a.objs = reinterpret_cast<const ObjDesc*>(base + B.objs);
  b->split = B.split;
  b->entropy_grid = (uint32_t)std::min<uint64_t>((3 * B.items + kBatchEntropyWarps - 1) / kBatchEntropyWarps, 8ull * idx[0]->num_sms);
  a.by_size = reinterpret_cast<const BatchSeg*>(base + B.by_size);
  a.by_level = reinterpret_cast<const BatchSeg*>(base + B.by_level);
  a.n_size = (uint32_t)by_size.size();
  a.n_level = (uint32_t)by_level.size();
  a.n_items = (uint32_t)B.items;
  a.window = b->L.chunk;
  a.warp_smem = b->L.smem[PASS_TOKENS];
  a.esc_cap = esc_cap(B.max_log2B);
  a.max_ntok = (uint32_t)B.max_ntok;
  a.sh = reinterpret_cast<ScratchHdr*>(base);
  a.timeout_ns = b->L.timeout;
  a.long_min = b->L.long_min;
  *out = b;
  return ACE_OK;
}

ace_status ace_decode_batch(const ace_batch* b, cudaStream_t s) {
  if (!b) return ACE_E_INVAL;
  if (!b->args.n_items) return ACE_OK;
  const Launch& L = b->L;
  if (L.schedule == ACE_SCHEDULE_FUSED && b->lv_done_bytes)
    CUDA_TRY(cudaMemsetAsync(b->d_scratch + b->lv_done_off, 0, b->lv_done_bytes, s));
  begin_call_kernel<<<1, 1, 0, s>>>(b->args.sh);
  if (L.schedule == ACE_SCHEDULE_FUSED)
    launch_fused(L, batch_decode_kernel<PASS_FUSED>, b->args, s);
  else if (b->split) {
    batch_entropy_kernel<<<b->entropy_grid, 32 * kBatchEntropyWarps,
                           kBatchEntropyWarps * job_smem_bytes(b->args.esc_cap, kRing), s>>>(b->args);
    batch_decode_kernel<PASS_PLACE><<<L.grid[PASS_MATCH], L.match_threads, L.smem[PASS_MATCH], s>>>(b->args);
  } else
    launch_passes(L, 7, batch_decode_kernel<PASS_TOKENS>, batch_decode_kernel<PASS_LITERALS>,
                  L.warp_match ? batch_decode_kernel<PASS_WARP> : batch_decode_kernel<PASS_MATCH>, b->args, s);
  CUDA_TRY(cudaGetLastError());
  return ACE_OK;
}

ace_status ace_batch_sync(const ace_batch* b, cudaStream_t s) {
  if (!b) return ACE_E_INVAL;
  ScratchHdr h;
  ace_status rc = read_header(b->d_scratch, &h, sizeof h, s);
  if (rc) return rc;
  if (h.status) {
    CUDA_TRY(cudaMemsetAsync(b->d_scratch, 0, 3 * sizeof(uint32_t), s));
    CUDA_TRY(cudaStreamSynchronize(s));
  }
  return (ace_status)h.status;
}

ace_status ace_batch_launch_shape(const ace_batch* b, uint32_t* grid, uint32_t* warps_per_cta, uint32_t* window) {
  if (!b) return ACE_E_INVAL;
  const bool fused = b->L.schedule == ACE_SCHEDULE_FUSED, split = b->split && !fused;
  if (grid) *grid = split ? b->entropy_grid : b->L.grid[fused ? PASS_FUSED : PASS_TOKENS];
  if (warps_per_cta) *warps_per_cta = split ? kBatchEntropyWarps : b->L.warps;
  if (window) *window = split ? 0 : b->L.chunk;
  return ACE_OK;
}

ace_status ace_batch_free(ace_batch* b) {
  delete b;
  return ACE_OK;
}

// ------------------------------------------------------ seek batches (host)

struct ace_cache {
  int device;
  uint32_t n_arcs, log2B, n_slots, front_cap, max_reqs;
  int num_sms;
  uint8_t* mem;
  uint64_t bytes;
  CacheArgs args;
  CacheDecodeArgs dargs;
  Launch L;
  uint64_t req_off;  // requests are staged here by ace_seek_batch_host
  uint64_t owner_off;  // per-slot owners, cleared by a reset
  int occ[4][9][9];
};

namespace {

struct CacheLayout {
  uint64_t arcs, minmax, front0, front1, work, taken, owner_arc, owner_blk, ref, use, reqs, slots, recs, total, max_ntok,
      max_work;
};

// Blocks one seek batch may decode at most (work items): 32 per request the
// batch may hold, at least 1024, at most the slots.  Its match records are
// sized by it rather than by the slot count, since only the blocks a batch
// decodes need records, and only while it runs.
inline uint64_t cache_max_work(uint64_t n_slots, uint32_t max_reqs) {
  return std::min<uint64_t>(n_slots, std::max<uint64_t>(1024, 32ull * max_reqs));
}

CacheLayout cache_layout(const ace_index* const* idx, uint32_t n, uint64_t n_slots, uint32_t max_reqs,
                         uint32_t log2B) {
  CacheLayout C;
  uint64_t max_ntok = 0;
  for (uint32_t i = 0; i < n; i++) max_ntok = std::max<uint64_t>(max_ntok, idx[i]->max_ntok);
  const uint64_t mw = cache_max_work(n_slots, max_reqs);
  uint64_t o = sizeof(CacheHdr);
  C.arcs = o;
  o = align256(o + n * sizeof(CacheArc));
  C.minmax = o;
  o = align256(o + 8ull * n);
  C.front0 = o;
  o = align256(o + 8 * mw);
  C.front1 = o;
  o = align256(o + 8 * mw);
  C.work = o;
  o = align256(o + 8 * mw);
  C.taken = o;
  o = align256(o + 4 * mw);
  C.owner_arc = o;
  o = align256(o + 4 * n_slots);
  C.owner_blk = o;
  o = align256(o + 4 * n_slots);
  C.ref = o;
  o = align256(o + 4 * n_slots);
  C.use = o;
  o = align256(o + 4 * n_slots);
  C.reqs = o;
  o = align256(o + sizeof(ace_seek_req) * (uint64_t)max_reqs);
  C.slots = o;
  o = align256(o + (n_slots << log2B));
  C.recs = o;
  o = align256(o + 16 * max_ntok * mw);
  C.total = o;
  C.max_ntok = max_ntok;
  C.max_work = mw;
  return C;
}

ace_status cache_check(const ace_index* const* idx, uint32_t n) {
  if (!idx || n == 0) return ACE_E_INVAL;
  for (uint32_t i = 0; i < n; i++)
    if (!idx[i] || idx[i]->device != idx[0]->device || idx[i]->h.log2_block != idx[0]->h.log2_block)
      return ACE_E_INVAL;  // one device, one block size per cache
  return ACE_OK;
}

}  // namespace

ace_status ace_cache_size(const ace_index* const* idx, uint32_t n, uint64_t n_slots, uint32_t max_reqs,
                          uint64_t* bytes) {
  ace_status rc = cache_check(idx, n);
  if (rc) return rc;
  if (!bytes || n_slots == 0 || n_slots > 0xFFFFFFF0ull || max_reqs == 0) return ACE_E_INVAL;
  *bytes = cache_layout(idx, n, n_slots, max_reqs, idx[0]->h.log2_block).total;
  return ACE_OK;
}

ace_status ace_archive_state_size(const ace_index* idx, uint64_t* bytes) {
  if (!idx || !bytes) return ACE_E_INVAL;
  uint64_t nb = idx->h.n_blocks;
  *bytes = align256(4 * nb) * 3 + align256(4 * ((nb + 31) / 32));  // ready, slot_of, wpos; marks
  return ACE_OK;
}

ace_status ace_cache_create(const ace_index* const* idx, uint32_t n, void* const* d_states, uint64_t n_slots,
                            uint32_t max_reqs, void* d_mem, uint64_t bytes, const ace_tune* tune, cudaStream_t s,
                            ace_cache** out) {
  ace_status rc = cache_check(idx, n);
  if (rc) return rc;
  if (!out || !d_states || !d_mem || !aligned(d_mem, 256) || n_slots == 0 || max_reqs == 0) return ACE_E_INVAL;
  const uint32_t log2B = idx[0]->h.log2_block;
  CacheLayout C = cache_layout(idx, n, n_slots, max_reqs, log2B);
  if (bytes < C.total) return ACE_E_NOMEM;
  uint8_t* base = static_cast<uint8_t*>(d_mem);
  std::vector<CacheArc> arcs(n);
  for (uint32_t i = 0; i < n; i++) {
    const ace_index* x = idx[i];
    if (!d_states[i] || !aligned(d_states[i], 256)) return ACE_E_INVAL;
    uint8_t* st = static_cast<uint8_t*>(d_states[i]);
    uint64_t nb = x->h.n_blocks;
    arcs[i] = CacheArc{x->d_arc,
                       reinterpret_cast<const ace_block_dir*>(x->d_arc + x->h.dir_off),
                       x->h.payload_off,
                       x->h.total_size,
                       x->d_dep_ptr,
                       x->d_dep_iv,
                       reinterpret_cast<uint32_t*>(st),
                       reinterpret_cast<uint32_t*>(st + align256(4 * nb)),
                       reinterpret_cast<uint32_t*>(st + 3 * align256(4 * nb)),
                       reinterpret_cast<uint32_t*>(st + 2 * align256(4 * nb)),
                       (uint32_t)nb,
                       x->h.off_width};
    uint64_t sb = 0;
    ace_archive_state_size(x, &sb);
    if (cudaMemsetAsync(st, 0, sb, s) != cudaSuccess) return ACE_E_CUDA;
  }
  ace_cache* c = new (std::nothrow) ace_cache();
  if (!c) return ACE_E_NOMEM;
  c->device = idx[0]->device;
  c->n_arcs = n;
  c->log2B = log2B;
  c->n_slots = (uint32_t)n_slots;
  c->front_cap = (uint32_t)C.max_work;
  c->max_reqs = max_reqs;
  c->num_sms = idx[0]->num_sms;
  c->mem = base;
  c->bytes = bytes;
  c->req_off = C.reqs;
  c->owner_off = C.owner_arc;
  // seek batches run the three passes (their work list is in block order,
  // not level order); the fused entry only sizes like the match pass
  rc = plan_launch(idx[0], tune, log2B, C.max_work, cache_decode_kernel<PASS_TOKENS>,
                   cache_decode_kernel<PASS_LITERALS>, cache_decode_kernel<PASS_MATCH>,
                   cache_decode_kernel<PASS_MATCH>, &c->occ[0][0][0], &c->L, kSeekRing, true, false);
  // header (epoch 1: no block is cached, since every ready flag starts at 0)
  CacheHdr h{};
  h.epoch = 1;
  // every slot free (owner archive ~0), reference bits and batch serials 0
  if (rc == ACE_OK &&
      (cudaMemcpyAsync(base, &h, sizeof h, cudaMemcpyHostToDevice, s) != cudaSuccess ||
       cudaMemcpyAsync(base + C.arcs, arcs.data(), n * sizeof(CacheArc), cudaMemcpyHostToDevice, s) != cudaSuccess ||
       cudaMemsetAsync(base + C.owner_arc, 0xff, 4 * n_slots, s) != cudaSuccess ||
       cudaMemsetAsync(base + C.ref, 0, C.reqs - C.ref, s) != cudaSuccess ||
       cudaStreamSynchronize(s) != cudaSuccess))
    rc = ACE_E_CUDA;
  if (rc) {
    delete c;
    return rc;
  }
  CacheArgs& a = c->args;
  a.h = reinterpret_cast<CacheHdr*>(base);
  a.arcs = reinterpret_cast<const CacheArc*>(base + C.arcs);
  a.n_arcs = n;
  a.log2B = log2B;
  a.n_slots = (uint32_t)n_slots;
  a.front_cap = (uint32_t)C.max_work;
  a.front0 = reinterpret_cast<uint32_t*>(base + C.front0);
  a.front1 = reinterpret_cast<uint32_t*>(base + C.front1);
  a.work = reinterpret_cast<uint32_t*>(base + C.work);
  a.taken = reinterpret_cast<uint32_t*>(base + C.taken);
  a.owner_arc = reinterpret_cast<uint32_t*>(base + C.owner_arc);
  a.owner_blk = reinterpret_cast<uint32_t*>(base + C.owner_blk);
  a.ref = reinterpret_cast<uint32_t*>(base + C.ref);
  a.use = reinterpret_cast<uint32_t*>(base + C.use);
  a.arc_minmax = reinterpret_cast<uint32_t*>(base + C.minmax);
  a.slots = base + C.slots;
  a.recs = reinterpret_cast<MatchRec*>(base + C.recs);
  a.reqs = nullptr;
  a.n_reqs = 0;
  CacheDecodeArgs& d = c->dargs;
  d.window = c->L.chunk;
  d.warp_smem = c->L.smem[PASS_TOKENS];
  d.esc_cap = esc_cap(log2B);
  d.max_ntok = (uint32_t)C.max_ntok;
  d.timeout_ns = c->L.timeout;
  d.long_min = c->L.long_min;
  *out = c;
  return ACE_OK;
}

}  // extern "C"

namespace {

// split: decode the batch's blocks a stream per warp
ace_status seek_batch(const ace_cache* c, const ace_seek_req* d_reqs, uint32_t n, void* d_pool, bool split,
                      cudaStream_t s) {
  CacheArgs a = c->args;
  a.reqs = d_reqs;
  a.n_reqs = n;
  cache_closure_kernel<<<kClosureCtas, 1024, 0, s>>>(a);
  CacheDecodeArgs d = c->dargs;
  d.c = a;
  const Launch& L = c->L;
  if (split) {
    const uint32_t grid = std::min(3 * c->front_cap, 16 * (uint32_t)c->num_sms);
    cache_entropy_kernel<<<grid, 32, job_smem_bytes(d.esc_cap, kSeekRing), s>>>(d);
    cache_decode_kernel<PASS_PLACE><<<L.grid[PASS_MATCH], L.match_threads, L.smem[PASS_MATCH], s>>>(d);
  } else {
    launch_passes(L, 7, cache_decode_kernel<PASS_TOKENS>, cache_decode_kernel<PASS_LITERALS>,
                  cache_decode_kernel<PASS_MATCH>, d, s);
  }
  // CTAs of 8 warps per request until there are about 8 per SM's worth
  const uint32_t per = std::max(1u, std::min(8u, 1024 / n));
  cache_copy_kernel<<<dim3(std::min<uint32_t>(n, 1024), per), 256, 0, s>>>(a, static_cast<uint8_t*>(d_pool));
  CUDA_TRY(cudaGetLastError());
  return ACE_OK;
}

}  // namespace

extern "C" {

ace_status ace_seek_batch(const ace_cache* c, const ace_seek_req* d_reqs, uint32_t n, void* d_pool, uint64_t pool_bytes,
                          cudaStream_t s) {
  if (!c || (!d_reqs && n) || (!d_pool && n)) return ACE_E_INVAL;
  if (n == 0) return ACE_OK;
  (void)pool_bytes;  // request ranges are validated on the host by ace_seek_batch_host
  return seek_batch(c, d_reqs, n, d_pool, n <= kSplitReqs, s);
}

ace_status ace_seek_batch_host(const ace_cache* c, const ace_seek_req* h_reqs, const uint64_t* h_totals, uint32_t n,
                               void* d_pool, uint64_t pool_bytes, cudaStream_t s) {
  if (!c || (!h_reqs && n)) return ACE_E_INVAL;
  if (n > c->max_reqs) return ACE_E_NOMEM;
  uint64_t blocks = 0;
  for (uint32_t i = 0; i < n; i++) {
    const ace_seek_req& q = h_reqs[i];
    if (q.archive >= c->n_arcs) return ACE_E_INVAL;
    if (q.len == 0 || (h_totals && (q.coord >= h_totals[q.archive] || q.len > h_totals[q.archive] - q.coord)))
      return ACE_E_RANGE;
    if (q.out_off + q.len > pool_bytes) return ACE_E_NOMEM;
    blocks += (q.len >> c->log2B) + 1;
  }
  ace_seek_req* d = reinterpret_cast<ace_seek_req*>(c->mem + c->req_off);
  if (n) CUDA_TRY(cudaMemcpyAsync(d, h_reqs, n * sizeof(ace_seek_req), cudaMemcpyHostToDevice, s));
  if (n == 0) return ACE_OK;
  if (!d_pool) return ACE_E_INVAL;
  return seek_batch(c, d, n, d_pool, blocks <= kSplitBatch, s);
}

ace_status ace_cache_sync(const ace_cache* c, cudaStream_t s) {
  if (!c) return ACE_E_INVAL;
  CacheHdr h;
  ace_status rc = read_header(c->mem, &h, sizeof h, s);
  if (rc) return rc;
  if (h.status) {
    CUDA_TRY(cudaMemsetAsync(c->mem, 0, 3 * sizeof(uint32_t), s));
    CUDA_TRY(cudaStreamSynchronize(s));
  }
  return (ace_status)h.status;
}

ace_status ace_cache_usage(const ace_cache* c, uint32_t* used_slots, uint32_t* n_slots, cudaStream_t s) {
  if (!c) return ACE_E_INVAL;
  CacheHdr h;
  ace_status rc = read_header(c->mem, &h, sizeof h, s);
  if (rc) return rc;
  if (used_slots) *used_slots = h.n_cached;
  if (n_slots) *n_slots = c->n_slots;
  return ACE_OK;
}

ace_status ace_cache_reset(const ace_cache* c, cudaStream_t s) {
  if (!c) return ACE_E_INVAL;
  cache_reset_kernel<<<1, 1, 0, s>>>(c->args.h);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemsetAsync(c->mem + c->owner_off, 0xff, 4ull * c->n_slots, s));
  return ACE_OK;
}

ace_status ace_cache_counters(const ace_cache* c, uint64_t* h_evicted, uint64_t* h_decoded, cudaStream_t s) {
  if (!c) return ACE_E_INVAL;
  CacheHdr h;
  ace_status rc = read_header(c->mem, &h, sizeof h, s);
  if (rc) return rc;
  if (h_evicted) *h_evicted = h.evicted;
  if (h_decoded) *h_decoded = h.decoded;
  return ACE_OK;
}

ace_status ace_cache_limits(const ace_cache* c, uint32_t* h_n_slots, uint32_t* h_max_work, uint32_t* h_max_reqs) {
  if (!c) return ACE_E_INVAL;
  if (h_n_slots) *h_n_slots = c->n_slots;
  if (h_max_work) *h_max_work = c->front_cap;
  if (h_max_reqs) *h_max_reqs = c->max_reqs;
  return ACE_OK;
}

ace_status ace_cache_free(ace_cache* c) {
  delete c;
  return ACE_OK;
}

// -------------------------------------------------- seek without allocation
//
// Some callers cannot allocate device memory at all: a host application
// that owns every byte of device memory through its own pool, a plug-in
// loaded into such an application, or a latency-critical request thread
// that must never reach the allocator.  ace_seek_noalloc serves them: it
// takes its scratch from a fixed array that lives in this library's device
// image, so the caller passes only the archive's index and the output.
//
// The array is kStaticScratchBytes (32 MiB) on every GPU that loads the
// library, held until the process exits.  It is shared by every call on a
// device and keeps the last call's contents; calls that overlap on the GPU
// race on it and must be ordered by the caller (one stream, or events).

namespace {

constexpr uint64_t kStaticScratchBytes = 32ull << 20;
constexpr int kMaxDevices = 64;

__device__ __align__(256) uint8_t g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mu;
uint8_t* g_static_ptr[kMaxDevices];  // device address of g_static_scratch, per device

// The host-side name g_static_scratch is a stand-in, not a device address:
// the address is looked up once per device, with that device current.
ace_status static_scratch(int device, uint8_t** out) {
  if (device < 0 || device >= kMaxDevices) return ACE_E_INVAL;
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[device]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return ACE_E_CUDA;
    g_static_ptr[device] = static_cast<uint8_t*>(p);
  }
  *out = g_static_ptr[device];
  return ACE_OK;
}

}  // namespace

ace_status ace_seek_noalloc(const ace_index* idx, uint64_t coord, uint64_t len, void* d_out, uint64_t out_bytes,
                            cudaStream_t s) {
  if (!idx || !d_out) return ACE_E_INVAL;
  if (len == 0 || coord >= idx->h.total_size || len > idx->h.total_size - coord) return ACE_E_RANGE;
  if (out_bytes < len) return ACE_E_NOMEM;
  int cur = -1;
  CUDA_TRY(cudaGetDevice(&cur));
  if (cur != idx->device) return ACE_E_INVAL;  // the index's device must be current
  uint8_t* base = nullptr;
  ace_status rc = static_scratch(cur, &base);
  if (rc) return rc;
  const uint64_t nb = idx->h.n_blocks;
  const uint32_t log2B = idx->h.log2_block;
  ScratchLayout S = scratch_layout(nb, log2B, 1, idx->max_ntok, 0);
  if (S.tail > kStaticScratchBytes) return ACE_E_NOMEM;  // archive too large for the fixed scratch
  uint64_t cap = std::min<uint64_t>(nb, (kStaticScratchBytes - S.tail) / slot_bytes(log2B, idx->max_ntok));
  uint64_t first = coord >> log2B, last = (coord + len - 1) >> log2B;
  if (last - first + 1 > cap) return ACE_E_NOMEM;  // more target blocks than slots
  ScratchHdr* sh = reinterpret_cast<ScratchHdr*>(base);
  // The array may hold what a call on another archive, with another layout,
  // left there.  The closure marks must start clear, and so must the ready
  // flags: a stale word equal to this call's epoch would pass a block outside
  // the closure as a member (epochs are never 0).
  CUDA_TRY(cudaMemsetAsync(base + S.ready, 0, S.slot_of - S.ready, s));
  CUDA_TRY(cudaMemsetAsync(base + S.marks, 0, S.front0 - S.marks, s));
  CUDA_TRY(cudaMemsetAsync(base, 0, 3 * sizeof(uint32_t), s));  // status word
  ClosureArgs c;
  c.dep_ptr = idx->d_dep_ptr;
  c.dep_iv = idx->d_dep_iv;
  c.sh = sh;
  c.marks = reinterpret_cast<uint32_t*>(base + S.marks);
  c.front0 = reinterpret_cast<uint32_t*>(base + S.front0);
  c.front1 = reinterpret_cast<uint32_t*>(base + S.front1);
  c.work = reinterpret_cast<uint32_t*>(base + S.work);
  c.slot_of = reinterpret_cast<uint32_t*>(base + S.slot_of);
  c.nb = nb;
  c.first = first;
  c.last = last;
  c.cap = cap;
  c.level = idx->by_levels ? idx->d_level : nullptr;
  c.n_levels = idx->n_levels;
  c.ready = reinterpret_cast<uint32_t*>(base + S.ready);
  Launch L;
  rc = plan_index_launch<true>(idx, nullptr, cap, &L);
  if (rc) return rc;
  if (!idx->by_levels) L.schedule = ACE_SCHEDULE_PASSES;
  c.lv_done = L.schedule == ACE_SCHEDULE_FUSED ? reinterpret_cast<uint32_t*>(base + S.lv_done) : nullptr;
  closure_kernel<<<kClosureCtas, 1024, 0, s>>>(c);
  DecodeArgs a{};
  a.arc = idx->d_arc;
  a.dir = reinterpret_cast<const ace_block_dir*>(idx->d_arc + idx->h.dir_off);
  a.payload_off = idx->h.payload_off;
  a.total = idx->h.total_size;
  a.nb = nb;
  a.log2B = log2B;
  a.w = idx->h.off_width;
  a.window = L.chunk;
  a.max_ntok = idx->max_ntok;
  a.esc_cap = esc_cap(log2B);
  a.warp_smem = L.smem[PASS_TOKENS];
  a.items = c.work;
  a.out = base + S.tail;
  a.sh = sh;
  a.ready = reinterpret_cast<uint32_t*>(base + S.ready);
  a.slot_of = c.slot_of;
  a.n_slots = (uint32_t)cap;
  a.slice = static_cast<uint8_t*>(d_out);
  a.coord = coord;
  a.len = len;
  a.timeout_ns = L.timeout;
  a.recs = reinterpret_cast<MatchRec*>(base + S.tail + (cap << log2B));
  a.match_ptr = nullptr;
  a.level = idx->d_level;
  a.closure_flags = true;
  a.long_min = L.long_min;
  a.lv_done = c.lv_done;
  launch_seek(idx, L, a, last - first + 1, s);
  CUDA_TRY(cudaGetLastError());
  // the status lives in the shared array, so the call waits for it
  uint32_t status = 0;
  rc = read_header(base, &status, sizeof status, s);
  if (rc) return rc;
  return (ace_status)status;
}

}  // extern "C"
