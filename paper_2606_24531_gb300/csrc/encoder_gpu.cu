// GPU encoder of the two-layer codec: the whole encode on the device, from
// input bytes in device memory to an archive in device memory, in the byte
// layout of ace_format.h (the same format the host encoder writes and every
// decoder reads).
//
// Match layer (Section 2: greedy parse with a global match search, absolute
// back-references): candidates are found for every position at once, a
// CTA per block -- the earliest earlier occurrence of the 16-byte keys
// around it (a table over the whole input, built with atomic minima) and
// the most recent repeats inside its block (hash chains in shared memory)
// -- then a warp per block walks its positions greedily, taking
// at each the longest candidate allowed there.  Windows of 64 blocks take
// no sources from each other: one of the first three windows takes its
// external sources from the windows before it, and every later block from
// those three, so dependency levels stay at most 3 as with the host encoder
// and no block waits on another's parse.  A match of a block's own earlier bytes resolves
// in waves (one reading only literals is wave 1, one reading wave-k bytes
// wave k + 1); candidates deeper than wave 3 are refused, and an external
// candidate nearly as long as the best is preferred.
// Entropy layer (Section 3): each block's literal, length and offset
// streams are rANS-coded, a warp per stream, with 32 interleaved states,
// 12-bit frequencies quantised as the host encoder does, byte
// renormalisation; with the adaptive option a stream rANS would not shrink
// is stored (Section 6.1).
//
// The parse differs from the host encoder's (another valid archive of the
// same input); every decoder reads either.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "ace.h"
#include "ace_device.cuh"
#include "ace_format.h"

using namespace ace;

namespace {

constexpr uint32_t kKey = 16;        // long-key length of the global table
constexpr uint32_t kStride = 8;      // positions whose keys enter the table
constexpr uint32_t kWin = 64;        // blocks of a window
constexpr uint32_t kHeadWins = 3;    // windows whose blocks may be sources
constexpr uint32_t kHead = kWin * kHeadWins;
constexpr uint32_t kCap = 32;        // match lengths measured by the candidate search (extended later)
constexpr uint32_t kHashBits4 = 12;  // in-block chains: hash of 4 bytes
constexpr uint32_t kMaxChain = 64;

// The blocks below which block b takes sources: those of the windows before its
// own, the first three windows at most.  So a block of window k has level k at
// most and no block one above 3, whatever is found, and the search and the
// walk of a block need nothing of any other's.
__device__ __forceinline__ uint64_t source_end(uint64_t b) { return min(b / kWin * kWin, (uint64_t)kHead); }

__host__ __device__ inline uint64_t align16(uint64_t v) { return (v + 15) & ~15ull; }

__device__ __forceinline__ uint64_t ld64u(const uint8_t* p) {
  uint64_t v = 0;
#pragma unroll
  for (int k = 0; k < 8; k++) v |= (uint64_t)p[k] << (8 * k);
  return v;
}

// The table's slot of a 16-byte key (its two halves, little endian).
__device__ __forceinline__ uint32_t hash_words(uint64_t lo, uint64_t hi, uint32_t bits) {
  const uint64_t a = lo * 0x9E3779B97F4A7C15ull, b = hi * 0xC2B2AE3D27D4EB4Full;
  return (uint32_t)(((a ^ ((b << 31) | (b >> 33))) * 0x165667B19E3779F9ull) >> (64 - bits));
}

// Common prefix of a and b (a precedes b), at most limit bytes.
__device__ __forceinline__ uint32_t common(const uint8_t* a, const uint8_t* b, uint32_t limit) {
  uint32_t l = 0;
  while (l + 8 <= limit) {
    const uint64_t x = ld64u(a + l) ^ ld64u(b + l);
    if (x) return l + (__ffsll((long long)x) - 1) / 8;
    l += 8;
  }
  while (l < limit && a[l] == b[l]) l++;
  return l;
}

struct EncArgs {
  const uint8_t* in;
  uint64_t n;
  uint32_t log2B, min_match, max_chain, w, adaptive, bits;
  unsigned long long* table;  // 2^bits: the earliest stride position with each key hash
  uint64_t c0;  // the launch's first block
  uint32_t* entries;  // per position: the candidate search's links and hashes (64 KiB blocks; smaller ones: shared memory)
  uint2* cand;        // per position: x = in-block candidate length (bits 0..7), external length (8..15), both
                      // capped at kCap, and the in-block source as an offset in the block (16..31); y = the external
                      // source (below kHead blocks, so below 2^24)
  uint32_t* tok;      // per chunk block: tok_cap x (lit_run, match_len, src lo, src hi)
  uint32_t tok_cap;
  uint32_t* ntok;     // per chunk block
  unsigned long long* stats;  // n_tokens, n_matches, literal, match, match_src bytes
};

// ---------------------------------------------------------------- the table

// Every stride position's 16-byte key: the table keeps the earliest.
__global__ void table_kernel(EncArgs a) {
  const uint64_t nkeys = a.n >= kKey ? (a.n - kKey) / kStride + 1 : 0;
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < nkeys; k += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t q = k * kStride;
    atomicMin(a.table + hash_words(ld64u(a.in + q), ld64u(a.in + q + 8), a.bits), (unsigned long long)q);
  }
}

// ------------------------------------------------------ candidate search

// Bytes from q a match of block b may read without entering a block it may
// not read (its own block, or blocks below source_end), at most want.
__device__ __forceinline__ uint32_t span(const EncArgs& a, uint64_t q, uint64_t b, uint32_t want) {
  uint64_t k = q >> a.log2B;
  uint32_t got = 0;
  while (got < want) {
    if (k != b && k >= source_end(b)) break;
    const uint64_t end = (k + 1) << a.log2B;
    got = (uint32_t)min((uint64_t)want, end - q);
    k++;
  }
  return got;
}

// The 32-bit word at byte o of a staged block (any alignment).
__device__ __forceinline__ uint32_t word_at(const uint32_t* sb, uint32_t o) {
  return __funnelshift_r(sb[o >> 2], sb[(o >> 2) + 1], 8 * (o & 3));
}

// Launch shape of the candidate search for a block size: threads of a CTA,
// the segments whose links warps build side by side, and whether the entries
// fit in shared memory beside the block (all but 64 KiB blocks).  16 KiB
// blocks: 112 KiB, so two CTAs of 16 warps fit an SM.
struct CandShape {
  uint32_t threads, segs;
  bool shared_entries;
  size_t smem;
};
constexpr uint32_t kPadBytes = 64;  // staged past the block: keys and compares read ahead

// One warp's arrays of the candidate walk (over the bucket heads, which are
// done with by then).
struct CandWarp {
  uint32_t key[64];       // the keys of the window's 32 positions and of those after it
  uint8_t found[64];      // those of them the table holds a usable position for
  uint32_t ext[32];       // per position, the best external source: length << 24 | (2^24 - 1 - source)
  uint32_t own[32];       // the best of the keys' sources in the block: length << 16 | (2^16 - 1 - offset)
};

__host__ __device__ inline CandShape cand_shape(uint32_t log2B) {
  CandShape c;
  c.threads = log2B >= 12 ? 512 : log2B >= 10 ? 128 : 64;
  c.segs = log2B >= 10 ? 4 : 1;
  c.shared_entries = log2B < 16;
  const size_t heads = (size_t)c.segs * (2u << kHashBits4), warps = c.threads / 32 * sizeof(CandWarp);
  c.smem = ((size_t)1 << log2B) + kPadBytes + (c.shared_entries ? (size_t)4 << log2B : 0) +
           (heads > warps ? heads : warps);
  return c;
}

constexpr uint32_t kNoKey = ~0u;
constexpr uint32_t kCandParts = 4;  // CTAs a block's positions are split over, at most
constexpr uint64_t kSplitEntries = 256;  // 64 KiB blocks whose entries fill scratch, where launches split

// A CTA per block, or (gridDim.y > 1) per part of its positions: for every
// position the best in-block candidate (its chain
// of earlier positions with the same 4-byte hash, most recent first,
// max_chain deep) and the best external one (earliest occurrences of the keys
// at p .. p + 7, shifted back), each the longest measured up to kCap bytes
// (ties: the more recent in the chain; among keys' sources the smaller one).
//
// The block is staged in shared memory, where every link and every in-block
// compare then reads.  Links: a position's is the nearest earlier one with its
// hash; warps build them for a segment of the block each (lanes grouped by
// __match_any_sync, else the segment's bucket heads), and a segment's firsts
// are looked up in the heads of the segments before.  An entry packs the link
// with 16 bits of a hash of as many of the position's first bytes as a match
// must have, so a chain step is one shared load, and a candidate that cannot
// reach min_match is nearly always dropped there.  Each key is looked up once,
// by the lane of its position, and shared with the seven positions before;
// positions a match may not read count as not found, and the pairs of a found
// key and a position before it are dealt evenly to the lanes.  Bound by issue and
// the chains' dependent steps: about 860 warp instructions per 32 positions of
// FASTQ, 1,940 of text, issued on 57% and 64% of cycles.  Byte loads from global
// memory, a launch for the links and eight lookups a position took 12.4 + 1.5 ms
// of the 64 MiB FASTQ encode; this takes 2.5 ms.
template <bool SHARED>
__global__ void __launch_bounds__(512, 2) candidate_kernel(EncArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const uint32_t B = 1u << a.log2B;
  const CandShape shape = cand_shape(a.log2B);
  const uint64_t b = a.c0 + blockIdx.x, bstart = b << a.log2B;
  const uint32_t blen = (uint32_t)min(a.n - bstart, (uint64_t)B);
  const uint32_t* sb = reinterpret_cast<const uint32_t*>(smem);
  uint32_t* ent = SHARED ? reinterpret_cast<uint32_t*>(smem + B + kPadBytes) : a.entries + (blockIdx.x * (uint64_t)gridDim.y + blockIdx.y) * B;
  uint8_t* after = smem + B + kPadBytes + (SHARED ? 4 * (size_t)B : 0);
  uint16_t* heads = reinterpret_cast<uint16_t*>(after);  // [segs][2^kHashBits4]
  CandWarp& w = reinterpret_cast<CandWarp*>(after)[wid];
  const uint32_t mm = a.min_match;

  // the block and the bytes after it (zero past the input)
  const uint64_t avail = a.n - bstart;
  if ((reinterpret_cast<uintptr_t>(a.in) & 15) == 0) {
    for (uint32_t o = 16 * tid; o < B + kPadBytes; o += 16 * nt) {
      if (o + 16 <= avail) {
        *reinterpret_cast<uint4*>(smem + o) = __ldg(reinterpret_cast<const uint4*>(a.in + bstart + o));
      } else {
        for (uint32_t k = o; k < o + 16; k++) smem[k] = k < avail ? a.in[bstart + k] : (uint8_t)0;
      }
    }
  } else {
    for (uint32_t k = tid; k < B + kPadBytes; k += nt) smem[k] = k < avail ? a.in[bstart + k] : (uint8_t)0;
  }
  for (uint32_t k = tid; k < shape.segs << (kHashBits4 - 1); k += nt) reinterpret_cast<uint32_t*>(heads)[k] = ~0u;
  __syncthreads();

  // entries: link distance (0: none) in the low half, the hash in the high half
  uint16_t* ent16 = reinterpret_cast<uint16_t*>(ent);
  const uint32_t seg = B / shape.segs;
  auto bucket = [&](uint32_t p) { return (word_at(sb, p) * 2654435761u) >> (32 - kHashBits4); };
  if (wid < shape.segs) {
    uint16_t* head = heads + (wid << kHashBits4);
    const uint32_t end = min((wid + 1) * seg, blen);
    uint32_t hn = bucket(wid * seg + lane);
    for (uint32_t c = wid * seg; c < end; c += 32) {
      const uint32_t p = c + lane;
      const bool valid = p + 4 <= blen;
      const uint32_t h = valid ? hn : (1u << kHashBits4) + lane;  // invalid lanes alone
      hn = bucket(min(p + 32, B));  // the next round's, beside this one's chain
      const uint32_t grp = __match_any_sync(kFull, h);
      const uint32_t below = grp & lanemask_lt();
      uint32_t pp = 0xffffu;  // no position with four bytes left is 0xffff
      if (valid) pp = below ? c + (31 - __clz(below)) : head[h];
      __syncwarp();
      if (valid && !(grp >> lane >> 1)) head[h] = (uint16_t)p;  // the group's last lane is the new head
      __syncwarp();
      if (p < blen) ent16[2 * p] = pp != 0xffffu ? (uint16_t)(p - pp) : (uint16_t)0;
    }
  }
  // (a CTA of few warps has the linking ones hash too)
  const uint32_t hw = nw > shape.segs ? nw - shape.segs : nw, hid = nw > shape.segs ? wid - shape.segs : wid;
  if (hid < hw)
    for (uint32_t p = 32 * hid + lane; p < blen; p += 32 * hw) {
      uint32_t x = word_at(sb, p) * 0x85EBCA6Bu;
      if (mm >= 8) x = ((x >> 15) ^ x ^ word_at(sb, p + 4)) * 0x85EBCA6Bu;
      if (mm >= 12) x = ((x >> 15) ^ x ^ word_at(sb, p + 8)) * 0x85EBCA6Bu;
      if (mm >= 16) x = ((x >> 15) ^ x ^ word_at(sb, p + 12)) * 0x85EBCA6Bu;
      ent16[2 * p + 1] = (uint16_t)((x ^ (x >> 13)) >> 12);
    }
  __syncthreads();
  for (uint32_t p = seg + tid; p + 4 <= blen; p += nt) {  // the segments' firsts
    if (ent16[2 * p]) continue;
    const uint32_t h = bucket(p);
    for (uint32_t k = p / seg; k-- > 0;) {
      const uint32_t v = heads[(k << kHashBits4) + h];
      if (v != 0xffffu) {
        ent16[2 * p] = (uint16_t)(p - v);
        break;
      }
    }
  }
  __syncthreads();

  // the table's position for the key at p: in this block as an offset with the
  // top bit set, in a block that may be a source (or up to 7 bytes past those,
  // for the shift back) as it is
  const uint64_t wend = source_end(b) << a.log2B;
  auto key_of = [&](uint32_t p) -> uint32_t {
    if (p + kKey > avail) return kNoKey;
    const uint32_t* t = sb + (p >> 2);
    const uint32_t sh = 8 * (p & 3), t1 = t[1], t2 = t[2], t3 = t[3];
    const uint32_t x0 = __funnelshift_r(t[0], t1, sh), x1 = __funnelshift_r(t1, t2, sh);
    const uint32_t x2 = __funnelshift_r(t2, t3, sh), x3 = __funnelshift_r(t3, t[4], sh);
    const unsigned long long q =
        __ldg(a.table + hash_words((uint64_t)x1 << 32 | x0, (uint64_t)x3 << 32 | x2, a.bits));
    if (q >= bstart) return q - bstart < 2 * (uint64_t)B ? 0x80000000u | (uint32_t)(q - bstart) : kNoKey;
    return q < wend + kStride ? (uint32_t)q : kNoKey;
  };
  // common prefix of q and p in the block, at most kCap (never past the staged bytes)
  auto common_in = [&](uint32_t q, uint32_t p) -> uint32_t {
    const uint32_t *s = sb + (q >> 2), *t = sb + (p >> 2);
    const uint32_t sh = 8 * (q & 3), th = 8 * (p & 3);
    uint32_t u = s[0], v = t[0];
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) {
      const uint32_t u2 = s[k + 1], v2 = t[k + 1];
      const uint32_t x = __funnelshift_r(u, u2, sh) ^ __funnelshift_r(v, v2, th);
      if (x) return 4 * k + ((__ffs(x) - 1) >> 3);
      u = u2;
      v = v2;
    }
    return kCap;
  };
  // common prefix of the input at q and the block's p, at most kCap
  auto common_ex = [&](uint32_t q, uint32_t p, uint32_t lim) -> uint32_t {
    const uintptr_t A = reinterpret_cast<uintptr_t>(a.in + q);
    // the aligned words around the source, where they lie in the input
    if (q < 4 || (uint64_t)q + 40 > a.n) return common(a.in + q, a.in + bstart + p, lim);
    const uint32_t* g = reinterpret_cast<const uint32_t*>(a.in + q - (A & 3));
    const uint32_t sh = 8 * (uint32_t)(A & 3);
    const uint32_t g0 = __ldg(g), g1 = __ldg(g + 1), g2 = __ldg(g + 2);
    const uint32_t x0 = __funnelshift_r(g0, g1, sh) ^ word_at(sb, p);
    const uint32_t x1 = __funnelshift_r(g1, g2, sh) ^ word_at(sb, p + 4);
    if (x0 | x1) return x0 ? (__ffs(x0) - 1) >> 3 : 4 + ((__ffs(x1) - 1) >> 3);
    uint32_t r[7] = {g2}, l = kCap;
#pragma unroll
    for (uint32_t i = 1; i < 7; i++) r[i] = __ldg(g + 2 + i);
#pragma unroll
    for (uint32_t i = 6; i-- > 0;) {
      const uint32_t x = __funnelshift_r(r[i], r[i + 1], sh) ^ word_at(sb, p + 8 + 4 * i);
      if (x) l = 8 + 4 * i + ((__ffs(x) - 1) >> 3);
    }
    return l;
  };
  // positions of a warp: of the CTA's part of the block, a multiple of 32
  const uint32_t per = max(B / (nw * gridDim.y), 32u), first = (blockIdx.y * nw + wid) * per;
  uint2* out = a.cand + (uint64_t)blockIdx.x * B;
  uint32_t next = first < blen ? key_of(first + lane) : kNoKey;
  for (uint32_t c = first; c < min(first + per, blen); c += 32) {
    const uint32_t p = c + lane;
    __syncwarp();
    w.key[lane] = next;
    w.ext[lane] = w.own[lane] = 0;
    next = key_of(p + 32);  // in flight during the chain walk
    uint32_t li = 0, qi = 0;
    const uint32_t lim = p < blen ? min(blen - p, kCap) : 0u;
    // one chain step for the whole warp at a time, so its lanes stay together
    uint32_t e = lim >= mm ? ent[p] : 0u, q = p;
    const uint32_t mine = e >> 16;
    uint32_t tail = 0;  // the position's bytes li - 3 .. li: a longer candidate has them too
    uint32_t P[kCap / 4];
    {
      const uint32_t* t = sb + (min(p, B - 1) >> 2);
      uint32_t v = t[0];
#pragma unroll
      for (uint32_t k = 0; k < kCap / 4; k++) {
        const uint32_t v2 = t[k + 1];
        P[k] = __funnelshift_r(v, v2, 8 * (p & 3));
        v = v2;
      }
    }
    for (uint32_t depth = 0; depth < a.max_chain && __any_sync(kFull, e & 0xffffu); depth++) {
      if (!(e & 0xffffu)) continue;
      q -= e & 0xffffu;
      e = ent[q];
      if (e >> 16 != mine || (li && word_at(sb, q + li - 3) != tail)) continue;
      // common prefix with p: eight bytes, then word by word
      const uint32_t* t = sb + (q >> 2);
      const uint32_t sh = 8 * (q & 3);
      uint32_t v = t[2], l = kCap;
      const uint32_t x0 = __funnelshift_r(t[0], t[1], sh) ^ P[0], x1 = __funnelshift_r(t[1], v, sh) ^ P[1];
      if (x0 | x1) {
        l = x0 ? (__ffs(x0) - 1) >> 3 : 4 + ((__ffs(x1) - 1) >> 3);
      } else {
#pragma unroll
        for (uint32_t k = 2; k < kCap / 4; k++) {
          const uint32_t v2 = t[k + 1], x = __funnelshift_r(v, v2, sh) ^ P[k];
          if (x) {
            l = 4 * k + ((__ffs(x) - 1) >> 3);
            break;
          }
          v = v2;
        }
      }
      l = min(l, lim);
      if (l >= mm && l > li) {
        li = l;
        qi = q;
        if (l == lim) e = 0;  // none is longer
        else tail = word_at(sb, p + l - 3);
      }
    }
    if (lane < kStride - 1) w.key[32 + lane] = next;
    __syncwarp();
    // the keys' sources: every key found serves the eight positions up to its
    // own, (key, shift) pairs dealt to the lanes 32 at a time
    const uint32_t f0 = __ballot_sync(kFull, w.key[lane] != kNoKey);
    const uint32_t f1 = __ballot_sync(kFull, lane < kStride - 1 && next != kNoKey);
    const uint32_t n = __popc(f0) + __popc(f1);
    if (f0 >> lane & 1) w.found[__popc(f0 & lanemask_lt())] = (uint8_t)lane;
    if (f1 >> lane & 1) w.found[__popc(f0) + __popc(f1 & lanemask_lt())] = (uint8_t)(32 + lane);
    __syncwarp();
    for (uint32_t it = lane; it < kStride * n; it += 32) {
      const uint32_t k = w.found[it / kStride], j = it % kStride, at = k - j, pq = c + at;
      if (at >= 32 || pq >= blen) continue;  // (k < j too)
      const uint32_t room = min(blen - pq, kCap);
      const uint32_t t = w.key[k], q0 = t & 0x7fffffffu;
      if (room < mm) continue;
      if (t >> 31 && q0 >= j) {  // an earlier occurrence inside the block
        const uint32_t s = q0 - j;
        if (s >= pq || (ent[s] ^ ent[pq]) >> 16) continue;
        const uint32_t l = min(common_in(s, pq), room);
        if (l >= mm) atomicMax(&w.own[at], l << 16 | (0xffffu - s));
      } else {
        const uint64_t q64 = (t >> 31 ? bstart : 0) + q0;
        // in a block that may be a source (its length beyond it: span)
        if (q64 < j || q64 - j >= wend) continue;
        const uint32_t s = (uint32_t)(q64 - j);
        uint32_t l = min(common_ex(s, pq, room), room);
        if (l >= mm) l = span(a, s, b, l);
        if (l >= mm) atomicMax(&w.ext[at], l << 24 | (0xffffffu - s));
      }
    }
    __syncwarp();
    const uint32_t o = w.own[lane], x = w.ext[lane];
    if (o >> 16 > li || (li && o >> 16 == li && 0xffffu - (o & 0xffffu) < qi)) {
      li = o >> 16;
      qi = 0xffffu - (o & 0xffffu);
    }
    if (p < blen) out[p] = make_uint2(li | (x >> 24 << 8) | (qi << 16), 0xffffffu - (x & 0xffffffu));
  }
}

// ----------------------------------------------------------- greedy parse

// Eight bytes of the input at pos (pos + 8 <= n), from the aligned words
// around them where those lie inside the input.
__device__ __forceinline__ uint64_t ld64_in(const EncArgs& a, uint64_t pos) {
  const uint8_t* p = a.in + pos;
  const uintptr_t A = reinterpret_cast<uintptr_t>(p);
  const uint32_t sh = 8 * (uint32_t)(A & 7);
  if (!sh) return *reinterpret_cast<const uint64_t*>(p);
  const uint8_t* al = p - (A & 7);
  if (al < a.in || al + 16 > a.in + a.n) return ld64u(p);
  const uint64_t* w = reinterpret_cast<const uint64_t*>(al);
  return (w[0] >> sh) | (w[1] << (64 - sh));
}

// Common prefix of the input at q and at p (q < p), at most limit bytes, by
// the warp: eight bytes per lane, 256 a round.
__device__ __forceinline__ uint32_t common_warp(const EncArgs& a, uint64_t q, uint64_t p, uint32_t limit,
                                                uint32_t lane) {
  for (uint32_t o = 0; o < limit; o += 256) {
    const uint32_t at = o + 8 * lane;
    uint32_t l = 8;  // equal bytes among this lane's
    if (at + 8 <= limit) {
      const uint64_t x = ld64_in(a, q + at) ^ ld64_in(a, p + at);
      if (x) l = (__ffsll((long long)x) - 1) >> 3;
    } else {
      l = 0;
      while (at + l < limit && a.in[q + at + l] == a.in[p + at + l]) l++;  // at most 7
    }
    const uint32_t stop = __ballot_sync(kFull, l < 8);
    if (stop) {
      const uint32_t f = __ffs(stop) - 1;
      return min(limit, o + 8 * f + __shfl_sync(kFull, l, f));
    }
  }
  return limit;
}

// Bits [lo, hi) of word i of a bit map (those of them the word holds).
__device__ __forceinline__ uint32_t word_mask(uint32_t i, uint32_t lo, uint32_t hi) {
  uint32_t m = kFull;
  if (i == lo >> 5) m <<= lo & 31;
  if (i == (hi - 1) >> 5) m &= kFull >> (31 - ((hi - 1) & 31));
  return m;
}

// Whether the external candidate (len 0: none) is taken over the in-block one
// (len 0: none or refused): the longer one, but a shallower one within
// max(4, len / 8) bytes of it; on a tie of both, the smaller source, which is
// the external one.
__device__ __forceinline__ bool external_wins(uint32_t li, uint32_t wi, uint32_t le, uint32_t we) {
  if (!li || !le) return le != 0;
  if (we < wi) return le + max(4u, max(le, li) / 8) >= li;
  if (we > wi) return le > li + max(4u, le / 8);
  return le >= li;
}

// The greedy walk over a block's positions, a warp per block: at the first
// position with an acceptable candidate a match, literals before it.  A
// match's resolution wave is 1 + the deepest wave among the bytes of its own
// block it reads (literals and bytes of earlier blocks are wave 0); deeper
// than 3 is refused.
//
// The walk is a serial chain of decisions, so its latency bounds it.  The
// warp therefore decides 32 positions at once, a lane each, as if every
// position before them were a literal: true for the first that accepts, and
// the others are decided again after it.  The waves are three bit maps in
// shared memory (bit: wave at least 1, 2, 3), so the wave of a source of at
// most kCap bytes is two words of each.  Only candidates that extend past the
// cap, or external sources that run into the block, take the warp as a whole
// (256 bytes compared a round).  The next 32 positions' candidates load ahead.
// A thread per block with a byte per wave took 14.5 ms of the 64 MiB FASTQ
// encode and 45.8 ms of the 11 MiB text one; a warp per block that decided one
// position at a time 4.2 ms of the text one; this takes 0.33 and 0.62 ms.
__global__ void __launch_bounds__(32) parse_kernel(EncArgs a) {
  extern __shared__ uint32_t planes[];  // [3][B / 32 + 1]
  const uint32_t lane = threadIdx.x;
  const uint64_t b = a.c0 + blockIdx.x;
  const uint64_t base = a.c0 << a.log2B, bstart = b << a.log2B;
  const uint32_t blen = (uint32_t)min(a.n - bstart, (uint64_t)1 << a.log2B);
  const uint32_t words = (1u << (a.log2B - 5)) + 1;  // one past the block, for two-word reads
  uint32_t* const w1 = planes;
  uint32_t* const w2 = w1 + words;
  uint32_t* const w3 = w2 + words;
  for (uint32_t i = lane; i < 3 * words; i += 32) planes[i] = 0;
  __syncwarp();
  const uint2* cd = a.cand + (bstart - base);
  uint4* tk = reinterpret_cast<uint4*>(a.tok) + blockIdx.x * (uint64_t)a.tok_cap;
  auto load = [&](uint32_t i) { return i < blen ? __ldcg(cd + i) : make_uint2(0u, 0u); };
  uint32_t nt = 0, lit = 0, lbytes = 0, msrc = 0;
  uint32_t p = 0, wb = 0;  // positions count from the block's start; the window is [wb, wb + 32)
  uint2 cur = load(lane), nxt = load(32 + lane);
  while (p < blen) {
    if (p >= wb + 32) {
      const uint32_t nb = p & ~31u;
      cur = nb == wb + 32 ? nxt : load(nb + lane);
      wb = nb;
      nxt = load(nb + 32 + lane);
    }
    // this lane's position: 0 refused or no candidate, 1 decided, 2 left to the warp
    const uint32_t pos = wb + lane;
    const uint32_t li = cur.x & 0xffu, le = (cur.x >> 8) & 0xffu;
    uint32_t state = 0, len = 0, wave = 1;
    bool ext = false;
    if (pos >= p && (li | le)) {
      if ((max(li, le) == kCap && pos + kCap < blen) || (le && cur.y + le > bstart)) {
        state = 2;
      } else {
        uint32_t l = li;
        if (li) {
          const uint32_t q = cur.x >> 16, i = q >> 5, sh = q & 31;
          const uint32_t m = kFull >> (32 - min(li, pos - q));
          if (__funnelshift_r(w1[i], w1[i + 1], sh) & m) wave = 2;
          if (__funnelshift_r(w2[i], w2[i + 1], sh) & m) wave = 3;
          if (__funnelshift_r(w3[i], w3[i + 1], sh) & m) l = 0;
        }
        ext = external_wins(l, wave, le, 1);
        len = ext ? le : l;
        if (ext) wave = 1;
        state = len != 0;
      }
    }
    uint32_t todo = __ballot_sync(kFull, state);
    const uint32_t slow = __ballot_sync(kFull, state == 2);
    while (todo) {
      const uint32_t f = __ffs(todo) - 1, at = wb + f;
      uint32_t mlen = __shfl_sync(kFull, len | wave << 8 | (uint32_t)ext << 16, f);
      const uint32_t cx = __shfl_sync(kFull, cur.x, f), cy = __shfl_sync(kFull, cur.y, f);
      uint32_t mw = (mlen >> 8) & 0xffu;
      bool mext = mlen >> 16;
      mlen &= 0xffu;
      const uint64_t P = bstart + at, qi = bstart + (cx >> 16);
      if (slow >> f & 1) {
        const uint32_t room = blen - at;
        uint32_t fi = cx & 0xffu, fe = (cx >> 8) & 0xffu;
        if (fi == kCap && room > kCap) fi = kCap + common_warp(a, qi + kCap, P + kCap, room - kCap, lane);
        if (fe == kCap && room > kCap)
          fe = span(a, cy, b, kCap + common_warp(a, cy + kCap, P + kCap, room - kCap, lane));
        // the waves of both sources: lanes 0..15 the in-block one's words, 16..31 the external one's
        const uint64_t q = lane < 16 ? qi : cy;
        const uint32_t l = lane < 16 ? fi : fe;
        const uint32_t lo = q > bstart ? (uint32_t)(q - bstart) : 0u;
        const uint32_t hi = q + l > bstart ? (uint32_t)min(q + l - bstart, (uint64_t)at) : 0u;
        uint32_t d1 = 0, d2 = 0, d3 = 0;
        if (l && lo < hi) {
          for (uint32_t i = (lo >> 5) + (lane & 15); i <= (hi - 1) >> 5; i += 16) {
            const uint32_t m = word_mask(i, lo, hi);
            d1 |= w1[i] & m;
            d2 |= w2[i] & m;
            d3 |= w3[i] & m;
          }
        }
        const uint32_t b1 = __ballot_sync(kFull, d1), b2 = __ballot_sync(kFull, d2), b3 = __ballot_sync(kFull, d3);
        const uint32_t wi = 1 + ((b1 & 0xffffu) != 0) + ((b2 & 0xffffu) != 0), we = 1 + ((b1 >> 16) != 0) + ((b2 >> 16) != 0);
        if (b3 & 0xffffu) fi = 0;
        if ((b3 >> 16) || fe < a.min_match) fe = 0;
        mext = external_wins(fi, wi, fe, we);
        mlen = mext ? fe : fi;
        mw = mext ? we : wi;
        if (!mlen) {  // refused: a literal like the positions before it
          todo &= todo - 1;
          continue;
        }
      }
      const uint64_t src = mext ? (uint64_t)cy : qi;
      const uint32_t end = at + mlen, run = lit + (at - p);
      if (lane == 0) tk[nt] = make_uint4(run, mlen, (uint32_t)src, (uint32_t)(src >> 32));
      nt++;
      __syncwarp();  // every lane has read the maps
      for (uint32_t i = (at >> 5) + lane; i <= (end - 1) >> 5; i += 32) {
        const uint32_t m = word_mask(i, at, end);
        w1[i] |= m;
        if (mw > 1) w2[i] |= m;
        if (mw > 2) w3[i] |= m;
      }
      __syncwarp();
      lbytes += run;
      msrc += (uint32_t)min((uint64_t)mlen, P - src);
      lit = 0;
      p = end;
      break;
    }
    if (!todo) {  // literals to the window's end
      const uint32_t e = min(wb + 32, blen);
      lit += e - p;
      p = e;
    }
  }
  if (lane) return;
  tk[nt] = make_uint4(lit, 0u, 0u, 0u);  // the last token: literals only
  a.ntok[blockIdx.x] = nt + 1;
  atomicAdd(a.stats + 0, (unsigned long long)(nt + 1));
  atomicAdd(a.stats + 1, (unsigned long long)nt);
  atomicAdd(a.stats + 2, (unsigned long long)(lbytes + lit));
  atomicAdd(a.stats + 3, (unsigned long long)(blen - lbytes - lit));
  atomicAdd(a.stats + 4, (unsigned long long)msrc);
}

// ------------------------------------------------------------ block coder

struct CodeArgs {
  EncArgs e;
  uint8_t* syms;       // per chunk block: sym_cap bytes, the three streams' symbols one after another
  uint32_t sym_cap;
  uint8_t* tmp;        // per chunk block: 2 sym_cap bytes, two for each symbol's pushes
  uint8_t* pay;        // per chunk block: pay_cap bytes, the block's payload
  uint32_t pay_cap;
  ace_block_dir* dir;  // per block of the archive (stream offsets relative to the block's payload for now)
  uint32_t* pay_bytes; // per chunk block
  uint32_t* iv;        // per block of the archive: up to kHead / 2 (first, last) pairs
  uint32_t* n_iv;      // per block of the archive
};

constexpr uint32_t kIvCap = kHead / 2;  // runs of set bits in a kHead-bit map

// Frequencies of a stream as the host encoder quantises them: f_s =
// max(1, floor(n_s 4096 / n)); a shortfall goes to the most frequent symbol
// (lowest on ties), an excess is taken one at a time from the largest
// frequency above 1 (lowest on ties).  cnt: the histogram in shared memory.
// Lane l holds symbols 8l .. 8l + 7: their frequencies in f.
__device__ void quantise_warp(const uint32_t* cnt, uint32_t n, uint32_t (&f)[8], uint32_t lane) {
  uint32_t sum = 0, best = 0, most = 0;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const uint32_t s = 8 * lane + j, c = cnt[s];
    f[j] = c ? max(1u, (uint32_t)(((uint64_t)c * ACE_SCALE) / n)) : 0u;
    sum += f[j];
    if (c > best) {
      best = c;
      most = s;
    }
  }
  // most frequent, lowest symbol on ties: (count, -symbol) maximal
#pragma unroll
  for (int d = 16; d; d >>= 1) {
    const uint32_t ob = __shfl_xor_sync(kFull, best, d), om = __shfl_xor_sync(kFull, most, d);
    if (ob > best || (ob == best && om < most)) {
      best = ob;
      most = om;
    }
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
  if (sum < ACE_SCALE && (most >> 3) == lane) {
#pragma unroll
    for (int j = 0; j < 8; j++)
      if (8 * lane + j == most) f[j] += ACE_SCALE - sum;
  }
  while (sum > ACE_SCALE) {  // warp-uniform: sum is the same on every lane
    uint32_t bf = 0, bs = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < 8; j++)
      if (f[j] > 1 && f[j] > bf) {
        bf = f[j];
        bs = 8 * lane + j;
      }
#pragma unroll
    for (int d = 16; d; d >>= 1) {
      const uint32_t of = __shfl_xor_sync(kFull, bf, d), os = __shfl_xor_sync(kFull, bs, d);
      if (of > bf || (of == bf && os < bs)) {
        bf = of;
        bs = os;
      }
    }
    if ((bs >> 3) == lane) {
#pragma unroll
      for (int j = 0; j < 8; j++)
        if (8 * lane + j == bs) f[j]--;
    }
    sum--;
  }
}

// ceil(2^(31 + l) / f), l = ceil(log2 f), for f = 1 .. 4096: for x < 2^31,
// floor(x / f) = floor(2 x m / 2^32) >> l (Granlund and Montgomery, "Division
// by invariant integers using multiplication", 1994: the rounded-up multiplier
// exceeds 2^(31 + l) / f by less than 2^l / f).
struct Reciprocals {
  uint32_t m[ACE_SCALE + 1];
  constexpr Reciprocals() : m() {
    for (uint32_t f = 1, l = 0; f <= ACE_SCALE; f++) {
      while ((1u << l) < f) l++;
      m[f] = (uint32_t)(((1ull << (31 + l)) + f - 1) / f);
    }
  }
};
__device__ const Reciprocals kRecip = Reciprocals();

// One symbol as the coder needs it: x the multiplier, y = f | c << 13 | l << 25.
__device__ __forceinline__ uint2 coder_entry(uint32_t f, uint32_t c) {
  return f ? make_uint2(kRecip.m[f], f | c << 13 | (32 - __clz(f - 1)) << 25) : make_uint2(0u, 0u);
}

// n bytes from src (any alignment, with the aligned words around it readable)
// to dst (16-byte aligned), zeros up to the next multiple of 16; by a warp.
__device__ __forceinline__ void copy_padded(uint8_t* dst, const uint8_t* src, uint32_t n, uint32_t lane) {
  const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 3), sh = 8 * off;
  const uint32_t* w = reinterpret_cast<const uint32_t*>(src - off);
  for (uint32_t i = lane; i < ((n + 15) & ~15u) / 4; i += 32) {
    uint32_t v = 0;
    if (4 * i < n) {
      v = __funnelshift_r(w[i], 4 * i + 4 - off < n ? w[i + 1] : 0u, sh);
      if (4 * i + 4 > n) v &= (1u << 8 * (n - 4 * i)) - 1;
    }
    reinterpret_cast<uint32_t*>(dst)[i] = v;
  }
}

// A stream between its two halves: coded, not yet placed.
struct Coded {
  uint32_t x;        // this lane's final state
  uint32_t f[8];     // frequencies of symbols 8 lane .. 8 lane + 7
  uint32_t pushes, present, head, bytes, mode;
};

// One stream of n symbols, by a warp: frequencies from the histogram, then the
// encode from the last symbol to the first, symbol i on state i mod 32,
// pushing a state's low byte while x >= 2^19 f_s, then x <- (x / f_s) 4096 +
// x mod f_s + c_s.  The pushes go straight to their places before end
// (backwards: a symbol's bytes before those of later ones, its last push
// first), which is the byte order the decoder reads.  The chain from round to
// round is a compare, a shift, a multiply-high and a multiply-add; the
// symbols and their entries load ahead of it.
__device__ Coded code_stream_warp(const uint8_t* sym, uint32_t n, uint8_t* end, const uint32_t* cnt, uint2* tab,
                                  bool adaptive, uint32_t lane) {
  Coded r;
  r.x = ACE_RANS_L;
  r.pushes = r.present = r.head = r.bytes = r.mode = 0;
  if (n == 0) return r;
  quantise_warp(cnt, n, r.f, lane);
  uint32_t tot = 0, np = 0;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    tot += r.f[j];
    np += r.f[j] != 0;
  }
  uint32_t c = warp_incl_sum(tot, lane) - tot;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    tab[8 * lane + j] = coder_entry(r.f[j], c);
    c += r.f[j];
  }
  r.present = __reduce_add_sync(kFull, np);
  r.head = ACE_STREAM_HEAD + ((2 * r.present + 15) & ~15u);
  __syncwarp();
  uint32_t x = ACE_RANS_L;
  const uint32_t gt = kFull << lane << 1;  // the lanes of later symbols
  auto round = [&](bool act, uint2 e) {
    const uint32_t f = e.y & 0x1fffu, lim = f << (ACE_SCALE_BITS + 7);  // (L / 4096) * 256 * f = 2^19 f
    const bool k1 = act && x >= lim, k2 = act && x >> 8 >= lim;          // x < 2^31: at most two pushes
    const uint32_t b1 = __ballot_sync(kFull, k1), b2 = __ballot_sync(kFull, k2);
    uint8_t* at = end - __popc(b1 & gt) - __popc(b2 & gt);
    if (k1) at[-1] = (uint8_t)x;
    if (k2) at[-2] = (uint8_t)(x >> 8);
    end -= __popc(b1) + __popc(b2);
    r.pushes += __popc(b1) + __popc(b2);
    if (act) {
      x >>= k2 ? 16 : k1 ? 8 : 0;
      const uint32_t q = __umulhi(2 * x, e.x) >> (e.y >> 25);
      x += q * (ACE_SCALE - f) + (e.y >> 13 & 0xfffu);
    }
  };
  uint32_t i = n / 32 * 32 + lane;  // full rounds end before it
  if (n & 31) {
    const bool act = i < n;
    round(act, act ? tab[sym[i]] : make_uint2(0u, 0u));
  }
  // full rounds, the symbols three rounds ahead and the entries one
  uint32_t s0 = 0, s1 = 0;
  uint2 e = make_uint2(0u, 0u);
  if (i >= 32 + lane) e = tab[sym[i - 32]];
  if (i >= 64 + lane) s0 = sym[i - 64];
  if (i >= 96 + lane) s1 = sym[i - 96];
  while (i >= 32 + lane) {
    i -= 32;
    const uint2 cur = e;
    e = tab[s0];
    s0 = s1;
    if (i >= 96 + lane) s1 = sym[i - 96];
    round(true, cur);
  }
  r.x = x;
  r.mode = adaptive && r.head + r.pushes >= n;  // stored: the symbols verbatim
  r.bytes = r.mode ? n : r.head + r.pushes;
  return r;
}

// The coded stream's payload into out (16-byte aligned): 32 final states (the
// decoder's entry point), present bitmap, frequencies, renormalisation bytes;
// or, stored, its symbols.
__device__ void place_stream_warp(const Coded& r, const uint8_t* sym, const uint8_t* renorm, uint8_t* out,
                                  uint32_t lane) {
  if (!r.bytes) return;
  if (r.mode) {
    copy_padded(out, sym, r.bytes, lane);
    return;
  }
  reinterpret_cast<uint32_t*>(out)[lane] = r.x;
  uint32_t bm = 0;
#pragma unroll
  for (int j = 0; j < 8; j++) bm |= r.f[j] ? 1u << j : 0u;
  out[128 + lane] = (uint8_t)bm;  // bitmap byte l holds symbols 8l .. 8l + 7
  const uint32_t np = __popc(bm);
  uint16_t* fq = reinterpret_cast<uint16_t*>(out + ACE_STREAM_HEAD);
  uint32_t k = warp_incl_sum(np, lane) - np;
#pragma unroll
  for (int j = 0; j < 8; j++)
    if (r.f[j]) fq[k++] = (uint16_t)r.f[j];
  for (uint32_t i = r.present + lane; i < (r.head - ACE_STREAM_HEAD) / 2; i += 32) fq[i] = 0;
  copy_padded(out + r.head, renorm, r.pushes, lane);
}

constexpr uint32_t kCodeWarps = 4;
constexpr uint32_t kLongRun = 16;  // literal runs from here on are copied by the whole warp

// A CTA per block.  All warps: the token streams (literals in output order;
// lengths: the escape values, then two codes per token; offsets: each match's
// absolute source, w bytes) from groups of 32 tokens whose places a scan of
// the groups' totals gives, their histograms, and the dependency runs (a bit
// per earlier block a match reads, all below the window start) with the
// block's level.  Then a warp per stream codes it, and the three payloads are
// laid one after another, 16-byte aligned, in the block's payload.
//
// A warp per block did all of this in series, with a divide per symbol and a
// second pass over the symbols for the bytes' places, 2.6 ms of the 64 MiB
// FASTQ encode and 1.3 ms of the 11 MiB text one; this takes 0.41 and 0.09 ms.
// Bound by the coder's chain where
// blocks are few, by issue where they are many.
__global__ void __launch_bounds__(32 * kCodeWarps) code_kernel(CodeArgs ca) {
  extern __shared__ uint32_t group[];  // [3][groups]: bytes, literals, escapes before each group of 32 tokens
  __shared__ uint2 s_tab[3][256];
  __shared__ uint32_t s_cnt[3][256], s_bits[kHead / 32 + 2], s_total[3], s_bytes[3];
  const EncArgs& a = ca.e;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint64_t cb = blockIdx.x, b = a.c0 + cb, bstart = b << a.log2B;
  const uint4* tk = reinterpret_cast<const uint4*>(a.tok) + cb * a.tok_cap;
  const uint32_t nt = a.ntok[cb], nm = nt - 1, w = a.w, ng = (nt + 31) / 32;
  for (uint32_t i = tid; i < 3 * 256; i += 32 * kCodeWarps) (&s_cnt[0][0])[i] = 0;
  if (tid < kHead / 32 + 2) s_bits[tid] = 0;
  for (uint32_t g = wid; g < ng; g += kCodeWarps) {
    const uint32_t t = 32 * g + lane;
    const uint4 v = t < nt ? tk[t] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t r0 = __reduce_add_sync(kFull, v.x + v.y), r1 = __reduce_add_sync(kFull, v.x);
    const uint32_t r2 = __reduce_add_sync(kFull, (uint32_t)(v.x >= 255) + (v.y >= 255));
    if (lane == 0) {
      group[g] = r0;
      group[ng + g] = r1;
      group[2 * ng + g] = r2;
    }
  }
  __syncthreads();
  if (wid < 3) {
    uint32_t carry = 0;
    for (uint32_t g0 = 0; g0 < ng; g0 += 32) {
      const uint32_t v = g0 + lane < ng ? group[wid * ng + g0 + lane] : 0u;
      const uint32_t incl = warp_incl_sum(v, lane);
      if (g0 + lane < ng) group[wid * ng + g0 + lane] = carry + incl - v;
      carry += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) s_total[wid] = carry;
  }
  __syncthreads();
  const uint32_t lit_total = s_total[1], esc_total = s_total[2];
  uint8_t* lit = ca.syms + cb * (uint64_t)ca.sym_cap;
  uint8_t* lenp = lit + lit_total;                // lengths stream: 2 esc_total + 2 nt bytes
  uint8_t* offp = lenp + 2 * esc_total + 2 * nt;  // offsets stream: w nm bytes
  for (uint32_t g = wid; g < ng; g += kCodeWarps) {
    const uint32_t t = 32 * g + lane;
    const uint4 v = t < nt ? tk[t] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t lr = v.x, ml = v.y, run = lr + ml, e = (uint32_t)(lr >= 255) + (ml >= 255);
    const uint64_t src = (uint64_t)v.z | ((uint64_t)v.w << 32);
    const uint32_t my_dst = group[g] + warp_incl_sum(run, lane) - run;
    const uint32_t my_lit = group[ng + g] + warp_incl_sum(lr, lane) - lr;
    uint32_t ec = group[2 * ng + g] + warp_incl_sum(e, lane) - e;
    const uint8_t* from = a.in + bstart;
    if (lr < kLongRun)
      for (uint32_t k = 0; k < lr; k++) {
        const uint8_t s = from[my_dst + k];
        lit[my_lit + k] = s;
        atomicAdd(&s_cnt[0][s], 1u);
      }
    for (uint32_t lng = __ballot_sync(kFull, lr >= kLongRun); lng; lng &= lng - 1) {
      const uint32_t f = __ffs(lng) - 1, n = __shfl_sync(kFull, lr, f), d = __shfl_sync(kFull, my_dst, f),
                     l = __shfl_sync(kFull, my_lit, f);
      for (uint32_t k = lane; k < n; k += 32) {
        const uint8_t s = from[d + k];
        lit[l + k] = s;
        atomicAdd(&s_cnt[0][s], 1u);
      }
    }
    if (t < nt) {
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const uint32_t x = q ? ml : lr, s = min(x, 255u);
        lenp[2 * esc_total + 2 * t + q] = (uint8_t)s;
        atomicAdd(&s_cnt[1][s], 1u);
        if (x >= 255) {
          const uint32_t y = x - 255;
          lenp[2 * ec] = (uint8_t)y;
          lenp[2 * ec + 1] = (uint8_t)(y >> 8);
          atomicAdd(&s_cnt[1][y & 255], 1u);
          atomicAdd(&s_cnt[1][y >> 8], 1u);
          ec++;
        }
      }
    }
    if (t < nm) {
      for (uint32_t k = 0; k < w; k++) {
        const uint8_t s = (uint8_t)(src >> (8 * k));
        offp[w * t + k] = s;
        atomicAdd(&s_cnt[2][s], 1u);
      }
      const uint64_t D = bstart + my_dst + lr;
      if (ml && src < bstart) {  // blocks before this one that the match reads
        const uint64_t rl = min((uint64_t)ml, D - src);
        const uint64_t k0 = src >> a.log2B, k1 = min((src + rl - 1) >> a.log2B, b - 1);
        for (uint64_t k = k0; k <= k1 && k < kHead; k++) atomicOr(&s_bits[k >> 5], 1u << (k & 31));
      }
    }
  }
  __syncthreads();
  const uint32_t ns[3] = {lit_total, 2 * esc_total + 2 * nt, w * nm};
  const uint32_t k = min(wid, 2u), sym_at = k == 0 ? 0u : k == 1 ? ns[0] : ns[0] + ns[1];
  const uint32_t n = k == 0 ? ns[0] : k == 1 ? ns[1] : ns[2];
  Coded r;
  uint8_t* end = ca.tmp + cb * 2 * (uint64_t)ca.sym_cap + 2 * (sym_at + n);
  if (wid < 3) {
    r = code_stream_warp(lit + sym_at, n, end, s_cnt[wid], s_tab[wid], a.adaptive != 0, lane);
    if (lane == 0) s_bytes[wid] = r.bytes;
  } else {
    // the block's dependency runs
    uint32_t* iv = ca.iv + b * (uint64_t)(2 * kIvCap);
    const uint32_t v = lane < kHead / 32 ? s_bits[lane] : 0u;
    const uint32_t before = __shfl_up_sync(kFull, v, 1) >> 31, after = __shfl_down_sync(kFull, v, 1) << 31;
    uint32_t starts = v & ~(v << 1 | (lane ? before : 0u)), ends = v & ~(v >> 1 | after);
    const uint32_t si = warp_incl_sum(__popc(starts), lane);
    uint32_t at = si - __popc(starts);
    for (; starts; starts &= starts - 1) iv[2 * at++] = 32 * lane + __ffs(starts) - 1;
    at = warp_incl_sum(__popc(ends), lane) - __popc(ends);
    for (; ends; ends &= ends - 1) iv[2 * at++ + 1] = 32 * lane + __ffs(ends) - 1;
    if (lane == 31) ca.n_iv[b] = si;
  }
  __syncthreads();
  const uint32_t p0 = (s_bytes[0] + 15) & ~15u, p1 = (s_bytes[1] + 15) & ~15u, p2 = (s_bytes[2] + 15) & ~15u;
  const uint32_t off = wid == 0 ? 0u : wid == 1 ? p0 : p0 + p1;
  if (wid < 3) {
    place_stream_warp(r, lit + sym_at, end - r.pushes, ca.pay + cb * (uint64_t)ca.pay_cap + off, lane);
    if (lane == 0) {
      ace_block_dir& d = ca.dir[b];
      d.stream_off[wid] = off;
      d.stream_bytes[wid] = r.bytes;
      d.nsym[wid] = n;
      d.mode[wid] = (uint8_t)r.mode;
    }
  } else if (lane == 0) {
    ace_block_dir& d = ca.dir[b];
    d.ntok = nt;
    d.nesc = esc_total;
    for (int q = 0; q < 5; q++) d.reserved[q] = 0;
    ca.pay_bytes[cb] = p0 + p1 + p2;
  }
}

// ------------------------------------------------------ payload placement

struct EncHdr {
  uint32_t status;
  uint32_t max_level;
  uint64_t payload;   // payload bytes placed so far
  uint64_t n_iv;      // dependency runs in the archive
  unsigned long long stats[5];
  uint8_t pad[256 - 64];
};
static_assert(sizeof(EncHdr) == 256, "encoder header");

struct PlaceArgs {
  EncHdr* h;
  const uint32_t* pay_bytes;  // per chunk block
  uint64_t* pay_off;          // per chunk block: offset from the payload's start
  ace_block_dir* dir;
  uint64_t c0, cn;            // the chunk's first block and block count
  const uint8_t* pay;
  uint32_t pay_cap;
  uint8_t* arc;               // the archive's buffer
  uint64_t arc_cap;
  uint64_t reserve;           // where the payload is assembled, or
  uint64_t fixed;             // (not 0) once the dependency runs are counted: it starts after these bytes and the runs
};

// Where the payload goes in the archive's buffer.
__device__ __forceinline__ uint64_t payload_start(const PlaceArgs& p) {
  return p.fixed ? align16(p.fixed + 8 * p.h->n_iv) : p.reserve;
}

// One CTA: the chunk's block payloads laid end to end after the payload so
// far (each a multiple of 16 bytes), their directory offsets made relative
// to the payload's start.
__global__ void place_scan_kernel(PlaceArgs p) {
  __shared__ unsigned long long carry, wsum[32];
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) carry = p.h->payload;
  __syncthreads();
  for (uint64_t c0 = 0; c0 < p.cn; c0 += blockDim.x) {
    const uint64_t i = c0 + threadIdx.x;
    const unsigned long long v = i < p.cn ? p.pay_bytes[i] : 0;
    unsigned long long incl = v;
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long u = __shfl_up_sync(kFull, incl, d);
      if (lane >= (uint32_t)d) incl += u;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      unsigned long long x = lane < nw ? wsum[lane] : 0, xi = x;
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long u = __shfl_up_sync(kFull, xi, d);
        if (lane >= (uint32_t)d) xi += u;
      }
      if (lane < nw) wsum[lane] = xi - x;
    }
    __syncthreads();
    const unsigned long long at = carry + wsum[wid] + incl - v;
    if (i < p.cn) {
      p.pay_off[i] = at;
      ace_block_dir& d = p.dir[p.c0 + i];
      for (int k = 0; k < 3; k++) d.stream_off[k] += at;
    }
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = at + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (payload_start(p) + carry > p.arc_cap) p.h->status = ACE_E_NOMEM;  // this chunk and later ones are not copied
    p.h->payload = carry;
  }
}

// A warp per block: its payload to its place (16-byte pieces).
__global__ void place_copy_kernel(PlaceArgs p) {
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint64_t i = blockIdx.x * (uint64_t)(blockDim.x >> 5) + wid;
  if (i >= p.cn || *(volatile uint32_t*)&p.h->status) return;
  const uint4* src = reinterpret_cast<const uint4*>(p.pay + i * (uint64_t)p.pay_cap);
  uint4* dst = reinterpret_cast<uint4*>(p.arc + payload_start(p) + p.pay_off[i]);
  const uint32_t n16 = p.pay_bytes[i] / 16;
  for (uint32_t k = lane; k < n16; k += 32) dst[k] = src[k];
}

// ---------------------------------------------------------------- assembly

struct AsmArgs {
  EncHdr* h;
  const uint32_t* n_iv;   // per block
  const uint32_t* iv;     // per block: kIvCap pairs
  uint32_t* dep_ptr;      // scratch: nb + 1
  uint32_t* level;        // per block
  uint64_t nb;
};

// A block's level by the warp: 1 + the deepest block it reads.
__device__ __forceinline__ void block_level(const AsmArgs& a, uint64_t b, uint32_t lane) {
  const uint2* runs = reinterpret_cast<const uint2*>(a.iv) + b * kIvCap;
  const uint32_t n = a.n_iv[b];
  uint32_t l = 0;
  for (uint32_t i = lane; i < n; i += 32) {
    const uint2 r = runs[i];
    for (uint32_t k = r.x; k <= r.y; k++) l = max(l, a.level[k] + 1);
  }
  l = __reduce_max_sync(kFull, l);
  if (lane == 0) a.level[b] = l;
}

// The levels: HEAD, one CTA over the windows that may be sources, one after
// another; without it the blocks after them, a warp per block.
template <bool HEAD>
__global__ void level_kernel(AsmArgs a) {
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (HEAD) {
    for (uint32_t w = 0; w < kHead; w += kWin) {
      for (uint64_t b = w + wid; b < min((uint64_t)w + kWin, a.nb); b += nw) block_level(a, b, lane);
      __syncthreads();
    }
  } else {
    const uint64_t b = kHead + blockIdx.x * (uint64_t)nw + wid;
    if (b < a.nb) block_level(a, b, lane);
  }
}

// One CTA: the dependency table's pointers (exclusive prefix of the runs),
// the total, and the deepest level.
__global__ void deps_scan_kernel(AsmArgs a) {
  __shared__ uint32_t carry, wsum[32], lmax;
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) {
    carry = 0;
    lmax = 0;
  }
  __syncthreads();
  for (uint64_t c0 = 0; c0 < a.nb; c0 += blockDim.x) {
    const uint64_t i = c0 + threadIdx.x;
    const uint32_t v = i < a.nb ? a.n_iv[i] : 0;
    if (i < a.nb) atomicMax(&lmax, a.level[i]);
    const uint32_t incl = warp_incl_sum(v, lane);
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      const uint32_t x = lane < nw ? wsum[lane] : 0, xi = warp_incl_sum(x, lane);
      if (lane < nw) wsum[lane] = xi - x;
    }
    __syncthreads();
    const uint32_t at = carry + wsum[wid] + incl - v;
    if (i < a.nb) a.dep_ptr[i] = at;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = at + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    a.dep_ptr[a.nb] = carry;
    a.h->n_iv = carry;
    a.h->max_level = lmax;
  }
}

// The directory and the dependency table into the archive, a warp per block:
// its directory entry, its pointer, and its runs at that pointer.  (A thread
// per block took 23 us for the 704 blocks of 11 MiB of text, 33 for the 4096 of
// 64 MiB of FASTQ; this takes 3 and 5.)
__global__ void deps_write_kernel(AsmArgs a, const ace_block_dir* dir, uint8_t* arc, uint64_t dir_off,
                                  uint64_t deps_off) {
  const uint32_t lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  uint32_t* const ptr = reinterpret_cast<uint32_t*>(arc + deps_off);
  for (uint64_t i = blockIdx.x * (uint64_t)nw + (threadIdx.x >> 5); i <= a.nb; i += (uint64_t)gridDim.x * nw) {
    const uint32_t at = a.dep_ptr[i];
    if (lane == 0) ptr[i] = at;
    if (i == a.nb) continue;
    static_assert(sizeof(ace_block_dir) == 64, "directory entry");
    if (lane < 16)
      reinterpret_cast<uint32_t*>(arc + dir_off + 64 * i)[lane] = reinterpret_cast<const uint32_t*>(dir + i)[lane];
    uint32_t* ivs = ptr + a.nb + 1 + 2ull * at;
    const uint32_t* src = a.iv + i * (uint64_t)(2 * kIvCap);
    for (uint32_t k = lane; k < 2 * a.n_iv[i]; k += 32) ivs[k] = src[k];
  }
}

}  // namespace

// --------------------------------------------------------------- host side

namespace {

struct EncLayout {
  uint64_t table, level, dir, iv, n_iv, dep_ptr, hdr, entries, cand, tok, ntok, syms, tmp, pay,
      pay_bytes, pay_off, total;
  uint64_t nb, chunk, reserve, arc_bound, entry_blocks;
  uint32_t bits, tok_cap, sym_cap, pay_cap;
};

inline uint64_t a256(uint64_t v) { return (v + 255) & ~255ull; }

ace_status enc_layout(uint64_t n, const ace_encode_params* p, EncLayout* L) {
  if (!p || p->log2_block < ACE_MIN_LOG2_BLOCK || p->log2_block > ACE_MAX_LOG2_BLOCK || p->min_match < 4 ||
      p->adaptive > 1 || p->max_chain > kMaxChain)
    return ACE_E_INVAL;
  if (p->off_width != 0 && p->off_width != 4 && p->off_width != 5) return ACE_E_INVAL;
  if (p->off_width == 4 && n > (1ull << 32)) return ACE_E_INVAL;
  const uint64_t B = 1ull << p->log2_block;
  L->nb = (n + B - 1) / B;
  if (L->nb > 0xFFFFFFF0ull) return ACE_E_INVAL;
  uint64_t want = std::max<uint64_t>(1, n / kStride);
  L->bits = 10;
  while (L->bits < 27 && (1ull << L->bits) < want) L->bits++;
  const uint64_t chunk = p->threads ? p->threads : std::max<uint64_t>(kWin, (64ull << 20) >> p->log2_block);
  L->chunk = std::max<uint64_t>(1, std::min<uint64_t>(chunk, std::max<uint64_t>(L->nb, 1)));
  L->tok_cap = (uint32_t)(B / p->min_match + 2);
  L->sym_cap = (uint32_t)align16(B + 11ull * L->tok_cap);
  L->pay_cap = (uint32_t)align16(3ull * (ACE_STREAM_HEAD + 2 * 256 + 16) + 2ull * L->sym_cap + 64);
  const uint64_t nb = L->nb, C = L->chunk, cb = C * B;
  uint64_t o = 0;
  L->hdr = o;
  o = a256(o + sizeof(EncHdr));
  L->table = o;
  o = a256(o + (8ull << L->bits));
  L->level = o;
  o = a256(o + 4 * nb);
  L->dir = o;
  o = a256(o + 64 * nb);
  L->iv = o;
  o = a256(o + 8ull * kIvCap * nb);
  L->n_iv = o;
  o = a256(o + 4 * nb);
  L->dep_ptr = o;
  o = a256(o + 4 * (nb + 1));
  L->entries = o;
  // (an array per part where a launch's blocks are split)
  L->entry_blocks = cand_shape(p->log2_block).shared_entries ? 0 : 2 * C <= kSplitEntries ? 2 * C : C;
  o = a256(o + 4 * B * L->entry_blocks);
  L->cand = o;
  o = a256(o + 8 * cb);
  L->tok = o;
  o = a256(o + 16ull * L->tok_cap * C);
  L->ntok = o;
  o = a256(o + 4 * C);
  L->syms = o;
  o = a256(o + (uint64_t)L->sym_cap * C);
  L->tmp = o;
  o = a256(o + 2ull * L->sym_cap * C);
  L->pay = o;
  o = a256(o + (uint64_t)L->pay_cap * C);
  L->pay_bytes = o;
  o = a256(o + 4 * C);
  L->pay_off = o;
  o = a256(o + 8 * C);
  L->total = o;
  // the payload is assembled after room for the largest header, directory
  // and dependency table, then moved down against the table's real size
  L->reserve = a256(sizeof(ace_file_header) + 64 * nb + 4 * (nb + 1) + 8ull * kIvCap * nb);
  L->arc_bound = L->reserve + nb * (uint64_t)L->pay_cap + 256;
  return ACE_OK;
}

}  // namespace

extern "C" {

ace_status ace_encode_gpu_size(uint64_t n, const ace_encode_params* params, uint64_t* scratch_bytes,
                               uint64_t* arc_bound) {
  EncLayout L;
  ace_status rc = enc_layout(n, params, &L);
  if (rc) return rc;
  if (scratch_bytes) *scratch_bytes = L.total;
  if (arc_bound) *arc_bound = L.arc_bound;
  return ACE_OK;
}

#define ENC_TRY(x)                              \
  do {                                          \
    if ((x) != cudaSuccess) return ACE_E_CUDA;  \
  } while (0)

ace_status ace_encode_gpu(const void* d_in, uint64_t n, const ace_encode_params* params, void* d_scratch,
                          uint64_t scratch_bytes, void* d_arc, uint64_t arc_cap, uint64_t* h_arc_len,
                          ace_encode_stats* h_stats, cudaStream_t s) {
  EncLayout L;
  ace_status rc = enc_layout(n, params, &L);
  if (rc) return rc;
  if ((!d_in && n) || !d_scratch || !d_arc || !h_arc_len) return ACE_E_INVAL;
  if ((reinterpret_cast<uintptr_t>(d_scratch) & 255) || (reinterpret_cast<uintptr_t>(d_arc) & 255))
    return ACE_E_INVAL;
  if (scratch_bytes < L.total || arc_cap < L.reserve + 256) return ACE_E_NOMEM;
  uint8_t* base = static_cast<uint8_t*>(d_scratch);
  uint8_t* arc = static_cast<uint8_t*>(d_arc);
  const uint64_t nb = L.nb, B = 1ull << params->log2_block;
  const uint32_t w = (n > (1ull << 32) || params->off_width == 5) ? 5 : 4;
  EncHdr* hdr = reinterpret_cast<EncHdr*>(base + L.hdr);
  ENC_TRY(cudaMemsetAsync(base + L.hdr, 0, sizeof(EncHdr), s));
  ENC_TRY(cudaMemsetAsync(base + L.table, 0xff, 8ull << L.bits, s));
  EncArgs e{};
  e.in = static_cast<const uint8_t*>(d_in);
  e.n = n;
  e.log2B = params->log2_block;
  e.min_match = params->min_match;
  e.max_chain = params->max_chain ? params->max_chain : 16;
  e.w = w;
  e.adaptive = params->adaptive;
  e.bits = L.bits;
  e.table = reinterpret_cast<unsigned long long*>(base + L.table);
  e.entries = reinterpret_cast<uint32_t*>(base + L.entries);
  e.cand = reinterpret_cast<uint2*>(base + L.cand);
  e.tok = reinterpret_cast<uint32_t*>(base + L.tok);
  e.tok_cap = L.tok_cap;
  e.ntok = reinterpret_cast<uint32_t*>(base + L.ntok);
  e.stats = hdr->stats;
  CodeArgs ca;
  ca.syms = base + L.syms;
  ca.sym_cap = L.sym_cap;
  ca.tmp = base + L.tmp;
  ca.pay = base + L.pay;
  ca.pay_cap = L.pay_cap;
  ca.dir = reinterpret_cast<ace_block_dir*>(base + L.dir);
  ca.pay_bytes = reinterpret_cast<uint32_t*>(base + L.pay_bytes);
  ca.iv = reinterpret_cast<uint32_t*>(base + L.iv);
  ca.n_iv = reinterpret_cast<uint32_t*>(base + L.n_iv);
  PlaceArgs pa;
  pa.h = hdr;
  pa.pay_bytes = ca.pay_bytes;
  pa.pay_off = reinterpret_cast<uint64_t*>(base + L.pay_off);
  pa.dir = ca.dir;
  pa.pay = ca.pay;
  pa.pay_cap = L.pay_cap;
  pa.arc = arc;
  pa.arc_cap = arc_cap;
  pa.reserve = L.reserve;
  if (n >= kKey) {
    const uint64_t nkeys = (n - kKey) / kStride + 1;
    table_kernel<<<(uint32_t)std::min<uint64_t>((nkeys + 255) / 256, 65535ull * 8), 256, 0, s>>>(e);
  }
  const CandShape shape = cand_shape(params->log2_block);
  int dev = 0, num_sms = 0;
  ENC_TRY(cudaGetDevice(&dev));
  ENC_TRY(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
  for (auto k : {candidate_kernel<true>, candidate_kernel<false>})  // the most either asks for, whatever the block size
    ENC_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)std::max(cand_shape(15).smem, cand_shape(16).smem)));
  AsmArgs aa;
  aa.h = hdr;
  aa.n_iv = ca.n_iv;
  aa.iv = ca.iv;
  aa.dep_ptr = reinterpret_cast<uint32_t*>(base + L.dep_ptr);
  aa.level = reinterpret_cast<uint32_t*>(base + L.level);
  aa.nb = nb;
  auto count_runs = [&] {
    level_kernel<true><<<1, 1024, 0, s>>>(aa);
    if (nb > kHead) level_kernel<false><<<(uint32_t)((nb - kHead + 7) / 8), 256, 0, s>>>(aa);
    deps_scan_kernel<<<1, 1024, 0, s>>>(aa);
  };
  // An input of one launch places its payload where it stays: the runs are
  // counted before.  One of several places it above room for the largest table
  // and moves it down in the end, in copies no longer than the gap between the
  // two (22 copies, 127 us, for 64 MiB of FASTQ).
  const bool whole = nb <= L.chunk;
  pa.fixed = whole ? sizeof(ace_file_header) + 64 * nb + 4 * (nb + 1) : 0;
  // As many blocks at once as the scratch holds.  Levels come after all of them,
  // so the first windows run beside the rest, where they had been four rounds
  // of launches, each as long as its slowest block: 11 MiB of text 3.75 ms, now 1.90; 64
  // MiB of FASTQ 5.1 and 3.7 ms.
  for (e.c0 = 0; e.c0 < nb; e.c0 += L.chunk) {
    const uint64_t cn = std::min(nb - e.c0, L.chunk);
    // a launch of few blocks splits each over CTAs until there are two per SM;
    // every part links the whole block again, so no further than needed (text:
    // 256 KiB 804 us split, 910 unsplit, 1 MiB 842 and 933, 3 MiB 1151 and 1133)
    uint32_t parts = 1;
    while (parts < kCandParts && cn * parts < 2ull * num_sms && B / shape.threads >= 2 * parts &&
           (shape.shared_entries || 2 * cn * parts <= L.entry_blocks))
      parts *= 2;
    (shape.shared_entries ? candidate_kernel<true> : candidate_kernel<false>)<<<dim3((uint32_t)cn, parts), shape.threads,
                                                                                shape.smem, s>>>(e);
    parse_kernel<<<(uint32_t)cn, 32, 3 * (B / 8 + 4), s>>>(e);  // at most 24.1 KB of bit maps
    ca.e = e;
    code_kernel<<<(uint32_t)cn, 32 * kCodeWarps, 12 * ((L.tok_cap + 31) / 32), s>>>(ca);
    pa.c0 = e.c0;
    pa.cn = cn;
    if (whole) count_runs();
    place_scan_kernel<<<1, 1024, 0, s>>>(pa);
    place_copy_kernel<<<(uint32_t)((cn + 7) / 8), 256, 0, s>>>(pa);
  }
  if (nb && !whole) count_runs();
  ENC_TRY(cudaGetLastError());
  EncHdr h;
  ENC_TRY(cudaMemcpyAsync(&h, hdr, sizeof h, cudaMemcpyDeviceToHost, s));
  ENC_TRY(cudaStreamSynchronize(s));
  if (h.status) return (ace_status)h.status;
  ace_file_header fh{};
  fh.magic = ACE_MAGIC;
  fh.version = ACE_VERSION;
  fh.n_streams = ACE_NSTREAMS;
  fh.n_states = ACE_NSTATES;
  fh.scale_bits = ACE_SCALE_BITS;
  fh.off_width = (uint8_t)w;
  fh.log2_block = (uint8_t)params->log2_block;
  fh.total_size = n;
  fh.n_blocks = nb;
  fh.dir_off = sizeof(ace_file_header);
  fh.deps_off = fh.dir_off + 64 * nb;
  fh.payload_off = align16(fh.deps_off + 4 * (nb + 1) + 8 * h.n_iv);
  fh.archive_bytes = align16(fh.payload_off + h.payload);
  if (fh.archive_bytes > arc_cap || fh.payload_off > L.reserve) return ACE_E_NOMEM;
  ENC_TRY(cudaMemsetAsync(arc, 0, fh.payload_off, s));
  if (nb) {
    deps_write_kernel<<<(uint32_t)std::min<uint64_t>((nb + 8) / 8, 65535), 256, 0, s>>>(aa, ca.dir, arc, fh.dir_off,
                                                                                           fh.deps_off);
    // the payload down to its place, in pieces no longer than the gap
    const uint64_t gap = whole ? 0 : L.reserve - fh.payload_off;
    for (uint64_t o = 0; o < h.payload;) {
      const uint64_t len = gap ? std::min(gap, h.payload - o) : h.payload;
      if (gap) ENC_TRY(cudaMemcpyAsync(arc + fh.payload_off + o, arc + L.reserve + o, len, cudaMemcpyDeviceToDevice, s));
      o += len;
    }
  }
  if (fh.archive_bytes > fh.payload_off + h.payload)
    ENC_TRY(cudaMemsetAsync(arc + fh.payload_off + h.payload, 0, fh.archive_bytes - fh.payload_off - h.payload, s));
  ENC_TRY(cudaMemcpyAsync(arc, &fh, sizeof fh, cudaMemcpyHostToDevice, s));
  ENC_TRY(cudaGetLastError());
  ENC_TRY(cudaStreamSynchronize(s));
  *h_arc_len = fh.archive_bytes;
  if (h_stats) {
    h_stats->n_tokens = h.stats[0];
    h_stats->n_matches = h.stats[1];
    h_stats->literal_bytes = h.stats[2];
    h_stats->match_bytes = h.stats[3];
    h_stats->match_src_bytes = h.stats[4];
    h_stats->n_dep_intervals = h.n_iv;
    h_stats->n_levels = nb ? h.max_level + 1 : 0;
    h_stats->reserved = 0;
  }
  return ACE_OK;
}

}  // extern "C"
