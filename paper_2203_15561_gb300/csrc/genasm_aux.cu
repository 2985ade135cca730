// Input stage of the hot path: ASCII -> 2-bit packer, and the output stage:
// dense CIGARs.
//
// Packer: each thread turns 16 ASCII bytes (one 16-byte load) into 4 packed
// bytes (one 4-byte store), four such chunks at a time, so both sides of the
// copy are fully coalesced. 1.25 bytes move per base: bound by memory, 185 us for
// a gigabase (6.76 TB/s, 99% of the measured copy rate). The integer ALU would
// take 360 at 28 operations per four bases (what a code and an exact test per
// letter took: 311 us a gigabase); the word-wide forms below take 9.
#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

#include "genasm_admit.h"
#include "genasm_internal.h"

namespace ga {

// A/a->0, C/c->1, G/g->2, T/t->3: bits 1-2 of the byte, with the G/T pair
// swapped by xoring bit 2 into bit 1. `ok` reports whether c is one of the
// eight accepted letters.
__device__ __forceinline__ uint32_t code_of(uint32_t c, bool& ok) {
  const uint32_t u = c | 0x20u;
  ok = u == 'a' || u == 'c' || u == 'g' || u == 't';
  return ok ? (((c >> 1) ^ (c >> 2)) & 3u) : 0u;
}

// The codes of a word's four letters, code q at bits 8q + 1 and 8q + 2 (bit 2
// of the letter, and bits 1 and 2 xored; other letters: anything).
__device__ __forceinline__ uint32_t word_codes(uint32_t w) { return (w ^ (w >> 1)) & 0x06060606u; }

// One multiplication brings the four codes together: the byte is bits 24..31.
// (Code q moves up by 23 - 6q bits; no two of the sixteen products overlap.)
__device__ __forceinline__ uint32_t gather_codes(uint32_t c) { return c * 0x820820u; }

// Zero in each byte that is an accepted letter. Those are 01x0 or 01x1 in the
// high half and, with b4 the bit that tells T from the others, b0 = !b4, b3 = 0
// and b4 = b2 & !b1. (Left shifts move bits of a byte into bit 4 of the same
// byte, whatever the neighbours hold.)
__device__ __forceinline__ uint32_t not_letters(uint32_t w) {
  const uint32_t x = w ^ ((w << 2) & ~(w << 3));  // bit 4: b4 ^ (b2 & !b1)
  const uint32_t v = x | ~(w ^ (w << 4));         // bit 4: that, or b4 = b0
  return (v & 0x10101010u) | ((w ^ 0x40404040u) & 0xC8C8C8C8u);
}

// word_codes with 0 for other letters, which are counted in `bad`.
__device__ __forceinline__ uint32_t checked_codes(uint32_t w, uint32_t& bad) {
  const uint32_t t = not_letters(w);
  const uint32_t no = (((t & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | t) & 0x80808080u;  // 0x80 in nonzero bytes
  bad += static_cast<uint32_t>(__popc(no));
  return word_codes(w) & ~((no >> 5) | (no >> 6));
}

// The four bases of a word as one byte (base q at bits 2q).
__device__ __forceinline__ uint32_t pack4(uint32_t w, uint32_t& bad) {
  return gather_codes(checked_codes(w, bad)) >> 24;
}

// Sixteen bases. Other letters are rare: the words are tested together, and only
// a chunk that holds one takes the exact form.
__device__ __forceinline__ uint32_t pack16(const uint4& v, uint32_t& bad) {
  uint32_t a = word_codes(v.x), b = word_codes(v.y), c = word_codes(v.z), d = word_codes(v.w);
  if ((not_letters(v.x) | not_letters(v.y)) | (not_letters(v.z) | not_letters(v.w))) {
    a = checked_codes(v.x, bad);
    b = checked_codes(v.y, bad);
    c = checked_codes(v.z, bad);
    d = checked_codes(v.w, bad);
  }
  return __byte_perm(__byte_perm(gather_codes(a), gather_codes(b), 0x0073),
                     __byte_perm(gather_codes(c), gather_codes(d), 0x0073), 0x5410);
}

// kLong: an input far larger than L2 (see launch_pack).
template <bool kLong>
__global__ void pack_kernel(const uint8_t* __restrict__ ascii, uint64_t n, uint8_t* __restrict__ out,
                            uint32_t* __restrict__ n_invalid) {
  const uint64_t chunks = n / 16;
  uint32_t bad = 0;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  const auto letters = [](const uint4* at) { return kLong ? __ldg(at) : __ldcs(at); };
  const uint4* in = reinterpret_cast<const uint4*>(ascii);
  uint32_t* to = reinterpret_cast<uint32_t*>(out);
  uint64_t q = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  // Four chunks per iteration: their 16-byte loads are in flight together.
  for (; q + 3 * stride < chunks; q += 4 * stride) {
    uint4 v[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) v[x] = letters(in + q + x * stride);
#pragma unroll
    for (int x = 0; x < 4; ++x) to[q + x * stride] = pack16(v[x], bad);
  }
  for (; q < chunks; q += stride) to[q] = pack16(letters(in + q), bad);
  // Tail (n % 16 bytes): one thread, byte by byte.
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (uint64_t x = chunks * 16; x < n; x += 4) {
      uint32_t byte = 0;
      for (uint64_t y = x; y < x + 4 && y < n; ++y) {
        bool ok;
        byte |= code_of(ascii[y], ok) << (2 * (y - x));
        bad += ok ? 0u : 1u;
      }
      out[x / 4] = static_cast<uint8_t>(byte);
    }
  }
  if (n_invalid && bad) atomicAdd(n_invalid, bad);
}

// ASCII at any address, the output 4-aligned. A thread's 16 letters lie in two
// aligned 16-byte blocks (the second is the next thread's first, in L1 by then):
// loaded whole and shifted into place, `shift` bytes (1..15). The letters of the
// blocks that are not wholly the sequence's, at its two ends, go byte by byte. A
// gigabase 214 us (the loads of L1 are twice the aligned form's), byte by byte 1,483.
__global__ void pack_shifted_kernel(const uint8_t* __restrict__ ascii, uint64_t n, uint32_t shift,
                                    uint8_t* __restrict__ out, uint32_t* __restrict__ n_invalid) {
  uint32_t bad = 0;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  const uint64_t first = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const uint4* in = reinterpret_cast<const uint4*>(ascii - shift);
  uint32_t* to = reinterpret_cast<uint32_t*>(out);
  // Chunk q is in blocks q and q + 1, which lie within the sequence for q = 1 ..
  // whole - 2 (block 0 begins before it, block `whole` ends past it).
  const uint64_t whole = (n + shift) / 16;
  const uint64_t end = whole >= 2 ? whole - 1 : 0;
  const bool by2 = (shift & 8u) != 0, by1 = (shift & 4u) != 0;
  const uint32_t bits = 8u * (shift & 3u);
  const auto chunk = [&](const uint4& x, const uint4& y) {
    // Words from shift / 4 on, then the bits.
    const uint32_t a0 = by2 ? x.z : x.x, a1 = by2 ? x.w : x.y, a2 = by2 ? y.x : x.z, a3 = by2 ? y.y : x.w,
                   a4 = by2 ? y.z : y.x, a5 = by2 ? y.w : y.y;
    const uint32_t b0 = by1 ? a1 : a0, b1 = by1 ? a2 : a1, b2 = by1 ? a3 : a2, b3 = by1 ? a4 : a3,
                   b4 = by1 ? a5 : a4;
    return make_uint4(__funnelshift_r(b0, b1, bits), __funnelshift_r(b1, b2, bits),
                      __funnelshift_r(b2, b3, bits), __funnelshift_r(b3, b4, bits));
  };
  uint64_t q = first + 1;
  for (; q + 3 * stride < end; q += 4 * stride) {
    uint4 v[4], u[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      v[x] = __ldg(in + q + x * stride);
      u[x] = __ldg(in + q + x * stride + 1);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) to[q + x * stride] = pack16(chunk(v[x], u[x]), bad);
  }
  for (; q < end; q += stride) to[q] = pack16(chunk(__ldg(in + q), __ldg(in + q + 1)), bad);
  // The first chunk and those from `end` on, a byte of four letters each.
  const uint64_t nb = (n + 3) / 4, head = min(nb, static_cast<uint64_t>(4));
  const uint64_t tail = max(head, 4 * end);
  if (first < head + (nb - tail)) {
    const uint64_t o = first < head ? first : tail + (first - head);
    uint32_t byte = 0;
    for (uint64_t y = 4 * o; y < 4 * o + 4 && y < n; ++y) {
      bool ok;
      byte |= code_of(ascii[y], ok) << (2 * (y - 4 * o));
      bad += ok ? 0u : 1u;
    }
    out[o] = static_cast<uint8_t>(byte);
  }
  if (n_invalid && bad) atomicAdd(n_invalid, bad);
}

// Any alignment: one thread per output byte.
__global__ void pack_bytes_kernel(const uint8_t* __restrict__ ascii, uint64_t n,
                                  uint8_t* __restrict__ out, uint32_t* __restrict__ n_invalid) {
  const uint64_t nb = (n + 3) / 4;
  uint32_t bad = 0;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t q = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < nb;
       q += stride) {
    uint32_t byte = 0;
    for (uint64_t y = 4 * q; y < 4 * q + 4 && y < n; ++y) {
      bool ok;
      byte |= code_of(ascii[y], ok) << (2 * (y - 4 * q));
      bad += ok ? 0u : 1u;
    }
    out[q] = static_cast<uint8_t>(byte);
  }
  if (n_invalid && bad) atomicAdd(n_invalid, bad);
}

// Many sequences at once: segment q packs segs[q].bytes ASCII bytes (a
// multiple of 4, starting 4-aligned) from ascii + segs[q].src into
// out + segs[q].dst, one output byte per four bases. Block row y handles
// segments y, y + gridDim.y, ...
__global__ void pack_segments_kernel(const uint8_t* __restrict__ ascii,
                                     const PackSegment* __restrict__ segs, uint32_t n_segs,
                                     uint8_t* __restrict__ out) {
  for (uint32_t q = blockIdx.y; q < n_segs; q += gridDim.y) {
    const PackSegment g = segs[q];
    const uint32_t* src = reinterpret_cast<const uint32_t*>(ascii + g.src);
    uint8_t* dst = out + g.dst;
    const uint64_t words = g.bytes / 4;
    uint32_t bad = 0;
    for (uint64_t w = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; w < words;
         w += static_cast<uint64_t>(gridDim.x) * blockDim.x)
      dst[w] = static_cast<uint8_t>(pack4(__ldcs(src + w), bad));
  }
}

cudaError_t launch_pack_segments(const uint8_t* ascii, const PackSegment* segs, uint32_t n_segs,
                                 uint64_t max_bytes, uint8_t* out, cudaStream_t s) {
  if (n_segs == 0) return cudaSuccess;
  const uint64_t words = max_bytes / 4;
  const uint32_t bx = static_cast<uint32_t>(std::min<uint64_t>((words + 255) / 256, 64));
  const uint32_t by = std::min<uint32_t>(n_segs, 4096);
  pack_segments_kernel<<<dim3(bx > 0 ? bx : 1, by), 256, 0, s>>>(ascii, segs, n_segs, out);
  count_launches(1);
  return cudaGetLastError();
}

__global__ void scatter_slots_kernel(const SlotRecord* __restrict__ recs, uint32_t n,
                                     uint64_t* __restrict__ read_off, uint64_t* __restrict__ ref_off,
                                     uint64_t* __restrict__ cigar_off, uint32_t* __restrict__ read_len,
                                     uint32_t* __restrict__ ref_len, uint32_t* __restrict__ cigar_cap,
                                     SlotState* __restrict__ state) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const SlotRecord r = recs[i];
    read_off[r.slot] = r.read_off;
    ref_off[r.slot] = r.ref_off;
    cigar_off[r.slot] = r.cigar_off;
    read_len[r.slot] = r.read_len;
    ref_len[r.slot] = r.ref_len;
    cigar_cap[r.slot] = r.cigar_cap;
    state[r.slot] = SlotState{};
  }
}

cudaError_t launch_scatter_slots(const SlotRecord* recs, uint32_t n, uint64_t* read_off,
                                 uint64_t* ref_off, uint64_t* cigar_off, uint32_t* read_len,
                                 uint32_t* ref_len, uint32_t* cigar_cap, SlotState* state,
                                 cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t blocks = std::min<uint32_t>((n + 255) / 256, 1024);
  scatter_slots_kernel<<<blocks, 256, 0, s>>>(recs, n, read_off, ref_off, cigar_off, read_len,
                                              ref_len, cigar_cap, state);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_pack(const uint8_t* ascii, uint64_t n, uint8_t* packed, uint32_t* n_invalid,
                        cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const uint64_t chunks = n / 16;
  const uint64_t want = (chunks + 255) / 256;
  // Eight resident blocks per SM, and letters marked as not to be kept, so that L2
  // holds the packed bases for the alignment. From 320 MB on 64 blocks, that start
  // as others end and keep the reads of all SMs close together, and plain loads
  // (us, both ways: 100 MB 31, 38; 200 MB 48, 51; 300 MB 70, 70; 400 MB 94, 86;
  // 600 MB 146, 118; 1 GB 234, 186).
  const bool lng = n >= 320'000'000ull;
  const uint64_t most = (lng ? 64ull : 8ull) * sms;
  const int blocks = static_cast<int>(want < 1 ? 1 : std::min(want, most));
  const bool aligned = (reinterpret_cast<uintptr_t>(ascii) % 16 == 0) &&
                       (reinterpret_cast<uintptr_t>(packed) % 4 == 0);
  if (aligned) {
    if (lng) pack_kernel<true><<<blocks, 256, 0, s>>>(ascii, n, packed, n_invalid);
    else pack_kernel<false><<<blocks, 256, 0, s>>>(ascii, n, packed, n_invalid);
  } else if (reinterpret_cast<uintptr_t>(packed) % 4 == 0) {
    pack_shifted_kernel<<<blocks, 256, 0, s>>>(ascii, n, static_cast<uint32_t>(reinterpret_cast<uintptr_t>(ascii) % 16),
                                               packed, n_invalid);
  } else {
    const uint64_t wb = ((n + 3) / 4 + 255) / 256;
    const int b2 = static_cast<int>(wb > 8ull * sms ? 8ull * sms : (wb < 1 ? 1 : wb));
    pack_bytes_kernel<<<b2, 256, 0, s>>>(ascii, n, packed, n_invalid);
  }
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace ga

// ---------------------------------------------------------------------------
// CIGAR compaction: gathers every pair's runs (written at fixed per-pair
// capacities by the alignment kernels) into one dense array, with the
// exclusive prefix sum of the run counts as offsets. Chunks of 1,024 pairs: one
// launch scans each chunk's counts (none for a single chunk, whose blocks scan them
// themselves), one does the rest: a block adds the chunks before its own to the
// offsets of its tile of pairs and copies the tile's runs.
// ---------------------------------------------------------------------------

namespace ga {

constexpr int kCompactThreads = 256;
constexpr uint32_t kCompactWarps = kCompactThreads / 32;
constexpr uint32_t kCompactChunk = 4 * kCompactThreads;  // pairs
constexpr uint32_t kCompactTile = 8 * kCompactWarps;     // most pairs of a tile

// Sums over the block's threads, in every thread. sh: a word per warp.
__device__ __forceinline__ uint64_t block_sum(uint64_t v, uint64_t* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  uint64_t t = 0;
#pragma unroll
  for (uint32_t w = 0; w < kCompactWarps; ++w) t += sh[w];
  return t;
}

// The counts of pairs p0 + 4 t .. + 3 (thread t) from their chunk's start on: c[x]
// before pair x of the four; returns the chunk's total. sh: a word per warp.
__device__ __forceinline__ uint64_t scan_chunk(const uint32_t* __restrict__ n_runs, uint32_t n, uint64_t p0,
                                               uint64_t* sh, uint64_t (&c)[4]) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t mine = 0;
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const uint64_t p = p0 + 4u * threadIdx.x + x;
    c[x] = mine;
    mine += p < n ? n_runs[p] : 0u;
  }
  uint64_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= static_cast<uint32_t>(o)) incl += y;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  uint64_t before = incl - mine, total = 0;
#pragma unroll
  for (uint32_t w = 0; w < kCompactWarps; ++w) {
    before += w < warp ? sh[w] : 0u;
    total += sh[w];
  }
#pragma unroll
  for (int x = 0; x < 4; ++x) c[x] += before;
  return total;
}

// Each chunk's pairs' offsets from its start, and its sum.
__global__ void __launch_bounds__(kCompactThreads)
    chunk_scan_kernel(const uint32_t* __restrict__ n_runs, uint32_t n, uint64_t* __restrict__ out_off,
                      uint64_t* __restrict__ sums) {
  __shared__ uint64_t sh[kCompactWarps];
  const uint64_t p0 = static_cast<uint64_t>(blockIdx.x) * kCompactChunk;
  uint64_t c[4];
  const uint64_t total = scan_chunk(n_runs, n, p0, sh, c);
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const uint64_t p = p0 + 4u * threadIdx.x + x;
    if (p < n) out_off[p] = c[x];
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// One block, for many chunks: exclusive scan of the chunk sums in place, their
// sum after them.
__global__ void __launch_bounds__(kCompactThreads) scan_sums_kernel(uint64_t* sums, uint32_t n_chunks) {
  __shared__ uint64_t sh[kCompactWarps];
  uint64_t carry = 0;
  for (uint32_t at = 0; at < n_chunks; at += kCompactThreads) {
    const uint32_t q = at + threadIdx.x;
    const uint64_t v = q < n_chunks ? sums[q] : 0u;
    uint64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if ((threadIdx.x & 31) >= static_cast<uint32_t>(o)) incl += y;
    }
    if ((threadIdx.x & 31) == 31) sh[threadIdx.x >> 5] = incl;
    __syncthreads();
    uint64_t before = carry + incl - v;
#pragma unroll
    for (uint32_t w = 0; w < kCompactWarps; ++w) {
      before += w < threadIdx.x >> 5 ? sh[w] : 0u;
      carry += sh[w];
    }
    if (q < n_chunks) sums[q] = before;
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[n_chunks] = carry;
}

// The runs of a tile's pairs, from cigar + at[q] to out + off[q]. The copy is bound by
// memory latency, not bandwidth: a lane has several loads in flight.
//
// Short CIGARs: a lane per run of the warp's `per` pairs (a power of two), which
// finds the run's pair in their offsets. (32 bits hold the runs of such a tile.)
__device__ __forceinline__ void copy_short(const uint32_t* __restrict__ cigar, const uint64_t* __restrict__ at,
                                           const uint64_t* off, uint32_t pairs, uint32_t per,
                                           uint32_t* __restrict__ out) {
  const uint32_t first = threadIdx.x / 32 * per, end = min(first + per, pairs);
  if (first >= pairs) return;
  const uint32_t begin = static_cast<uint32_t>(off[first]);
  const uint32_t runs = static_cast<uint32_t>(off[end]) - begin;
  out += off[first];
  for (uint32_t x = threadIdx.x & 31; x < runs; x += 128) {
    uint32_t v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t y = x + 32 * u;
      if (y < runs) {
        uint32_t q = first;  // the last pair that begins at run y or before
        for (uint32_t step = per / 2; step > 0; step /= 2)
          if (q + step < end && static_cast<uint32_t>(off[q + step]) - begin <= y) q += step;
        v[u] = __ldcs(cigar + at[q] + (y - (static_cast<uint32_t>(off[q]) - begin)));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (x + 32 * u < runs) out[x + 32 * u] = v[u];
  }
}

// Long ones: a warp per pair.
__device__ __forceinline__ void copy_long(const uint32_t* __restrict__ cigar, const uint64_t* __restrict__ at,
                                         const uint64_t* off, uint32_t pairs, uint32_t* __restrict__ out) {
  for (uint32_t q = threadIdx.x / 32; q < pairs; q += kCompactWarps) {
    const uint32_t* src = cigar + at[q];
    uint32_t* dst = out + off[q];
    const uint64_t cnt = off[q + 1] - off[q];
    uint64_t x = threadIdx.x & 31;
    uint32_t v[8];
    for (; x + 224 < cnt; x += 256) {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcs(src + x + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u) dst[x + 32 * u] = v[u];
    }
    if (x < cnt) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (x + 32 * u < cnt) v[u] = __ldcs(src + x + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (x + 32 * u < cnt) dst[x + 32 * u] = v[u];
    }
  }
}

// Block b: tile b % tiles (of `tile` pairs, a divisor of the chunk) of chunk
// b / tiles. out_off holds each pair's offset from its chunk's start (kOne, the only
// chunk: nothing yet) and receives its offset. `scanned`: sums holds the chunks'
// exclusive scan and the total. 32 registers a thread, so that an SM holds eight
// blocks: the loads in flight are what the copy lives by (500,000 CIGARs of 120 runs
// 111 us, with 72 registers 170).
template <bool kOne>
__global__ void __launch_bounds__(kCompactThreads, 8)
    compact_kernel(const uint32_t* __restrict__ cigar, const uint64_t* __restrict__ cigar_off,
                   const uint32_t* __restrict__ n_runs, uint32_t n, uint32_t tile,
                   uint32_t tiles, const uint64_t* __restrict__ sums, uint32_t n_chunks, bool scanned,
                   uint64_t* out_off, uint64_t out_cap, uint32_t* __restrict__ out) {
  __shared__ uint64_t sh[2 * kCompactWarps];
  // The offsets of the tile's pairs from the chunk's start (kOne: all pairs').
  __shared__ uint64_t offs[(kOne ? kCompactChunk : kCompactTile) + 1];
  const uint32_t chunk = kOne ? 0u : blockIdx.x / tiles;
  const uint32_t first = kOne ? blockIdx.x * tile : blockIdx.x % tiles * tile;
  const uint64_t p0 = static_cast<uint64_t>(chunk) * kCompactChunk + first;  // the tile's first pair
  if (p0 >= n) return;
  const uint32_t pairs = static_cast<uint32_t>(n - p0 < tile ? n - p0 : tile);
  uint64_t base = 0, total = 0;  // the chunks before this one, and all of them
  const uint64_t* off = offs;
  if constexpr (kOne) {
    uint64_t c[4];
    total = scan_chunk(n_runs, n, 0u, sh, c);
#pragma unroll
    for (int x = 0; x < 4; ++x) offs[4u * threadIdx.x + x] = c[x];
    if (threadIdx.x == 0) offs[kCompactChunk] = total;
    off += first;
  } else {
    if (threadIdx.x < pairs) {
      const uint64_t o = out_off[p0 + threadIdx.x];
      offs[threadIdx.x] = o;
      if (threadIdx.x == pairs - 1) offs[pairs] = o + n_runs[p0 + threadIdx.x];
    }
    if (scanned) {
      base = sums[chunk];
      total = sums[n_chunks];
    } else {
      uint64_t lo = 0, all = 0;
      for (uint32_t q = threadIdx.x; q < n_chunks; q += kCompactThreads) {
        const uint64_t v = sums[q];
        all += v;
        lo += q < chunk ? v : 0u;
      }
      base = block_sum(lo, sh);
      total = block_sum(all, sh + kCompactWarps);
    }
  }
  __syncthreads();
  if (threadIdx.x < pairs) out_off[p0 + threadIdx.x] = base + off[threadIdx.x];
  if (p0 + pairs == n && threadIdx.x == 0) out_off[n] = total;
  if (total > out_cap) return;  // caller's buffer too small: copy nothing
  // Two loads a lane and pair, as many as a warp per pair has in a CIGAR of 64 runs.
  if (off[pairs] - off[0] < 64u * pairs) {
    copy_short(cigar, cigar_off + p0, off, pairs, tile / kCompactWarps, out + base);
  } else {
    copy_long(cigar, cigar_off + p0, off, pairs, out + base);
  }
}

size_t compact_workspace_bytes(uint32_t n_pairs) {
  const size_t chunks = (static_cast<size_t>(n_pairs) + kCompactChunk - 1) / kCompactChunk;
  return 256 + sizeof(uint64_t) * (chunks + 1);
}

cudaError_t launch_compact(const uint32_t* cigar, const uint64_t* cigar_off, const uint32_t* n_runs,
                           uint32_t n, uint32_t* out, uint64_t out_cap, uint64_t* out_off, void* ws,
                           cudaStream_t s) {
  if (n == 0) {
    const cudaError_t e = cudaMemsetAsync(out_off, 0, sizeof(uint64_t), s);
    return e;
  }
  uint64_t* sums = static_cast<uint64_t*>(ws);
  const uint32_t chunks = static_cast<uint32_t>((static_cast<uint64_t>(n) + kCompactChunk - 1) / kCompactChunk);
  // Tiles of one pair per warp while that makes no more than a block for each
  // resident one (152 SMs of eight), then of two, four, eight. From cold caches, us
  // with tiles of 8 up to 32,768 pairs and of 64 past that and each block scanning
  // its chunk again, and now: 32,000 CIGARs of 30 runs 33, 24, of 600 58, 51; 500,000
  // of 30 runs 103, 68, of 120 runs 201, 122.
  uint32_t tile = kCompactWarps;
  while (tile < kCompactTile && n > 1250u * tile) tile *= 2u;
  const uint32_t tiles = (std::min(n, kCompactChunk) + tile - 1) / tile;
  if (chunks == 1) {
    compact_kernel<true><<<tiles, kCompactThreads, 0, s>>>(cigar, cigar_off, n_runs, n, tile, tiles, sums,
                                                           1u, false, out_off, out_cap, out);
    count_launches(1);
    return cudaGetLastError();
  }
  // Past 256 chunks the blocks would spend more on adding them up than a scan of
  // them costs (500,000 pairs of one run: 39 us, without the scan 43).
  const bool scanned = chunks > 256;
  chunk_scan_kernel<<<chunks, kCompactThreads, 0, s>>>(n_runs, n, out_off, sums);
  if (scanned) scan_sums_kernel<<<1, kCompactThreads, 0, s>>>(sums, chunks);
  compact_kernel<false><<<chunks * tiles, kCompactThreads, 0, s>>>(
      cigar, cigar_off, n_runs, n, tile, tiles, sums, chunks, scanned, out_off, out_cap, out);
  count_launches(scanned ? 3 : 2);
  return cudaGetLastError();
}

}  // namespace ga
