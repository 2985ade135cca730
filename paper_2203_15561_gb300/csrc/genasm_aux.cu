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
// launch sums each chunk's counts (none for a single chunk), one does the rest:
// a block scans its chunk's counts, adds the chunks before it, writes the
// offsets of its tile of the chunk and copies the tile's runs. (Recounting a
// chunk in each of its blocks costs 4 KB of reads from L2 and two barriers; the
// two launches it saves cost more on small batches and as much on large ones.)
// ---------------------------------------------------------------------------

namespace ga {

constexpr int kCompactThreads = 256;
constexpr uint32_t kCompactChunk = 4 * kCompactThreads;  // pairs

// Sum over the block's threads, in every thread. sh: one word per warp.
__device__ __forceinline__ uint64_t block_sum(uint64_t v, uint64_t* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  uint64_t t = 0;
#pragma unroll
  for (int w = 0; w < kCompactThreads / 32; ++w) t += sh[w];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(kCompactThreads) chunk_sum_kernel(const uint32_t* __restrict__ n_runs,
                                                                    uint32_t n,
                                                                    uint64_t* __restrict__ sums) {
  __shared__ uint64_t sh[kCompactThreads / 32];
  uint64_t v = 0;
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const uint64_t p = static_cast<uint64_t>(blockIdx.x) * kCompactChunk + x * kCompactThreads + threadIdx.x;
    v += p < n ? n_runs[p] : 0u;
  }
  v = block_sum(v, sh);
  if (threadIdx.x == 0) sums[blockIdx.x] = v;
}

// One block, for many chunks: exclusive scan of the chunk sums in place, their
// sum after them.
__global__ void __launch_bounds__(kCompactThreads) scan_sums_kernel(uint64_t* sums, uint32_t n_chunks) {
  __shared__ uint64_t sh[kCompactThreads / 32];
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
    for (uint32_t w = 0; w < kCompactThreads / 32; ++w) {
      before += w < threadIdx.x >> 5 ? sh[w] : 0u;
      carry += sh[w];
    }
    if (q < n_chunks) sums[q] = before;
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[n_chunks] = carry;
}

// Block b: tile b % tiles (of `tile` pairs, a divisor of the chunk) of chunk
// b / tiles. `scanned`: sums holds the chunks' exclusive scan and the total.
__global__ void __launch_bounds__(kCompactThreads)
    compact_kernel(const uint32_t* __restrict__ cigar, const uint64_t* __restrict__ cigar_off,
                   const uint32_t* __restrict__ n_runs, uint32_t n, uint32_t tile,
                   uint32_t tiles, const uint64_t* __restrict__ sums, uint32_t n_chunks, bool scanned,
                   uint64_t* __restrict__ out_off, uint64_t out_cap, uint32_t* __restrict__ out) {
  __shared__ uint64_t sh[kCompactThreads / 32];
  __shared__ uint64_t off[kCompactChunk + 1];  // the chunk's pairs' offsets, from the chunk's start
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t chunk = blockIdx.x / tiles;
  const uint64_t p0 = static_cast<uint64_t>(chunk) * kCompactChunk;
  const uint32_t first = blockIdx.x % tiles * tile;
  if (p0 + first >= n) return;
  // Each thread's four counts, their scan over the block.
  uint64_t c[4], mine = 0;
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
  for (uint32_t w = 0; w < kCompactThreads / 32; ++w) {
    before += w < warp ? sh[w] : 0u;
    total += sh[w];
  }
#pragma unroll
  for (int x = 0; x < 4; ++x) off[4u * threadIdx.x + x] = before + c[x];
  if (threadIdx.x == 0) off[kCompactChunk] = total;
  __syncthreads();
  // The chunks before this one, and all of them.
  uint64_t base = 0;
  if (scanned) {
    base = sums[chunk];
    total = sums[n_chunks];
  } else if (n_chunks > 1) {
    uint64_t lo = 0, all = 0;
    for (uint32_t q = threadIdx.x; q < n_chunks; q += kCompactThreads) {
      const uint64_t v = sums[q];
      all += v;
      lo += q < chunk ? v : 0u;
    }
    base = block_sum(lo, sh);
    total = block_sum(all, sh);
  }
  const uint32_t in_chunk = static_cast<uint32_t>(n - p0 < kCompactChunk ? n - p0 : kCompactChunk);
  const uint32_t last = first + tile < in_chunk ? first + tile : in_chunk;
  for (uint32_t q = first + threadIdx.x; q < last; q += kCompactThreads) out_off[p0 + q] = base + off[q];
  if (p0 + last == n && threadIdx.x == 0) out_off[n] = total;
  if (total > out_cap) return;  // caller's buffer too small: copy nothing
  const uint64_t runs = off[last] - off[first];
  if (runs < 32u * (last - first)) {
    // Short CIGARs: a thread per run, its pair found in the offsets.
    for (uint64_t x = threadIdx.x; x < runs; x += kCompactThreads) {
      const uint64_t at = off[first] + x;
      uint32_t a = first, b = last;  // off[a] <= at < off[b]
      while (b - a > 1) {
        const uint32_t m = (a + b) >> 1;
        if (off[m] <= at) a = m;
        else b = m;
      }
      out[base + at] = __ldcs(cigar + cigar_off[p0 + a] + (at - off[a]));
    }
    return;
  }
  for (uint32_t q = first + warp; q < last; q += kCompactThreads / 32) {
    const uint32_t* src = cigar + cigar_off[p0 + q];
    uint32_t* dst = out + base + off[q];
    const uint64_t cnt = off[q + 1] - off[q];
    // Eight loads in flight per lane (the copy is bound by memory latency, not
    // bandwidth, with one warp per pair).
    uint64_t x = lane;
    for (; x + 224 < cnt; x += 256) {
      uint32_t v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcs(src + x + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u) dst[x + 32 * u] = v[u];
    }
    for (; x < cnt; x += 32) dst[x] = __ldcs(src + x);
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
  // Tiles of one pair per warp while that makes no more than a few thousand
  // blocks, else of eight. Past a million pairs the blocks would spend more on
  // adding up the chunks than a scan of them costs.
  const uint32_t tile = n <= 32768 ? 8u : 64u;
  const uint32_t tiles = (std::min(n, kCompactChunk) + tile - 1) / tile;
  const bool scanned = chunks > 1024;
  if (chunks > 1) {
    chunk_sum_kernel<<<chunks, kCompactThreads, 0, s>>>(n_runs, n, sums);
    count_launches(1);
  }
  if (scanned) {
    scan_sums_kernel<<<1, kCompactThreads, 0, s>>>(sums, chunks);
    count_launches(1);
  }
  compact_kernel<<<chunks * tiles, kCompactThreads, 0, s>>>(cigar, cigar_off, n_runs, n, tile, tiles,
                                                            sums, chunks, scanned, out_off, out_cap,
                                                            out);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace ga
