// Plain GPU GenASM: one pair per 32-thread block (each lane a strip of 2 text
// columns), one launch, pairs in index order, no queue, no tuning, no
// workspace. The improved algorithm in its row form (genasm_window.cuh): the
// yardstick the batched kernel is measured against.
#include <cstdint>

#include <cuda_runtime.h>

#include "genasm_internal.h"
#include "genasm_pair.cuh"
#include "genasm_window.cuh"

namespace ga {

namespace {

constexpr int kPlainG = 32;
// The worst-case table (65 rows x 66 entries) and the PM[T[i]] columns.
constexpr int kTableEntries = kMaxRows * kMaxStride;
constexpr size_t kPlainSmem = sizeof(uint64_t) * (kTableEntries + kPmCols);

__device__ __forceinline__ void plain_window(const AlignParams& p, int r, PairState& st,
                                             uint64_t* table, uint64_t* pmcol) {
  constexpr int G = kPlainG;
  const bool writer = r == 0;
  const int commit = p.W - p.O;
  const int wp = static_cast<int>(min(static_cast<uint32_t>(p.W), st.m - st.pos_p));
  const int wt = static_cast<int>(min(static_cast<uint32_t>(p.W), st.n - st.pos_t));
  const bool last = st.pos_p + static_cast<uint32_t>(wp) == st.m;
  const int ncols = last ? wt + 1 : min(wt, commit) + 1;  // columns the traceback can reach
  const int S = table_stride(ncols);
  build_masks<G>(r, 0, true, st.read, st.pos_p, wp, st.ref, st.pos_t, wt, pmcol);
  __syncwarp();
  uint64_t pm[64 / G];
#pragma unroll
  for (int x = 0; x < 64 / G; ++x) pm[x] = pmcol[r * (64 / G) + x];
  __syncwarp();
  const int dmin = dc_window<G, true>(r, 0, true, wp, wt, p.kmax, ncols, S, kMaxRows, pm, table);
  __syncwarp();
  int cp = 0, ct = 0;
  const bool ok = tb_window<G>(r, 0, dmin >= 0, wp, wt, dmin, last, commit, ncols, S, p.tb_table,
                               pmcol, table, st.rw, writer, cp, ct, st.edits);
  __syncwarp();
  if (dmin < 0) {
    st.status = kPairExceedsK;
  } else if (!ok || cp + ct == 0) {
    st.status = kPairTbStuck;
  } else if (st.rw.full) {
    st.status = kPairCigarFull;
  } else {
    ++st.windows;
    st.cells += static_cast<uint64_t>(wt) * static_cast<uint64_t>(dmin + 1);
    st.pos_p += static_cast<uint32_t>(cp);
    st.pos_t += static_cast<uint32_t>(ct);
  }
  if (st.status != kPairOk || st.pos_p >= st.m) finish_pair(p, st, writer);
}

__global__ void __launch_bounds__(32) align_plain_kernel(const AlignParams p) {
  extern __shared__ __align__(16) uint64_t smem[];
  const int r = threadIdx.x;
  PairState st;
  begin_pair(p, blockIdx.x, st, r == 0);
  while (st.busy) plain_window(p, r, st, smem, smem + kTableEntries);
}

}  // namespace

cudaError_t launch_plain(const AlignParams& p, cudaStream_t s) {
  if (p.n_pairs == 0) return cudaSuccess;
  align_plain_kernel<<<p.n_pairs, 32, kPlainSmem, s>>>(p);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace ga
