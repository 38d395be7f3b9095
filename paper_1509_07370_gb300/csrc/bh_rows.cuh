// Lists by row: a lane serves a row of four cells of the octant (same y and
// z) and steps through the nodes that a cell of its row accepts (or opens),
// for the walks whose interactions cost more than gathering them (binary64,
// periodic).  Two lanes, the halves, share a row.
#pragma once
#include "bh_lists.cuh"

namespace bhg {
namespace {

// The lane's row: a nibble of the 64-bit masks (bit 16 (y >> 1) + 8 (z & 1) +
// 4 (y & 1) + x of word z >> 1).
struct Row {
  int half, y, z, word, shift;
  __device__ __forceinline__ explicit Row(int lane) {
    const int r = lane & 15;
    half = lane >> 4;
    y = 2 * ((r >> 2) & 1) + (r & 1);
    z = 2 * (r >> 3) + ((r >> 1) & 1);
    word = r >> 3;
    shift = 4 * (r & 7);
  }
};

// Which of n <= 64 N entries with masks {lo, hi} have a target of the lane's
// row, found by ballots; steps: the most that any lane has.
template <int N>
struct RowList {
  unsigned long long left[N];
  int mine, steps;
  bool taken;
  __device__ __forceinline__ RowList(const uint32_t *lo, const uint32_t *hi, int n, int lane) {
    uint32_t m[2 * N];
#pragma unroll
    for (int w = 0; w < 2 * N; ++w) {
      const int j = 32 * w + lane;
      const uint32_t l = j < n ? lo[j] : 0u, h = j < n ? hi[j] : 0u;
      m[w] = 0u;
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const unsigned b = __ballot_sync(kFull, (((r < 8 ? l : h) >> (4 * (r & 7))) & 15u) != 0u);
        if ((lane & 15) == r) m[w] = b;
      }
    }
    mine = 0;
#pragma unroll
    for (int w = 0; w < N; ++w) {
      left[w] = ((unsigned long long)m[2 * w + 1] << 32) | m[2 * w];
      mine += __popcll(left[w]);
    }
    steps = (int)__reduce_max_sync(kFull, (unsigned)mine);
    taken = false;
  }
  // The lower half of the entries for half 0 (taken from the bottom), the
  // upper for half 1 (from the top).
  __device__ __forceinline__ void halve(int half) {
    mine = half ? mine / 2 : mine - mine / 2;
    steps = (int)__reduce_max_sync(kFull, (unsigned)mine);
  }
  // The next entry (0 with taken = false when the lane has none left).
  __device__ __forceinline__ int from_bottom() {
    taken = mine > 0;
    --mine;
    int w = 0;  // the lowest word with an entry left
#pragma unroll
    for (int i = N - 1; i >= 0; --i) w = left[i] ? i : w;
    int j = 0;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i == w) {
        j = taken ? 64 * i + __ffsll((long long)left[i]) - 1 : 0;
        left[i] &= left[i] - 1ull;
      }
    return j;
  }
  __device__ __forceinline__ int from_top() {
    taken = mine > 0;
    --mine;
    int w = 0;  // the highest
#pragma unroll
    for (int i = 0; i < N; ++i) w = left[i] ? i : w;
    int j = 0;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i == w) {
        j = taken ? 64 * i + 63 - __clzll((long long)left[i]) : 0;
        left[i] &= ~(1ull << (j & 63));
      }
    return j;
  }
};

}  // namespace
}  // namespace bhg
