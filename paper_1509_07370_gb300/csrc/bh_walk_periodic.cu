// The Barnes-Hut walk with periodic boundaries (App. A).
//
// The traversal is that of bh_lists.cuh (eight siblings tested at a time, one
// child per lane); what changes is the geometry and the term:
//  * every displacement is the minimum image: each box-unit component of
//    t - R is wrapped into [-1/2, 1/2] (dx > 0.5 -> dx - 1, dx < -0.5 ->
//    dx + 1, both exact in binary32), for the opening test of Eq. 4 and for
//    the term;
//  * an accepted node or another cell adds M psi(d) = M (1/d + chi(d)), chi
//    the smooth part of the Ewald field interpolated quadratically from the
//    table (bh_ewald.cuh);
//  * the target's own cell adds its mass times chi(0): the field of its
//    periodic copies (the direct part 1/d is absent, as in the isolated walk).
//
// What bounds it: the table.  A lookup reads one 64-byte entry and contracts
// its 27 coefficients, and lanes with different entries each cost the L1 data
// stage a wavefront per load (2 per interaction in the walk that stepped 64
// targets together: 69 % of it busy at 11.6 ms, and half of its lanes idle).
// So a lane serves a row of four cells (same y and z) and half of the nodes a
// cell of the row accepts (lists by row, as in bh_walk_f64.cu): the y and z
// indices and fractions are shared, and an entry is read and contracted over z
// and y (24 FMAs) once for all targets of the row that fall on its centre --
// each then takes two FMAs.  Where the cells are finer than the table (four of
// them span two centres on the finest level of the 2M-cell spheroid) a row
// needs two or three entries instead of four.  Measured (that spheroid, theta
// 0.7): 11.57 -> 8.7 ms; the L1 data stage is still what bounds it (75 % busy:
// two wavefronts an entry and lane), the issue slots are 60 % used.  72 or 64
// registers instead of 91 change nothing, 8 warps per CTA instead of 4 take
// 13 % longer.
#include "bh_rows.cuh"
#include "bh_ewald.cuh"

namespace bhg {
namespace {

constexpr int kPWarpsPerCta = 4;
constexpr int kPMaxThreads = 512;
constexpr int kPStage = 64;      // staged nodes, evaluated once a further step's might not fit
constexpr int kPBottoms = 64;    // opened bottom nodes, likewise

struct PeriodicMem {             // of one warp
  Front front;
  float4 node[kPStage];          // px, py, pz, m of the staged nodes
  uint32_t mask[2][kPStage];     // the accepting targets
  float4 centre[kPBottoms];      // opened bottom nodes: geometric centre, half a cell,
  uint32_t bottom[3][kPBottoms]; // index, O (two words)
};

__device__ __forceinline__ float min_image(float d) {
  return d > 0.5f ? __fsub_rn(d, 1.0f) : (d < -0.5f ? __fadd_rn(d, 1.0f) : d);
}

// A row's interactions with one source of mass m at (px, py, pz): targets at
// tx[i], ty, tz for the bits of m4; own: the target's own cell (d = 0) has no
// direct part (nodes: no target sits on one it accepts).
template <bool KAHAN>
__device__ __forceinline__ void row_terms(const unsigned char *__restrict__ tab, int n, float s,
                                          float px, float py, float pz, float m, uint32_t m4,
                                          const float tx[4], float ty, float tz, float sum[4],
                                          float comp[4]) {
  const float dy = min_image(__fsub_rn(ty, py)), dz = min_image(__fsub_rn(tz, pz));
  const float h = __fmaf_rn(dz, dz, __fmul_rn(dy, dy));
  float fy, fz, fx[4], chi[4];
  const int cy = ewald_axis(fabsf(dy), s, n, fy), cz = ewald_axis(fabsf(dz), s, n, fz);
  const unsigned row0 = (unsigned)(((cz - 1) * n + (cy - 1)) * n) - 1u;
  int c[4];
  float r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float dx = min_image(__fsub_rn(tx[i], px));
    const float d2 = __fmaf_rn(dx, dx, h);
    r[i] = d2 > 0.0f ? rsqrt_approx(d2) : 0.0f;
    c[i] = ewald_axis(fabsf(dx), s, n, fx[i]);
    if (!(m4 & (1u << i))) c[i] = 0x7fffffff;  // not taking part
    chi[i] = 0.0f;
  }
  for (;;) {  // the entries that some target falls on, in order
    const int at = min(min(c[0], c[1]), min(c[2], c[3]));
    if (at == 0x7fffffff) break;
    float k[3];
    ewald_row(tab, row0 + (unsigned)at, fy, fz, k);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool hit = c[i] == at;
      chi[i] = hit ? __fmaf_rn(fx[i], __fmaf_rn(fx[i], k[2], k[1]), k[0]) : chi[i];
      c[i] = hit ? 0x7fffffff : c[i];
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float t = (m4 & (1u << i)) ? __fmul_rn(m, __fadd_rn(r[i], chi[i])) : 0.0f;
    const float v = __fadd_rn(sum[i], t);  // compensated as accumulate2
    if (KAHAN) comp[i] = __fadd_rn(comp[i], __fadd_rn(__fsub_rn(sum[i], v), t));
    sum[i] = v;
  }
}

// Walk of octant u & 7 of sorted block u >> 3.
template <bool KAHAN, bool COUNTS>
__device__ __forceinline__ void walk_octant_periodic(
    unsigned u, int lane, PeriodicMem &S, const WalkRec *__restrict__ rec, const SibArgs &sib,
    const int4 *__restrict__ blk, const int *__restrict__ orig, const int4 *__restrict__ fld,
    const int *__restrict__ flev, const double *__restrict__ invL,
    const unsigned long long *__restrict__ mmax, const unsigned char *__restrict__ tab, int n,
    double G, float *__restrict__ out, int32_t *__restrict__ n_int, int32_t *__restrict__ n_test,
    int32_t *__restrict__ n_leaf) {
  const unsigned p = u >> 3;
  const int o = (int)(u & 7);
  const int4 B = blk[p], F = fld[p];
  const Octant O = octant_at(B, o);
  front_start(S.front, O, F, p, lane, rec, sib.tops);
  const Row R(lane);
  const unsigned lower = (1u << lane) - 1u;
  const float s = (float)(2 * n);
  float tx[4], sum[4] = {0.0f, 0.0f, 0.0f, 0.0f}, comp[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  int na[4] = {0, 0, 0, 0}, nb[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 4; ++i) tx[i] = O.centre(O.ox + i);
  const float ty = O.centre(O.oy + R.y), tz = O.centre(O.oz + R.z);

  int depth = 1, staged = 0, nbot = 0;
  const int pop4 = stack_pop4(flev[F.w]);
  const unsigned tops = (unsigned)sib.tops;
  while (depth > 0) {
    const Tested t = front_step<false, true>(S.front, depth, pop4, tops, lane, sib.sib);
    const bool accepted = (t.alo | t.ahi) != 0u;
    const unsigned acc = __ballot_sync(kFull, accepted);
    if (accepted) {
      const int slot = staged + __popc(acc & lower);
      S.node[slot] = t.rec;
      S.mask[0][slot] = t.alo;
      S.mask[1][slot] = t.ahi;
    }
    staged += __popc(acc);
    const bool bottom = (t.olo | t.ohi) != 0u && (t.kids & kBottomBit) != 0u;
    const unsigned bot = __ballot_sync(kFull, bottom);
    if (bottom) {
      const int slot = nbot + __popc(bot & lower);
      S.bottom[0][slot] = t.kids & ~kBottomBit;
      S.bottom[1][slot] = t.olo;
      S.bottom[2][slot] = t.ohi;
    }
    nbot += __popc(bot);
    __syncwarp();
    const bool last = depth == 0;
    if (staged > kPStage - 32 || (last && staged)) {
      RowList<1> list(S.mask[0], S.mask[1], staged, lane);
      list.halve(R.half);
      for (int it = 0; it < list.steps; ++it) {
        const int j = R.half ? list.from_top() : list.from_bottom();
        const uint32_t m4 = list.taken ? S.mask[R.word][j] >> R.shift : 0u;
        if (COUNTS) {
#pragma unroll
          for (int i = 0; i < 4; ++i) na[i] += (m4 >> i) & 1u;
        } else {
          const float4 q = S.node[j];
          row_terms<KAHAN>(tab, n, s, q.x, q.y, q.z, q.w, m4, tx, ty, tz, sum, comp);
        }
      }
      staged = 0;
      __syncwarp();
    }
    if (nbot > kPBottoms - 32 || (last && nbot)) {
      for (int j = lane; j < nbot; j += 32) S.centre[j] = bottom_centre(S.bottom[0][j], blk);
      __syncwarp();
      RowList<1> list(S.bottom[1], S.bottom[2], nbot, lane);
      for (int it = 0; it < list.steps; ++it) {  // the lane's half: the four cells of one z
        const int j = list.from_bottom();
        const uint32_t m4 = list.taken ? S.bottom[1 + R.word][j] >> R.shift : 0u;
        if (COUNTS) {
#pragma unroll
          for (int i = 0; i < 4; ++i) nb[i] += (m4 >> i) & 1u;
          continue;
        }
        const float4 m = __ldg(reinterpret_cast<const float4 *>(sib.cmass) +
                               2 * (size_t)S.bottom[0][j] + R.half);
        const float4 c = S.centre[j];
        const float cz = R.half ? __fadd_rn(c.z, c.w) : __fsub_rn(c.z, c.w);
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
          const float px = (k & 1) ? __fadd_rn(c.x, c.w) : __fsub_rn(c.x, c.w);
          const float py = (k & 2) ? __fadd_rn(c.y, c.w) : __fsub_rn(c.y, c.w);
          const float mk = (k & 2) ? ((k & 1) ? m.w : m.z) : ((k & 1) ? m.y : m.x);
          row_terms<KAHAN>(tab, n, s, px, py, cz, mk, m4, tx, ty, tz, sum, comp);
        }
      }
      nbot = 0;
      __syncwarp();
    }
  }
  const int64_t cell = (int64_t)orig[p] * kCellsPerBlock + (4 * (o >> 2) + R.z) * 64 +
                       (4 * ((o >> 1) & 1) + R.y) * 8 + 4 * (o & 1);
  if (COUNTS) {  // as the isolated walk counts (bh_walk.cu)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int a = na[i] + __shfl_xor_sync(kFull, na[i], 16);
      if ((i >> 1) != R.half) continue;
      const int cells = 8 * nb[i] - 1;
      n_int[cell + i] = a + cells;
      n_test[cell + i] = (8 * (a + nb[i]) - 1) / 7;
      if (n_leaf) n_leaf[cell + i] = cells;
    }
    return;
  }
  const float scale = (float)(-G * invL[F.w] * pow2i(mass_exponent(mmax[F.w])));
#pragma unroll
  for (int i = 0; i < 4; ++i) {  // the two halves' sums, by TwoSum
    const float a = sum[i], b = __shfl_xor_sync(kFull, sum[i], 16);
    const float v = __fadd_rn(a, b);
    float total = v;
    if (KAHAN) {
      const float bb = __fsub_rn(v, a);
      const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(v, bb)), __fsub_rn(b, bb));
      total = __fadd_rn(v, __fadd_rn(__fadd_rn(comp[i], __shfl_xor_sync(kFull, comp[i], 16)), e));
    }
    if ((i >> 1) == R.half) out[cell + i] = __fmul_rn(total, scale);
  }
}

// One warp per octant: octant order[warp] when an order is given (the
// octants sorted by the time of their walks, longest first, so that the
// CTAs, issued in index order, start with the long walks and each holds
// octants of about equal length).  With `cycles`, lane 0 stores the SM clock
// cycles its octant's walk took.
template <bool KAHAN, bool COUNTS>
__global__ void __launch_bounds__(kPMaxThreads)
    k_walk_periodic(unsigned nunits, const unsigned *__restrict__ order,
                    unsigned long long *__restrict__ cycles, const WalkRec *__restrict__ rec,
                    const SibArgs sib, const int4 *__restrict__ blk, const int *__restrict__ orig,
                    const int4 *__restrict__ fld, const int *__restrict__ flev,
                    const double *__restrict__ invL, const unsigned long long *__restrict__ mmax,
                    const unsigned char *__restrict__ tab, int n, double G,
                    float *__restrict__ out, int32_t *__restrict__ n_int,
                    int32_t *__restrict__ n_test, int32_t *__restrict__ n_leaf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PeriodicMem &S = reinterpret_cast<PeriodicMem *>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (warp >= nunits) return;  // whole warps only
  const unsigned u = order ? order[warp] : warp;
  const long long t0 = cycles ? clock64() : 0;
  walk_octant_periodic<KAHAN, COUNTS>(u, lane, S, rec, sib, blk, orig, fld, flev, invL, mmax, tab,
                                      n, G, out, n_int, n_test, n_leaf);
  if (cycles && lane == 0) cycles[u] = (unsigned long long)(clock64() - t0);
}

template <bool KAHAN, bool COUNTS>
cudaError_t go_periodic(cudaStream_t s, int nb, const WalkRec *rec, const SibArgs &sib,
                        const int4 *blk, const int *orig, const FieldArgs &fa,
                        const unsigned char *tab, int n, double G, void *out, int32_t *ni,
                        int32_t *nt, int32_t *nl, int wpc, const unsigned *order,
                        unsigned long long *cycles) {
  const unsigned nunits = (unsigned)nb * 8u;
  const int w = wpc > 0 ? wpc : kPWarpsPerCta;
  const int grid = (int)((nunits + w - 1) / w);
  k_walk_periodic<KAHAN, COUNTS><<<grid, 32 * w, w * sizeof(PeriodicMem), s>>>(
      nunits, order, cycles, rec, sib, blk, orig, fa.fld, fa.flev, fa.invL, fa.mmax, tab, n, G,
      (float *)out, ni, nt, nl);
  return cudaGetLastError();
}

}  // namespace

cudaError_t prepare_periodic_kernels() {
  const int bytes = kPMaxThreads / 32 * (int)sizeof(PeriodicMem);
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(k_walk_periodic<true, false>, attr, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_walk_periodic<false, false>, attr, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_walk_periodic<false, true>, attr, bytes);
  return e;
}

cudaError_t launch_walk_periodic(cudaStream_t s, const bh_options &opt, int nb,
                                 const WalkRec *rec, const SibArgs &sib, const int4 *blk,
                                 const int *orig, const FieldArgs &fa, const unsigned char *tab,
                                 int n, double G, void *out, int32_t *n_int, int32_t *n_test,
                                 int32_t *n_leaf, int wpc, const unsigned *order,
                                 unsigned long long *cycles) {
  if (n_int)
    return go_periodic<false, true>(s, nb, rec, sib, blk, orig, fa, tab, n, G, out, n_int, n_test,
                                    n_leaf, wpc, order, nullptr);
  return opt.kahan ? go_periodic<true, false>(s, nb, rec, sib, blk, orig, fa, tab, n, G, out,
                                              nullptr, nullptr, nullptr, wpc, order, cycles)
                   : go_periodic<false, false>(s, nb, rec, sib, blk, orig, fa, tab, n, G, out,
                                               nullptr, nullptr, nullptr, wpc, order, cycles);
}

}  // namespace bhg
