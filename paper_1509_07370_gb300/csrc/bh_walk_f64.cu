// The binary64 walk: the traversal of bh_lists.cuh (the binary32 opening test,
// so the decisions are those of every other walk) with the interactions in
// binary64 from the FP64 moments.
//
// What bounds it: GB300 issues two binary64 operations per clock and SM, and a
// warp-wide one takes 16 clocks whether 32, 8 or 1 of its lanes need it.  So
// the lanes are kept busy and the operations few:
//  * a lane serves a row of four cells (same y and z; lane & 15) and takes
//    half of the nodes that a cell of the row accepts (lane >> 4): the row's
//    accepted nodes are gathered by ballots over the staged ones, so a lane
//    steps through its own list (83-92 % of the 4 targets of a step take
//    part, against 44 % when 32 cells step together), and dy, dz and their
//    squares are shared by the row;
//  * 1/d by one approximation on the special-function unit and one third-order
//    step (Householder's method): y (1 + e (1/2 + 3/8 e)), e = 1 - d2 y y, five
//    operations instead of a square root and a division (some 9 each).  The
//    approximation's 2^-20 makes e at most 2^-19, so 5/16 e^3, 2^-58.7, is left
//    out; with the roundings 1/d is within 1.6 2^-53.
// An interaction then takes 9 operations (7.9 with a cell) instead of 26.
// Measured (32^3 cells, theta 0.5): 3.07 -> 1.43 ms; error against exact sums
// 1.12e-15 -> 1.07e-15 of the potential.  That is 36 operations per step of a
// lane's 4 targets against the FP64 rate's 1.04 ms (four octants on the
// fullest SM): the rest is rows waiting for the longest list of their warp.
#include "bh_rows.cuh"

namespace bhg {
namespace {

constexpr int kF64Warps = 4;       // per CTA
// Staged nodes and opened bottom nodes, evaluated once a further step's might
// not fit: rows wait less for the longest list of their warp in long lists.
// 96 and 128 entries against 64 and 64: 1.59 -> 1.43 ms on 32^3 cells, 13.1 ->
// 12.2 on a core at theta 0.7; with quadrupoles (more shared memory an entry)
// 2 % slower.
template <bool QUAD>
constexpr int kF64Stage = QUAD ? 64 : 96;
template <bool QUAD>
constexpr int kF64Bottoms = QUAD ? 64 : 128;

template <bool QUAD>
struct F64Mem {                    // of one warp
  Front front;
  double4_32a node[kF64Stage<QUAD>];     // centre of mass and mass
  double quad[QUAD ? 6 * kF64Stage<QUAD> : 2];
  uint32_t mask[2][kF64Stage<QUAD>];     // the accepting targets
  float4 centre[kF64Bottoms<QUAD>];      // opened bottom nodes: geometric centre, half a cell,
  uint32_t bottom[3][kF64Bottoms<QUAD>]; // index, O (two words)
};

// 1/sqrt(d) for normal d > 0.
__device__ __forceinline__ double rsqrt64(double d) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-(d * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

template <bool QUAD, bool VOTE>
__global__ void __launch_bounds__(32 * kF64Warps)
    k_walk_f64(unsigned nunits, const WalkRec *__restrict__ rec, const SibArgs sib,
               const int4 *__restrict__ blk, const int *__restrict__ orig,
               const int4 *__restrict__ fld, const int *__restrict__ flev,
               const double *__restrict__ invL, double G, double *__restrict__ out) {
  extern __shared__ __align__(32) unsigned char smem_raw[];
  F64Mem<QUAD> &S = reinterpret_cast<F64Mem<QUAD> *>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned u = blockIdx.x * kF64Warps + (threadIdx.x >> 5);
  if (u >= nunits) return;  // whole warps only
  const unsigned p = u >> 3;
  const int o = (int)(u & 7);
  const int4 B = blk[p], F = fld[p];
  const Octant O = octant_at(B, o);
  front_start(S.front, O, F, p, lane, rec, sib.tops);
  const Row R(lane);
  const unsigned lower = (1u << lane) - 1u;
  double tx[4], sum[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 4; ++i) tx[i] = (double)O.centre(O.ox + i);
  const double ty = (double)O.centre(O.oy + R.y), tz = (double)O.centre(O.oz + R.z);

  int depth = 1, staged = 0, nbot = 0;
  const int pop4 = stack_pop4(flev[F.w]);
  const unsigned tops = (unsigned)sib.tops;
  while (depth > 0) {
    const Tested t = front_step<VOTE>(S.front, depth, pop4, tops, lane, sib.sib);
    const bool accepted = (t.alo | t.ahi) != 0u;
    const unsigned acc = __ballot_sync(kFull, accepted);
    if (accepted) {
      const int slot = staged + __popc(acc & lower);
      copy_async<16>(&S.node[slot], sib.mom + t.node);
      copy_async<16>(&S.node[slot].z, &sib.mom[t.node].z);
      if (QUAD) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
          copy_async<16>(&S.quad[6 * slot + 2 * i], sib.q64 + 6 * (size_t)t.node + 2 * i);
      }
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
    if (staged > kF64Stage<QUAD> - 32 || (last && staged)) {
      copy_async_wait();
      __syncwarp();
      double part[4] = {0.0, 0.0, 0.0, 0.0};  // (short sums of their own: less rounding)
      RowList<(kF64Stage<QUAD> + 63) / 64> list(S.mask[0], S.mask[1], staged, lane);
      list.halve(R.half);
      for (int it = 0; it < list.steps; ++it) {
        const int j = R.half ? list.from_top() : list.from_bottom();
        const uint32_t m4 = list.taken ? S.mask[R.word][j] >> R.shift : 0u;
        const double4_32a n = S.node[j];
        const double dz = tz - n.z, dy = ty - n.y, h = fma(dy, dy, dz * dz);
        double qu = 0.0, qc = 0.0, qx = 0.0;
        if (QUAD) {  // d^T Q d / 2 = dx (Qxx/2 dx + qu) + qc
          const double *Q = &S.quad[6 * j];
          qx = 0.5 * Q[0];
          qu = fma(Q[3], dy, Q[4] * dz);
          qc = fma(dy, fma(0.5 * Q[1], dy, Q[5] * dz), (0.5 * Q[2] * dz) * dz);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double dx = tx[i] - n.x, d2 = fma(dx, dx, h);
          double y = rsqrt64(d2);
          y = (m4 & (1u << i)) ? y : 0.0;
          double w = n.w;
          if (QUAD) {
            const double hq = fma(dx, fma(qx, dx, qu), qc), y2 = y * y;
            w = fma(hq, y2 * y2, w);
          }
          part[i] = fma(w, y, part[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) sum[i] += part[i];
      staged = 0;
      __syncwarp();
    }
    if (nbot > kF64Bottoms<QUAD> - 32 || (last && nbot)) {
      for (int j = lane; j < nbot; j += 32) S.centre[j] = bottom_centre(S.bottom[0][j], blk);
      __syncwarp();
      double part[4] = {0.0, 0.0, 0.0, 0.0};
      RowList<(kF64Bottoms<QUAD> + 63) / 64> list(S.bottom[1], S.bottom[2], nbot, lane);
      for (int it = 0; it < list.steps; ++it) {  // the lane's half: the four cells of one z
        const int j = list.from_bottom();
        const uint32_t m4 = list.taken ? S.bottom[1 + R.word][j] >> R.shift : 0u;
        const double *cm = sib.cmass64 + 8 * (size_t)S.bottom[0][j] + 4 * R.half;
        const double2 m01 = __ldg(reinterpret_cast<const double2 *>(cm));
        const double2 m23 = __ldg(reinterpret_cast<const double2 *>(cm) + 1);
        const float4 c = S.centre[j];  // (cell centres are exact in binary32)
        const double dz = tz - (double)(R.half ? __fadd_rn(c.z, c.w) : __fsub_rn(c.z, c.w));
        const double dzz = dz * dz;
        const double xc[2] = {(double)__fsub_rn(c.x, c.w), (double)__fadd_rn(c.x, c.w)};
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const double dy = ty - (double)(y ? __fadd_rn(c.y, c.w) : __fsub_rn(c.y, c.w));
          const double h = fma(dy, dy, dzz);
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const double mc = y ? (x ? m23.y : m23.x) : (x ? m01.y : m01.x);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const double dx = tx[i] - xc[x], d2 = fma(dx, dx, h);
              // every cell but the target's own (d2 = 0)
              double r = rsqrt64(d2);
              r = (m4 & (1u << i)) && d2 > 0.0 ? r : 0.0;
              part[i] = fma(mc, r, part[i]);
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) sum[i] += part[i];
      nbot = 0;
      __syncwarp();
    }
  }
  const double scale = -G * invL[F.w];  // physical FP64 moments
  const int64_t cell = (int64_t)orig[p] * kCellsPerBlock + (4 * (o >> 2) + R.z) * 64 +
                       (4 * ((o >> 1) & 1) + R.y) * 8 + 4 * (o & 1);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double s = sum[i] + __shfl_xor_sync(kFull, sum[i], 16);
    if ((i >> 1) == R.half) out[cell + i] = s * scale;
  }
}

template <bool QUAD, bool VOTE>
cudaError_t go_f64(cudaStream_t s, int nb, const WalkRec *rec, const SibArgs &sib, const int4 *blk,
                   const int *orig, const FieldArgs &fa, double G, double *out) {
  const unsigned nunits = (unsigned)nb * 8u;
  constexpr int smem = kF64Warps * (int)sizeof(F64Mem<QUAD>);
  static_assert(smem <= 48 * 1024, "within the default dynamic shared-memory limit");
  k_walk_f64<QUAD, VOTE><<<(nunits + kF64Warps - 1) / kF64Warps, 32 * kF64Warps, smem, s>>>(
      nunits, rec, sib, blk, orig, fa.fld, fa.flev, fa.invL, G, out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_walk_f64(cudaStream_t s, const bh_options &opt, int nb, const WalkRec *rec,
                            const SibArgs &sib, const int4 *blk, const int *orig,
                            const FieldArgs &fa, double G, void *out) {
  const bool vote = opt.criterion == BH_CRIT_WARP_VOTE;
  double *o = (double *)out;
  if (opt.quadrupole)
    return vote ? go_f64<true, true>(s, nb, rec, sib, blk, orig, fa, G, o)
                : go_f64<true, false>(s, nb, rec, sib, blk, orig, fa, G, o);
  return vote ? go_f64<false, true>(s, nb, rec, sib, blk, orig, fa, G, o)
              : go_f64<false, false>(s, nb, rec, sib, blk, orig, fa, G, o);
}

}  // namespace bhg
