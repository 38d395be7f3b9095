// The Barnes-Hut walk: potential at every cell centre (Sec. 3.3).
//
// The paper walks node by node with a shared-memory stack and an all() vote
// (Sec. 3.3).  Here one warp walks for the 64 cells of a 4x4x4 octant of a
// block in two alternating phases that need no per-node control flow:
//
// 1. Testing.  The warp pops up to four opened nodes from its stack in shared
//    memory and tests their 32 children, one child per lane: the lane forms
//    the opening test of Eq. 4 for all 64 targets and gets a 64-bit mask.
//    Siblings lie together (WalkSib), so that 8 lanes read 8 neighbours.  With
//    P the targets that opened the parent, the targets accepting the child
//    are A = P & mask, those opening it O = P & ~mask.  A child with A != 0
//    is staged in shared memory; a child with O != 0 goes on the stack with P
//    = O, or, if it is a bottom node (its 8 children are cells), to the list
//    of opened bottom nodes.  Cells are never tested.
// 2. Evaluating.  Four sub-bricks of 16 cells (4x2x2) each have a list of the
//    staged nodes that one of their cells accepts, with the 16-bit mask.  8
//    lanes serve a sub-brick: lane bits 0-1 take every fourth list entry, bit
//    2 is the cell's z within the sub-brick, and a lane owns the 8 cells (4 in
//    x, 2 in y) of that z.  So a warp evaluates 16 different (node, 8 cells)
//    pairs at a time, each lane loading a record once for 8 interactions.
//    Opened bottom nodes are met row by row (eval_cells).
//
// Each target visits exactly the nodes of its own recursive walk and takes
// the decisions of the per-cell definition (or, with the warp vote, those of
// its 32-cell brick: the two words of the mask are the octant's two bricks).
// The order in which a target's terms are added depends on its octant's lists
// only -- not on the launch shape, the other fields of a batch or timing -- so
// every launch shape gives the same bits.
//
// What bounds it.  An interaction costs one rsqrt on the special-function
// unit (16 lanes per clock and SM: 4 clocks per 64 interactions) and, packed
// in f32x2 pairs, about 13 (monopole) or 25 (quadrupole) FMA-pipe clocks per
// 64 and scheduler.  What the lists save against a walk in which 64 targets
// share every step: at theta 0.75 on the 2M-cell spheroid a target accepts
// 401 nodes and opens 11 bottom nodes, its octant's union is 687 nodes and 61
// bottom nodes, a 16-cell sub-brick's 554 and 35 (groups of 4: 483 and 20,
// but then every lane reads its own record, and the shared-memory return path
// bounds the quadrupole walk).
//
// Measured (2,039,808-cell spheroid, persistent grid of 4-warp CTAs, groups in
// their own order; ms, with in brackets the walk that stepped 64 targets, or
// 32 with the vote, through the tree together, on its plain grid): quadrupole
// theta 0.75 0.96 (1.85), monopole 0.5 1.92 (3.2) and 0.24 10.7 (15.5), vote
// with quadrupole 0.8 0.91 (2.49); 16.3M-cell core, monopole 0.5 18.6 (27.4);
// 32^3 cells 0.085 (0.45): there a step tests 32 nodes per chain of dependent
// loads instead of one, and two warps share an octant (k_walk_shared).
//
// The opening test is evaluated in binary32 with the operation order stated
// in the public header; the interaction uses the same d2 formed again.  (The
// binary64 walk, bh_walk_f64.cu, and the periodic one share the traversal.)
#include "bh_lists.cuh"

namespace bhg {
namespace {

constexpr int kMaxWalkThreads = 512;  // largest tunable CTA
// Registers.  Monopole: 80, 24 warps per SM (97 without a bound, 20 warps: 8 %
// slower; 72 spills: 2-5 % slower).  Quadrupole: shared memory allows 16 warps
// whatever the registers, so 112 (80: 3.6 % slower; 128: 1 %).
constexpr int walk_regs(bool quad) { return quad ? 112 : 80; }

__global__ void k_prepare_sib_s2(int64_t n, WalkSib *__restrict__ sib, float inv_theta) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float s = __fadd_rn(__fmul_rn(sib[i].l, inv_theta), sib[i].delta);
  sib[i].s2 = __fmul_rn(s, s);
}

__global__ void k_prepare_s2(int64_t n, const float2 *__restrict__ aux, WalkRec *__restrict__ rec,
                             float inv_theta) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float2 a = aux[i];
  const float s = __fadd_rn(__fmul_rn(a.x, inv_theta), a.y);  // l/theta + delta
  rec[i].s2 = __fmul_rn(s, s);
}

// ---- binary32 walk -----------------------------------------------------------
// Staged nodes (a ring; room for one more step's is kept) and opened bottom
// nodes (evaluated once a step's might not fit).  Longer lists lose less where
// the sub-bricks' or rows' lists differ in length, and are evaluated in fewer
// and longer runs, which is worth more than the warps per SM that their shared
// memory costs (quadrupole 24 -> 16): 64 and 64 entries take 5.5 % longer on the
// core and the spheroid at theta 0.5, 7 % on the quadrupole walk.
constexpr int kRing = 128;
constexpr int kBottoms = 96;

struct QuadRest {                    // second half of a staged quadrupole (16-byte stride)
  float qxz, qyz, unused[2];
};
template <bool QUAD>
struct WalkMem {                     // of one warp
  Front front;
  float4 node[kRing];                // px, py, pz, m of the staged nodes
  float4 quad[QUAD ? kRing : 1];     // Qxx/2, Qyy/2, Qzz/2, Qxy
  QuadRest quad2[QUAD ? kRing : 1];  // Qxz, Qyz
  uint32_t list[4][kRing];           // per sub-brick, a ring: 16 slot | mask << 16
  float4 centre[kBottoms];           // opened bottom nodes: geometric centre, half a cell,
  uint32_t bottom[3][kBottoms];      // index, O (two words)
};

// Per-lane state of the evaluation: the lane's 8 targets as four x pairs, pair
// 2 r + k: row r (y = 2 (sub-brick & 1) + r), x = 2 k, 2 k + 1.  A walk shared
// by SPLIT warps leaves each its x pair k0 of both rows (SPLIT = 2: 4 targets)
// or of row r0 (SPLIT = 4: 2 targets).
constexpr int split_rows(int split) { return split == 4 ? 1 : 2; }
constexpr int split_pairs(int split) { return split == 1 ? 2 : 1; }  // x pairs of a row
template <bool COUNTS, int SPLIT>
struct Lane {
  u64 sum[4 / SPLIT], comp[4 / SPLIT];    // compensated pair sums
  int na[COUNTS ? 8 : 1], nb[COUNTS ? 8 : 1];  // accepted nodes, opened bottom nodes
};

// 1/sqrt(d) if m has the bit, else 0.
__device__ __forceinline__ float rsqrt_if(float d, uint32_t m, uint32_t bit) {
  float r;
  asm("{\n.reg .pred p;\n.reg .b32 t;\nand.b32 t, %2, %3;\nsetp.ne.b32 p, t, 0;\n"
      "mov.f32 %0, 0f00000000;\n@p rsqrt.approx.ftz.f32 %0, %1;\n}"
      : "=f"(r)
      : "f"(d), "r"(m), "r"(bit));
  return r;
}

// 1/sqrt(d) if d > least, else 0.
__device__ __forceinline__ float rsqrt_above(float d, float least) {
  float r;
  asm("{\n.reg .pred p;\nsetp.gt.f32 p, %1, %2;\nmov.f32 %0, 0f00000000;\n"
      "@p rsqrt.approx.ftz.f32 %0, %1;\n}"
      : "=f"(r)
      : "f"(d), "f"(least));
  return r;
}

// sum + comp += a b, compensated, the product unrounded: s = the sum with it
// added, err = (sum - s) + a b, exact where the sum is the larger (all terms
// are positive).  So that it is from the first term on, a lane's sums start
// from sum_base, which is taken off before they are merged.  Relative error
// of the potential against binary64 on 32^3 cells at theta 0.5: 2.757e-8, of
// which rounding the result is 2.5e-8; from zero 2.763e-8 (the early terms of
// four lanes' sums, where the walk that kept a target in one lane had 2.762e-8);
// two products to a compensation, 2 % faster, 2.765e-8.
template <bool KAHAN>
__device__ __forceinline__ void accumulate_product2(u64 &sum, u64 &comp, u64 a, u64 b) {
  const u64 s = fma2(a, b, sum);
  if (KAHAN) comp = add2(comp, fma2(a, b, sub2(sum, s)));
  sum = s;
}
// Four times the power of two at or below the field's mass: above any term
// (a mass over a distance) but those of a few cells next to a target that
// hold most of the field's mass, and a power of two, so that sum - sum_base
// is exact.  Zero for an octant with a cell of half the field's mass or more
// (cells: its 64 masses): that cell is no term of its own sum, which may then
// be far below the base, where comp would do all the adding, uncompensated (a
// cell of 10^7 times the rest's mass: error 8e-8 from the base, 3e-8 from
// zero).  A sum without a cell of half the mass is at least mass / (2 sqrt(3)).
template <bool KAHAN>
__device__ __forceinline__ u64 sum_base(float mass, const float *__restrict__ cells, int lane) {
  if (!KAHAN) return 0ull;
  const float2 m = __ldg(reinterpret_cast<const float2 *>(cells) + lane);
  const unsigned most = __reduce_max_sync(kFull, __float_as_uint(fmaxf(m.x, m.y)));  // (m >= 0)
  if (__uint_as_float(most) >= 0.5f * mass) return 0ull;
  const float b = 4.0f * __uint_as_float(__float_as_uint(mass) & 0x7f800000u);
  return pk(b, b);
}

template <int NR, int NK>  // rows, x pairs of a row
struct Targets {          // of one lane, read back before every evaluation
  u64 tx[NK];             // {x0, x1}, {x2, x3}
  float ty[NR], tz;
};

// A list entry as a lane evaluates it: the staged record (mass and x pairs
// duplicated for the packed operations) and the parts shared by a row.
template <bool QUAD, int NK>
struct Entry {
  u64 dx[NK], mm;      // {x0, x1} - px, {x2, x3} - px; {m, m}
  float py, dz;
  float4 q;            // Qxx/2, Qyy/2, Qzz/2, Qxy
  float2 q2;           // Qxz, Qyz
  uint32_t m8;         // bit 4 r + x: target x of row r takes part
  float h, qu, qc;     // of the current row

  template <int NR>
  __device__ __forceinline__ void load(const WalkMem<QUAD> &S, uint32_t v, int zsh,
                                       const Targets<NR, NK> &T) {
    const char *at = reinterpret_cast<const char *>(S.node) + (v & 0xffffu);
    const float4 n = *reinterpret_cast<const float4 *>(at);
    if (QUAD) {
      q = *reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(S.quad) + (v & 0xffffu));
      q2 = *reinterpret_cast<const float2 *>(reinterpret_cast<const char *>(S.quad2) + (v & 0xffffu));
    }
    m8 = v >> zsh;
    const u64 px = pk(n.x, n.x);
#pragma unroll
    for (int k = 0; k < NK; ++k) dx[k] = sub2(T.tx[k], px);
    mm = pk(n.w, n.w);
    py = n.y;
    dz = __fsub_rn(T.tz, n.z);
  }
  __device__ __forceinline__ void row(float ty) {
    const float dy = __fsub_rn(ty, py);
    h = __fmaf_rn(dz, dz, __fmul_rn(dy, dy));
    if (QUAD) {  // d^T Q d / 2 = dx (Qxx/2 dx + qu) + qc
      qu = __fmaf_rn(q2.x, dz, __fmul_rn(q.w, dy));
      const float v = __fmaf_rn(q.y, dy, __fmul_rn(q2.y, dz));
      qc = __fmaf_rn(dy, v, __fmul_rn(__fmul_rn(q.z, dz), dz));
    }
  }
  // The terms of targets 2 k, 2 k + 1 of row r as products rr t.
  __device__ __forceinline__ void terms(int r, int k, u64 &rr, u64 &t) const {
    float da, db;
    upk(fma2(dx[k], dx[k], pk(h, h)), da, db);
    rr = pk(rsqrt_if(da, m8, 1u << (4 * r + 2 * k)), rsqrt_if(db, m8, 2u << (4 * r + 2 * k)));
    t = mm;
    if (QUAD) {  // M rinv + (d^T Q d / 2) rinv^5
      const u64 hq = fma2(dx[k], fma2(pk(q.x, q.x), dx[k], pk(qu, qu)), pk(qc, qc));
      const u64 r2 = mul2(rr, rr);
      t = fma2(hq, mul2(r2, r2), mm);
    }
  }
};

// 8 entries of every sub-brick's list from ring position `at` (a multiple of
// 8): the lane takes entries par and par + 4.
template <bool KAHAN, bool COUNTS, bool QUAD, int SPLIT>
__device__ __forceinline__ void eval_nodes(
    const WalkMem<QUAD> &S, int sb, unsigned at, int par, int zsh,
    const Targets<split_rows(SPLIT), split_pairs(SPLIT)> &T, Lane<COUNTS, SPLIT> &L) {
  constexpr int NR = split_rows(SPLIT), NK = split_pairs(SPLIT);
  const uint32_t *list = &S.list[sb][(at & (kRing - 1)) + par];
  const uint32_t v0 = list[0], v1 = list[4];
  if (COUNTS) {
#pragma unroll
    for (int i = 0; i < 8; ++i) L.na[i] += ((v0 >> (zsh + i)) & 1u) + ((v1 >> (zsh + i)) & 1u);
    return;
  }
  Entry<QUAD, NK> a, b;
  a.load(S, v0, zsh, T);
  b.load(S, v1, zsh, T);
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    a.row(T.ty[r]);
    b.row(T.ty[r]);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      u64 ra, ta, rb, tb;
      a.terms(r, k, ra, ta);
      b.terms(r, k, rb, tb);
      accumulate_product2<KAHAN>(L.sum[NK * r + k], L.comp[NK * r + k], ra, ta);
      accumulate_product2<KAHAN>(L.sum[NK * r + k], L.comp[NK * r + k], rb, tb);
    }
  }
}

// TwoSum (Knuth): s + e = a + b exactly.
__device__ __forceinline__ u64 two_sum2(u64 a, u64 b, u64 &e) {
  const u64 s = add2(a, b), bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return s;
}

// The cells of the n opened bottom nodes.  Here a lane serves one row of four
// targets (row = lane & 15: y = 2 (row >> 2 & 1) + (row & 1), z = 2 (row >> 3)
// + (row >> 1 & 1)) and four cells of a bottom node (lane >> 4: its z half),
// and walks through the bottom nodes that a target of its row opened: few
// targets open a bottom node (19 % of the octant's 64, 32 % of a sub-brick's
// 16, 56 % of a row's 4 at theta 0.75), and one costs 8 interactions each.
// Every cell but the target's own (d2 > 0); a node's four terms are added
// plainly and join a compensated sum, which joins the lanes' totals at the end.
template <bool KAHAN, bool COUNTS, bool QUAD, int SPLIT>
__device__ __forceinline__ void eval_cells(const WalkMem<QUAD> &S,
                                           const float4 *__restrict__ cmass, int n, int lane,
                                           int r0, int k0, u64 base, Lane<COUNTS, SPLIT> &L) {
  constexpr int W = kBottoms / 32, NR = split_rows(SPLIT), NK = split_pairs(SPLIT);
  constexpr unsigned row_bits = SPLIT == 1 ? 15u : 3u;
  const bool serves = SPLIT != 4 || (lane & 1) == r0;  // (the row's y & 1)
  const int row = lane & 15, word = 1 + (row >> 3), sh = 4 * (row & 7) + 2 * k0, zhalf = lane >> 4;
  uint32_t mine[W];  // bottom nodes some target of the row opened
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int j = 32 * w + lane;
    const uint32_t lo = j < n ? S.bottom[1][j] : 0u, hi = j < n ? S.bottom[2][j] : 0u;
    mine[w] = 0u;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const unsigned b = __ballot_sync(kFull, (((r < 8 ? lo : hi) >> (4 * (r & 7) + 2 * k0)) & row_bits) != 0u);
      if (row == r) mine[w] = serves ? b : 0u;
    }
  }
  int left = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) left += __popc(mine[w]);
  const int steps = (int)__reduce_max_sync(kFull, (unsigned)left);
  u64 sum[NK], comp[NK], tx[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    sum[k] = base;
    comp[k] = 0ull;
    tx[k] = pk(S.front.tx[k0 + k].x, S.front.tx[k0 + k].z);
  }
  int nb[4] = {0, 0, 0, 0};
  const float ty = S.front.coord(16 + 2 * ((row >> 2) & 1) + (row & 1));
  const float tz = S.front.coord(8 + 4 * (row >> 3) + (row & 2));
#pragma unroll 2
  for (int it = 0; it < steps; ++it) {
    int j = 0;  // the next of the row's bottom nodes (none left: node 0 with an empty mask)
    const bool any = it < left;
#pragma unroll
    for (int w = W - 1; w >= 0; --w) j = mine[w] ? 32 * w + __ffs((int)mine[w]) - 1 : j;
#pragma unroll
    for (int w = 0, done = 0; w < W; ++w) {
      const uint32_t m = mine[w];
      mine[w] = done ? m : m & (m - 1u);
      done = done || m != 0u;
    }
    const uint32_t m4 = any ? S.bottom[word][j] >> sh : 0u;
    if (COUNTS) {
#pragma unroll
      for (int i = 0; i < 4; ++i) nb[i] += (m4 >> i) & 1u;
      continue;
    }
    // masses of the cells (x0, y0), (x1, y0), (x0, y1), (x1, y1) of the lane's z
    const float4 m = __ldg(cmass + 2 * (size_t)S.bottom[0][j] + zhalf);
    const float4 c = S.centre[j];
    float least[2 * NK];  // a target takes part where d2 > least: 0, or never
#pragma unroll
    for (int i = 0; i < 2 * NK; ++i) least[i] = (m4 & (1u << i)) ? 0.0f : __int_as_float(0x7f800000);
    const float dz = __fsub_rn(tz, zhalf ? __fadd_rn(c.z, c.w) : __fsub_rn(c.z, c.w));
    const float dzz = __fmul_rn(dz, dz);
    const float xl = __fsub_rn(c.x, c.w), xh = __fadd_rn(c.x, c.w);
    u64 dx[2][NK], part[NK];
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      dx[0][k] = sub2(tx[k], pk(xl, xl));
      dx[1][k] = sub2(tx[k], pk(xh, xh));
      part[k] = 0ull;
    }
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const float dy = __fsub_rn(ty, y ? __fadd_rn(c.y, c.w) : __fsub_rn(c.y, c.w));
      const float h = __fmaf_rn(dy, dy, dzz);
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const float mc = y ? (x ? m.w : m.z) : (x ? m.y : m.x);
#pragma unroll
        for (int k = 0; k < NK; ++k) {
          float da, db;
          upk(fma2(dx[x][k], dx[x][k], pk(h, h)), da, db);
          part[k] = fma2(pk(mc, mc), pk(rsqrt_above(da, least[2 * k]), rsqrt_above(db, least[2 * k + 1])),
                         part[k]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NK; ++k) accumulate2<KAHAN>(sum[k], comp[k], part[k]);
  }
  // to the lanes that own the targets: rows 2 (lane >> 2) and the next; the
  // two z halves are added, one lane of the four that share the targets takes them
  const int from = 2 * (lane >> 2);
  if (COUNTS) {
#pragma unroll
    for (int i = 0; i < 8; ++i) L.nb[i] += __shfl_sync(kFull, nb[i & 3], from + (i >> 2));
    return;
  }
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    u64 e = 0ull;
    sum[k] = sub2(sum[k], base);
    const u64 o = __shfl_xor_sync(kFull, sum[k], 16);
    if (KAHAN) {
      sum[k] = (lane & 16) ? two_sum2(o, sum[k], e) : two_sum2(sum[k], o, e);
      comp[k] = add2(add2(comp[k], __shfl_xor_sync(kFull, comp[k], 16)), e);
    } else {
      sum[k] = add2(sum[k], o);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const u64 v = __shfl_sync(kFull, sum[k], from + r0 + r);
      const u64 c = KAHAN ? __shfl_sync(kFull, comp[k], from + r0 + r) : 0ull;
      if ((lane & 3) == 0) {
        if (KAHAN) {
          L.sum[NK * r + k] = two_sum2(L.sum[NK * r + k], v, e);
          L.comp[NK * r + k] = add2(add2(L.comp[NK * r + k], c), e);
        } else {
          L.sum[NK * r + k] = add2(L.sum[NK * r + k], v);
        }
      }
    }
  }
}

// The sums of the four lanes that share the targets (lane bits 0 and 1).
template <bool KAHAN>
__device__ __forceinline__ void merge_lanes(u64 &sum, u64 &comp) {
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    const u64 v = __shfl_xor_sync(kFull, sum, o);
    if (KAHAN) {
      u64 e;  // (exact, so both lanes of a pair get the same)
      sum = (threadIdx.x & o) ? two_sum2(v, sum, e) : two_sum2(sum, v, e);
      comp = add2(add2(comp, __shfl_xor_sync(kFull, comp, o)), e);
    } else {
      sum = add2(sum, v);
    }
  }
}

struct WalkArgs {
  const WalkRec *rec;           // (the root's only)
  SibArgs sib;
  const int4 *blk;
  const int *orig;
  const int4 *fld;
  const double *invL;
  const unsigned long long *mmax;
  double G;
  float *out;
  int32_t *n_int, *n_test, *n_leaf;
  const int *flev;              // deepest block level per field
};

// Walk of octant u & 7 of sorted block u >> 3; with SPLIT > 1 by the SPLIT warps
// of the CTA, each for its part of the targets (r0, k0; else 0).  They test
// their part alone and join the masks (`joint`: two buffers, of which a warp
// overwrites one only after a barrier that follows the others' reads), so
// that all take the same steps and make the same lists.
template <bool KAHAN, bool COUNTS, bool QUAD, bool VOTE, int SPLIT = 1>
__device__ __forceinline__ void walk_octant(unsigned u, int lane, WalkMem<QUAD> &S,
                                            const WalkArgs &A, int r0 = 0, int k0 = 0,
                                            uint2 (*joint)[SPLIT][32] = nullptr) {
  constexpr int NR = split_rows(SPLIT), NK = split_pairs(SPLIT), NP = NR * NK;
  const unsigned p = u >> 3;
  const int o = (int)(u & 7);
  const int4 B = A.blk[p], F = A.fld[p];
  const int par = lane & 3, zl = (lane >> 2) & 1, sb = lane >> 3;
  const unsigned lower = (1u << lane) - 1u;
  front_start(S.front, octant_at(B, o), F, p, lane, A.rec, A.sib.tops);
  const u64 base = sum_base<KAHAN>(A.rec[F.x].m, A.sib.cmass + ((size_t)u << 6), lane);
  Lane<COUNTS, SPLIT> L;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    L.sum[i] = base;
    L.comp[i] = 0ull;
  }
#pragma unroll
  for (int i = 0; i < (COUNTS ? 8 : 1); ++i) L.na[i] = L.nb[i] = 0;
  const int zsh = 16 + 8 * zl + 4 * r0 + 2 * k0;
  unsigned turn = 0u;

  // warp-uniform: stack entries; staged nodes ever and the oldest still needed;
  // list positions (written ever per sub-brick, evaluated ever); opened bottom nodes
  int depth = 1, nbot = 0;
  const int pop4 = stack_pop4(A.flev[F.w]);
  const unsigned tops = (unsigned)A.sib.tops;
  unsigned staged = 0u, oldest = 0u, head = 0u, tail[4] = {0u, 0u, 0u, 0u};
  while (depth > 0) {
    const Tested t = front_step<VOTE>(
        S.front, depth, pop4, tops, lane, A.sib.sib, [&](const float4 &a, float s2, uint32_t *m) {
          if (SPLIT == 1) {
            test64<false>(S.front, a.x, a.y, a.z, s2, m);
            return;
          }
          test_part<SPLIT>(S.front, r0, k0, a.x, a.y, a.z, s2, m);
          joint[turn][threadIdx.x >> 5][lane] = make_uint2(m[0], m[1]);
          __syncthreads();
#pragma unroll
          for (int i = 0; i < SPLIT; ++i) {
            const uint2 o = joint[turn][i][lane];
            m[0] |= o.x;
            m[1] |= o.y;
          }
          turn ^= 1u;
        });
    const unsigned acc = __ballot_sync(kFull, (t.alo | t.ahi) != 0u);
    if (acc) {
      const unsigned slot = (staged + __popc(acc & lower)) & (kRing - 1);
      if (t.alo | t.ahi) {
        S.node[slot] = t.rec;
        if (QUAD) {
          copy_async<16>(&S.quad[slot], A.sib.quad + t.node);
          copy_async<8>(&S.quad2[slot], &A.sib.quad[t.node].qxz);
        }
      }
      staged += __popc(acc);
#pragma unroll
      for (int g = 0; g < 4; ++g) {  // to the lists of the sub-bricks with an accepting cell
        const uint32_t w = g < 2 ? t.alo : t.ahi;
        const uint32_t mk = (g & 1) ? (w & 0xffff0000u) : (w << 16);
        const unsigned c = __ballot_sync(kFull, mk != 0u);
        if (mk) S.list[g][(tail[g] + __popc(c & lower)) & (kRing - 1)] = mk | (16u * slot);
        tail[g] += __popc(c);
      }
    }
    const bool bottom = (t.olo | t.ohi) != 0u && (t.kids & kBottomBit) != 0u;
    const unsigned bot = __ballot_sync(kFull, bottom);
    if (bot) {
      const int slot = nbot + __popc(bot & lower);
      if (bottom) {
        S.bottom[0][slot] = t.kids & ~kBottomBit;
        S.bottom[1][slot] = t.olo;
        S.bottom[2][slot] = t.ohi;
      }
      nbot += __popc(bot);
    }
    __syncwarp();
    const bool last = depth == 0;
    if (staged - oldest > kRing - 32 || last) {
      // Evaluate listed nodes until a further chunk's fit the ring (at the
      // end: all).  All lists are read at the same position, 8 entries at a
      // time: while every list has 8, and then with the short ones filled up
      // by empty entries.
      if (QUAD) {
        copy_async_wait();
        __syncwarp();
      }
      Targets<NR, NK> T;
#pragma unroll
      for (int k = 0; k < NK; ++k) T.tx[k] = pk(S.front.tx[k0 + k].x, S.front.tx[k0 + k].z);
#pragma unroll
      for (int r = 0; r < NR; ++r) T.ty[r] = S.front.coord(16 + 2 * (sb & 1) + r0 + r);
      T.tz = S.front.coord(8 + 4 * (sb >> 1) + 2 * zl);
      for (;;) {
        const unsigned full = (min(min(tail[0], tail[1]), min(tail[2], tail[3])) - head) / 8u;
        for (unsigned i = 0; i < full; ++i, head += 8u)
          eval_nodes<KAHAN, COUNTS, QUAD, SPLIT>(S, sb, head, par, zsh, T, L);
        const unsigned mine = sb < 2 ? (sb ? tail[1] : tail[0]) : (sb == 2 ? tail[2] : tail[3]);
        // the oldest staged node still listed
        unsigned age = staged - oldest;
        if (mine != head) age = ((S.list[sb][head & (kRing - 1)] >> 4) - oldest) & (kRing - 1);
        oldest += __reduce_min_sync(kFull, age);
        if (last ? oldest == staged : staged - oldest <= kRing - 32) break;
        if ((int)(mine - head) < 8) {  // the 8 lanes of the sub-brick: one entry each
          const unsigned at = head + (lane & 7);
          if ((int)(at - mine) >= 0) S.list[sb][at & (kRing - 1)] = 0u;
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) tail[g] = (int)(tail[g] - head) < 8 ? head + 8u : tail[g];
        __syncwarp();
      }
      __syncwarp();
    }
    if (nbot > kBottoms - 32 || (last && nbot)) {
      for (int j = lane; j < nbot; j += 32) S.centre[j] = bottom_centre(S.bottom[0][j], A.blk);
      __syncwarp();
      eval_cells<KAHAN, COUNTS, QUAD, SPLIT>(S, reinterpret_cast<const float4 *>(A.sib.cmass), nbot,
                                             lane, r0, k0, base, L);
      nbot = 0;
      __syncwarp();
    }
  }
  // each of the four lanes writes two of the shared 8 targets: row par >> 1,
  // x = 2 (par & 1) and the next (of a shared walk two lanes or one)
  const int r = SPLIT == 4 ? r0 : (SPLIT == 2 ? par & 1 : par >> 1);
  const int k = SPLIT == 1 ? par & 1 : k0;
  const int64_t cell = (int64_t)A.orig[p] * kCellsPerBlock + (4 * (o >> 2) + 2 * (sb >> 1) + zl) * 64 +
                       (4 * ((o >> 1) & 1) + 2 * (sb & 1) + r) * 8 + 4 * (o & 1) + 2 * k;
  if (COUNTS) {
    int na[2] = {0, 0}, nb[2] = {0, 0};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      int v = L.na[i];  // every lane of the four counted the entries it took
      v += __shfl_xor_sync(kFull, v, 1);
      v += __shfl_xor_sync(kFull, v, 2);
      if ((i >> 1) == par) {
        na[i & 1] = v;
        nb[i & 1] = L.nb[i];
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      // t tests: the root and 8 for every opened node above the bottom ones;
      // each ends in an accepted, an opened bottom or another opened node:
      // t = 1 + 8 (t - na - nb)
      const int cells = 8 * nb[i] - 1;  // not its own
      A.n_int[cell + i] = na[i] + cells;
      A.n_test[cell + i] = (8 * (na[i] + nb[i]) - 1) / 7;
      if (A.n_leaf) A.n_leaf[cell + i] = cells;
    }
  } else {
    // -G/L times the field's binary32 mass unit 2^e (exact), rounded once
    const float scale = (float)(-A.G * A.invL[F.w] * pow2i(mass_exponent(A.mmax[F.w])));
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      L.sum[i] = sub2(L.sum[i], base);
      merge_lanes<KAHAN>(L.sum[i], L.comp[i]);
      if (i == par) {
        float sa, sb_;
        upk(finish2<KAHAN>(L.sum[i], L.comp[i]), sa, sb_);
        A.out[cell] = __fmul_rn(sa, scale);
        A.out[cell + 1] = __fmul_rn(sb_, scale);
      }
    }
  }
}

// A unit of work is one octant (np = 1) or two neighbouring ones, walked one
// after the other (np = 2).  Plain grid: warp i walks unit order[i] (or i).
template <bool KAHAN, bool COUNTS, bool QUAD, bool VOTE>
__global__ void __maxnreg__(walk_regs(QUAD))
    k_walk_lists(unsigned nunits, int np, const unsigned *__restrict__ order, const WalkArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WalkMem<QUAD> &S = reinterpret_cast<WalkMem<QUAD> *>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (warp >= nunits) return;  // whole warps only
  const unsigned u = order ? order[warp] : warp;
  for (int k = 0; k < np; ++k) walk_octant<KAHAN, COUNTS, QUAD, VOTE>(u * np + k, lane, S, A);
}

// The octants of a small mesh, one per CTA of SPLIT warps, each for its part of
// the targets: every target's terms are added in the same order as by one
// warp, so the bits are the same.  Where a warp has a scheduler to itself, the
// chain of a step and of its entries is what takes the time, and most
// schedulers are idle; a part's tests and evaluations take 1/SPLIT of it.
template <bool QUAD, int SPLIT>
struct SharedMem {
  WalkMem<QUAD> warp[SPLIT];
  uint2 joint[2][SPLIT][32];
};
template <bool KAHAN, bool QUAD, bool VOTE, int SPLIT>
__global__ void __launch_bounds__(32 * SPLIT) k_walk_shared(const WalkArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SharedMem<QUAD, SPLIT> &S = *reinterpret_cast<SharedMem<QUAD, SPLIT> *>(smem_raw);
  const int w = threadIdx.x >> 5;
  walk_octant<KAHAN, false, QUAD, VOTE, SPLIT>(blockIdx.x, threadIdx.x & 31, S.warp[w], A, w >> 1,
                                               w & 1, S.joint);
}
// The same walk on a persistent grid: each warp takes `per_ticket`
// consecutive units at a time from the work counter (one atomic add by lane
// 0; no waiting on other warps) until every unit is taken.  In the units'
// own order, consecutive units are neighbouring octants; with `order` (the
// units sorted by the time of their walks, longest first) the long walks
// start first and the short ones fill the end, so that fewer warps are left
// running alone at the end of the launch.  cycles (or null): the SM clock
// cycles of each unit's walk, the measurement that order is made from.
template <bool KAHAN, bool COUNTS, bool QUAD, bool VOTE>
__global__ void __maxnreg__(walk_regs(QUAD))
    k_walk_queue(unsigned nunits, int np, unsigned per_ticket, unsigned *__restrict__ counter,
                 const unsigned *__restrict__ order, unsigned long long *__restrict__ cycles,
                 const WalkArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WalkMem<QUAD> &S = reinterpret_cast<WalkMem<QUAD> *>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  for (;;) {
    unsigned u0 = 0u;
    if (lane == 0) u0 = atomicAdd(counter, per_ticket);
    u0 = __shfl_sync(kFull, u0, 0);
    if (u0 >= nunits) return;
    const unsigned u1 = u0 + per_ticket < nunits ? u0 + per_ticket : nunits;
    for (unsigned i = u0; i < u1; ++i) {
      const unsigned u = order ? order[i] : i;
      const long long c0 = cycles ? clock64() : 0;
      for (int k = 0; k < np; ++k) walk_octant<KAHAN, COUNTS, QUAD, VOTE>(u * np + k, lane, S, A);
      if (cycles && lane == 0) cycles[u] = (unsigned long long)(clock64() - c0);
    }
  }
}

template <bool KAHAN, bool COUNTS, bool QUAD, bool VOTE>
cudaError_t go_lists(cudaStream_t s, int nb, const WalkArgs &a, const WalkShape &shape) {
  const int np = shape.pairs > 0 ? shape.pairs : 1;
  const unsigned nunits = (unsigned)nb * (8u / (unsigned)np);
  const int w = shape.warps > 0 ? shape.warps : kDefaultWalkWarps;
  const int smem = w * (int)sizeof(WalkMem<QUAD>);
  // (whatever the shape: the bits are the same, and no counter is needed)
  const int split = COUNTS || shape.cycles ? 1 : walk_split(nb);
  if (split == 4) {
    k_walk_shared<KAHAN, QUAD, VOTE, 4><<<8 * nb, 128, (int)sizeof(SharedMem<QUAD, 4>), s>>>(a);
    return cudaGetLastError();
  }
  if (split == 2) {
    k_walk_shared<KAHAN, QUAD, VOTE, 2><<<8 * nb, 64, (int)sizeof(SharedMem<QUAD, 2>), s>>>(a);
    return cudaGetLastError();
  }
  if (shape.ticket > 0 && shape.counter) {  // persistent: the CTAs that fit at once
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &per_sm, k_walk_queue<KAHAN, COUNTS, QUAD, VOTE>, 32 * w, smem);
    if (e != cudaSuccess) return e;
    const unsigned warps_needed = (nunits + (unsigned)shape.ticket - 1) / (unsigned)shape.ticket;
    const unsigned ctas_needed = (warps_needed + (unsigned)w - 1) / (unsigned)w;
    const unsigned resident = (unsigned)(sms * (per_sm > 0 ? per_sm : 1));
    const unsigned grid = ctas_needed < resident ? ctas_needed : resident;
    e = cudaMemsetAsync(shape.counter, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    k_walk_queue<KAHAN, COUNTS, QUAD, VOTE><<<grid, 32 * w, smem, s>>>(
        nunits, np, (unsigned)shape.ticket, shape.counter, shape.order, shape.cycles, a);
    return cudaGetLastError();
  }
  const int grid = (int)((nunits + w - 1) / w);
  k_walk_lists<KAHAN, COUNTS, QUAD, VOTE><<<grid, 32 * w, smem, s>>>(nunits, np, shape.order, a);
  return cudaGetLastError();
}

template <bool KAHAN, bool COUNTS, bool QUAD>
cudaError_t go_criterion(cudaStream_t s, bool vote, int nb, const WalkArgs &a,
                         const WalkShape &shape) {
  return vote ? go_lists<KAHAN, COUNTS, QUAD, true>(s, nb, a, shape)
              : go_lists<KAHAN, COUNTS, QUAD, false>(s, nb, a, shape);
}

// CTAs of up to 16 warps take more dynamic shared memory than the default limit.
template <bool KAHAN, bool COUNTS, bool QUAD, bool VOTE>
cudaError_t raise_smem() {
  const int bytes = (kMaxWalkThreads / 32) * (int)sizeof(WalkMem<QUAD>);
  cudaError_t e = cudaFuncSetAttribute(k_walk_lists<KAHAN, COUNTS, QUAD, VOTE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_walk_queue<KAHAN, COUNTS, QUAD, VOTE>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && !COUNTS)
    e = cudaFuncSetAttribute(k_walk_shared<KAHAN, QUAD, VOTE, 4>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SharedMem<QUAD, 4>));
  return e;
}

}  // namespace

// Up to two warps to each scheduler an octant is shared by 4 or 2 warps (152
// SMs: 38 and 76 blocks).  Above, the doubled traversal costs more than the idle
// schedulers (us, walk alone; persistent grid, 2 warps, 4 warps): 8 octants 36,
// 29, 27; 64: 67, 55, 50; 120: 80, 67, 60; 512: 93, 85, 83 (quadrupole, 568:
// 54, 48, 51); 792: 167, 199, 258.
int walk_split(int nb) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  const int64_t warps = 4 * 2 * (int64_t)sms;
  for (int split = 4; split > 1; split /= 2)
    if (8 * (int64_t)nb * split <= warps) return split;
  return 1;
}

cudaError_t prepare_walk_kernels() {
  cudaError_t e = raise_smem<true, false, false, false>();
  if (e == cudaSuccess) e = raise_smem<true, false, false, true>();
  if (e == cudaSuccess) e = raise_smem<true, false, true, false>();
  if (e == cudaSuccess) e = raise_smem<true, false, true, true>();
  if (e == cudaSuccess) e = raise_smem<false, false, false, false>();
  if (e == cudaSuccess) e = raise_smem<false, false, false, true>();
  if (e == cudaSuccess) e = raise_smem<false, false, true, false>();
  if (e == cudaSuccess) e = raise_smem<false, false, true, true>();
  if (e == cudaSuccess) e = raise_smem<false, true, false, false>();
  if (e == cudaSuccess) e = raise_smem<false, true, false, true>();
  return e;
}

cudaError_t launch_prepare_s2(cudaStream_t s, int64_t n_nodes, const float2 *aux, WalkRec *rec,
                              float inv_theta) {
  const int threads = 256;
  k_prepare_s2<<<(unsigned)((n_nodes + threads - 1) / threads), threads, 0, s>>>(n_nodes, aux, rec,
                                                                               inv_theta);
  return cudaGetLastError();
}

cudaError_t launch_prepare_sib_s2(cudaStream_t s, int64_t entries, WalkSib *sib, float inv_theta) {
  const int threads = 256;
  k_prepare_sib_s2<<<(unsigned)((entries + threads - 1) / threads), threads, 0, s>>>(entries, sib,
                                                                                   inv_theta);
  return cudaGetLastError();
}

// Picks the kernel instance for the options.  The counting walk takes the
// same decisions as every walk of the same criterion (the opening test does
// not depend on precision, summation or the quadrupole term).
cudaError_t launch_walk(cudaStream_t s, const bh_options &opt, int nb, const WalkRec *rec,
                        const SibArgs &sib, const int4 *blk, const int *orig, const FieldArgs &fa,
                        double G, void *out, int32_t *n_int, int32_t *n_test, int32_t *n_leaf,
                        WalkShape shape) {
  WalkArgs a;
  a.rec = rec;
  a.sib = sib;
  a.blk = blk;
  a.orig = orig;
  a.fld = fa.fld;
  a.invL = fa.invL;
  a.mmax = fa.mmax;
  a.G = G;
  a.out = (float *)out;
  a.n_int = n_int;
  a.n_test = n_test;
  a.n_leaf = n_leaf;
  a.flev = fa.flev;
  const bool vote = opt.criterion == BH_CRIT_WARP_VOTE;
  if (n_int) return go_criterion<false, true, false>(s, vote, nb, a, shape);
  if (opt.precision == BH_PREC_F64)
    return launch_walk_f64(s, opt, nb, rec, sib, blk, orig, fa, G, out);
  if (opt.quadrupole)
    return opt.kahan ? go_criterion<true, false, true>(s, vote, nb, a, shape)
                     : go_criterion<false, false, true>(s, vote, nb, a, shape);
  return opt.kahan ? go_criterion<true, false, false>(s, vote, nb, a, shape)
                   : go_criterion<false, false, false>(s, vote, nb, a, shape);
}

}  // namespace bhg
