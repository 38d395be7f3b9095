// Traversal of the octree for a warp's 64 targets (a 4x4x4 octant of a block)
// by testing eight siblings at a time, one child per lane, shared by the walks
// that collect lists (bh_walk.cu describes the method).
#pragma once
#include "bh_walk_common.cuh"

namespace bhg {
namespace {

// ---- stack of opened nodes ---------------------------------------------------
// It never overflows: popping a node pushes at most its 8 children, and the
// nodes pushed have levels 1 .. max_block_level + 1 (the children of the
// deepest are bottom nodes), so from any state a depth-first descent by
// single pops adds at most 7 (max_block_level + 1); any four nodes are popped
// while the 28 that this can add leave room for such a descent.  Fuller, four
// are popped if all are block roots or level-one nodes and the 28 fit: what
// they push are level-one nodes at most, which push nothing, and the nodes
// below them on the stack have the room that they had.  (In a mesh of 18
// levels there is no room for any four, and single pops keep a quarter of the
// lanes at work: 3,452 blocks refined about four corners, theta 0.35, 4.49 ms
// before the lists, 5.33 by single pops, 3.87 so.  The level is the field's
// own, and a node's kind the same in every batch, so that a field's sums do
// not depend on the other fields.)
constexpr int kStack = 160;
constexpr int stack_pop4(int max_block_level) { return kStack - 28 - 7 * (max_block_level + 1); }
static_assert(kStack >= 1 + 7 * (kMaxBlockLevel + 1), "stack must hold a descent by single pops");

struct Front {                       // of one warp, in shared memory
  uint2 waiting[kStack];             // P of the opened nodes (two words),
  uint32_t kids[kStack];             // where their children start
  float4 tx[2], tz[2], ty;           // {x0, x0, x1, x1}, ..., {y0, y1, y2, y3} of the octant
  // float i of tx (0-7: x i/2), tz (8-15: z (i-8)/2), ty (16-19: y i-16)
  __device__ __forceinline__ float coord(int i) const {
    return reinterpret_cast<const float *>(tx)[i];
  }
};

// mask << 1 | sign bit of v
__device__ __forceinline__ uint32_t push_sign(uint32_t mask, float v) {
  return __funnelshift_l(__float_as_uint(v), mask, 1);
}

// The minimum image of a pair of box-unit displacements in (-1, 1): d minus the
// nearest whole number (the two magic additions round to even at one half, so
// +-1/2 stay; all three steps are exact for what they are used for).
__device__ __forceinline__ u64 wrap2(u64 d) {
  const u64 magic = pk(12582912.0f, 12582912.0f);  // 1.5 2^23
  return sub2(d, sub2(add2(d, magic), magic));
}

// The opening test of one node for the 64 targets: bit 16 (y >> 1) + 8 (z & 1)
// + 4 (y & 1) + x of m[z >> 1] is set iff d2 > s2, d2 = fma(dx, dx, fma(dz,
// dz, dy dy)) (the header's rounding), read off the sign of s2 - d2, which
// rounding to nearest keeps exact (and which a NaN has clear: not accepted).
// 4 dx, 4 dz, 2 pairs of dy; 8 packed FMAs give the 16 (y, z) parts, then a
// packed FMA, a packed subtraction and two funnel shifts per two targets:
// 148 instructions for 32 nodes x 64 targets (WRAP, minimum-image
// displacements: 178).
template <bool WRAP>
__device__ __forceinline__ void test64(const Front &S, float px, float py, float pz,
                                       float s2, uint32_t m[2]) {
  const float4 x01 = S.tx[0], x23 = S.tx[1], z01 = S.tz[0], z23 = S.tz[1], yy = S.ty;
  const u64 pxx = pk(px, px), pyy = pk(py, py), pzz = pk(pz, pz), ss = pk(s2, s2);
  u64 dx[4] = {sub2(pk(x01.x, x01.y), pxx), sub2(pk(x01.z, x01.w), pxx),
                     sub2(pk(x23.x, x23.y), pxx), sub2(pk(x23.z, x23.w), pxx)};
  u64 dz[4] = {sub2(pk(z01.x, z01.y), pzz), sub2(pk(z01.z, z01.w), pzz),
                     sub2(pk(z23.x, z23.y), pzz), sub2(pk(z23.z, z23.w), pzz)};
  u64 dya = sub2(pk(yy.x, yy.y), pyy), dyb = sub2(pk(yy.z, yy.w), pyy);
  if (WRAP) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      dx[i] = wrap2(dx[i]);
      dz[i] = wrap2(dz[i]);
    }
    dya = wrap2(dya);
    dyb = wrap2(dyb);
  }
  const u64 ya = mul2(dya, dya), yb = mul2(dyb, dyb);
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    uint32_t v = 0u;
#pragma unroll
    for (int yh = 1; yh >= 0; --yh)
#pragma unroll
      for (int zl = 1; zl >= 0; --zl) {
        const u64 h = fma2(dz[2 * w + zl], dz[2 * w + zl], yh ? yb : ya);
        float lo[4], hi[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) upk(sub2(ss, fma2(dx[x], dx[x], h)), lo[x], hi[x]);
#pragma unroll
        for (int x = 3; x >= 0; --x) v = push_sign(v, hi[x]);
#pragma unroll
        for (int x = 3; x >= 0; --x) v = push_sign(v, lo[x]);
      }
    m[w] = v;
  }
}

// The same test for the part of the targets that one of SPLIT warps holds: x =
// 2 k0, 2 k0 + 1 and, with SPLIT = 4, y = r0, r0 + 2; the other bits are clear.
template <int SPLIT>
__device__ __forceinline__ void test_part(const Front &S, int r0, int k0, float px, float py,
                                          float pz, float s2, uint32_t m[2]) {
  const float4 xx = S.tx[k0], z01 = S.tz[0], z23 = S.tz[1];
  const u64 pyy = pk(py, py), pzz = pk(pz, pz), ss = pk(s2, s2);
  const u64 dx[2] = {sub2(pk(xx.x, xx.y), pk(px, px)), sub2(pk(xx.z, xx.w), pk(px, px))};
  const u64 dz[4] = {sub2(pk(z01.x, z01.y), pzz), sub2(pk(z01.z, z01.w), pzz),
                     sub2(pk(z23.x, z23.y), pzz), sub2(pk(z23.z, z23.w), pzz)};
  constexpr int NY = SPLIT == 4 ? 1 : 2;  // y pairs {r0, r0 + 2} or {0, 1}, {2, 3}
  u64 yy[NY];
#pragma unroll
  for (int i = 0; i < NY; ++i) {
    const u64 dy = sub2(SPLIT == 4 ? pk(S.coord(16 + r0), S.coord(18 + r0))
                                   : pk(S.coord(16 + 2 * i), S.coord(17 + 2 * i)), pyy);
    yy[i] = mul2(dy, dy);
  }
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    float v[4][2][2];  // [y][z & 1][x]
#pragma unroll
    for (int zl = 0; zl < 2; ++zl)
#pragma unroll
      for (int i = 0; i < NY; ++i) {
        const u64 h = fma2(dz[2 * w + zl], dz[2 * w + zl], yy[i]);
#pragma unroll
        for (int x = 0; x < 2; ++x)
          upk(sub2(ss, fma2(dx[x], dx[x], h)), v[2 * i][zl][x], v[2 * i + 1][zl][x]);
      }
    uint32_t b = 0u;
#pragma unroll
    for (int yh = 1; yh >= 0; --yh)
#pragma unroll
      for (int zl = 1; zl >= 0; --zl)
#pragma unroll
        for (int r = NY - 1; r >= 0; --r) {
          const int y = SPLIT == 4 ? yh : 2 * yh + r;
          b = push_sign(push_sign(b << (SPLIT == 4 ? 6 : 2), v[y][zl][1]), v[y][zl][0]);
        }
    m[w] = b << ((SPLIT == 4 ? 4 * r0 : 0) + 2 * k0);
  }
}

// One octant's place in the mesh.
struct Octant {
  int ox, oy, oz;   // lowest cell of the octant in its level's lattice
  float hh;         // 2^-(level+1)
  // cell centre in box units, exact in binary32: (2 i + 1) 2^-(level+1)
  __device__ __forceinline__ float centre(int i) const {
    return __fmul_rn((float)(2 * i + 1), hh);
  }
};
__device__ __forceinline__ Octant octant_at(int4 B, int o) {
  return {8 * B.y + 4 * (o & 1), 8 * B.z + 4 * ((o >> 1) & 1), 8 * B.w + 4 * (o >> 2),
          pow2f(-(B.x + 3 + 1))};
}

// Starts the traversal of octant o of sorted block p (field F): coordinates,
// and the root opened by all (it contains every target, so no target accepts
// it, theta <= 1).  Its children: a top node's by its slot (the record's spare
// word), a field's only block's by p.  Ends with the warp in step.
__device__ __forceinline__ void front_start(Front &S, const Octant &O, int4 F, unsigned p, int lane,
                                            const WalkRec *__restrict__ rec, int64_t tops) {
  __syncwarp();  // the last octant's data has been read
  if (lane < 20) {  // tx (8 floats), tz (8), ty (4)
    const int i = lane < 16 ? (lane & 7) >> 1 : lane - 16;
    reinterpret_cast<float *>(S.tx)[lane] =
        O.centre((lane < 8 ? O.ox : lane < 16 ? O.oz : O.oy) + i);
  }
  if (lane == 0) {
    const WalkRec r = rec[F.x];
    S.waiting[0] = make_uint2(kFull, kFull);
    S.kids[0] = r.skip - (unsigned)F.x == (unsigned)kNodesPerBlock
                    ? (unsigned)kSibsPerBlock * p
                    : (unsigned)tops + 8u * __float_as_uint(r.pad[0]);
  }
  __syncwarp();
}

// What a lane found out about its child of this step.
struct Tested {
  float4 rec;              // px, py, pz, m
  unsigned node, kids;     // its sibling-order index, its children's (kBottomBit)
  uint32_t alo, ahi;       // targets that accept it
  uint32_t olo, ohi;       // targets that open it
};

// Pops up to four opened nodes, tests their children, and pushes those that
// some target opens (bottom nodes excepted).  With VOTE the targets of each
// 32-cell brick (a word of the mask) accept only together.  tops: where the
// top nodes' children start (below: children of block roots and level-one
// nodes).  test(a, s2, m) makes the mask.
template <bool VOTE, class Test>
__device__ __forceinline__ Tested front_step(Front &S, int &depth, int pop4, unsigned tops, int lane,
                                             const WalkSib *__restrict__ sib, const Test &test) {
  int pop = depth < 4 ? depth : 4;
  if (depth > pop4) {
    const bool inside = S.kids[max(depth - 1 - (lane & 3), 0)] < tops;
    pop = __all_sync(kFull, inside) && depth <= kStack - 28 ? pop : 1;
  }
  const bool valid = (lane >> 3) < pop;
  uint2 P = make_uint2(0u, 0u);
  float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
  Tested t;
  t.node = 0u;
  if (valid) {
    const int at = depth - 1 - (lane >> 3);
    t.node = S.kids[at] + (lane & 7);
    a = __ldg(reinterpret_cast<const float4 *>(sib + t.node));
    b = __ldg(reinterpret_cast<const float4 *>(sib + t.node) + 1);  // s2, kids
    P = S.waiting[at];
  }
  depth -= pop;
  uint32_t m[2];
  test(a, b.x, m);
  if (VOTE) {
    m[0] = m[0] == kFull ? kFull : 0u;
    m[1] = m[1] == kFull ? kFull : 0u;
  }
  t.rec = a;
  t.kids = __float_as_uint(b.y);
  t.alo = P.x & m[0];
  t.ahi = P.y & m[1];
  t.olo = P.x & ~m[0];
  t.ohi = P.y & ~m[1];
  const bool open = (t.olo | t.ohi) != 0u && !(t.kids & kBottomBit);
  __syncwarp();  // the popped entries have been read
  const unsigned push = __ballot_sync(kFull, open);
  if (open) {
    const int at = depth + __popc(push & ((1u << lane) - 1u));
    S.waiting[at] = make_uint2(t.olo, t.ohi);
    S.kids[at] = t.kids;
  }
  depth += __popc(push);
  return t;
}

template <bool VOTE, bool WRAP = false>
__device__ __forceinline__ Tested front_step(Front &S, int &depth, int pop4, unsigned tops, int lane,
                                             const WalkSib *__restrict__ sib) {
  return front_step<VOTE>(S, depth, pop4, tops, lane, sib,
                          [&](const float4 &a, float s2, uint32_t *m) {
                            test64<WRAP>(S, a.x, a.y, a.z, s2, m);
                          });
}

// Geometric centre and half a cell of the bottom node 64 p + q.
__device__ __forceinline__ float4 bottom_centre(unsigned at, const int4 *__restrict__ blk) {
  const unsigned q = at & 63u;
  const int4 Q = blk[at >> 6];
  const float half = pow2f(-(Q.x + 4)), side = pow2f(-(Q.x + 3));
  auto mid = [side](int block, unsigned hi, unsigned lo) {  // exact in binary32
    return __fmul_rn((float)(2 * (4 * block + (int)(2u * (hi & 1u) + (lo & 1u))) + 1), side);
  };
  return make_float4(mid(Q.y, q >> 3, q), mid(Q.z, q >> 4, q >> 1), mid(Q.w, q >> 5, q >> 2), half);
}

}  // namespace
}  // namespace bhg
