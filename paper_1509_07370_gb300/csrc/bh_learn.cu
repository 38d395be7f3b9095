// Learned residual correction of accepted nodes (not in the paper).
//
// The walk accepts a node and adds its monopole M/d.  The correction
// multiplies that term by (1 + s^2 y), y = MLP(x), s = l/d, where x holds ten
// features of the (target, node) pair:
//   u = d/|d| (3), s, s^2, s^3, delta/l, u^T Q u / (M l^2), |Q|_F / (M l^2),
//   s^2 u^T Q u / (M l^2)
// (Q: the node's traceless quadrupole about its centre of mass, so the
// quadrupole option's records are needed).  The network is 10 -> 64 -> 64 -> 1
// with tanh-form GELU activations.
//
// This file holds what trains it, on the GPU:
//   * k_pairs_list / k_pairs_eval: the method's own residuals -- for sampled
//     target cells, every internal node their per-cell walk accepts (the same
//     binary32 opening test as the walk), and for each pair the node's exact
//     contribution summed over its cells in FP64: eps = exact/(M/d) - 1;
//   * k_mlp_grad / k_mlp_adam: forward and backward passes of the MLP over a
//     batch (mean squared error against z = eps/s^2) and an Adam update, in
//     FP32 on the CUDA cores;
// and bh_set_mlp, which rounds trained weights to bf16 for the tensor-core
// evaluation inside the walk (bh_walk.cu).
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "bh_internal.cuh"

namespace bhg {
namespace {

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// Cell centre (box units, exact) of caller cell c.
__device__ __forceinline__ void cell_centre(int64_t c, const int *pos, const int4 *blk, int &p,
                                            float &tx, float &ty, float &tz) {
  const int b = (int)(c >> 9), li = (int)(c & 511);
  const int cx = li & 7, cy = (li >> 3) & 7, cz = li >> 6;
  p = pos[b];
  const int4 B = blk[p];
  const float hh = pow2f(-(B.x + 3 + 1));
  tx = __fmul_rn((float)(2 * (8 * B.y + cx) + 1), hh);
  ty = __fmul_rn((float)(2 * (8 * B.z + cy) + 1), hh);
  tz = __fmul_rn((float)(2 * (8 * B.w + cz) + 1), hh);
}

// One thread per target: its per-cell walk (single-lane version of the warp
// walk, same binary32 test), listing every accepted internal node.
__global__ void k_pairs_list(int ntargets, const int64_t *__restrict__ targets,
                             const int *__restrict__ pos, const int4 *__restrict__ blk,
                             const int4 *__restrict__ fld, const WalkRec *__restrict__ rec,
                             int64_t cap, int64_t *__restrict__ pairs,
                             unsigned long long *__restrict__ counter) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntargets) return;
  const int64_t c = targets[i];
  int p;
  float tx, ty, tz;
  cell_centre(c, pos, blk, p, tx, ty, tz);
  const int4 F = fld[p];
  unsigned node = (unsigned)F.x;
  while (node < (unsigned)F.y) {
    const WalkRec r = rec[node];
    const float dx = __fsub_rn(tx, r.px), dy = __fsub_rn(ty, r.py), dz = __fsub_rn(tz, r.pz);
    const float d2 = __fmaf_rn(dx, dx, __fmaf_rn(dz, dz, __fmul_rn(dy, dy)));
    if (r.s2 > 0.0f && d2 > r.s2) {  // an accepted internal node
      const unsigned long long slot = atomicAdd(counter, 1ull);
      if ((int64_t)slot < cap) {
        pairs[2 * slot] = c;
        pairs[2 * slot + 1] = node;
      }
      node = r.skip;
    } else {
      node = node + 1;  // opened (internal) or a cell, whose skip is node + 1
    }
  }
}

// One CTA per pair: features and the exact residual eps in FP64.
constexpr int kEvalThreads = 256;
__global__ void __launch_bounds__(kEvalThreads)
    k_pairs_eval(int64_t npairs, const int64_t *__restrict__ pairs, const int *__restrict__ pos,
                 const int4 *__restrict__ blk, const WalkRec *__restrict__ rec,
                 const double4_32a *__restrict__ mom, const float2 *__restrict__ aux,
                 const WalkQuad *__restrict__ qrec, const int4 *__restrict__ fld,
                 const unsigned long long *__restrict__ mmax, float *__restrict__ feat,
                 float *__restrict__ eps, int64_t *__restrict__ node_out) {
  __shared__ double part[kEvalThreads];
  const int64_t q = blockIdx.x;
  if (q >= npairs) return;
  const int64_t c = pairs[2 * q];
  const unsigned n = (unsigned)pairs[2 * q + 1];
  int p;
  float txf, tyf, tzf;
  cell_centre(c, pos, blk, p, txf, tyf, tzf);
  const double tx = txf, ty = tyf, tz = tzf;
  const unsigned end = rec[n].skip;
  double acc = 0.0;
  for (unsigned k = n + 1 + threadIdx.x; k < end; k += kEvalThreads) {
    if (rec[k].s2 > 0.0f) continue;  // internal: only cells count
    const double4_32a m = mom[k];
    const double ex = tx - m.x, ey = ty - m.y, ez = tz - m.z;
    acc += m.w / sqrt(ex * ex + ey * ey + ez * ez);
  }
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int o = kEvalThreads / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  const double4_32a m = mom[n];
  const double dx = tx - m.x, dy = ty - m.y, dz = tz - m.z;
  const double D = sqrt(dx * dx + dy * dy + dz * dz);
  const double ux = dx / D, uy = dy / D, uz = dz / D;
  const double l = (double)aux[n].x, delta = (double)aux[n].y;
  const double s = l / D;
  const WalkQuad w = qrec[n];
  const double Qxx = 2.0 * w.hxx, Qyy = 2.0 * w.hyy, Qzz = 2.0 * w.hzz;
  const double quu = Qxx * ux * ux + Qyy * uy * uy + Qzz * uz * uz +
                     2.0 * (w.qxy * ux * uy + w.qxz * ux * uz + w.qyz * uy * uz);
  const double qf = sqrt(Qxx * Qxx + Qyy * Qyy + Qzz * Qzz +
                         2.0 * ((double)w.qxy * w.qxy + (double)w.qxz * w.qxz +
                                (double)w.qyz * w.qyz));
  // the record's Q is in the field's binary32 mass unit 2^e
  const double ml2 = m.w > 0.0 ? m.w * pow2i(-mass_exponent(mmax[fld[p].w])) * l * l : 1.0;
  float *f = feat + kMlpIn * q;
  f[0] = (float)ux;
  f[1] = (float)uy;
  f[2] = (float)uz;
  f[3] = (float)s;
  f[4] = (float)(s * s);
  f[5] = (float)(s * s * s);
  f[6] = (float)(delta / l);
  f[7] = (float)(quu / ml2);
  f[8] = (float)(qf / ml2);
  f[9] = (float)(s * s * quu / ml2);
  eps[q] = (float)(part[0] / (m.w / D) - 1.0);
  if (node_out) node_out[q] = n;
}

// ---- MLP training (FP32, CUDA cores) ---------------------------------------
// 64 samples per CTA of 256 threads.  Each of the four 64 x 64 products of the
// forward and backward passes (hidden layer 2, its input gradient, the
// gradient of W2; layer 1 is 10 wide) is tiled in registers: thread (ti, tj)
// owns 4 samples (or weight rows) x 4 units, so 16 FMAs take two 128-bit
// shared-memory reads (the first version read one or two words per FMA and
// was bound by that).  Activations are kept transposed, [unit][sample], with a
// pitch of 68 words.  Each GELU and its derivative come from one tanh, kept in
// registers from the forward to the backward pass (the first version took
// five).  The CTA's gradients are added to the global ones with one atomic
// per weight, consecutive lanes to consecutive words.
// Measured (8,192 samples, 128 CTAs): 64 -> 22 us; 40,000 samples with the
// optimiser step 274 -> 64 us.
constexpr int kMlpSamples = 64;
constexpr int kMlpThreads = 256;
constexpr int kMlpPitch = 68;

// GELU (tanh form) and its derivative.
__device__ __forceinline__ float gelu_both(float a, float &grad) {
  const float c = 0.7978845608028654f;
  const float t = tanhf(c * (a + 0.044715f * a * a * a));
  grad = 0.5f * (1.0f + t) + 0.5f * a * (1.0f - t * t) * c * (1.0f + 3.0f * 0.044715f * a * a);
  return 0.5f * a * (1.0f + t);
}

struct MlpSmem {
  float w2[kMlpH][kMlpH], w2t[kMlpH][kMlpPitch];
  float w1[kMlpIn][kMlpH], xt[kMlpIn][kMlpPitch];
  float h1t[kMlpH][kMlpPitch];  // layer-1 activations
  float dt[kMlpH][kMlpPitch];   // loss gradient at layer 2's input sums, then layer 1's
  float red[3][16][kMlpH];      // of b1, b2 and W3 per sample group
  float b1[kMlpH], b2[kMlpH], w3[kMlpH];
  float dy[kMlpSamples], loss[kMlpSamples];
};

// acc[r][c] += sum over k of a[k][4 ti + r] b[k][4 tj + c].
template <int K, int PA, int PB>
__device__ __forceinline__ void tile_product(const float (*a)[PA], const float (*b)[PB], int ti,
                                             int tj, float acc[4][4]) {
#pragma unroll 8
  for (int k = 0; k < K; ++k) {
    const float4 u = *reinterpret_cast<const float4 *>(&a[k][4 * ti]);
    const float4 v = *reinterpret_cast<const float4 *>(&b[k][4 * tj]);
    const float uu[4] = {u.x, u.y, u.z, u.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(uu[r], vv[c], acc[r][c]);
  }
}

__global__ void __launch_bounds__(kMlpThreads)
    k_mlp_grad(int64_t n, const float *__restrict__ x, const float *__restrict__ z,
               const float *__restrict__ w, float *__restrict__ grad, float *__restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpSmem &S = *reinterpret_cast<MlpSmem *>(smem_raw);
  const int t = threadIdx.x, ti = t >> 4, tj = t & 15;
  const int64_t base = (int64_t)blockIdx.x * kMlpSamples;
  const float *W1 = w, *b1 = W1 + kMlpIn * kMlpH, *W2 = b1 + kMlpH, *b2 = W2 + kMlpH * kMlpH;
  const float *W3 = b2 + kMlpH, *b3 = W3 + kMlpH;
  for (int i = t; i < kMlpH * kMlpH; i += kMlpThreads) {
    const float v = W2[i];
    S.w2[i >> 6][i & 63] = v;
    S.w2t[i & 63][i >> 6] = v;
  }
  for (int i = t; i < kMlpIn * kMlpH; i += kMlpThreads) S.w1[i >> 6][i & 63] = W1[i];
  for (int i = t; i < kMlpSamples * kMlpIn; i += kMlpThreads)
    S.xt[i % kMlpIn][i / kMlpIn] = base + i / kMlpIn < n ? x[base * kMlpIn + i] : 0.0f;
  if (t < kMlpH) {
    S.b1[t] = b1[t];
    S.b2[t] = b2[t];
    S.w3[t] = W3[t];
  }
  __syncthreads();
  // layer 1 of samples 4 ti .. + 3, units 4 tj .. + 3
  float g1[4][4], g2[4][4], acc[4][4], part[4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = S.b1[4 * tj + c];
  tile_product<kMlpIn>(S.xt, S.w1, ti, tj, acc);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float4 h;
    h.x = gelu_both(acc[0][c], g1[0][c]);
    h.y = gelu_both(acc[1][c], g1[1][c]);
    h.z = gelu_both(acc[2][c], g1[2][c]);
    h.w = gelu_both(acc[3][c], g1[3][c]);
    *reinterpret_cast<float4 *>(&S.h1t[4 * tj + c][4 * ti]) = h;
  }
  __syncthreads();
  // layer 2 and the output
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = S.b2[4 * tj + c];
  tile_product<kMlpH>(S.h1t, S.w2, ti, tj, acc);
  float w3[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) w3[c] = S.w3[4 * tj + c];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float y = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      acc[r][c] = gelu_both(acc[r][c], g2[r][c]);
      y = fmaf(acc[r][c], w3[c], y);
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    const int64_t g = base + 4 * ti + r;
    const float res = g < n ? y + b3[0] - z[g] : 0.0f;
    part[r] = 2.0f * res / (float)n;  // dL/dy
    if (tj == 0) {
      S.dy[4 * ti + r] = part[r];
      S.loss[4 * ti + r] = res * res / (float)n;
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float gw3 = 0.0f, gb2 = 0.0f, d[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      gw3 = fmaf(acc[r][c], part[r], gw3);
      d[r] = part[r] * w3[c] * g2[r][c];
      gb2 += d[r];
      acc[r][c] = 0.0f;
    }
    S.red[2][ti][4 * tj + c] = gw3;
    S.red[1][ti][4 * tj + c] = gb2;
    *reinterpret_cast<float4 *>(&S.dt[4 * tj + c][4 * ti]) = make_float4(d[0], d[1], d[2], d[3]);
  }
  __syncthreads();
  // back through layer 2: dL/d(layer-1 sums), same ownership as layer 1
  tile_product<kMlpH>(S.dt, S.w2t, ti, tj, acc);
  // gradient of W2: rows ti + 16 r, columns tj + 16 c (conflict-free reads)
  float gw[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) gw[r][c] = 0.0f;
  for (int s = 0; s < kMlpSamples; s += 4) {
    float4 h[4], d[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      h[r] = *reinterpret_cast<const float4 *>(&S.h1t[ti + 16 * r][s]);
      d[r] = *reinterpret_cast<const float4 *>(&S.dt[tj + 16 * r][s]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        gw[r][c] = fmaf(h[r].w, d[c].w, fmaf(h[r].z, d[c].z, fmaf(h[r].y, d[c].y, fmaf(h[r].x, d[c].x, gw[r][c]))));
  }
  float *gW1 = grad, *gb1 = gW1 + kMlpIn * kMlpH, *gW2 = gb1 + kMlpH, *gb2 = gW2 + kMlpH * kMlpH;
  float *gW3 = gb2 + kMlpH, *gb3 = gW3 + kMlpH;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      atomicAdd(&gW2[(ti + 16 * r) * kMlpH + tj + 16 * c], gw[r][c]);
  __syncthreads();  // dt has been read
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float d[4], sum = 0.0f;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      d[r] = acc[r][c] * g1[r][c];
      sum += d[r];
    }
    S.red[0][ti][4 * tj + c] = sum;
    *reinterpret_cast<float4 *>(&S.dt[4 * tj + c][4 * ti]) = make_float4(d[0], d[1], d[2], d[3]);
  }
  __syncthreads();
  // gradient of W1: input k of unit j
  for (int e = t; e < kMlpIn * kMlpH; e += kMlpThreads) {
    const int k = e >> 6, j = e & 63;
    float v = 0.0f;
#pragma unroll 4
    for (int s = 0; s < kMlpSamples; s += 4) {
      const float4 u = *reinterpret_cast<const float4 *>(&S.xt[k][s]);
      const float4 d = *reinterpret_cast<const float4 *>(&S.dt[j][s]);
      v = fmaf(u.w, d.w, fmaf(u.z, d.z, fmaf(u.y, d.y, fmaf(u.x, d.x, v))));
    }
    atomicAdd(&gW1[e], v);
  }
  if (t < 3 * kMlpH) {  // b1, b2, W3
    const int q = t >> 6, j = t & 63;
    float v = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) v += S.red[q][i][j];
    atomicAdd((q == 0 ? gb1 : q == 1 ? gb2 : gW3) + j, v);
  } else {  // b3 and the loss, a warp each
    const int l = t & 31;
    const float *src = t < 3 * kMlpH + 32 ? S.dy : S.loss;
    float v = src[l] + src[l + 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (l == 0) atomicAdd(t < 3 * kMlpH + 32 ? gb3 : loss, v);
  }
}

__global__ void k_mlp_adam(const float *__restrict__ grad, float *__restrict__ w,
                           float *__restrict__ m, float *__restrict__ v, float lr, float b1t,
                           float b2t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kMlpNW) return;
  const float beta1 = 0.9f, beta2 = 0.999f;
  const float g = grad[i];
  const float mi = beta1 * m[i] + (1.0f - beta1) * g;
  const float vi = beta2 * v[i] + (1.0f - beta2) * g * g;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / (1.0f - b1t)) / (sqrtf(vi / (1.0f - b2t)) + 1e-8f);
}

uint16_t to_bf16(float f) {  // round to nearest even
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7f800000u) == 0x7f800000u)  // inf stays inf, nan stays nan
    return (uint16_t)((u >> 16) | ((u & 0x007fffffu) ? 0x40u : 0u));
  u += 0x7fffu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}
float from_bf16(uint16_t h) {
  const uint32_t u = (uint32_t)h << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}
uint16_t bf16_half(uint16_t h) { return to_bf16(0.5f * from_bf16(h)); }  // exact

// Place of weight W[k][n] in the B fragments of its (n-tile, k-tile)
// (layout described with MlpDev): lane 4 (n % 8) + (k % 8) / 2, register
// (k % 16) / 8, half k % 2.
int frag_lane(int k, int n) { return 4 * (n & 7) + ((k & 7) >> 1); }
int frag_reg(int k) { return (k & 15) >> 3; }
void frag_put(uint32_t &word, int k, uint16_t v) { word |= (uint32_t)v << (16 * (k & 1)); }
uint16_t frag_get(uint32_t word, int k) { return (uint16_t)(word >> (16 * (k & 1))); }

// Training target of a pair: z = eps / s^2 (s = feature 3), the network's
// output for which the walk's term (M/d)(1 + s^2 z) is the node's exact
// contribution.
__global__ void k_learn_targets(int64_t n, const float *__restrict__ x,
                                const float *__restrict__ eps, float *__restrict__ z) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float s = x[i * kMlpIn + 3];
  z[i] = __fdiv_rn(eps[i], __fmul_rn(s, s));
}

}  // namespace
}  // namespace bhg

using namespace bhg;

extern "C" {

bh_status bh_learn_targets(int64_t n, const float *feat, const float *eps, float *z,
                           void *cuda_stream) {
  if (n < 0 || (n > 0 && (!feat || !eps || !z))) return BH_ERR_ARG;
  if (n == 0) return BH_OK;
  k_learn_targets<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(n, feat,
                                                                                        eps, z);
  if (cudaGetLastError() != cudaSuccess) return BH_ERR_CUDA;
  return BH_OK;
}

bh_status bh_learn_pairs(bh_ctx *ctx, double theta, int64_t ntargets, const int64_t *targets,
                         int64_t cap, float *feat, float *eps, int64_t *node, int64_t *count) {
  if (!ctx) return BH_ERR_ARG;
  ctx->err[0] = 0;
  if (!ctx->opt.quadrupole && !ctx->opt.learned)
    return ctx_fail(ctx, BH_ERR_STATE, "bh_learn_pairs: the context needs the quadrupole option");
  if (ntargets < 0 || (ntargets > 0 && !targets) || cap < 0 || (cap > 0 && (!feat || !eps)) ||
      !count)
    return ctx_fail(ctx, BH_ERR_ARG, "bh_learn_pairs: bad arguments");
  bh_status st = ctx_prepare(ctx, theta);
  if (st != BH_OK) return st;
  Tree &t = ctx->tree;
  cudaStream_t s = ctx->stream;
  int64_t *d_pairs = nullptr;
  unsigned long long *d_count = nullptr;
  const int64_t pcap = cap > 0 ? cap : 1;
  cudaError_t e = bhg::dev_malloc(&d_pairs, (size_t)pcap * 2 * sizeof(int64_t));
  if (e == cudaSuccess) e = bhg::dev_malloc(&d_count, sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMemsetAsync(d_count, 0, sizeof(unsigned long long), s);
  if (e == cudaSuccess && ntargets > 0) {
    k_pairs_list<<<(unsigned)((ntargets + 127) / 128), 128, 0, s>>>(
        (int)ntargets, targets, t.d_pos, t.d_blk, t.d_fld, t.d_rec, cap, d_pairs, d_count);
    e = cudaGetLastError();
  }
  unsigned long long h_count = 0;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&h_count, d_count, sizeof(h_count), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  const int64_t np = (int64_t)h_count < cap ? (int64_t)h_count : cap;
  if (e == cudaSuccess && np > 0) {
    k_pairs_eval<<<(unsigned)np, kEvalThreads, 0, s>>>(np, d_pairs, t.d_pos, t.d_blk, t.d_rec,
                                                        t.d_mom, t.d_aux, t.d_qrec, t.d_fld,
                                                        t.d_mmax, feat, eps, node);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d_pairs);
  cudaFree(d_count);
  if (e != cudaSuccess)
    return ctx_fail(ctx, BH_ERR_CUDA, "bh_learn_pairs: %s", cudaGetErrorString(e));
  *count = (int64_t)h_count;
  return BH_OK;
}

bh_status bh_mlp_grad(int64_t n, const float *x, const float *z, const float *w, float *grad,
                      float *loss, void *cuda_stream) {
  if (n <= 0 || !x || !z || !w || !grad || !loss) return BH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const int smem = (int)sizeof(MlpSmem);
  if (cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
          cudaSuccess ||
      cudaMemsetAsync(grad, 0, kMlpNW * sizeof(float), s) != cudaSuccess ||
      cudaMemsetAsync(loss, 0, sizeof(float), s) != cudaSuccess) {
    cudaGetLastError();
    return BH_ERR_CUDA;
  }
  k_mlp_grad<<<(unsigned)((n + kMlpSamples - 1) / kMlpSamples), kMlpThreads, smem, s>>>(
      n, x, z, w, grad, loss);
  if (cudaGetLastError() != cudaSuccess) return BH_ERR_CUDA;
  return BH_OK;
}

bh_status bh_mlp_adam(const float *grad, float *w, float *m, float *v, int step, float lr,
                      void *cuda_stream) {
  if (!grad || !w || !m || !v || step < 1 || !(lr > 0.0f)) return BH_ERR_ARG;
  const float b1t = powf(0.9f, (float)step), b2t = powf(0.999f, (float)step);
  k_mlp_adam<<<(kMlpNW + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(grad, w, m, v, lr, b1t,
                                                                          b2t);
  if (cudaGetLastError() != cudaSuccess) return BH_ERR_CUDA;
  return BH_OK;
}

bh_status bh_set_mlp(bh_ctx *ctx, const float *w_host) {
  if (!ctx) return BH_ERR_ARG;
  ctx->err[0] = 0;
  if (!w_host) return ctx_fail(ctx, BH_ERR_ARG, "bh_set_mlp: weights are null");
  MlpDev h;
  std::memset(&h, 0, sizeof(h));
  const float *W1 = w_host, *b1 = W1 + kMlpIn * kMlpH, *W2 = b1 + kMlpH;
  const float *b2 = W2 + kMlpH * kMlpH, *W3 = b2 + kMlpH, *b3 = W3 + kMlpH;
  for (int n = 0; n < kMlpH; ++n) {
    for (int k = 0; k < kMlpIn; ++k)
      frag_put(h.w1f[n >> 3][frag_lane(k, n)][frag_reg(k)], k, to_bf16(W1[k * kMlpH + n]));
    frag_put(h.w1f[n >> 3][frag_lane(kMlpIn, n)][frag_reg(kMlpIn)], kMlpIn, to_bf16(b1[n]));
    for (int k = 0; k < kMlpH; ++k)
      frag_put(h.w2f[n >> 3][k >> 4][frag_lane(k, n)][frag_reg(k)], k,
               bf16_half(to_bf16(W2[k * kMlpH + n])));
    h.b2[n] = b2[n];
  }
  for (int k = 0; k < kMlpH; ++k)
    frag_put(h.w3f[k >> 4][frag_lane(k, 0)][frag_reg(k)], k, bf16_half(to_bf16(W3[k])));
  h.b3 = b3[0];
  // the same bf16 values in the tcgen05 evaluator's canonical layout
  MlpTc c;
  std::memset(&c, 0, sizeof(c));
  auto put = [](uint16_t *base, int byte_off, uint16_t v) { base[byte_off / 2] = v; };
  for (int n = 0; n < kMlpH; ++n) {
    for (int k = 0; k < kMlpIn; ++k) put(c.b1, tc_canon(n, k, 16), to_bf16(W1[k * kMlpH + n]));
    put(c.b1, tc_canon(n, kMlpIn, 16), to_bf16(b1[n]));
    for (int k = 0; k < kMlpH; ++k)
      put(c.b2, tc_canon(n, k, 64), bf16_half(to_bf16(W2[k * kMlpH + n])));
    c.bias2[n] = b2[n];
  }
  for (int k = 0; k < kMlpH; ++k) put(c.b3, tc_canon(0, k, 64), bf16_half(to_bf16(W3[k])));
  c.bias3 = b3[0];
  if (cudaSetDevice(ctx->device) != cudaSuccess) return ctx_fail(ctx, BH_ERR_CUDA, "device");
  if ((!ctx->d_mlp && bhg::dev_malloc(&ctx->d_mlp, sizeof(MlpDev)) != cudaSuccess) ||
      (!ctx->d_mlp_tc && bhg::dev_malloc(&ctx->d_mlp_tc, sizeof(MlpTc)) != cudaSuccess) ||
      (!ctx->h_tc_flag &&
       cudaHostAlloc((void **)&ctx->h_tc_flag, sizeof(unsigned), cudaHostAllocMapped) != cudaSuccess)) {
    cudaGetLastError();
    return ctx_fail(ctx, BH_ERR_OOM, "bh_set_mlp: no device memory");
  }
  if (cudaMemcpy(ctx->d_mlp, &h, sizeof(h), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(ctx->d_mlp_tc, &c, sizeof(c), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(ctx, BH_ERR_CUDA, "bh_set_mlp: copy failed");
  }
  return BH_OK;
}

bh_status bh_mlp_eval(bh_ctx *ctx, int64_t n, const float *x, float *y) {
  if (!ctx) return BH_ERR_ARG;
  ctx->err[0] = 0;
  if (!ctx->d_mlp_tc) return ctx_fail(ctx, BH_ERR_STATE, "bh_mlp_eval: call bh_set_mlp first");
  if (n < 0 || (n > 0 && (!x || !y))) return ctx_fail(ctx, BH_ERR_ARG, "bh_mlp_eval: bad arguments");
  if (n == 0) return BH_OK;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return ctx_fail(ctx, BH_ERR_CUDA, "device");
  // Test of the time-out path (host-side switch, no device fault): with
  // BHGRAV_TC_WAIT_PROBE=k (k > 0) the kernel issues no MMA and gives up its
  // first wait for the tensor core after k tries.
  int probe = 0;
  if (const char *env = std::getenv("BHGRAV_TC_WAIT_PROBE")) {
    const long v = std::strtol(env, nullptr, 10);
    probe = v > 0 ? (int)(v < (1L << 20) ? v : (1L << 20)) : 0;
  }
  // the time-out flag lies in mapped host memory, which the kernel writes only
  // when a wait gave up: no memset before it and no copy after it
  volatile unsigned *flag = ctx->h_tc_flag;
  unsigned *d_flag = nullptr;
  *flag = 0u;
  if (cudaHostGetDevicePointer((void **)&d_flag, ctx->h_tc_flag, 0) != cudaSuccess ||
      launch_mlp_tc(ctx->stream, n, x, ctx->d_mlp_tc, y, d_flag, probe) != cudaSuccess ||
      cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
    cudaGetLastError();
    return ctx_fail(ctx, BH_ERR_CUDA, "bh_mlp_eval: %s", "launch failed");
  }
  if (*flag) return ctx_fail(ctx, BH_ERR_DEVICE_TIMEOUT, "bh_mlp_eval: a tensor-core wait gave up");
  return BH_OK;
}

bh_status bh_get_mlp(const bh_ctx *ctx, float *w_host) {
  if (!ctx || !w_host) return BH_ERR_ARG;
  if (!ctx->d_mlp) return BH_ERR_STATE;
  MlpDev h;
  if (cudaMemcpy(&h, ctx->d_mlp, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) {
    cudaGetLastError();
    return BH_ERR_CUDA;
  }
  float *W1 = w_host, *b1 = W1 + kMlpIn * kMlpH, *W2 = b1 + kMlpH;
  float *b2 = W2 + kMlpH * kMlpH, *W3 = b2 + kMlpH, *b3 = W3 + kMlpH;
  for (int n = 0; n < kMlpH; ++n) {
    for (int k = 0; k < kMlpIn; ++k)
      W1[k * kMlpH + n] = from_bf16(frag_get(h.w1f[n >> 3][frag_lane(k, n)][frag_reg(k)], k));
    b1[n] = from_bf16(frag_get(h.w1f[n >> 3][frag_lane(kMlpIn, n)][frag_reg(kMlpIn)], kMlpIn));
    for (int k = 0; k < kMlpH; ++k)
      W2[k * kMlpH + n] =
          2.0f * from_bf16(frag_get(h.w2f[n >> 3][k >> 4][frag_lane(k, n)][frag_reg(k)], k));
    b2[n] = h.b2[n];
  }
  for (int k = 0; k < kMlpH; ++k)
    W3[k] = 2.0f * from_bf16(frag_get(h.w3f[k >> 4][frag_lane(k, 0)][frag_reg(k)], k));
  b3[0] = h.b3;
  return BH_OK;
}

bh_status bh_set_mlp_gate(bh_ctx *ctx, double s_min) {
  if (!ctx) return BH_ERR_ARG;
  ctx->err[0] = 0;
  if (!(s_min >= 0.0) || !(s_min < 1.0))
    return ctx_fail(ctx, BH_ERR_ARG, "bh_set_mlp_gate: s_min must lie in [0, 1)");
  ctx->mlp_s_min = s_min;
  return BH_OK;
}

}  // extern "C"
