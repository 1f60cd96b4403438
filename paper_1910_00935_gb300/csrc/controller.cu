// controller.cu -- the closed-loop controller of the actuated bodies (the neural-network
// controllers of Section 4.1): at every step the sensors of the current state feed a
// small MLP whose outputs are the actuation of the groups, and the reverse pass carries
// the actuation adjoint back through the MLP to its weights and to the sensed state.
//
//   inputs u (n_in = K + 2 d G): sin(2 pi k t / P + phi) for k = 1..K, then per group g
//     the offset of its centre of mass from the body's (d values) and its mean velocity
//     (d values); an empty group reads zeros
//   h = tanh(W1 u + b1) (H units), a_g = scale tanh(W2 h + b2)_g
//   theta per scene = [W1 (H x n_in, row-major) | b1 (H) | W2 (G x H, row-major) | b2 (G)]
//
// Weights arrive in FP32; a tile's sensor sums are FP32, the sums over tiles and the dot products
// compensated FP32 pairs (value and correction, ~48 bits: FP64 runs at 1/64 of the FP32 rate on
// this part, and a few thousand FP64 operations a step were most of these kernels' time; a sum that
// leaves FP32's range is formed again in FP64; on 12 batches of 1-4 robots, 7-64 hidden units and 128-256
// steps the deterministic states and gradients are bitwise those of FP64 sums), the inputs and what is kept for the reverse FP64, the activations tanh in FP32.  Every sum runs in a
// fixed order (a warp's lanes by butterfly, a tile's warps and a scene's tiles in order), so the
// controller adds nothing order-dependent to a deterministic run.
//
// One CTA a scene runs the MLP or its reverse: what bounds it is the chain of barriers and round trips to
// the L2, so every independent read is issued at the start and the sums over tiles are trees.
// The G2P pass of a controlled step leaves its tiles' sensor sums (sense_tile), and the G2P
// adjoint adds the sensors' adjoints as it reads the state's (AdjArgs::sense_add).  Measured on
// 4 x 27,648 particles, 32 hidden units (us a launch under ncu): sensing 8.3 -> in the G2P pass, MLP
// 19.3 -> 10.6, reverse 25.5 -> 14.5, adding the sensors' adjoints 7.3 -> in the adjoint pass.
#include <cfloat>

#include "mpm_internal.h"
#include "mpm_kernels.cuh"

namespace mpm {

namespace {

constexpr int kCtrlThreads = 1024;    // one CTA per scene for the MLP passes
constexpr int kSenseVals = 7;       // x (d), v (d), count: at most 7
constexpr int kSenseSlots = kMaxGroups + 1;  // slot 0: particles in no group

// a value and its correction, hi + lo to ~48 bits (TwoSum, TwoProd)
struct Pair {
  float h, l;
};
__device__ __forceinline__ Pair pair_norm(float s, float e) {
  const float h = ef_add(s, e);
  return {h, ef_add(e, -ef_add(h, -s))};
}
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  return pair_norm(s, e + (a.l + b.l));
}
__device__ __forceinline__ Pair pair_of(double d) {
  const float h = (float)d;
  return {h, (float)(d - (double)h)};
}
__device__ __forceinline__ double pair_value(Pair a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ Pair pair_mul(float w, Pair u) {  // w * (h + l)
  float p, e;
  two_prod(w, u.h, p, e);
  return pair_norm(p, fmaf(w, u.l, e));
}
// whether a sum stayed within FP32's range (once beyond it, a pair never comes back)
__device__ __forceinline__ bool in_range(Pair a) { return fabsf(a.h) <= FLT_MAX; }
// sum over the lanes of aligned groups of LANES, the same order on every run (all lanes call it)
template <int LANES>
__device__ __forceinline__ Pair lanes_sum(Pair v) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1)
    v = pair_add(v, {__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
  return v;
}

// sum over i < n of w[i * stride] * u[i] in FP64 by a whole warp: the way out of a pair that left its
// range (out of line: what never happens in earnest holds no registers)
__device__ __noinline__ double dot_fp64(const float* w, int stride, const double* u, int n) {
  double z = 0.0;
  for (int i = threadIdx.x & 31; i < n; i += 32) z += (double)w[i * stride] * u[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  return z;
}
// sum over t in [t0, t1) of a[t * nv] in FP64 by one thread
__device__ __noinline__ double rows_fp64(const float* a, int t0, int t1, int nv) {
  double z = 0.0;
  for (int t = t0; t < t1; ++t) z += (double)a[(int64_t)t * nv];
  return z;
}

// out[j] = sum over t in [t0, t1) of a[t * nv + j] for j < nv, by the whole CTA: thread (r, j)
// sums rows t0 + r, t0 + r + R, ... (R = blockDim / nv, all reads issued before the first sum),
// then four lanes a value sum its R partials in order and combine.  The order depends only on
// (t0, t1), so the sums are reproducible.  scratch: kCtrlThreads pairs; out: shared, nv doubles.
// 4 nv <= blockDim.  Ends with a barrier.
__device__ void block_tile_sums(float* a, int t0, int t1, int nv, Pair* scratch, double* out) {
  const int R = blockDim.x / nv;
  const int r = threadIdx.x / nv, j = threadIdx.x - r * nv;
  Pair acc = {0.0f, 0.0f};
  if (r < R) {
    constexpr int U = 8;
    for (int t = t0 + r; t < t1; t += U * R) {
      float q[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool in = t + u * R < t1;
        float* e = a + (int64_t)(in ? t + u * R : t) * nv + j;
        q[u] = in ? *e : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) acc = pair_add(acc, {q[u], 0.0f});
    }
  }
  scratch[threadIdx.x] = acc;
  __syncthreads();
  const int v = threadIdx.x >> 2, q4 = threadIdx.x & 3;
  if ((int)(threadIdx.x & ~31u) < 4 * nv) {  // whole warps (the combine shuffles)
    Pair p = {0.0f, 0.0f};
    const int per = (R + 3) >> 2;
    if (v < nv)
      for (int k = q4 * per; k < R && k < (q4 + 1) * per; ++k) p = pair_add(p, scratch[k * nv + v]);
    p = lanes_sum<4>(p);
    if (v < nv && q4 == 0) out[v] = in_range(p) ? pair_value(p) : rows_fp64(a + v, t0, t1, nv);
  }
  __syncthreads();
}

// Per-tile sensor sums of the initial state (every later state's come from its G2P pass)
template <int D>
__global__ void __launch_bounds__(kTile) ctrl_sense_kernel(int G, int64_t N, const int4* tiles, const float* st,
                                                           const int* group, float* part) {
  __shared__ float scratch[kWarps * kSenseSlots * (2 * D + 1)];
  const int4 tile = tiles[blockIdx.x];
  const bool active = (int)threadIdx.x < tile.z;
  const int64_t p = (int64_t)tile.y + (active ? threadIdx.x : 0);
  float x[D], v[D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    x[a] = st[(int64_t)a * N + p];  // fixed-point position rows
    v[a] = st[(int64_t)(D + a) * N + p];
  }
  sense_tile<D>(G, true, group[p], active, x, v, scratch, part + (int64_t)blockIdx.x * (G + 1) * (2 * D + 1));
}

// One CTA per scene: reduce the scene's tile sums in order, form the inputs, run the MLP
// and store u, h, y = tanh(W2 h + b2) (kept for the reverse pass), the actuation
// a = scale y, and the group sizes.
__global__ void __launch_bounds__(kCtrlThreads) ctrl_forward_kernel(CtrlStep cs, const int* tile_off, float* part,
                                    const float* theta, double* u_out, double* h_out,
                                    double* y_out, float* act_out, double* cnt_out) {
  __shared__ double sums[kSenseSlots * kSenseVals];
  __shared__ double inv_n[kSenseSlots], mean[3];  // 1 / group sizes (0: empty; slot 0: the body), the body's mean
  __shared__ Pair u[kCtrlMaxInputs];
  __shared__ float hs[kCtrlMaxHidden];
  __shared__ Pair scratch[kCtrlThreads];
  const int s = blockIdx.x;
  const int dim = cs.dim, G = cs.G, K = cs.K, H = cs.H;
  const int nv = 2 * dim + 1, ns = G + 1;
  const int n_in = K + 2 * dim * G;
  const int n_par = H * n_in + H + G * H + G;
  const float* th = theta + (int64_t)s * n_par;
  const float* W1 = th;
  const float* b1 = th + H * n_in;
  const float* W2 = b1 + H;
  const float* b2 = W2 + G * H;
  // one warp per hidden unit (then per output): its lanes take the dot product's terms and
  // a butterfly sums them; the first round's weights are read before the sums they meet
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  float w1[kCtrlMaxInputs / 32 + 1], w2[2];
#pragma unroll
  for (int q = 0; q <= kCtrlMaxInputs / 32; ++q) w1[q] = warp < H && lane + 32 * q < n_in ? W1[warp * n_in + lane + 32 * q] : 0.0f;
#pragma unroll
  for (int q = 0; q < 2; ++q) w2[q] = warp < G && lane + 32 * q < H ? W2[warp * H + lane + 32 * q] : 0.0f;
  const float bias1 = warp < H ? b1[warp] : 0.0f, bias2 = warp < G ? b2[warp] : 0.0f;
  const int t0 = tile_off[s], t1 = tile_off[s + 1];
  pass_wait();
  pass_ready();
  block_tile_sums(part, t0, t1, ns * nv, scratch, sums);
  if ((int)threadIdx.x < ns) {
    const int g = threadIdx.x;
    double n = sums[g * nv + 2 * dim];
    cnt_out[s * ns + g] = n;
    if (g == 0)
      for (int q = 1; q < ns; ++q) n += sums[q * nv + 2 * dim];
    inv_n[g] = n > 0.0 ? 1.0 / n : 0.0;
  } else if ((int)threadIdx.x >= 32 && (int)threadIdx.x < 32 + dim) {
    double tot = 0.0;
    for (int q = 0; q < ns; ++q) tot += sums[q * nv + threadIdx.x - 32];
    mean[threadIdx.x - 32] = tot;
  }
  __syncthreads();
  // inputs: the time basis, then per group (centre offset, mean velocity)
  for (int i = threadIdx.x; i < n_in; i += blockDim.x) {
    double val;
    if (i < K) {
      val = cs.basis[i];
    } else {
      const int r = i - K, g = r / (2 * dim), c = r % (2 * dim);
      val = sums[(g + 1) * nv + c] * inv_n[g + 1];
      if (c < dim && inv_n[g + 1] > 0.0) val -= mean[c] * inv_n[0];
    }
    u[i] = pair_of(val);
    u_out[(int64_t)s * n_in + i] = val;
  }
  __syncthreads();
  for (int j = warp; j < H; j += n_warps) {
    Pair z = {0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q <= kCtrlMaxInputs / 32; ++q) {
      const int i = lane + 32 * q;
      if (i < n_in) z = pair_add(z, pair_mul(j == warp ? w1[q] : W1[j * n_in + i], u[i]));
    }
    z = pair_add(lanes_sum<32>(z), {j == warp ? bias1 : b1[j], 0.0f});
    float zj = z.h + z.l;
    if (!in_range(z)) zj = (float)(dot_fp64(W1 + j * n_in, 1, u_out + (int64_t)s * n_in, n_in) + (double)b1[j]);
    if (lane == 0) {
      // the activation in FP32: FP64 transcendentals run on the FP64 pipe
      const float hj = tanhf(zj);
      hs[j] = hj;
      h_out[(int64_t)s * H + j] = (double)hj;
    }
  }
  __syncthreads();
  if (warp < G) {  // G <= kMaxGroups warps
    Pair z = {0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (lane + 32 * q < H) z = pair_add(z, pair_mul(w2[q], {hs[lane + 32 * q], 0.0f}));
    z = pair_add(lanes_sum<32>(z), {bias2, 0.0f});
    float zg = z.h + z.l;
    if (!in_range(z)) zg = (float)(dot_fp64(W2 + warp * H, 1, h_out + (int64_t)s * H, H) + (double)bias2);
    if (lane == 0) {
      const double y = (double)tanhf(zg);
      y_out[(int64_t)s * G + warp] = y;
      act_out[(int64_t)s * G + warp] = (float)((double)cs.scale * y);
    }
  }
}
static_assert(kMaxGroups <= kCtrlThreads / 32, "one warp per output");
static_assert(kCtrlMaxHidden <= 64, "two hidden units a lane");
static_assert(4 * kSenseSlots * kSenseVals <= kCtrlThreads, "four lanes a sensor sum");

// One CTA per scene, reverse of the controller at one step: abar_g = the scene's per-tile
// actuation adjoints summed in tile order (and the tile slots cleared for the next step);
// dL/dtheta accumulates in FP64 (thbar); the sensor adjoint becomes per-slot additions to
// the state adjoint: add[scene][slot][0..d) to xbar, [d..2d) to vbar.
__global__ void __launch_bounds__(kCtrlThreads) ctrl_backward_kernel(CtrlStep cs, const int* tile_off, float* abar_tile,
                                     const float* theta, const double* u_in, const double* h_in,
                                     const double* y_in, const double* cnt, double* thbar,
                                     float* add) {
  __shared__ double z2b[kMaxGroups], z1b[kCtrlMaxHidden], n_s[kSenseSlots], inv_n[kSenseSlots + 1], us[kCtrlMaxInputs], hsd[kCtrlMaxHidden], ub[kCtrlMaxInputs];
  __shared__ double body[3];
  __shared__ Pair scratch[kCtrlThreads], z1p[kCtrlMaxHidden];
  __shared__ double abar[kMaxGroups];
  __shared__ float w2s[kMaxGroups * kCtrlMaxHidden];
  const int s = blockIdx.x;
  const int dim = cs.dim, G = cs.G, K = cs.K, H = cs.H;
  const int ns = G + 1;
  const int n_in = K + 2 * dim * G;
  const int n_par = H * n_in + H + G * H + G;
  const float* th = theta + (int64_t)s * n_par;
  const float* W1 = th;
  const float* W2 = th + H * n_in + H;
  double* W1b = thbar + (int64_t)s * n_par;
  double* b1b = W1b + H * n_in;
  double* W2b = b1b + H;
  double* b2b = W2b + G * H;
  const int tid = threadIdx.x, t0 = tile_off[s], t1 = tile_off[s + 1];
  // the forward's records and the weights, read while the tiles' adjoints are summed
  for (int i = tid; i < n_in; i += kCtrlThreads) us[i] = u_in[(int64_t)s * n_in + i];
  if (tid < H) hsd[tid] = h_in[(int64_t)s * H + tid];
  if (tid < G * H) w2s[tid] = W2[tid];
  if (tid < ns) n_s[tid] = cnt[s * ns + tid];
  const double y = tid < G ? y_in[(int64_t)s * G + tid] : 0.0;
  // one warp per input, four at a time over the lanes' hidden units
  const int warp = tid >> 5, lane = tid & 31;
  constexpr int RI = (kCtrlMaxInputs + kCtrlThreads / 32 - 1) / (kCtrlThreads / 32);
  float w1[RI][2];
#pragma unroll
  for (int q = 0; q < RI; ++q)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = warp + q * (kCtrlThreads / 32), j = lane + 32 * k;
      w1[q][k] = i < n_in && j < H ? W1[j * n_in + i] : 0.0f;
    }
  pass_wait();
  pass_ready();
  block_tile_sums(abar_tile, t0, t1, G, scratch, abar);
  if (tid < G) {
    const double zb = abar[tid] * (double)cs.scale * (1.0 - y * y);
    z2b[tid] = zb;
    b2b[tid] += zb;
  } else if (tid >= 32 && tid <= 32 + ns) {  // 1 / group sizes (0: empty), last: 1 / the body's
    double n = tid < 32 + ns ? n_s[tid - 32] : 0.0;
    if (tid == 32 + ns)
      for (int q = 0; q < ns; ++q) n += n_s[q];
    inv_n[tid - 32] = n > 0.0 ? 1.0 / n : 0.0;
  }
  __syncthreads();
  if (tid < H) {
    double hb = 0.0;
    for (int g = 0; g < G; ++g) hb += (double)w2s[g * H + tid] * z2b[g];
    const double zb = hb * (1.0 - hsd[tid] * hsd[tid]);
    z1b[tid] = zb;
    z1p[tid] = pair_of(zb);
    b1b[tid] += zb;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < RI; ++q) {
    const int i = warp + q * (kCtrlThreads / 32);
    if (i >= n_in) break;
    Pair acc = {0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (lane + 32 * k < H) acc = pair_add(acc, pair_mul(w1[q][k], z1p[lane + 32 * k]));
    acc = lanes_sum<32>(acc);
    const double ubi = in_range(acc) ? pair_value(acc) : dot_fp64(W1 + i, n_in, z1b, H);
    if (lane == 0) ub[i] = ubi;
  }
  // the weights' adjoints: nothing below reads them
  for (int e = tid; e < G * H; e += kCtrlThreads) W2b[e] += z2b[e / H] * hsd[e % H];
  for (int e = tid; e < H * n_in; e += kCtrlThreads) W1b[e] += z1b[e / n_in] * us[e % n_in];
  __syncthreads();
  // u_xg = mean_{p in g} x_p - mean_p x_p: every particle carries -sum_g ub_xg / N, and
  // its own group's ub_xg / N_g; u_vg = mean_{p in g} v_p: ub_vg / N_g
  if (tid < dim) {
    double tot = 0.0;
    for (int g = 0; g < G; ++g)
      if (inv_n[g + 1] > 0.0) tot += ub[K + g * 2 * dim + tid];
    body[tid] = tot * inv_n[ns];
  }
  __syncthreads();
  for (int j = tid; j < ns * 2 * dim; j += kCtrlThreads) {
    const int sl = j / (2 * dim), c = j % (2 * dim);
    double v = 0.0;
    if (c < dim) v = -body[c];
    if (sl > 0) v += ub[K + (sl - 1) * 2 * dim + c] * inv_n[sl];
    add[((int64_t)s * ns + sl) * 2 * dim + c] = (float)v;
  }
  // the tile slots, consumed, start the next step at zero
  for (int64_t e = (int64_t)t0 * G + tid; e < (int64_t)t1 * G; e += kCtrlThreads) abar_tile[e] = 0.0f;
}

// xbar_p += add[scene][slot(p)][0..d), vbar_p += add[scene][slot(p)][d..2d): one CTA per
// particle tile (the initial state's; the other states' are added by their G2P adjoint)
__global__ void ctrl_sensor_adjoint_kernel(int dim, int G, int64_t N, const int4* tiles,
                                           const int* group, const float* add, float* adj) {
  const int4 tile = tiles[blockIdx.x];
  if ((int)threadIdx.x >= tile.z) return;
  const int64_t p = (int64_t)tile.y + threadIdx.x;
  const int g = group[p];
  const int sl = (g >= 0 && g < G) ? g + 1 : 0;
  const float* a = add + ((int64_t)tile.x * (G + 1) + sl) * 2 * dim;
  for (int c = 0; c < 2 * dim; ++c) adj[(int64_t)c * N + p] += a[c];
}

// gw[scene][i] = thbar[scene][i] (FP64 -> FP32)
__global__ void ctrl_grad_out_kernel(int64_t n, const double* thbar, float* gw) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    gw[i] = (float)thbar[i];
}

}  // namespace

namespace {
// one CTA a scene; early: as a programmatic dependent of the pass before it
template <typename... KArgs, typename... Args>
cudaError_t launch_ctrl(void (*k)(KArgs...), int n_scenes, bool early, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_scenes);
  cfg.blockDim = dim3(kCtrlThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, KArgs(args)...);
}
}  // namespace

cudaError_t launch_ctrl_forward(const CtrlStep& cs, int n_scenes, int n_tiles, int64_t N,
                                const int4* tiles, const int* tile_off, const float* st,
                                const int* group, float* part, const float* theta, double* u,
                                double* h, double* y, float* act, double* cnt, bool early, cudaStream_t s) {
  if (st) {
    if (cs.dim == 2) ctrl_sense_kernel<2><<<n_tiles, kTile, 0, s>>>(cs.G, N, tiles, st, group, part);
    else ctrl_sense_kernel<3><<<n_tiles, kTile, 0, s>>>(cs.G, N, tiles, st, group, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    early = false;
  }
  return launch_ctrl(ctrl_forward_kernel, n_scenes, early, s, cs, tile_off, part, theta, u, h, y, act, cnt);
}

cudaError_t launch_ctrl_backward(const CtrlStep& cs, int n_scenes, int n_tiles, int64_t N,
                                 const int4* tiles, const int* tile_off, const int* group,
                                 float* abar_tile, const float* theta, const double* u,
                                 const double* h, const double* y, const double* cnt,
                                 double* thbar, float* add, float* adj, bool early, cudaStream_t s) {
  cudaError_t e = launch_ctrl(ctrl_backward_kernel, n_scenes, early, s, cs, tile_off, abar_tile, theta, u, h, y, cnt,
                              thbar, add);
  if (e != cudaSuccess || !adj) return e;
  ctrl_sensor_adjoint_kernel<<<n_tiles, kTile, 0, s>>>(cs.dim, cs.G, N, tiles, group, add, adj);
  return cudaGetLastError();
}

cudaError_t launch_ctrl_grad_out(int64_t n, const double* thbar, float* gw, cudaStream_t s) {
  ctrl_grad_out_kernel<<<(int)((n + 255) / 256 > 1024 ? 1024 : (n + 255) / 256), 256, 0, s>>>(n, thbar, gw);
  return cudaGetLastError();
}

}  // namespace mpm
