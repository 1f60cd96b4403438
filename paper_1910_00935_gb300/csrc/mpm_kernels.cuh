// mpm_kernels.cuh -- the particle passes of one MLS-MPM step and of its adjoint
// (Appendix D: p2g, grid_op, g2p and their .grad counterparts).
//
// There are no separate grid passes.  grid_op (v = p/m + dt g, sticky walls) and its
// adjoint (pbar = ubar/m, mbar = -ubar.p/m^2) are node-local, so the particle pass that
// consumes a grid applies them to every node it gathers.  Grids are accumulation
// buffers handed out by the host's ring allocator: a pass scatters into a clean buffer,
// records the touched box per scene, and a later pass zeroes that box once the buffer's
// last reader has finished (each buffer keeps two parity copies of its box so that a box
// is never reset while another CTA may still read it).
//
// Particle passes run one CTA per tile of up to kTile particles of one scene
// (particles are sorted per scene at set-up, so a tile covers a compact block of cells, ~8
// particles per cell in 3D, and a warp's 32 particles are two runs along the last axis).
// Thread t owns particle t: gathers, stress and state I/O are coalesced rows.  Scatters hand a
// warp's 32 particles to columns of lanes that walk them in order and sum the particles that
// share a node in registers before one float4 reduction to the grid (scatter_runs); the
// records cross between the two through shared memory, warp by warp.  Gathers read a shared
// gather box filled once per CTA (grid functions applied while filling), or the grid directly.
//
// Stencil loops are separable: the weight of node (i, j, k) is w0[i] w1[j] w2[k] and
// dpos = (dp0[i], dp1[j], dp2[k]), so partial products over (i) and (i, j) are hoisted.
#pragma once

#include <climits>

#include "mpm_common.cuh"

namespace mpm {

// particle-pass modes
enum StepMode : int {
  kP2GOnly = 0,      // full state in -> P2G
  kG2PP2G = 1,       // G2P (writes x, F) then P2G of the new state
  kG2PP2GFull = 2,   // same, also writes v and C
  kG2POnlyFull = 3,  // G2P, writes the full state
};
enum AdjMode : int {
  kAdjG2P = 0,    // G2P-adjoint of step s from the full adjoint of state s+1
  kAdjFused = 1,  // P2G-adjoint of step s+1, then G2P-adjoint of step s
  kAdjP2G = 2,    // P2G-adjoint of step s+1 only (s+1 = 0), writes the full adjoint
};

// a dirty grid buffer to zero over its recorded per-scene boxes
struct ClearJob {
  float4* grid;     // scene-major dense grids
  const int* box;   // [scene][8]: lo[3], hi[3]
};
constexpr int kMaxClears = 3;
struct Clears {
  ClearJob job[kMaxClears];
  int n;
  int words;  // float4 slots per node (1, or 2 for fixed-point grids)
};

struct StepArgs {
  const int4* tiles;       // {scene, first particle, count, rank of the tile in its scene}
  const int* scene_tiles;  // tiles per scene
  int N;                   // row stride (total particles)
  const float* in;         // state rows x, v, C, F - f_diag I (component-major)
  float* out;
  const float* mu;
  const float* la;
  const int* group;
  const int* matid;        // per-particle material (kMixed scenes) or null
  const float* wact;       // [scene][group][basis]
  const float4* PMr;       // grid (m, p) of step t-1, read by G2P (null: P2G only)
  float4* PMw;             // grid of step t, accumulated by P2G (null: G2P only)
  double* Rw;              // [9][N] polar factors (polar_to_cache) of the P2G's states, written (or null)
  int* box_w;              // [scene][8] box of PMw for this use
  int* box_reset;          // [scene][8] the other parity box of PMw, reset here (or null)
  Clears clears;
  unsigned* err;
  unsigned long long* box_stats;  // [2]: gather boxes staged, of which too large for the shared
                                  // box (read from the grid instead); null: not counted
  float* sense;            // closed-loop controller: per-tile sensor sums [tile][slot][value] (or null)
  int early;               // launched as a programmatic dependent (host only)
};

struct AdjArgs {
  const int4* tiles;
  const int* scene_tiles;
  int N;
  const float* st1;   // state s+1 (full)
  const float* st0;   // state s (x and F rows)
  const float* stm;   // state s-1 (full) for the recomputed P2G of step s-1, or null
  float* adj;         // adjoint rows x, v, C, F
  const float* mu;
  const float* la;
  float2* mubar;      // dL/dmu, dL/dlambda per particle, summed over the steps as compensated
  float2* labar;      // FP32 (value, correction) pairs: the per-step terms oscillate in sign
                      // over a long run and mostly cancel, so the sum needs ~48 bits
  const int* group;
  const int* matid;   // per-particle material (kMixed scenes) or null
  const float* wact;
  float* wbar_tile;   // [tile][group][basis] per-tile dL/dw partial sums (this pass adds)
  const float4* PM1;  // grid (m, p) of step s+1 (P2G-adjoint)
  const float4* UB1;  // grid-velocity adjoint of step s+1
  const float4* PM0;  // grid of step s (G2P-adjoint)
  float4* UB0;        // grid-velocity adjoint of step s (accumulated)
  int* box_ub;
  int* box_ub_reset;
  float4* PMm;        // grid of step s-1 (recomputed P2G) or null
  unsigned* ub_m0;    // deterministic mode: largest velocity-adjoint contribution bound of
                      // the backward's first scatter (FP32 bits; the measuring pass raises it,
                      // every pass derives the fixed-point scale of the ubar grids from it)
  int measure;        // 1: this kAdjG2P pass only measures that bound (no scatter, no writes)
  const double* R1;   // [9][N] cached polar factors of state s+1 (or null: recompute)
  const double* Rm;   // same for state s-1
  int* box_m;
  int* box_m_reset;
  Clears clears;
  unsigned* err;
  const float* sense_add;  // kAdjG2P: sensor adjoints [scene][slot][2D] added to xbar, vbar (or null)
  int early;  // launched as a programmatic dependent (host only)
  int early_states;  // no state is written by a pass that may still run when this one starts
};

// Grid reads in the particle passes are coherent loads: a pass may be resident while the pass
// before it still scatters into the grid that it will gather (see pass_wait), or run in the same
// persistent launch, so the read-only path (__ldg), which is defined for memory that nothing writes while
// a kernel runs and whose loads may be moved above the wait, is not for them.  As one ordered
// 16-byte load they take the same time as through that path (1,024 steps and reverse of a
// 262,144-particle cube 95.4 ms both, its first 256 steps 8.30, 16 x 65,536 fixed-corotated 57.3); left to
// the compiler they gain 1.5% on the two shorter runs and lose 2.4% on the long forward (27.1 -> 27.8 ms).
__device__ __forceinline__ float4 grid_load(const float4* p) {
  float4 r;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "l"(p) : "memory");
  return r;
}
// Node `node` of a scene's (m, p) grid as floats (DET: fixed-point grid).
template <bool DET>
__device__ __forceinline__ float4 pm_load(const float4* g, int64_t node, const SimParams& P) {
  if (DET) return fix_load(g, node, P.unfix_m, P.unfix_p);
  return grid_load(g + node);
}
// fixed-point scale pair of this backward's velocity-adjoint grids (deterministic mode)
__device__ __forceinline__ void ub_scales(const unsigned* m0, float& fix, float& unfix) {
  fix_scales_from(__uint_as_float(*(const volatile unsigned*)m0), fix, unfix);
}
// node of a scene's velocity-adjoint grid
template <bool DET>
__device__ __forceinline__ float4 ub_load(const float4* g, int64_t node, const SimParams& P,
                                          const unsigned* m0) {
  if (DET) {
    float fix, unfix;
    ub_scales(m0, fix, unfix);
    return fix_load(g, node, unfix, unfix);
  }
  return grid_load(g + node);
}
// Programmatic launch: a pass may start while the pass before it on its stream drains.  wait: every
// access to what another pass writes comes after it (it returns once that pass has completed and
// its writes are visible; at once in a normal launch); it precedes ready, so a pass that
// starts early finds all passes but the last one complete.  ready: the next pass may be placed on the SMs
// once every CTA has said so -- after a tile's first box is loaded, so that waiting CTAs do not
// hold slots that the other stream of an overlapped backward could use.  A small scene's pass
// is ~4 us of latency, 1 of them the launch: 4,096 2D particles over 128 steps 0.712 -> 0.647 ms,
// 3,477 forward and reverse over 384 steps 4.50 -> 4.11; 262,144 particles 0.5%.
__device__ __forceinline__ void pass_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pass_ready() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Packed FP32 pairs: one instruction for two independent operations, each rounded as on its own.
// Used where a pass is short of issue slots: the 3D adjoint gathers (16 warps an SM; fused pass of
// 16 x 65,536 fixed-corotated particles 276 -> 270 us, adjoint of the last step 138 -> 130).  In the
// forward gather and the scatter they measured no gain.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ float f2_lo(F2 p) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
  return a;
}
__device__ __forceinline__ float f2_hi(F2 p) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
  return b;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

struct NodePair {
  float4 ub, pm;
};
// a scene's grid inside a buffer of per-scene grids
__device__ __forceinline__ float4* scene_grid(float4* g, int scene, const SimParams& P) {
  return g + (int64_t)scene * P.nnodes * P.node_words;
}
__device__ __forceinline__ const float4* scene_grid(const float4* g, int scene, const SimParams& P) {
  return g + (int64_t)scene * P.nnodes * P.node_words;
}

template <int D>
struct Rows {
  static constexpr int X = 0, V = D, C = 2 * D, F = 2 * D + D * D, Q = 2 * D + 2 * D * D;
};

// scatter records: kQuads float4 per particle, [quad][kTile] (see put_record)
template <int D>
struct Rec {
  static constexpr int kQuads = D == 3 ? 6 : 4;
  static constexpr int kFloats = 4 * kQuads * kTile;
};

// per-warp group sums of the dL/dw reduction
constexpr int kWbarSlots = (kTile / 32) * kMaxGroups;

// Particle rows staged ahead of use with asynchronous copies (cp.async, no registers held
// while in flight): stage row r holds component r of the CTA's particles at
// [r * kTile + threadIdx.x]; each thread copies and later reads only its own column.
template <int D>
struct Stage {
  static constexpr int kStep = 3;                   // mu, la, group (read by the P2G stress)
  static constexpr int kAdjB = D + D * D;           // x, F rows of state s (G2P-adjoint)
  static constexpr int kAdjC = 2 * D + 2 * D * D;   // full state s-1 (recomputed P2G)
  static constexpr int kAdj = kAdjB + kAdjC + 3;    // + mu, la, group
};
__device__ __forceinline__ void stage_row(float* stage, int r, const float* src) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(stage + r * kTile + threadIdx.x);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
// a float2 of each particle into rows r and r + 1
__device__ __forceinline__ void stage_pair(float* stage, int r, const float2* src) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(stage + r * kTile + 2 * threadIdx.x);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// wait until at most N of this thread's copy groups are still in flight (the passes use
// N = 0 before the first read of any staged row)
template <int N>
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ float2 staged_pair(const float* stage, int r) {
  return *reinterpret_cast<const float2*>(stage + r * kTile + 2 * threadIdx.x);
}
__device__ __forceinline__ float staged(const float* stage, int r) { return stage[r * kTile + threadIdx.x]; }

// dynamic shared memory of a particle pass: gather box (4 floats per node), scatter records,
// staged rows
__host__ __device__ inline int box_floats(int gather_cap) { return 4 * (gather_cap > 0 ? gather_cap : 1); }
template <int D>
inline size_t step_smem_bytes(int gather_cap) {
  return sizeof(float) * ((size_t)box_floats(gather_cap) + Rec<D>::kFloats + Stage<D>::kStep * kTile);
}
template <int D>
inline size_t adj_smem_bytes(int gather_cap) {
  return sizeof(float) * ((size_t)box_floats(gather_cap) + Rec<D>::kFloats + Stage<D>::kAdj * kTile);
}

// Bounds of the stencil bases of a warp's valid lanes, written by lane 0 as two int4 (lo, hi) into
// the warp's own slot, so that nothing has to be reset beforehand and no shared atomics are
// needed; readers fold the warps' slots after the CTA's next barrier.
constexpr int kWarps = kTile / 32;
struct WarpBounds {
  int4 lo[kWarps], hi[kWarps];
};
// static shared memory of a tile
struct TileShared {
  WarpBounds gather[2], scatter[2];  // at most two gathers and two scatters (adjoint passes)
  int clear_box[8 * kMaxClears];     // scene boxes of the clear jobs
};
template <int D>
__device__ __forceinline__ void warp_bounds(bool valid, const int base[D], WarpBounds& wb) {
  int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    lo[a] = __reduce_min_sync(0xffffffffu, valid ? base[a] : INT_MAX);
    hi[a] = __reduce_max_sync(0xffffffffu, valid ? base[a] : INT_MIN);
  }
  if ((threadIdx.x & 31) == 0) {
    wb.lo[threadIdx.x >> 5] = make_int4(lo[0], lo[1], lo[2], 0);
    wb.hi[threadIdx.x >> 5] = make_int4(hi[0], hi[1], hi[2], 0);
  }
}

// Thread a (lo) or 4 + a (hi), a < D, folds the CTA's bound (stencil bases wb, whose last node is
// base + 2) into the scene box.  seen: that bound as the CTA read it when it started (box_seen);
// one that it already covers needs no atomic.  (Six atomics of every CTA on one scene's box
// serialise in the L2: they cost the plain P2G pass of a 2,048-tile cube 6 of 29 us.)
__device__ __forceinline__ int box_seen(const int* bbox_scene) {
  return threadIdx.x < 8 ? __ldcg(bbox_scene + threadIdx.x) : 0;
}
template <int D>
__device__ __forceinline__ void cta_bbox_flush(const WarpBounds& wb, int* bbox_scene, int seen) {
  if (threadIdx.x >= 8 || (threadIdx.x & 3) >= D) return;
  const bool is_lo = threadIdx.x < 4;
  const int* b = reinterpret_cast<const int*>(is_lo ? wb.lo : wb.hi) + (threadIdx.x & 3);
  int v = b[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) v = is_lo ? min(v, b[4 * w]) : max(v, b[4 * w]);
  if (is_lo) {
    if (v != INT_MAX && v < seen) atomicMin(bbox_scene + threadIdx.x, v);
  } else {
    if (v != INT_MIN && v + 2 > seen) atomicMax(bbox_scene + threadIdx.x, v + 2);
  }
}

template <int D>
__device__ __forceinline__ int pack_base(const int b[D]) {
  return D == 2 ? (b[0] << 16) | b[D - 1] : (b[0] << 20) | (b[1] << 10) | b[D - 1];
}
template <int D>
__device__ __forceinline__ void unpack_base(int v, int b[D]) {
  if (D == 2) {
    b[0] = v >> 16;
    b[D - 1] = v & 0xFFFF;
  } else {
    b[0] = v >> 20;
    b[1] = (v >> 10) & 0x3FF;
    b[D - 1] = v & 0x3FF;
  }
}

// flat node index inside one scene grid
template <int D>
__device__ __forceinline__ int node_flat(const int idx[D], int n) {
  int r = idx[0];
#pragma unroll
  for (int a = 1; a < D; ++a) r = r * n + idx[a];
  return r;
}

// flat offset of stencil node (i, j, k) from the stencil base
template <int D>
__device__ __forceinline__ int stencil_off(int i, int j, int k, int n) {
  return D == 2 ? i * n + j : (i * n + j) * n + k;
}

// The gathers sum over a stencil axis by axis -- the last axis's three nodes, then the rows of a
// plane, then the planes -- with the axis weights applied to the partial sums, so a node costs
// its differences and the last axis's products only (3D: 9 multiply-adds a node for W d and its
// moments against 15 with W formed per node).  In the 3D adjoint passes the planes run in a loop:
// a third of the code and of the values in flight, which at 128 registers measured 5% faster on
// 16 x 65,536 fixed-corotated particles (333 -> 316 us a fused pass) and 2% on the neo-Hookean
// cube; unrolled, the forward passes' planes overlap and measured 1% faster.
// wp: weight times dpos per axis (the first axis's come from axis_at).
template <int D>
struct GatherAxes {
  float wp[D][3];
  __device__ __forceinline__ explicit GatherAxes(const Axes<D>& s) {
#pragma unroll
    for (int a = 1; a < D; ++a)
#pragma unroll
      for (int o = 0; o < 3; ++o) wp[a][o] = s.w[a][o] * s.dp[a][o];
  }
};

template <int D>
__device__ __forceinline__ bool is_wall(const int idx[D], const SimParams& P) {
  bool wall = false;
#pragma unroll
  for (int a = 0; a < D; ++a) wall = wall || (unsigned)(idx[a] - P.wall) >= (unsigned)(P.n_grid - 2 * P.wall);
  return wall;
}

// ---------------------------------------------------------------------------
// CTA-cooperative node box in shared memory
// ---------------------------------------------------------------------------
template <int D>
struct BoxInfo {
  int lo[D], dim[D];
  int vol;
  bool use_tile;
};

// Extent of the node box covering the stencils of the CTA's valid particles.  Every thread of
// the CTA must call this; wb has not been used since an earlier barrier.  Holds one barrier,
// which also orders every earlier read of the shared node box before the box_load that follows.
template <int D>
__device__ __forceinline__ BoxInfo<D> box_extent(bool valid, const int base[D], int cap, WarpBounds& wb) {
  warp_bounds<D>(valid, base, wb);
  __syncthreads();
  int4 lo = wb.lo[0], hi = wb.hi[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) {
    const int4 l = wb.lo[w], h = wb.hi[w];
    lo = make_int4(min(lo.x, l.x), min(lo.y, l.y), min(lo.z, l.z), 0);
    hi = make_int4(max(hi.x, h.x), max(hi.y, h.y), max(hi.z, h.z), 0);
  }
  const int l3[3] = {lo.x, lo.y, lo.z}, h3[3] = {hi.x, hi.y, hi.z};
  const bool any = hi.x >= lo.x;
  BoxInfo<D> b;
  int vol = 1;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    b.lo[a] = l3[a];
    b.dim[a] = any ? h3[a] - l3[a] + 3 : 0;
    vol *= b.dim[a];
  }
  b.vol = vol;
  b.use_tile = any && vol <= cap;
  return b;
}

// Fill the shared gather box (float4 per node, box-local order), one node per thread: raw(f)
// reads what node f of the scene's grid needs, value(raw, wall) turns it into the gathered
// quantity.  BATCH nodes a thread are read before the first is used, so the box of a tile
// costs one round trip to the L2.  Called right after box_extent (whose barrier separates it
// from earlier readers of the box); synchronises after.
template <int D, int BATCH, typename Raw, typename Value>
__device__ __forceinline__ void box_load(const BoxInfo<D>& b, float4* sm4, const SimParams& P, Raw&& raw,
                                         Value&& value) {
  if (b.use_tile) {
    // box-local index -> node by float reciprocals: with q the quotient and d the divisor, the
    // quotient's error is below 3e-7 q and its distance to the next integer at least 0.5 / d,
    // so the truncation is exact while q d < 1.6e6 (a box holds at most 12,288 nodes)
    const float rz = __fdividef(1.0f, (float)b.dim[D - 1]), ry = D == 3 ? __fdividef(1.0f, (float)b.dim[1]) : 0.0f;
#pragma unroll 1
    for (int l0 = threadIdx.x; l0 < b.vol; l0 += BATCH * kTile) {
      decltype(raw(0)) r[BATCH];
      bool wall[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int l = l0 + u * kTile;
        if (l < b.vol) {
          int idx[D];
          int q = (int)(((float)l + 0.5f) * rz);
          idx[D - 1] = b.lo[D - 1] + (l - q * b.dim[D - 1]);
          if (D == 3) {
            const int x = (int)(((float)q + 0.5f) * ry);
            idx[1] = b.lo[1] + (q - x * b.dim[1]);
            q = x;
          }
          idx[0] = b.lo[0] + q;
          wall[u] = is_wall<D>(idx, P);
          r[u] = raw(node_flat<D>(idx, P.n_grid));
        }
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u)
        if (l0 + u * kTile < b.vol) sm4[l0 + u * kTile] = value(r[u], wall[u]);
    }
  }
  __syncthreads();
}

// Run body(load) with load(i, j, k) returning value(base + (i, j, k)): from the shared
// gather box when it holds the CTA's stencils, else computed from global memory.
template <int D, typename Raw, typename Value, typename Body>
__device__ __forceinline__ void with_nodes(const BoxInfo<D>& b, const float4* sm4, const int base[D], const SimParams& P,
                                           Raw&& raw, Value&& value, Body&& body) {
  if (b.use_tile) {
    int lb = base[0] - b.lo[0];
#pragma unroll
    for (int c = 1; c < D; ++c) lb = lb * b.dim[c] + (base[c] - b.lo[c]);
    const int s1 = D == 2 ? 1 : b.dim[D - 1];
    const int s0 = b.dim[1] * s1;
    const float4* p = sm4 + lb;
    body([&](int i, int j, int k) { return p[i * s0 + j * s1 + k]; });
  } else {
    body([&](int i, int j, int k) {
      int idx[D];
      idx[0] = base[0] + i;
      idx[1] = base[1] + j;
      if (D == 3) idx[D - 1] = base[D - 1] + k;
      return value(raw(node_flat<D>(idx, P.n_grid)), is_wall<D>(idx, P));
    });
  }
}

// ---------------------------------------------------------------------------
// Run-merged scatter: node (i, j, k) of a particle's stencil receives
//   mass  W * mass_c          (when WITH_MASS)
//   vec   W * (a + B dpos)
// A particle's 3^D nodes are 3^(D-1) columns along the grid's last axis.  Each warp scatters
// its own 32 particles: lane (slot, column) walks its slot's third (3D) or eighth (2D) of them
// in order, sums their contributions to its column's three nodes in registers, and where the
// stencil base moves by one node along the last axis reduces only the node that falls out
// of the window into the grid; any other move reduces all three.  The particle order makes
// runs of such moves (sort_keys_kernel), but nothing depends on it.
//
// Why: a pass with one float4 reduction per particle and node is bound by the L2's reduction
// rate (~3.4e11 a second here, 7.1 M a pass on a 262,144-particle cube, about 20 us of its
// 48 us).  On lattice rows of half cells the walk issues 6-8 reductions a particle in 3D
// (27 before) and ~4 in 2D (9).  Three slots of nine columns keep 27 of 32 lanes busy; the
// column's weights and affine value cost ~30 instructions per particle and lane, paid by
// passes that issued only 38% of the time.  Per launch, between two events (us, before ->
// after): 262,144-particle neo-Hookean cube fused step 48.5 -> 38.6, fused adjoint (half of
// them with a recomputed P2G) 107.9 -> 92.0; 16 x 65,536 fixed-corotated 171.7 -> 153.7 and
// 431 -> 377; 64 uneven 2D scenes (391,000 particles) 27.9 -> 23.4 and 52.5 -> 47.2; the cube
// in the deterministic mode, whose every node takes four 64-bit integer atomics,
// 101.6 -> 51.9 (89,505 particles).
// ---------------------------------------------------------------------------

// Write this thread's scatter record: the B-spline weights per axis, the affine value at the
// stencil's centre node a + B dpos(1, 1, 1), its increment per node B dx, and the packed base
// (-1: no scatter, whatever its weights and values).  Every thread writes its record.
template <int D>
__device__ __forceinline__ void put_record(float4* rec, bool valid, const Axes<D>& s, const float a[D],
                                           const float B[D][D], float dx) {
  float ac[D], Bd[D][D];
#pragma unroll
  for (int c = 0; c < D; ++c) {
    ac[c] = a[c];
#pragma unroll
    for (int b = 0; b < D; ++b) {
      Bd[c][b] = B[c][b] * dx;
      ac[c] += Bd[c][b] * (1.0f - s.f[b]);
    }
  }
  const float (&w)[D][3] = s.w;
  const float base = __int_as_float(valid ? pack_base<D>(s.base) : -1);
  float4* r = rec + threadIdx.x;
  r[0] = make_float4(w[0][0], w[0][1], w[0][2], 0.0f);
  if (D == 3) {
    constexpr int z = D - 1;
    r[kTile] = make_float4(w[1][0], w[1][1], w[1][2], 0.0f);
    r[2 * kTile] = make_float4(w[z][0], w[z][1], w[z][2], ac[0]);
    r[3 * kTile] = make_float4(ac[1], ac[z], Bd[0][0], Bd[0][1]);
    r[4 * kTile] = make_float4(Bd[0][z], Bd[1][0], Bd[1][1], Bd[1][z]);
    r[5 * kTile] = make_float4(Bd[z][0], Bd[z][1], Bd[z][z], base);
  } else {
    r[kTile] = make_float4(w[1][0], w[1][1], w[1][2], base);
    r[2 * kTile] = make_float4(ac[0], ac[1], Bd[0][0], Bd[0][1]);
    r[3 * kTile] = make_float4(Bd[1][0], Bd[1][1], 0.0f, 0.0f);
  }
}

// a node's running sums in registers: weight (or nothing) and vector
template <int D, bool WITH_MASS, bool DET>
struct NodeSum {
  static constexpr int kCh = D + (WITH_MASS ? 1 : 0);
  float v[kCh];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int c = 0; c < kCh; ++c) v[c] = 0.0f;
  }
  __device__ __forceinline__ void add(float W, const float q[D], float, float, float, unsigned&) {
    if (WITH_MASS) v[0] += W;
#pragma unroll
    for (int c = 0; c < D; ++c) v[c + (WITH_MASS ? 1 : 0)] += W * q[c];
  }
  __device__ __forceinline__ void reduce(float4* g, int node, float mass_c) const {
    const float x = WITH_MASS ? v[0] * mass_c : v[0];
    atomicAdd(g + node, make_float4(x, v[1], kCh > 2 ? v[kCh > 2 ? 2 : 0] : 0.0f, kCh > 3 ? v[kCh > 3 ? 3 : 0] : 0.0f));
  }
};
// Deterministic mode: every contribution is rounded once, exactly as a reduction of its own
// would round it (fix_round), and the integers are summed: h * 2^28 + l per channel with
// |l| <= 2^27, |h| <= 2^27 a contribution, so the at most 11 of a walk fit 32 bits each.
template <int D, bool WITH_MASS>
struct NodeSum<D, WITH_MASS, true> {
  static constexpr int kCh = D + (WITH_MASS ? 1 : 0);
  int h[kCh], l[kCh];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int c = 0; c < kCh; ++c) h[c] = l[c] = 0;
  }
  __device__ __forceinline__ void add(float W, const float q[D], float mass_c, float fix0, float fix1,
                                      unsigned& err) {
    float c[kCh];
    if (WITH_MASS) c[0] = W * mass_c * fix0;
#pragma unroll
    for (int a = 0; a < D; ++a) c[a + (WITH_MASS ? 1 : 0)] = W * q[a] * (WITH_MASS || a > 0 ? fix1 : fix0);
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
      const bool in = fabsf(c[k]) <= kFixLimit;
      if (!in) err |= kErrRange;
      int hi, lo;
      fix_split(in ? c[k] : 0.0f, hi, lo);
      h[k] += hi;
      l[k] += lo;
    }
  }
  __device__ __forceinline__ void reduce(float4* g, int node, float) const {
    unsigned long long* q = reinterpret_cast<unsigned long long*>(g + 2 * (int64_t)node);
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
      const long long v = fix_join(h[k], l[k]);
      if (v != 0) atomicAdd(q + k, (unsigned long long)v);
    }
  }
};

// Scatter the warp's 32 records (written by its own lanes, __syncwarp'ed) into grid g.  Slots: three
// of nine columns in 3D (27 lanes, 10 or 11 particles each), eight of three in 2D (24 lanes, four
// particles each, so that the slots' moves fall on the same turns).
template <int D, bool WITH_MASS, bool DET>
__device__ __forceinline__ void scatter_runs(const float4* rec, float4* g, int n, float mass_c, float fix0,
                                             float fix1, unsigned& err) {
  constexpr int COLS = D == 3 ? 9 : 3, SLOTS = D == 3 ? 3 : 8;
  const int lane = threadIdx.x & 31;
  const int slot = lane / COLS, col = lane - slot * COLS;
  if (slot >= SLOTS) return;
  const int i = D == 3 ? col / 3 : col, j = D == 3 ? col - 3 * i : 0;
  const float si = (float)(i - 1), sj = (float)(j - 1);
  const int off = D == 3 ? (i * n + j) * n : i * n;
  const float4* r = rec + (threadIdx.x & ~31u) + (slot * 32) / SLOTS;
  const float4* end = rec + (threadIdx.x & ~31u) + ((slot + 1) * 32) / SLOTS;
  NodeSum<D, WITH_MASS, DET> a0, a1, a2;
  a0.zero();
  a1.zero();
  a2.zero();
  int cur = -2, node = 0;  // (no base, nor the -1 of a refused particle: even a walk's first record is compared)
#pragma unroll 1
  for (; r < end; ++r) {
    const float* w0 = reinterpret_cast<const float*>(r);
    float wc, wz[3], qc[D], Bz[D];  // weight of the column, along the last axis; value at its centre, increment
    int base;
    if (D == 3) {
      const float4 q2 = r[2 * kTile], q3 = r[3 * kTile], q4 = r[4 * kTile], q5 = r[5 * kTile];
      wc = w0[i] * w0[4 * kTile + j];
      wz[0] = q2.x;
      wz[1] = q2.y;
      wz[2] = q2.z;
      qc[0] = q2.w + si * q3.z + sj * q3.w;
      qc[1] = q3.x + si * q4.y + sj * q4.z;
      qc[D - 1] = q3.y + si * q5.x + sj * q5.y;
      Bz[0] = q4.x;
      Bz[1] = q4.w;
      Bz[D - 1] = q5.z;
      base = __float_as_int(q5.w);
    } else {
      const float4 q1 = r[kTile], q2 = r[2 * kTile];
      const float2 q3 = *reinterpret_cast<const float2*>(r + 3 * kTile);
      wc = w0[i];
      wz[0] = q1.x;
      wz[1] = q1.y;
      wz[2] = q1.z;
      base = __float_as_int(q1.w);
      qc[0] = q2.x + si * q2.z;
      qc[1] = q2.y + si * q3.x;
      Bz[0] = q2.w;
      Bz[1] = q3.y;
    }
    if (base != cur) {
      if (base < 0) continue;  // no scatter
      // base and cur hold the last axis in their low bits and differ by at least 3 across rows
      // (the last axis stays below its field's range), so a difference of one is a move along it
      const int d = base - cur;
      if (cur >= 0 && d == 1) {
        a0.reduce(g, node, mass_c);
        a0 = a1;
        a1 = a2;
        a2.zero();
        node += 1;
      } else if (cur >= 0 && d == -1) {
        a2.reduce(g, node + 2, mass_c);
        a2 = a1;
        a1 = a0;
        a0.zero();
        node -= 1;
      } else {
        if (cur >= 0) {
          a0.reduce(g, node, mass_c);
          a1.reduce(g, node + 1, mass_c);
          a2.reduce(g, node + 2, mass_c);
          a0.zero();
          a1.zero();
          a2.zero();
        }
        int b[D];
        unpack_base<D>(base, b);
        node = node_flat<D>(b, n) + off;
      }
      cur = base;
    }
    float q[D];
#pragma unroll
    for (int c = 0; c < D; ++c) q[c] = qc[c] - Bz[c];
    a0.add(wc * wz[0], q, mass_c, fix0, fix1, err);
    a1.add(wc * wz[1], qc, mass_c, fix0, fix1, err);
#pragma unroll
    for (int c = 0; c < D; ++c) q[c] = qc[c] + Bz[c];
    a2.add(wc * wz[2], q, mass_c, fix0, fix1, err);
  }
  if (cur >= 0) {
    a0.reduce(g, node, mass_c);
    a1.reduce(g, node + 1, mass_c);
    a2.reduce(g, node + 2, mass_c);
  }
}

// actuation of a particle of group g (< 0 or >= n_groups: none) at a step with the given basis; axis:
// the fibre's.  The group comes by an asynchronous copy issued before a pass waits for the one before it
// (staged_group), so that its round trip is not on the chain of the stress.
__device__ __forceinline__ float particle_act(const SimParams& P, const float* basis, int g,
                                              const float* wact, int scene, int dim, int& axis) {
  axis = 0;
  if (g < 0 || g >= P.n_groups) return 0.0f;
  axis = g % dim;
  const float* w = wact + ((int64_t)scene * P.n_groups + g) * P.n_basis;
  float a = 0.0f;
#pragma unroll
  for (int k = 0; k < kMaxBasis; ++k)
    if (k < P.n_basis) a += w[k] * basis[k];
  return a;
}

// the particle's group from its staged row (-1: no groups)
__device__ __forceinline__ int staged_group(const SimParams& P, const float* stage, int r) {
  return P.n_groups > 0 ? __float_as_int(staged(stage, r)) : -1;
}

template <int D>
__device__ __forceinline__ void load_E(const float* rows, int64_t N, int64_t p, float f_diag,
                                       float E[D][D]) {
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j)
      E[i][j] = rows[(Rows<D>::F + i * D + j) * N + p] - (i == j ? f_diag : 0.0f);
}

// ---------------------------------------------------------------------------
// grid functions applied at gather time
// ---------------------------------------------------------------------------
// grid_op: v = p/m + dt g for m > 0 off the sticky walls, else 0 (w keeps m).  Rounding is
// spelled out (no compiler-chosen contraction), so a node gives the same bits whether it
// is staged in the shared gather box or read directly.
template <int D>
__device__ __forceinline__ float4 node_velocity(float4 pm, bool wall, const SimParams& P) {
  float4 u = make_float4(0.0f, 0.0f, 0.0f, pm.x);
  if (pm.x > 0.0f && !wall) {
    const float im = __frcp_rn(pm.x);
    u.x = __fmaf_rn(pm.y, im, __fmul_rn(P.dt, P.gravity[0]));
    u.y = __fmaf_rn(pm.z, im, __fmul_rn(P.dt, P.gravity[1]));
    if (D == 3) u.z = __fmaf_rn(pm.w, im, __fmul_rn(P.dt, P.gravity[2]));
  }
  return u;
}

// grid_op.grad: pbar = ubar / m and mbar = -ubar . (p / m) / m for m > 0 off the walls
// (rounding spelled out as in node_velocity)
template <int D>
__device__ __forceinline__ float4 node_adjoint(float4 ub, float4 pm, bool wall, const SimParams& P) {
  float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (pm.x > 0.0f && !wall) {
    const float im = __frcp_rn(pm.x);
    r.x = __fmul_rn(ub.x, im);
    r.y = __fmul_rn(ub.y, im);
    float dot = __fmaf_rn(ub.y, pm.z, __fmul_rn(ub.x, pm.y));
    if (D == 3) {
      r.z = __fmul_rn(ub.z, im);
      dot = __fmaf_rn(ub.z, pm.w, dot);
    }
    r.w = __fmul_rn(__fmul_rn(-dot, im), im);
  }
  return r;
}

// ---------------------------------------------------------------------------
// clears and box resets (each CTA takes its share of its own scene)
// ---------------------------------------------------------------------------
// The boxes of the jobs are copied to shared memory at the start of a tile (stage_clears:
// asynchronous, 8 threads a job) and the clears run after a later barrier, off the chain of loads that
// the tile starts with.
__device__ __forceinline__ void stage_clears(const Clears& C, int scene, int* boxes) {
  if ((int)threadIdx.x < 8 * C.n) {
    const int* src = C.job[threadIdx.x >> 3].box + scene * 8 + (threadIdx.x & 7);
    const unsigned dst = (unsigned)__cvta_generic_to_shared(boxes + threadIdx.x);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
  }
}
template <int D>
__device__ __forceinline__ void run_clears(const Clears& C, const int* boxes, int scene, int rank, int nranks,
                                           int nnodes, int n) {
  for (int c = 0; c < C.n; ++c) {
    const int* bb = boxes + 8 * c;
    // An empty box (lo = INT_MAX, hi = INT_MIN: a buffer that was allocated but never
    // scattered into, e.g. after a pass that gave up) clears nothing; hi - lo is formed
    // only for a non-empty box, and the box is clipped to the grid.
    int lo[D], ext[D], vol = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      lo[a] = bb[a] > 0 ? bb[a] : 0;
      const int hi = bb[4 + a] < n - 1 ? bb[4 + a] : n - 1;
      ext[a] = hi >= lo[a] ? hi - lo[a] + 1 : 0;
      vol *= ext[a];
    }
    const int w = C.words;
    float4* g = C.job[c].grid + (int64_t)scene * nnodes * w;
    for (int l = rank * blockDim.x + threadIdx.x; l < vol; l += nranks * blockDim.x) {
      int idx[D], r = l;
#pragma unroll
      for (int a = D - 1; a >= 0; --a) {
        idx[a] = lo[a] + r % ext[a];
        r /= ext[a];
      }
      float4* q = g + (int64_t)node_flat<D>(idx, n) * w;
      q[0] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (w == 2) q[1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
  }
}

__device__ __forceinline__ void reset_box(int* box, int scene) {
  if (box && threadIdx.x < 8) box[scene * 8 + threadIdx.x] = (threadIdx.x & 4) ? INT_MIN : INT_MAX;
}

// ---------------------------------------------------------------------------
// closed-loop controller: a tile's sums of x, v and the particle count by group slot (slot 0:
// particles in no group), out[slot][x_0.., v_0.., count], in a fixed order: each warp sums
// its lanes of one slot at a time (butterfly), then the warps are added in order.  Every
// thread calls it.  scratch: kWarps * slots * (2D + 1) floats.
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ void sense_tile(int G, bool xfix, int g, bool active, const float x[D], const float v[D],
                                           float* scratch, float* out) {
  constexpr int NV = 2 * D + 1;
  const int lane = threadIdx.x & 31, ns = G + 1;
  const int slot = !active ? -1 : (g >= 0 && g < G) ? g + 1 : 0;
  float q[2 * D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    q[a] = xfix ? (float)__float_as_int(x[a]) * (1.0f / kFixPos) : x[a];
    q[D + a] = v[a];
  }
  float* w = scratch + (threadIdx.x >> 5) * ns * NV;
  for (int l = lane; l < ns * NV; l += 32) w[l] = 0.0f;
  __syncwarp();
  unsigned left = __ballot_sync(0xffffffffu, active);
  while (left) {  // usually one or two slots a warp
    const int s = __shfl_sync(0xffffffffu, slot, __ffs(left) - 1);
    const bool in = slot == s;
    const unsigned mask = __ballot_sync(0xffffffffu, in);
#pragma unroll
    for (int c = 0; c < 2 * D; ++c) {
      float t = in ? q[c] : 0.0f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == c) w[s * NV + c] = t;
    }
    if (lane == 2 * D) w[s * NV + 2 * D] = (float)__popc(mask);
    left &= ~mask;
  }
  __syncthreads();
  for (int l = threadIdx.x; l < ns * NV; l += kTile) {
    float t = scratch[l];
#pragma unroll
    for (int k = 1; k < kWarps; ++k) t += scratch[k * ns * NV + l];
    out[l] = t;
  }
}

// ---------------------------------------------------------------------------
// P2G of the CTA's particles: stress, affine matrix A = kappa tau + m C, scatter
// (m, m v + A dpos) into the scene grid g, fold the touched box into box_scene.
// Every thread calls it; wb has not been used since an earlier barrier.
// ---------------------------------------------------------------------------
template <int D, int MAT, bool DET>
__device__ __forceinline__ void p2g_pass(const SimParams& P, const float* basis, bool active, int scene,
                                         int64_t p, int grp, const float x[D], const float v[D],
                                         const float C[D][D], const float E[D][D], float mu_p,
                                         float la_p, int mat_p, const float* wact, float4* g, int* box_scene, float4* rec, WarpBounds& wb,
                                         int seen, unsigned& err, const double* R_in, double* R_out, int64_t N) {
  Axes<D> s;
  bool ok = make_axes<D>(x, P, s) && active;
  if (active && !ok) err |= kErrOOB;
  float Am[D][D], mv[D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    mv[i] = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) Am[i][j] = 0.0f;
  }
  if (ok) {
    int axis;
    const float act = particle_act(P, basis, grp, wact, scene, D, axis);
    float tau[D][D];
    StressCache<D> sc;
    if (!kirchhoff<D, MAT>(E, mu_p, la_p, act, axis, tau, sc, R_in, N, p, mat_p)) {
      err |= kErrNonFinite;
      ok = false;
    }
    // the polar cache is a 3D fixed-corotated feature
    if (D == 3 && (MAT == kFixedCorotated || (MAT == kMixed && mat_p == kFixedCorotated)) && R_out && active)
      polar_to_cache<D>(R_out, N, p, sc.pol);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      mv[i] = P.p_mass * v[i];
#pragma unroll
      for (int j = 0; j < D; ++j) Am[i][j] = P.kappa * tau[i][j] + P.p_mass * C[i][j];
    }
  }
  __syncwarp();  // the warp's records may still be read by its earlier scatter
  put_record<D>(rec, ok, s, mv, Am, P.dx);
  warp_bounds<D>(ok, s.base, wb);
  __syncwarp();
  scatter_runs<D, true, DET>(rec, g, P.n_grid, P.p_mass, P.fix_m, P.fix_p, err);
  __syncthreads();  // every warp's share of the box
  cta_bbox_flush<D>(wb, box_scene, seen);
}

// ---------------------------------------------------------------------------
// forward particle pass: [G2P of step t-1] then [P2G of step t]
// ---------------------------------------------------------------------------
// One tile of a forward pass; every thread of the CTA calls it.  sm: dynamic shared memory
// (step_smem_bytes).  OWN: the pass is a launch of its own (it then waits for the one before it), not
// one of a persistent launch.  A CTA that runs several tiles must synchronise between them.
//
// A tile is a chain of dependent round trips to the L2 -- its entry, its particles' rows, its
// box of grid nodes -- and a 2,048-tile cube runs in two waves of 7 tiles per SM, so what is
// not part of the chain stays off it: the clear jobs' boxes, mu and la come by asynchronous
// copies, the bounds of a box need one barrier and no reset, all nodes of a box are read
// before the first is used, and a warp scatters without waiting for the others.
template <int D, int MAT, int MODE, bool OWN, bool DET>
__device__ __forceinline__ void step_tile(const SimParams& P, const StepArgs& A, int tile_index,
                                          float* sm, TileShared& sh) {
  using R = Rows<D>;
  constexpr int kBatch = 3;
  float4* rec = reinterpret_cast<float4*>(sm + box_floats(P.gather_capacity));
  const int4 tile = A.tiles[tile_index];
  const int scene = tile.x;
  const bool active = (int)threadIdx.x < tile.z;
  const int64_t p = (int64_t)tile.y + (active ? threadIdx.x : 0);
  const int64_t N = A.N;
  const int n = P.n_grid;
  unsigned err = 0;
  // what no pass writes: before the wait for the pass before
  float* stage = reinterpret_cast<float*>(rec) + Rec<D>::kFloats;
  if (MODE != kG2POnlyFull) {
    stage_row(stage, 0, A.mu + p);
    stage_row(stage, 1, A.la + p);
  }
  if (P.n_groups > 0) stage_row(stage, 2, reinterpret_cast<const float*>(A.group) + p);
  const int nranks = A.scene_tiles[scene];
  if (OWN) pass_wait();
  const int seen = MODE != kG2POnlyFull ? box_seen(A.box_w + scene * 8) : 0;
  // the particle's rows first: in flight while the clears below read their boxes
  float x[D], v[D], C[D][D], E[D][D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    x[a] = A.in[(R::X + a) * N + p];
    if (MODE == kP2GOnly) v[a] = A.in[(R::V + a) * N + p];
  }
  if (MODE == kP2GOnly)
#pragma unroll
    for (int i = 0; i < D * D; ++i) C[i / D][i % D] = A.in[(R::C + i) * N + p];
  load_E<D>(A.in, N, p, P.f_diag, E);
  stage_clears(A.clears, scene, sh.clear_box);
  if (tile.w == 0) reset_box(A.box_reset, scene);
  stage_commit();

  if (MODE != kP2GOnly) {
    // ---- G2P: v' = sum W u, C' = 4/dx^2 sum W (u - u_c) dpos^T, x' = x + dt v',
    //      E' = E + dt C' (I + E), with u = grid_op(PM of step t-1) at each node
    float xo[D], Eo[D][D];
#pragma unroll
    for (int a = 0; a < D; ++a) xo[a] = x[a];
#pragma unroll
    for (int i = 0; i < D * D; ++i) Eo[i / D][i % D] = E[i / D][i % D];
    Axes<D> s;
    const bool ok = make_axes<D>(xo, P, s) && active;
    if (active && !ok) err |= kErrOOB;
    float B[D][D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      v[a] = 0.0f;
#pragma unroll
      for (int b = 0; b < D; ++b) B[a][b] = 0.0f;
    }
    const float4* PMg = scene_grid(A.PMr, scene, P);
    stage_wait<0>();  // (this thread's share of the clear boxes, before the barrier below)
    auto raw = [&](int f) { return pm_load<DET>(PMg, f, P); };
    auto velocity = [&](float4 pm, bool wall) { return node_velocity<D>(pm, wall, P); };
    BoxInfo<D> gbx;
    gbx.use_tile = false;
    if (P.gather_capacity > 0) {
      gbx = box_extent<D>(ok, s.base, P.gather_capacity, sh.gather[0]);
      if (A.box_stats && threadIdx.x == 0 && gbx.vol > 0) {
        atomicAdd(A.box_stats, 1ull);
        if (!gbx.use_tile) atomicAdd(A.box_stats + 1, 1ull);
      }
      box_load<D, kBatch>(gbx, reinterpret_cast<float4*>(sm), P, raw, velocity);
    } else {
      __syncthreads();
    }
    if (OWN) pass_ready();
    run_clears<D>(A.clears, sh.clear_box, scene, tile.w, nranks, P.nnodes, n);
    if (ok) {
      // centred on the stencil's centre node: equal because sum W dpos = 0, and
      // accurate in FP32 when u is nearly uniform over the stencil
      with_nodes<D>(gbx, reinterpret_cast<const float4*>(sm), s.base, P, raw, velocity, [&](auto load) {
        const float4 uc4 = load(1, 1, D == 3 ? 1 : 0);
        const float uc[3] = {uc4.x, uc4.y, uc4.z};
        GatherAxes<D> g(s);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          float wi, dwi, dpi, t[D], tb[D][D];  // sums over the plane: W d, and W d dpos_b (b >= 1)
          axis_at(i, s.f[0], P.dx, wi, dwi, dpi);
#pragma unroll
          for (int a = 0; a < D; ++a) {
            t[a] = 0.0f;
#pragma unroll
            for (int b = 1; b < D; ++b) tb[a][b] = 0.0f;
          }
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            float r[D], rb[D];  // the same along the last axis
            if (D == 3) {
#pragma unroll
              for (int a = 0; a < D; ++a) r[a] = rb[a] = 0.0f;
#pragma unroll
              for (int k = 0; k < 3; ++k) {
                const float4 u4 = load(i, j, k);
                const float u[3] = {u4.x, u4.y, u4.z};
#pragma unroll
                for (int a = 0; a < D; ++a) {
                  const float d = u[a] - uc[a];
                  r[a] += s.w[D - 1][k] * d;
                  rb[a] += g.wp[D - 1][k] * d;
                }
              }
            } else {
              const float4 u4 = load(i, j, 0);
              r[0] = u4.x - uc[0];
              r[1] = u4.y - uc[1];
            }
#pragma unroll
            for (int a = 0; a < D; ++a) {
              t[a] += s.w[1][j] * r[a];
              tb[a][1] += g.wp[1][j] * r[a];
              if (D == 3) tb[a][D - 1] += s.w[1][j] * rb[a];
            }
          }
          const float wpi = wi * dpi;
#pragma unroll
          for (int a = 0; a < D; ++a) {
            v[a] += wi * t[a];
            B[a][0] += wpi * t[a];
#pragma unroll
            for (int b = 1; b < D; ++b) B[a][b] += wi * tb[a][b];
          }
        }
#pragma unroll
        for (int a = 0; a < D; ++a) v[a] += uc[a];  // sum W = 1
      });
    }
    const float c4 = 4.0f * P.inv_dx * P.inv_dx;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int b = 0; b < D; ++b) C[a][b] = c4 * B[a][b];
#pragma unroll
    for (int a = 0; a < D; ++a) x[a] = P.xfix ? pos_advance(xo[a], P.dt * v[a]) : xo[a] + P.dt * v[a];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) {
        float g = P.dt * C[i][j];  // dt C' (I + E)
#pragma unroll
        for (int k = 0; k < D; ++k) g += P.dt * C[i][k] * Eo[k][j];
        E[i][j] = Eo[i][j] + g;
      }
    if (active) {
#pragma unroll
      for (int a = 0; a < D; ++a) A.out[(R::X + a) * N + p] = x[a];
#pragma unroll
      for (int i = 0; i < D * D; ++i)
        A.out[(R::F + i) * N + p] = E[i / D][i % D] + (i / D == i % D ? P.f_diag : 0.0f);
      if (MODE == kG2PP2GFull || MODE == kG2POnlyFull) {
#pragma unroll
        for (int a = 0; a < D; ++a) A.out[(R::V + a) * N + p] = v[a];
#pragma unroll
        for (int i = 0; i < D * D; ++i) A.out[(R::C + i) * N + p] = C[i / D][i % D];
      }
    }
  }

  if (MODE == kG2POnlyFull && A.sense)
    sense_tile<D>(P.n_groups, P.xfix, staged_group(P, stage, 2), active, x, v, reinterpret_cast<float*>(rec),
                  A.sense + (int64_t)tile_index * (P.n_groups + 1) * (2 * D + 1));
  if (MODE != kG2POnlyFull) {
    stage_wait<0>();
    if (OWN && MODE == kP2GOnly) pass_ready();
    p2g_pass<D, MAT, DET>(P, P.basis, active, scene, p, staged_group(P, stage, 2), x, v, C, E, staged(stage, 0),
                          staged(stage, 1), MAT == kMixed ? A.matid[p] : MAT, A.wact, scene_grid(A.PMw, scene, P), A.box_w + scene * 8, rec, sh.scatter[0], seen, err, nullptr, A.Rw, N);
    if (MODE == kP2GOnly) run_clears<D>(A.clears, sh.clear_box, scene, tile.w, nranks, P.nnodes, n);
  }
  if (err) atomicOr(A.err, err);
}

// resident CTAs per SM the adjoint passes are compiled for
template <int D>
constexpr int adj_ctas_per_sm() {
  return D == 2 ? MPM_ADJ_CTAS_PER_SM_2D : MPM_ADJ_CTAS_PER_SM_3D;
}
// resident CTAs per SM the forward passes are compiled for
template <int D, int MAT>
constexpr int step_ctas_per_sm() {
  return D == 2 ? MPM_STEP_CTAS_PER_SM_2D
                : (MAT == kFixedCorotated || MAT == kMixed) ? MPM_STEP_CTAS_PER_SM_3D_POLAR
                                                           : MPM_STEP_CTAS_PER_SM_3D;
}

template <int D, int MAT, int MODE, bool DET>
__global__ void __launch_bounds__(kTile, step_ctas_per_sm<D, MAT>())
    step_kernel(const __grid_constant__ SimParams P, const __grid_constant__ StepArgs A) {
  extern __shared__ __align__(16) float sm[];
  __shared__ TileShared sh;
  step_tile<D, MAT, MODE, true, DET>(P, A, blockIdx.x, sm, sh);
}

// ---------------------------------------------------------------------------
// adjoint particle pass: [P2G-adjoint of step s+1] [G2P-adjoint of step s]
// [recomputed P2G of step s-1, the grid the next adjoint pass needs (Appendix D.1)]
// ---------------------------------------------------------------------------
// One tile of an adjoint pass (same calling rules as step_tile; s_wbar: kWbarSlots floats).
template <int D, int MAT, int MODE, bool OWN, bool DET>
__device__ __forceinline__ void adjoint_tile(const SimParams& P, const AdjArgs& A, int tile_index,
                                             float* sm, TileShared& sh, float* s_wbar) {
  using R = Rows<D>;
  constexpr int kBatch = 3;
  float4* rec = reinterpret_cast<float4*>(sm + box_floats(P.gather_capacity));
  const int4 tile = A.tiles[tile_index];
  const int scene = tile.x;
  const bool active = (int)threadIdx.x < tile.z;
  const int64_t p = (int64_t)tile.y + (active ? threadIdx.x : 0);
  const int64_t N = A.N;
  const int n = P.n_grid;
  const float c4 = 4.0f * P.inv_dx * P.inv_dx;
  unsigned err = 0;
  const int nranks = A.scene_tiles[scene];
  float* stage = reinterpret_cast<float*>(rec) + Rec<D>::kFloats;
  if (P.n_groups > 0) stage_row(stage, Stage<D>::kAdj - 1, reinterpret_cast<const float*>(A.group) + p);
  stage_commit();

  constexpr bool kStress = MODE != kAdjG2P;
  constexpr bool kLate = D == 3;
  constexpr bool kCarried = D == 3 && MODE != kAdjG2P;
  constexpr int kSums = D + 2 * D * D;
  static_assert(D == 2 || kSums + 4 <= Stage<D>::kAdj - 1 - Stage<D>::kAdjB, "the carried rows fit");
  const bool carried = kCarried && !A.stm;
  int seen_ub = 0, seen_m = 0;
  auto stage_rest = [&]() {
    seen_ub = MODE != kAdjP2G && A.box_ub ? box_seen(A.box_ub + scene * 8) : 0;
    seen_m = MODE != kAdjP2G && A.stm ? box_seen(A.box_m + scene * 8) : 0;
    stage_clears(A.clears, scene, sh.clear_box);
    stage_commit();
    if (tile.w == 0) {
      reset_box(A.box_ub_reset, scene);
      reset_box(A.box_m_reset, scene);
    }
    // stage what the G2P-adjoint (state s: x, F) and the recomputed P2G (state s-1, mu, la)
    // read, so that those loads are in flight during the P2G-adjoint
    if (MODE != kAdjP2G) {
#pragma unroll
      for (int a = 0; a < D; ++a) stage_row(stage, a, A.st0 + (int64_t)(R::X + a) * N + p);
#pragma unroll
      for (int i = 0; i < D * D; ++i) stage_row(stage, D + i, A.st0 + (int64_t)(R::F + i) * N + p);
    }
    stage_commit();
    if (MODE != kAdjP2G && A.stm) {  // the recomputed P2G runs whenever state s-1 is given
#pragma unroll
      for (int r = 0; r < R::Q; ++r) stage_row(stage, Stage<D>::kAdjB + r, A.stm + (int64_t)r * N + p);
      stage_row(stage, Stage<D>::kAdjB + R::Q, A.mu + p);
      stage_row(stage, Stage<D>::kAdjB + R::Q + 1, A.la + p);
    }
    // without it, its rows hold what the P2G-adjoint needs after its gather: the carried adjoint, C
    // of state s+1, the material sums -- at four CTAs an SM each exposed round trip is ~3% of a
    // tile's 33,000 cycles (with the group ahead of the chain and nothing waiting for the dL/dw
    // slot, 16 x 65,536 fixed-corotated: fused pass 263 -> 250 us, last P2G-adjoint 215 -> 199)
    if (carried) {
      constexpr int b = Stage<D>::kAdjB;
#pragma unroll
      for (int a = 0; a < D; ++a) stage_row(stage, b + a, A.adj + (int64_t)(R::X + a) * N + p);
#pragma unroll
      for (int i = 0; i < D * D; ++i) {
        stage_row(stage, b + D + i, A.adj + (int64_t)(R::F + i) * N + p);
        stage_row(stage, b + D + D * D + i, A.st1 + (int64_t)(R::C + i) * N + p);
      }
      stage_pair(stage, b + kSums, A.mubar + p);
      stage_pair(stage, b + kSums + 2, A.labar + p);
    }
    stage_commit();
  };
  // adjoint of state s+1: xb, vb, Cb, Fb (Fb = dL/dE = dL/dF); C1 = C of state s+1.  In 3D,
  // after a P2G-adjoint the carried xb, Fb and the rows of state s+1 needed again (C, E,
  // mu, la, the polar factor) are read after its gather -- fresh loads, as the gather's
  // barriers order them -- so that none of them holds a register across the gather (in 2D
  // they fit: loaded once, before it)
  float xb[D], vb[D], Cb[D][D], Fb[D][D], C1[D][D];
  auto load_carried = [&]() {
    if (carried) {
      stage_wait<0>();
      constexpr int b = Stage<D>::kAdjB;
#pragma unroll
      for (int a = 0; a < D; ++a) xb[a] = staged(stage, b + a);
#pragma unroll
      for (int i = 0; i < D * D; ++i) {
        Fb[i / D][i % D] = staged(stage, b + D + i);
        C1[i / D][i % D] = staged(stage, b + D + D * D + i);
      }
      return;
    }
#pragma unroll
    for (int a = 0; a < D; ++a) xb[a] = A.adj[(R::X + a) * N + p];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) {
        Fb[i][j] = A.adj[(R::F + i * D + j) * N + p];
        if (kLate || !kStress) C1[i][j] = A.st1[(R::C + i * D + j) * N + p];
      }
  };

  // State s+1 and its stress: a quarter of a tile's time that needs nothing of the pass before when
  // that is an adjoint pass (states are written by step passes: early_states).  It then goes ahead
  // of the wait, its rows read through the L2 (nothing that an SM kept from another pass).  Forward
  // and reverse: 49,152 liquid particles over 256 steps 6.38 -> 5.97 ms, 3,477 in 2D over 384 steps
  // 3.93 -> 3.72, the 262,144-particle neo-Hookean cube 28.68 -> 28.17.  2D passes of many waves
  // lose 1% (the launch decides); 3D fixed-corotated ones lose 0.5% (the rows are read again
  // after the gather, then from the L1) and keep the wait first.
  constexpr bool kMayLead = OWN && kStress && (D == 2 || MAT == kNeoHookean || MAT == kLiquid);
  const bool early = kMayLead && A.early_states;
  if (!early) {
    if (OWN) pass_wait();
    stage_rest();
    if (MODE == kAdjG2P || !kLate) load_carried();
  }
  float x[D], v[D], E[D][D], Am[D][D], mv[D];
  Axes<D> s;
  StressCache<D> sc;
  bool ok = false;
  int axis = 0, grp = -1, mat_p = MAT;
  float act = 0.0f;
  if constexpr (kStress) {
    auto row = [&](int r) {
      const float* at = A.st1 + (int64_t)r * N + p;
      return kMayLead ? __ldcg(at) : *at;
    };
#pragma unroll
    for (int a = 0; a < D; ++a) {
      x[a] = row(R::X + a);
      v[a] = row(R::V + a);
    }
#pragma unroll
    for (int i = 0; i < D * D; ++i) {
      E[i / D][i % D] = row(R::F + i) - (i / D == i % D ? P.f_diag : 0.0f);
      C1[i / D][i % D] = row(R::C + i);
    }
    const float mu = A.mu[p], la = A.la[p];
    ok = make_axes<D>(x, P, s) && active;
    if (active && !ok) err |= kErrOOB;
    if (early) stage_wait<0>();  // this thread's group
    else stage_wait<3>();
    grp = staged_group(P, stage, Stage<D>::kAdj - 1);
    act = particle_act(P, P.basis, grp, A.wact, scene, D, axis);
    float tau[D][D];
    if (MAT == kMixed) mat_p = A.matid[p];
    if (!kirchhoff<D, MAT>(E, mu, la, act, axis, tau, sc, A.R1, N, p, mat_p) && ok) {
      err |= kErrNonFinite;
      ok = false;
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
      mv[i] = P.p_mass * v[i];
#pragma unroll
      for (int j = 0; j < D; ++j) Am[i][j] = P.kappa * tau[i][j] + P.p_mass * C1[i][j];
    }
    if (early) {
      pass_wait();
      stage_rest();
      if (!kLate) load_carried();
    }
  }
  if (MODE == kAdjG2P) {
#pragma unroll
    for (int a = 0; a < D; ++a) vb[a] = A.adj[(R::V + a) * N + p];
#pragma unroll
    for (int i = 0; i < D * D; ++i) Cb[i / D][i % D] = A.adj[(R::C + i) * N + p];
    if (A.sense_add) {
      stage_wait<2>();
      const int grp = staged_group(P, stage, Stage<D>::kAdj - 1);
      const float* add = A.sense_add + ((int64_t)scene * (P.n_groups + 1) + ((grp >= 0 && grp < P.n_groups) ? grp + 1 : 0)) * 2 * D;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        xb[a] += add[a];
        vb[a] += add[D + a];
      }
    }
  } else {
    // ---- P2G adjoint of step s+1: gather (pbar, mbar) = grid_op.grad(ubar, (m, p)) ----
    float Ab[D][D], xg[D], sw[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      vb[a] = 0.0f;
      xg[a] = 0.0f;
      sw[a] = 0.0f;
#pragma unroll
      for (int b = 0; b < D; ++b) Ab[a][b] = 0.0f;
    }
    const float4* UBg = scene_grid(A.UB1, scene, P);
    const float4* PMg = scene_grid(A.PM1, scene, P);
    auto raw = [&](int f) { return NodePair{ub_load<DET>(UBg, f, P, A.ub_m0), pm_load<DET>(PMg, f, P)}; };
    auto pbar = [&](const NodePair& g, bool wall) { return node_adjoint<D>(g.ub, g.pm, wall, P); };
    BoxInfo<D> gbx;
    gbx.use_tile = false;
    if (P.gather_capacity > 0) {
      gbx = box_extent<D>(ok, s.base, P.gather_capacity, sh.gather[0]);
      stage_wait<2>();  // this thread's share of the clear boxes, before the box's barrier
      box_load<D, 2>(gbx, reinterpret_cast<float4*>(sm), P, raw, pbar);
    } else {
      stage_wait<2>();
      __syncthreads();
    }
    run_clears<D>(A.clears, sh.clear_box, scene, tile.w, nranks, P.nnodes, n);
    if (ok) with_nodes<D>(gbx, reinterpret_cast<const float4*>(sm), s.base, P, raw, pbar, [&](auto load) {
      // pbar - pbar_c and mbar - mbar_c (centre node) in the moment and weight-gradient
      // terms: equal to the plain sums because sum W dpos = 0, sum grad W = 0 and
      // sum grad W dpos^T = I, without the FP32 cancellation of a smooth pbar field
      const float4 gc = load(1, 1, D == 3 ? 1 : 0);
      const float pc[3] = {gc.x, gc.y, gc.z};
      GatherAxes<D> ga(s);
      if constexpr (D == 3) {
        constexpr int Z = D - 1;
        // pairs: components (0, 1) and (2, mass)
        const F2 nc = f2(-gc.x, -gc.y), ncm = f2(-gc.z, -gc.w), z2 = f2(0.0f);
        const F2 A0 = f2(Am[0][0], Am[1][0]), A1 = f2(Am[0][1], Am[1][1]), A2 = f2(Am[0][Z], Am[1][Z]);
        F2 sw01 = z2, Ab0 = z2, Ab1 = z2, Ab2 = z2;
        float swz = 0.0f, Ab0z = 0.0f, Ab1z = 0.0f, Ab2z = 0.0f;
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {
          float wi, dwi, dpi;
          axis_at(i, s.f[0], P.dx, wi, dwi, dpi);
          const F2 qi = f2_fma(A0, f2(dpi), f2(mv[0], mv[1]));
          const float qiz = mv[Z] + Am[Z][0] * dpi;
          F2 t = z2, t1 = z2, t2 = z2;
          float tz = 0.0f, t1z = 0.0f, t2z = 0.0f, e[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const F2 qij = f2_fma(A1, f2(s.dp[1][j]), qi);
            const float qijz = qiz + Am[Z][1] * s.dp[1][j];
            F2 r = z2, rb = z2;
            float rz = 0.0f, rbz = 0.0f, e0 = 0.0f, e1 = 0.0f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const float4 g4 = load(i, j, k);
              const F2 d = f2_add(f2(g4.x, g4.y), nc), dm = f2_add(f2(g4.z, g4.w), ncm);
              const F2 q = f2_fma(A2, f2(s.dp[Z][k]), qij);
              const F2 m = f2_fma(dm, f2(qijz + Am[Z][Z] * s.dp[Z][k], P.p_mass), f2_mul(d, q));
              const float Wbar = f2_lo(m) + f2_hi(m), dz = f2_lo(dm);
              r = f2_fma(f2(s.w[Z][k]), d, r);
              rb = f2_fma(f2(ga.wp[Z][k]), d, rb);
              rz += s.w[Z][k] * dz;
              rbz += ga.wp[Z][k] * dz;
              e0 += s.w[Z][k] * Wbar;
              e1 += s.dw[Z][k] * Wbar;
            }
            const F2 w1 = f2(s.w[1][j]);
            t = f2_fma(w1, r, t);
            t1 = f2_fma(f2(ga.wp[1][j]), r, t1);
            t2 = f2_fma(w1, rb, t2);
            tz += s.w[1][j] * rz;
            t1z += ga.wp[1][j] * rz;
            t2z += s.w[1][j] * rbz;
            e[0] += s.w[1][j] * e0;
            e[1] += s.dw[1][j] * e0;
            e[2] += s.w[1][j] * e1;
          }
          const float wpi = wi * dpi;
          const F2 w0 = f2(wi);
          sw01 = f2_fma(w0, t, sw01);
          Ab0 = f2_fma(f2(wpi), t, Ab0);
          Ab1 = f2_fma(w0, t1, Ab1);
          Ab2 = f2_fma(w0, t2, Ab2);
          swz += wi * tz;
          Ab0z += wpi * tz;
          Ab1z += wi * t1z;
          Ab2z += wi * t2z;
          xg[0] += dwi * e[0];
          xg[1] += wi * e[1];
          xg[Z] += wi * e[2];
        }
        sw[0] = f2_lo(sw01);
        sw[1] = f2_hi(sw01);
        sw[Z] = swz;
        Ab[0][0] = f2_lo(Ab0);
        Ab[1][0] = f2_hi(Ab0);
        Ab[Z][0] = Ab0z;
        Ab[0][1] = f2_lo(Ab1);
        Ab[1][1] = f2_hi(Ab1);
        Ab[Z][1] = Ab1z;
        Ab[0][Z] = f2_lo(Ab2);
        Ab[1][Z] = f2_hi(Ab2);
        Ab[Z][Z] = Ab2z;
      } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float wi, dwi, dpi, qi[D], t[D], tb[D][D], e[D];
        axis_at(i, s.f[0], P.dx, wi, dwi, dpi);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          qi[c] = mv[c] + Am[c][0] * dpi;
          t[c] = e[c] = 0.0f;  // e[b]: sum of W-bar times the weight, differentiated along b >= 1
#pragma unroll
          for (int b = 1; b < D; ++b) tb[c][b] = 0.0f;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          float qij[D], r[D], rb[D], e0 = 0.0f, e1 = 0.0f;
#pragma unroll
          for (int c = 0; c < D; ++c) {
            qij[c] = qi[c] + Am[c][1] * s.dp[1][j];
            r[c] = rb[c] = 0.0f;
          }
#pragma unroll
          for (int k = 0; k < (D == 3 ? 3 : 1); ++k) {
            const float4 g4 = load(i, j, k);
            const float pb[3] = {g4.x, g4.y, g4.z};
            float Wbar = P.p_mass * (g4.w - gc.w);
#pragma unroll
            for (int c = 0; c < D; ++c) {
              const float d = pb[c] - pc[c];
              Wbar += d * (D == 3 ? qij[c] + Am[c][D - 1] * s.dp[D - 1][k] : qij[c]);
              if (D == 3) {
                r[c] += s.w[D - 1][k] * d;
                rb[c] += ga.wp[D - 1][k] * d;
              } else {
                r[c] = d;
              }
            }
            if (D == 3) {
              e0 += s.w[D - 1][k] * Wbar;
              e1 += s.dw[D - 1][k] * Wbar;
            } else {
              e0 = Wbar;
            }
          }
#pragma unroll
          for (int c = 0; c < D; ++c) {
            t[c] += s.w[1][j] * r[c];
            tb[c][1] += ga.wp[1][j] * r[c];
            if (D == 3) tb[c][D - 1] += s.w[1][j] * rb[c];
          }
          e[0] += s.w[1][j] * e0;
          e[1] += s.dw[1][j] * e0;
          if (D == 3) e[D - 1] += s.w[1][j] * e1;
        }
        const float wpi = wi * dpi;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          sw[c] += wi * t[c];
          Ab[c][0] += wpi * t[c];
#pragma unroll
          for (int b = 1; b < D; ++b) Ab[c][b] += wi * tb[c][b];
        }
        xg[0] += dwi * e[0];
#pragma unroll
        for (int b = 1; b < D; ++b) xg[b] += wi * e[b];
      }
      }
#pragma unroll
      for (int c = 0; c < D; ++c) vb[c] = pc[c] + sw[c];  // sum W = 1
    });
    if (kLate) load_carried();
    // x += inv_dx sum Wbar gradW - A^T sum W dpbar
#pragma unroll
    for (int b = 0; b < D; ++b) {
      float atw = 0.0f;
#pragma unroll
      for (int a = 0; a < D; ++a) atw += Am[a][b] * sw[a];
      xb[b] += P.inv_dx * xg[b] - atw;
      vb[b] *= P.p_mass;
    }
    float tb[D][D];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) {
        Cb[i][j] = P.p_mass * Ab[i][j];
        tb[i][j] = P.kappa * Ab[i][j];
      }
    float mub = 0.0f, lab = 0.0f, abar = 0.0f;
    if (kLate) load_E<D>(A.st1, N, p, P.f_diag, E);
    if (kLate && (MAT == kFixedCorotated || MAT == kMixed)) {
      // the polar factor again (from the cache, or recomputed where the state has no cached
      // factor: one adjoint pass per segment), so that it holds no registers across the
      // gather; the stress itself is not needed again
      float tau_again[D][D];
      kirchhoff<D, MAT>(E, A.mu[p], A.la[p], act, axis, tau_again, sc, A.R1, N, p, mat_p);
    }
    if (ok) abar = kirchhoff_adjoint<D, MAT>(E, A.mu[p], A.la[p], act, axis, sc, tb, Fb, mub, lab, mat_p);
    if (active) {
      float2 ms = carried ? staged_pair(stage, Stage<D>::kAdjB + kSums) : A.mubar[p];
      float2 ls = carried ? staged_pair(stage, Stage<D>::kAdjB + kSums + 2) : A.labar[p];
      compensated_add(ms, mub);
      compensated_add(ls, lab);
      A.mubar[p] = ms;
      A.labar[p] = ls;
    }
    if (P.n_groups > 0) {
      // dL/dw_gk += basis_k * sum of abar over this tile's particles of group g, reduced in
      // a fixed order (warp butterfly, then warps in order) into the tile's own slot, so
      // the result does not depend on scheduling; the tiles are summed in order at the end
      const int g = ok && grp < P.n_groups ? grp : -1;
      const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
      if (lane < kMaxGroups) s_wbar[warp * kMaxGroups + lane] = 0.0f;
      __syncwarp();
      unsigned left = __ballot_sync(0xffffffffu, g >= 0);
      while (left) {  // the groups of the warp's particles: usually one
        const int gg = __shfl_sync(0xffffffffu, g, __ffs(left) - 1);
        float v = (g == gg) ? abar : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) s_wbar[warp * kMaxGroups + gg] = v;
        left &= ~__ballot_sync(0xffffffffu, g == gg);
      }
      __syncthreads();
      const int GK = P.n_groups * P.n_basis;
      if ((int)threadIdx.x < GK) {
        const int gg = threadIdx.x / P.n_basis, k = threadIdx.x % P.n_basis;
        float sum = 0.0f;
        for (int w = 0; w < kTile / 32; ++w) sum += s_wbar[w * kMaxGroups + gg];
        // (the tile's own slot: a reduction only so that nothing waits for the value)
        atomicAdd(A.wbar_tile + (int64_t)tile_index * GK + threadIdx.x, sum * P.basis[k]);
      }
    }
    if (MODE == kAdjP2G) {
      if (active) {
#pragma unroll
        for (int a = 0; a < D; ++a) {
          A.adj[(R::X + a) * N + p] = xb[a];
          A.adj[(R::V + a) * N + p] = vb[a];
        }
#pragma unroll
        for (int i = 0; i < D * D; ++i) {
          A.adj[(R::C + i) * N + p] = Cb[i / D][i % D];
          A.adj[(R::F + i) * N + p] = Fb[i / D][i % D];
        }
      }
      if (err) atomicOr(A.err, err);
      return;
    }
  }

  if (OWN) pass_ready();
  // ---- G2P adjoint of step s: x' = x + dt v', E' = E + dt C' (I + E) ----
  {
    float x0[D], E0[D][D];
    stage_wait<0>();
#pragma unroll
    for (int a = 0; a < D; ++a) x0[a] = staged(stage, a);
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) E0[i][j] = staged(stage, D + i * D + j) - (i == j ? P.f_diag : 0.0f);
    float vt[D], Ct[D][D], Fb0[D][D], xb0[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      vt[a] = vb[a] + P.dt * xb[a];
      xb0[a] = xb[a];
    }
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) {
        float g = Fb[i][j], h = Cb[i][j] + P.dt * Fb[i][j];
#pragma unroll
        for (int k = 0; k < D; ++k) {
          g += P.dt * C1[k][i] * Fb[k][j];  // (I + dt C')^T Fbar'
          h += P.dt * Fb[i][k] * E0[j][k];  // Cbar' + dt Fbar' (I + E)^T
        }
        Fb0[i][j] = g;
        Ct[i][j] = h;
      }
    Axes<D> s;
    const bool ok = make_axes<D>(x0, P, s) && active;
    if (active && !ok) err |= kErrOOB;
    if (MODE == kAdjG2P && DET && A.measure) {
      // bound of this particle's ubar contributions W (vt + c4 Ct dpos), W <= 1, |dpos| <= 1.5 dx
      float bound = 0.0f;
      if (ok) {
#pragma unroll
        for (int a = 0; a < D; ++a) {
          float r = fabsf(vt[a]);
#pragma unroll
          for (int b = 0; b < D; ++b) r += 1.5f * P.dx * c4 * fabsf(Ct[a][b]);
          bound = fmaxf(bound, r);
        }
        if (!(bound <= 3.0e38f)) {
          err |= kErrNonFinite;
          bound = 0.0f;
        }
      }
      // non-negative floats order like their bit patterns
      const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(bound));
      if ((threadIdx.x & 31) == 0 && mb != 0u) atomicMax(A.ub_m0, mb);
      if (err) atomicOr(A.err, err);
      __syncthreads();
      run_clears<D>(A.clears, sh.clear_box, scene, tile.w, nranks, P.nnodes, n);
      return;
    }
    const float4* PMg = scene_grid(A.PM0, scene, P);
    auto raw = [&](int f) { return pm_load<DET>(PMg, f, P); };
    auto velocity = [&](float4 pm, bool wall) { return node_velocity<D>(pm, wall, P); };
    BoxInfo<D> gbx;
    gbx.use_tile = false;
    if (P.gather_capacity > 0) {
      gbx = box_extent<D>(ok, s.base, P.gather_capacity, sh.gather[1]);
      box_load<D, kBatch>(gbx, reinterpret_cast<float4*>(sm), P, raw, velocity);
    } else if (MODE == kAdjG2P) {
      __syncthreads();
    }
    if (MODE == kAdjG2P) run_clears<D>(A.clears, sh.clear_box, scene, tile.w, nranks, P.nnodes, n);
    if (ok) with_nodes<D>(gbx, reinterpret_cast<const float4*>(sm), s.base, P, raw, velocity, [&](auto load) {
      // x-adjoint terms on u - u_c (centre node), by the same B-spline identities
      const float4 uc4 = load(1, 1, D == 3 ? 1 : 0);
      const float uc[3] = {uc4.x, uc4.y, uc4.z};
      float xg[D], sw[D];
#pragma unroll
      for (int a = 0; a < D; ++a) xg[a] = sw[a] = 0.0f;
      if constexpr (D == 3) {
        constexpr int Z = D - 1;
        const F2 nc = f2(-uc[0], -uc[1]), z2 = f2(0.0f);
        const F2 A0 = f2(c4 * Ct[0][0], c4 * Ct[1][0]), A1 = f2(c4 * Ct[0][1], c4 * Ct[1][1]), A2 = f2(c4 * Ct[0][Z], c4 * Ct[1][Z]);
        F2 sw01 = z2;
        float swz = 0.0f;
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {
          float wi, dwi, dpi;
          axis_at(i, s.f[0], P.dx, wi, dwi, dpi);
          const F2 qi = f2_fma(A0, f2(dpi), f2(vt[0], vt[1]));
          const float qiz = vt[Z] + c4 * Ct[Z][0] * dpi;
          F2 t = z2;
          float tz = 0.0f, e[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const F2 qij = f2_fma(A1, f2(s.dp[1][j]), qi);
            const float qijz = qiz + c4 * Ct[Z][1] * s.dp[1][j];
            F2 r = z2;
            float rz = 0.0f, e0 = 0.0f, e1 = 0.0f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const float4 u4 = load(i, j, k);
              const F2 d = f2_add(f2(u4.x, u4.y), nc);
              const float dz = u4.z - uc[2];
              const F2 m = f2_mul(d, f2_fma(A2, f2(s.dp[Z][k]), qij));
              const float Wbar = dz * (qijz + c4 * Ct[Z][Z] * s.dp[Z][k]) + (f2_lo(m) + f2_hi(m));
              r = f2_fma(f2(s.w[Z][k]), d, r);
              rz += s.w[Z][k] * dz;
              e0 += s.w[Z][k] * Wbar;
              e1 += s.dw[Z][k] * Wbar;
            }
            t = f2_fma(f2(s.w[1][j]), r, t);
            tz += s.w[1][j] * rz;
            e[0] += s.w[1][j] * e0;
            e[1] += s.dw[1][j] * e0;
            e[2] += s.w[1][j] * e1;
          }
          sw01 = f2_fma(f2(wi), t, sw01);
          swz += wi * tz;
          xg[0] += dwi * e[0];
          xg[1] += wi * e[1];
          xg[Z] += wi * e[2];
        }
        sw[0] = f2_lo(sw01);
        sw[1] = f2_hi(sw01);
        sw[Z] = swz;
      } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float wi, dwi, dpi, qi[D], t[D], e[D];
        axis_at(i, s.f[0], P.dx, wi, dwi, dpi);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          qi[c] = vt[c] + c4 * Ct[c][0] * dpi;
          t[c] = e[c] = 0.0f;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          float qij[D], r[D], e0 = 0.0f, e1 = 0.0f;
#pragma unroll
          for (int c = 0; c < D; ++c) {
            qij[c] = qi[c] + c4 * Ct[c][1] * s.dp[1][j];
            r[c] = 0.0f;
          }
#pragma unroll
          for (int k = 0; k < (D == 3 ? 3 : 1); ++k) {
            const float4 u4 = load(i, j, k);
            const float u[3] = {u4.x, u4.y, u4.z};
            float Wbar = 0.0f;
#pragma unroll
            for (int c = 0; c < D; ++c) {
              const float d = u[c] - uc[c];
              Wbar += d * (D == 3 ? qij[c] + c4 * Ct[c][D - 1] * s.dp[D - 1][k] : qij[c]);
              r[c] = D == 3 ? r[c] + s.w[D - 1][k] * d : d;
            }
            if (D == 3) {
              e0 += s.w[D - 1][k] * Wbar;
              e1 += s.dw[D - 1][k] * Wbar;
            } else {
              e0 = Wbar;
            }
          }
#pragma unroll
          for (int c = 0; c < D; ++c) t[c] += s.w[1][j] * r[c];
          e[0] += s.w[1][j] * e0;
          e[1] += s.dw[1][j] * e0;
          if (D == 3) e[D - 1] += s.w[1][j] * e1;
        }
#pragma unroll
        for (int c = 0; c < D; ++c) sw[c] += wi * t[c];
        xg[0] += dwi * e[0];
#pragma unroll
        for (int b = 1; b < D; ++b) xg[b] += wi * e[b];
      }
      }
#pragma unroll
      for (int b = 0; b < D; ++b) {
        float ctu = 0.0f;
#pragma unroll
        for (int a = 0; a < D; ++a) ctu += Ct[a][b] * sw[a];
        xb0[b] += P.inv_dx * xg[b] - c4 * ctu;
      }
    });
    if (active) {
#pragma unroll
      for (int a = 0; a < D; ++a) A.adj[(R::X + a) * N + p] = xb0[a];
#pragma unroll
      for (int i = 0; i < D * D; ++i) A.adj[(R::F + i) * N + p] = Fb0[i / D][i % D];
    }
    // ---- scatter ubar_i += W (vt + c4 Ct dpos) ----
    float Bs[D][D];
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) Bs[i][j] = c4 * Ct[i][j];
    float4* UBs = scene_grid(A.UB0, scene, P);
    float fix_u = 1.0f, unfix_u = 1.0f;
    if (DET) ub_scales(A.ub_m0, fix_u, unfix_u);
    put_record<D>(rec, ok, s, vt, Bs, P.dx);
    warp_bounds<D>(ok, s.base, sh.scatter[0]);
    __syncwarp();
    scatter_runs<D, false, DET>(rec, UBs, n, 0.0f, fix_u, fix_u, err);
    __syncthreads();  // every warp's share of the box
    cta_bbox_flush<D>(sh.scatter[0], A.box_ub + scene * 8, seen_ub);
  }

  // ---- recomputed P2G of step s-1 (the grid of the next adjoint pass) ----
  if (A.stm) {
    float x[D], v[D], C[D][D], E[D][D];
    stage_wait<0>();
    constexpr int b = Stage<D>::kAdjB;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      x[a] = staged(stage, b + R::X + a);
      v[a] = staged(stage, b + R::V + a);
    }
#pragma unroll
    for (int i = 0; i < D * D; ++i) C[i / D][i % D] = staged(stage, b + R::C + i);
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) E[i][j] = staged(stage, b + R::F + i * D + j) - (i == j ? P.f_diag : 0.0f);
    p2g_pass<D, MAT, DET>(P, P.basis2, active, scene, p, staged_group(P, stage, Stage<D>::kAdj - 1), x, v, C, E,
                          staged(stage, b + R::Q), staged(stage, b + R::Q + 1), MAT == kMixed ? A.matid[p] : MAT, A.wact,
                          scene_grid(A.PMm, scene, P), A.box_m + scene * 8, rec, sh.scatter[1], seen_m, err, A.Rm, nullptr, N);
  }
  if (err) atomicOr(A.err, err);
}

template <int D, int MAT, int MODE, bool DET>
__global__ void __launch_bounds__(kTile, adj_ctas_per_sm<D>())
    adjoint_kernel(const __grid_constant__ SimParams P, const __grid_constant__ AdjArgs A) {
  extern __shared__ __align__(16) float sm[];
  __shared__ TileShared sh;
  __shared__ float s_wbar[kWbarSlots];
  adjoint_tile<D, MAT, MODE, true, DET>(P, A, blockIdx.x, sm, sh, s_wbar);
}

// ---------------------------------------------------------------------------
// persistent launches: one co-resident (cooperative) grid runs a list of passes of one
// kind with a grid-wide barrier between consecutive passes.  The list is recorded on the
// host by the same code that issues the one-launch-per-pass form, so the two run the
// same passes on the same buffers in the same order.
// ---------------------------------------------------------------------------
enum PassKind : int { kPassStep = 0, kPassAdjoint = 1 };

struct __align__(16) PassEntry {
  int kind;  // PassKind
  int mode;  // StepMode or AdjMode
  int pad[2];
  SimParams P;
  StepArgs S;  // kPassStep
  AdjArgs A;   // kPassAdjoint
};

struct GridSync {
  unsigned arrived;  // CTA arrivals at the barriers of this launch (reset before it)
  unsigned abort;    // set by a CTA whose wait ran out; every CTA then leaves
};

struct PersistCtl {
  GridSync* sync;
  unsigned* tickets;     // [n_pass] tile tickets (reset before the launch)
  unsigned* err;
  long long timeout_ns;  // limit of one barrier wait
  unsigned extra;        // arrivals a barrier waits for beyond the grid's own (0; a nonzero
                         // value makes every wait run out: the timeout path's test hook)
};

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ld_relaxed_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid-wide barrier: returns when `target` arrivals have been counted, or false when the
// wait ran out (err |= kErrTimeout, abort raised) or another CTA aborted.  The wait is
// bounded twice: by the global nanosecond timer and by the SM cycle counter (4 cycles per
// ns of limit, at least twice the limit at any SM clock up to 2 GHz), so it ends even if
// one of the two clocks stalls.
__device__ __forceinline__ bool grid_barrier(const PersistCtl& c, unsigned target, int* s_go) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();  // this CTA's grid and state writes before its arrival
    atomicAdd(&c.sync->arrived, 1u);
    int go = 1;
    const unsigned long long t0 = globaltimer_ns();
    const long long c0 = clock64();
    const long long cycle_limit = 4 * c.timeout_ns;
    for (unsigned it = 1;; ++it) {
      if (ld_acquire_gpu(&c.sync->arrived) >= target) break;
      if (ld_relaxed_gpu(&c.sync->abort)) {
        go = 0;
        break;
      }
      if ((it & 15u) == 0 && ((long long)(globaltimer_ns() - t0) > c.timeout_ns ||
                              clock64() - c0 > cycle_limit)) {
        atomicExch(&c.sync->abort, 1u);
        atomicOr(c.err, kErrTimeout);
        go = 0;
        break;
      }
      __nanosleep(128);
    }
    __threadfence();
    *s_go = go;
  }
  __syncthreads();
  return *s_go != 0;
}

// Copy a 16-byte-multiple object to shared memory with the whole CTA (no barrier).
template <typename T>
__device__ __forceinline__ void cta_copy(T* dst, const T* src) {
  static_assert(sizeof(T) % 16 == 0, "16-byte multiple");
  const int4* s4 = reinterpret_cast<const int4*>(src);
  int4* d4 = reinterpret_cast<int4*>(dst);
  for (int i = threadIdx.x; i < (int)(sizeof(T) / 16); i += blockDim.x) d4[i] = s4[i];
}

// Next tile of pass i for this CTA (tickets in tile order, so tiles are taken in the order
// the hardware would dispatch one CTA per tile, and a CTA that finishes early takes more);
// a value >= n_tiles ends the pass.  Synchronises the CTA.
__device__ __forceinline__ int next_tile(const PersistCtl& c, int i, int* s_tile) {
  if (threadIdx.x == 0) *s_tile = (int)atomicAdd(&c.tickets[i], 1u);
  __syncthreads();
  return *s_tile;
}

// Forward-kind passes plan[0..n_pass), all of pass mode MODE (the launcher splits runs at
// mode changes, so each interpreter compiles one pass body, as the one-launch-per-pass kernel
// does), tiles handed out by tickets.
template <int D, int MAT, int MODE, bool DET>
__global__ void __launch_bounds__(kTile, step_ctas_per_sm<D, MAT>())
    step_persistent_kernel(const PassEntry* plan, int n_pass, int n_tiles, PersistCtl ctl) {
  extern __shared__ __align__(16) float sm[];
  __shared__ TileShared sh;
  __shared__ int s_go, s_tile;
  __shared__ PassEntry e;
  // a barrier of an earlier launch of this sequence gave up: its passes never finished, so
  // this launch would only run on an incomplete state
  if (*(volatile unsigned*)ctl.err & kErrTimeout) return;
  for (int i = 0; i < n_pass; ++i) {
    if (i > 0 && !grid_barrier(ctl, (unsigned)i * gridDim.x + ctl.extra, &s_go)) return;
    __syncthreads();
    cta_copy(&e, plan + i);
    for (int t; (t = next_tile(ctl, i, &s_tile)) < n_tiles;) {
      step_tile<D, MAT, MODE, false, DET>(e.P, e.S, t, sm, sh);
      __syncthreads();
    }
  }
}

// Adjoint-kind passes plan[0..n_pass), all of mode MODE.
template <int D, int MAT, int MODE, bool DET>
__global__ void __launch_bounds__(kTile, adj_ctas_per_sm<D>())
    adjoint_persistent_kernel(const PassEntry* plan, int n_pass, int n_tiles, PersistCtl ctl) {
  extern __shared__ __align__(16) float sm[];
  __shared__ TileShared sh;
  __shared__ float s_wbar[kWbarSlots];
  __shared__ int s_go, s_tile;
  __shared__ PassEntry e;
  // a barrier of an earlier launch of this sequence gave up: its passes never finished, so
  // this launch would only run on an incomplete state
  if (*(volatile unsigned*)ctl.err & kErrTimeout) return;
  for (int i = 0; i < n_pass; ++i) {
    if (i > 0 && !grid_barrier(ctl, (unsigned)i * gridDim.x + ctl.extra, &s_go)) return;
    __syncthreads();
    cta_copy(&e, plan + i);
    for (int t; (t = next_tile(ctl, i, &s_tile)) < n_tiles;) {
      adjoint_tile<D, MAT, MODE, false, DET>(e.P, e.A, t, sm, sh, s_wbar);
      __syncthreads();
    }
  }
}

// Zero the dirty boxes of the clear jobs (end of a launch sequence); blockIdx.y = scene.
template <int D>
__global__ void clear_kernel(const __grid_constant__ Clears C, int nnodes, int n) {
  __shared__ int boxes[8 * kMaxClears];
  if ((int)threadIdx.x < 8 * C.n) boxes[threadIdx.x] = C.job[threadIdx.x >> 3].box[blockIdx.y * 8 + (threadIdx.x & 7)];
  __syncthreads();
  run_clears<D>(C, boxes, blockIdx.y, blockIdx.x, gridDim.x, nnodes, n);
}

// The same for a run of buffers (blockIdx.z), grid_stride float4s and box_stride ints apart.
template <int D>
__global__ void clear_run_kernel(int words, float4* grid, int64_t grid_stride, const int* box, int box_stride, int nnodes,
                                 int n) {
  __shared__ int boxes[8];
  Clears C;
  C.n = 1;
  C.words = words;
  C.job[0].grid = grid + blockIdx.z * grid_stride;
  if (threadIdx.x < 8) boxes[threadIdx.x] = box[(int64_t)blockIdx.z * box_stride + blockIdx.y * 8 + threadIdx.x];
  __syncthreads();
  run_clears<D>(C, boxes, blockIdx.y, blockIdx.x, gridDim.x, nnodes, n);
}

}  // namespace mpm
