// CUDA kernels of the wavelet-domain MAP tomography solve (sm_103a).
//
// Per PCG iteration (Sec. 5.1 of the paper) four launches cover the operator
// (W P^T Gamma^T C^-1 Gamma P W^-1 + alpha D) p and the (P)CG vector updates:
//
//   k_synthesis  beta from the r.z partials, p <- J^-1 r + beta p,
//                phi = W^-1 p                                    [cluster per layer]
//   k_forward    psi = P phi on sensor corners, Fried slopes,
//                C^-1 weighting, Gamma^T; tip/tilt sums          [tile per sensor]
//   k_analysis   g = sum_m P_m^T v_m (gather + pupil-edge list),
//                q = W g + alpha D p, p.q partials               [cluster per layer]
//   k_update     alpha from the p.q partials, x += alpha p,
//                r -= alpha q, r.J^-1 r partials                 [chunk per CTA]
//
// The periodic 2-D DWT of one layer runs inside one thread-block cluster: CTA c
// owns N/C consecutive rows; the row pass is local, and before the column pass
// each CTA copies the Lf-2 halo rows it needs from its neighbours' shared memory
// (distributed shared memory) next to its own rows.  The coarse levels (from a
// block of transform_coarse_side on) are finished by CTA 0 alone.  Each CTA loads every coefficient it
// owns in one round trip at its start (with the PCG direction update fused in).
//
// Reductions are FP64: warp shuffle -> block -> one partial per CTA; the
// consumer kernel (every CTA of it) sums the producer's partials in a fixed
// order, so no kernel waits on a "last CTA" and results do not depend on
// scheduling.  Kernels are launched with programmatic dependent launch: each
// triggers its dependents at entry and waits (griddepcontrol.wait) only before
// touching data the previous kernel wrote.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "common.h"
#include "device_util.cuh"
#include "launch.h"
#include "transform.cuh"
#include "adjoint.cuh"

namespace cg = cooperative_groups;

namespace tomo {

// ------------------------------------------------------------------ helpers

// The two halves of a cluster barrier (cluster.sync() is both): every thread
// of every CTA in the cluster alternates arrive and wait.  arrive releases the
// thread's earlier shared-memory accesses (including reads of other CTAs'
// shared memory); wait returns once all threads of the cluster have arrived.
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// A forward tile's two partial sums in its 16-byte partial slot: doubles for
// FP64 plans, double-float pairs (hi, lo, hi, lo) for FP32 plans.
__device__ __forceinline__ void store_tile_partial(double *slot, Acc<double> a, Acc<double> b) {
  const double2 s = block_sum2(a, b);
  if (threadIdx.x == 0) *reinterpret_cast<double2 *>(slot) = s;
}
__device__ __forceinline__ void store_tile_partial(double *slot, Acc<float> a, Acc<float> b) {
  const float4 s = block_sum2_df(a, b);
  if (threadIdx.x == 0) *reinterpret_cast<float4 *>(slot) = s;
}


// ------------------------------------------------------------ k_forward
// MODE 0: operator, z = Gamma P phi.  MODE 1: residual, z = s - Gamma P phi.
// MODE 2: data only, z = s (phi = 0).  MODE 3: the noise-free measurement A phi
// itself (eq. atm_tomo) into io.out0: the slopes, and a tip/tilt-only sensor's
// two means (by its first chunk's CTA alone); nothing of the plan is written.
// Otherwise writes the corner field
// v_m = Gamma_m^T sigma^-2 z_m and, with tip/tilt removal, each tile's sums of z
// (the analysis subtracts the means on the pupil edge, Sec. 4.3 eq. widehatc).
// A tip/tilt-only sensor writes its weighted mean slopes (e_x, e_y).
// io.in0: layer grids (NULL = the plan's phi); io.in1: slopes (MODE 1, 2).
// EL: some sensor of the launch has elongated spots (Sec. 4.3); without it the
// elongation code is compiled out.
//
// A tile is kFwdCols x kFwdRows corners of a sensor.  The ray-trace covers the
// tile and a halo of one corner, kFwdLanes columns (one per lane) by kFwdPsi
// rows, RS consecutive rows per warp.  Down a column the corners' traced rows
// follow each other on the layer grid, mostly one node row apart or, under the
// cone effect, in the same one, so the interpolation along x of a node row is
// formed once for the corner rows above and below it: RS + 1 node rows are read
// per layer instead of 2 RS, all requested before any is used.
//
// RS = kFwdStrip (4, FP64 2: kFwdThreads threads) for big launches, RS = 1 (a warp
// per row, no reuse, less work in a chain) for small ones.  The steps that feed
// the tile's partial sums (the slopes' sums and the tip/tilt-only chunks) keep a
// fixed kFwdThreads-thread mapping, so the partials, and every result, are
// bitwise the same at either block size.  In a small launch without elongated
// spots the slopes themselves are formed by every warp, a row each, and taken to
// the four summing warps through shared memory (with elongated spots, whose
// sums are four, that costs more than it saves: 114 x 114, one layer, 22.8 ->
// 23.6 us an operator); the loop over the layers and the pairs of a tip/tilt-only
// chunk hold no branch, so all their loads are in flight at once, and a last
// layer alone is not padded to a batch of four (E-ELT solve 409 -> 403 us).
// Normal operator of one system (GB300, us): four warps forming the slopes, a
// break after the last layer and a branch per pair 20.0, this form 19.1 (9 layers
// of 64 x 64, 9 sensors); 19.7 and 18.7 (7 layers, 7 sensors); 17.7 and 16.8 (8
// layers of 32 x 32, 6 sensors).
//
// Bound by the latency of its grid loads (16 E-ELT systems: SM at 45%, L1 at 49% of their
// peaks; of the reasons a warp waits, the loads are the first).
// Against one corner per thread on 18 x 18 corners, four loads per corner and
// layer (GB300, cold launch): 16 E-ELT systems 49.2 -> 29 us, 64 uneven systems
// 50.9 -> 29 us, the 100 m system 54.0 -> 43 us.
// What a small launch asks of an SM.  The kernels of a frame overlap by programmatic launch: an
// analysis CTA (up to 108 KB) can start beside the forward CTAs only if the SM's split between L1
// and shared memory holds both.  A forward CTA alone (about 14 KB) asks for a small split; small
// launches ask for 72% (164 KB, which leaves 64 KB of L1).  59 systems of 9 to 120 subapertures,
// FP32, geometric means of the time (GB300) against 64 KB of unused shared memory per CTA and the
// driver's split, normal operator and solve of 10 iterations: 50% 1.003 and 0.996, 72% 0.992 and
// 0.993, 86% 0.999 and 0.997; neither 0.999 and 1.001.
// Where an analysis CTA takes 64 KB itself, so that where it starts matters more, each forward CTA
// takes 64 KB as well (at 72%, us without and with: 67 x 67, 3 layers 36.1 and 32.6 an operator;
// 104 x 104, 5 layers 26.6 and 26.2, and 399 and 390 a solve; E-ELT 31.9 and 31.7; smaller analysis
// CTAs lose: 82 x 82, 1 layer 300 and 314 a solve, 64 x 64, 5 layers 274 and 292).
constexpr int kFwdCarveout = 72;
constexpr size_t kFwdBesideSmem = 64 * 1024;
// FP64: an SM's FP64 pipe is slow enough that CTAs sharing an SM while others are idle cost more
// than anything, so a launch of up to one and a half CTAs per SM of 152 asks for 100 KB each: one
// forward CTA per SM.  Normal operator (us, without and with): 4 sensors of 88 x 88 (180 CTAs) 77
// and 59, 6 of 60 x 60 (200) 108 and 104, 6 of 31 x 31 57 and 44; 6 of 84 x 84 (300 CTAs) would
// go from 122 to 126.
constexpr size_t kFwdAloneSmem = 100 * 1024;
constexpr int kFwdAloneLaunch = 228;
constexpr int kFwdLanes = kFwdCols + 2;
template <typename T>
constexpr int kFwdRows = fwd_rows(sizeof(T) == 8);
template <typename T>
constexpr int kFwdPsi = kFwdRows<T> + 2;
// rows per warp of big launches (kFwdThreads threads)
template <typename T>
constexpr int kFwdStrip = kFwdPsi<T> * 32 / kFwdThreads;

// Shared memory of the staged corner tables of L layers: per layer the grid
// side and offset, the columns' node index and fraction, and per corner row
// (first node row, fraction).  Copied asynchronously: one memory latency for
// all of them, however many layers there are.
template <typename T>
struct FwdRow {
  int y0;
  T f;
};
template <typename T>
__host__ __device__ constexpr size_t fwd_table_bytes(int L) {
  return L * (kFwdPsi<T> * sizeof(FwdRow<T>) + kFwdLanes * sizeof(T) + (kFwdLanes + 2) * sizeof(int)) + 16;
}

__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// (1 - f) a + f b, rounded the same way wherever it is used.
__device__ __forceinline__ float lerp(float f, float a, float b) {
  return __fmaf_rn(__fsub_rn(1.f, f), a, __fmul_rn(f, b));
}
__device__ __forceinline__ double lerp(double f, double a, double b) {
  return __fma_rn(__dsub_rn(1.0, f), a, __dmul_rn(f, b));
}

// The corners' phase psi = sum_l phi_l(traced corner) for RS rows from corner
// row w of the tile's psi rows, lane = column; layers in order.
template <typename T, int RS>
__device__ __forceinline__ void trace_strip(const T *__restrict__ phi, int L, int w, const int *s_N, const int *s_off,
                                            const int *s_x0, const T *s_fx, const FwdRow<T> *s_row, T (&val)[RS]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < RS; ++j) val[j] = T(0);
  if constexpr (RS == 1) {
    // NB layers from l0, their loads in flight together, the sums predicated rather than left by a break
    auto batch = [&](int l0, auto nb) {
      constexpr int NB = decltype(nb)::value;
      T v00[NB], v01[NB], v10[NB], v11[NB], fx[NB], fy[NB];
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        const int l = l0 + q < L ? l0 + q : L - 1;
        const int N = s_N[l], x0 = s_x0[l * kFwdLanes + lane];
        const FwdRow<T> row = s_row[l * kFwdPsi<T> + w];
        const int x1 = (x0 + 1) & (N - 1), y1 = (row.y0 + 1) & (N - 1);
        const T *p = phi + s_off[l];
        fx[q] = s_fx[l * kFwdLanes + lane];
        fy[q] = row.f;
        v00[q] = p[row.y0 * N + x0];
        v01[q] = p[row.y0 * N + x1];
        v10[q] = p[y1 * N + x0];
        v11[q] = p[y1 * N + x1];
      }
#pragma unroll
      for (int q = 0; q < NB; ++q)
        if (l0 + q < L) val[0] += lerp(fy[q], lerp(fx[q], v00[q], v01[q]), lerp(fx[q], v10[q], v11[q]));
    };
    int l0 = 0;
    for (; l0 + 1 < L; l0 += 4) batch(l0, std::integral_constant<int, 4>());
    if (l0 < L) batch(l0, std::integral_constant<int, 1>());   // (a last layer alone: no loads for padding)
    return;
  }
  // layers whose loads are in flight together
  constexpr int kBatch = 2;
  for (int l0 = 0; l0 < L; l0 += kBatch) {
    T v0[kBatch][RS + 1], v1[kBatch][RS + 1], fx[kBatch], fy[kBatch][RS];
    int r0[kBatch][RS];
    bool odd = false;
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int l = l0 + q < L ? l0 + q : L - 1;
      const int N = s_N[l], x0 = s_x0[l * kFwdLanes + lane];
      fx[q] = s_fx[l * kFwdLanes + lane];
      const int mask = N * N - 1;
      const int lgN = 31 - __clz(N);
      const T *p0 = phi + s_off[l] + x0, *p1 = phi + s_off[l] + ((x0 + 1) & (N - 1));
      int last = 0;
#pragma unroll
      for (int j = 0; j < RS; ++j) {
        const FwdRow<T> row = s_row[l * kFwdPsi<T> + w + j];
        const int rj = row.y0 << lgN, r1 = (rj + N) & mask;
        r0[q][j] = rj;
        fy[q][j] = row.f;
        if (j == 0) {
          v0[q][0] = p0[rj];
          v1[q][0] = p1[rj];
        } else {
          odd = odd || (rj != last && rj != r0[q][j - 1]);
        }
        v0[q][j + 1] = p0[r1];
        v1[q][j + 1] = p1[r1];
        last = r1;
      }
    }
    const bool skips = __any_sync(0xffffffffu, odd);   // (the same in every lane)
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      if (l0 + q >= L) break;
      T h0 = lerp(fx[q], v0[q][0], v1[q][0]);
      T h1 = lerp(fx[q], v0[q][1], v1[q][1]);
#pragma unroll
      for (int j = 0; j < RS; ++j) {
        if (j > 0) {
          if (skips) {
            // a node row between is skipped somewhere (subapertures larger than the layer's cells)
            const int l = l0 + q, N = s_N[l], x0 = s_x0[l * kFwdLanes + lane];
            const T *p = phi + s_off[l] + r0[q][j];
            h0 = lerp(fx[q], p[x0], p[(x0 + 1) & (N - 1)]);
          } else {
            h0 = r0[q][j] == r0[q][j - 1] ? h0 : h1;
          }
          h1 = lerp(fx[q], v0[q][j + 1], v1[q][j + 1]);
        }
        val[j] += lerp(fy[q][j], h0, h1);
      }
    }
  }
}

template <typename T, int MODE, bool EL, int RS>
__global__ void __launch_bounds__(32 * kFwdPsi<T> / RS, RS == 1 ? 2 : (sizeof(T) == 4 ? 8 : 4))
    k_forward(const InstDev *__restrict__ insts, const FwdItem *__restrict__ items, IoArgs io) {
  extern __shared__ __align__(16) unsigned char fsm[];
  __shared__ T s_psi[kFwdPsi<T>][kFwdLanes + 1];
  __shared__ T s_ex[kFwdRows<T> + 1][kFwdLanes];
  __shared__ T s_ey[kFwdRows<T> + 1][kFwdLanes];
  // the slopes of a small launch, formed by every warp, for the four summing warps
  constexpr bool kAllWarps = RS == 1 && !EL;
  __shared__ T s_z[2][kAllWarps ? kFwdRows<T> + 1 : 1][kFwdLanes];
  pdl_trigger();
  const FwdItem it = items[blockIdx.x];
  if (io.active && !io.active[it.inst]) return;
  const InstDev &I = insts[it.inst];
  const WfsDev W = I.wfs[it.wfs];   // (by value: nothing of it is read again after the dependency wait)
  const T *phi = io.in0[it.inst] ? static_cast<const T *>(io.in0[it.inst]) : static_cast<const T *>(I.phi);
  const T *dat = static_cast<const T *>(io.in1[it.inst]);
  const int nc = W.nc, n = W.n, tid = threadIdx.x, nt = blockDim.x, L = I.n_layers;
  const int *pi = I.pos_i0 + it.pos;   // the sensor's corner tables: per layer nc columns, then nc rows
  const T *pf = static_cast<const T *>(I.pos_f) + it.pos;
  double *part = I.part + W.part_off;
  T *v = static_cast<T *>(I.v) + W.v_off;

  if (it.a0 < 0) {
    // Tip/tilt-only sensor: the sum of its Fried slopes over the valid
    // subapertures is <Gamma^T 1, psi>, which lives on the pupil-edge corners;
    // (edge corner, layer) terms, one FP64 partial per chunk of kFwdChunk.
    if (MODE == 2) return;   // data only: the model term is zero
    if constexpr (MODE == 3) {
      if (it.tile != 0) return;
      pdl_wait();
      // (the measurement's sums are FP64 in FP32 plans too: one CTA per sensor, a term or two per thread)
      Acc<double> ax, ay;
      constexpr int kBatch = 5;   // layers whose loads a thread issues together
      for (int e = tid; e < W.n_edge; e += nt) {
        const int c = I.edge_idx[W.edge_off + e], a = c % nc, b = c / nc;
        const T *et = static_cast<const T *>(I.edge_t) + 2 * (W.edge_off + e);
        const T tx = et[0], ty = et[1];
        T ps = T(0);
        for (int l0 = 0; l0 < L; l0 += kBatch) {
          T v00[kBatch], v01[kBatch], v10[kBatch], v11[kBatch], fx[kBatch], fy[kBatch];
          int x0[kBatch], y0[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int po = 2 * min(l0 + q, L - 1) * nc;
            x0[q] = pi[po + a];
            y0[q] = pi[po + nc + b];
            fx[q] = pf[po + a];
            fy[q] = pf[po + nc + b];
          }
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const LayerDev &Y = I.layers[min(l0 + q, L - 1)];
            const int N = Y.N, x1 = (x0[q] + 1) & (N - 1), y1 = (y0[q] + 1) & (N - 1);
            const T *g = phi + Y.off;
            v00[q] = g[y0[q] * N + x0[q]];
            v01[q] = g[y0[q] * N + x1];
            v10[q] = g[y1 * N + x0[q]];
            v11[q] = g[y1 * N + x1];
          }
#pragma unroll
          for (int q = 0; q < kBatch; ++q)
            if (l0 + q < L) ps += lerp(fy[q], lerp(fx[q], v00[q], v01[q]), lerp(fx[q], v10[q], v11[q]));
        }
        ax.add_prod(double(tx), double(ps));
        ay.add_prod(double(ty), double(ps));
      }
      const double2 m = block_sum2(ax, ay);
      if (tid == 0) {
        T *out = static_cast<T *>(io.out0[it.inst]);
        out[W.slope_off] = T(m.x / W.S);
        out[W.slope_off + 1] = T(m.y / W.S);
      }
      return;
    }
    constexpr int U = kFwdChunk / kFwdThreads;
    const int pairs = W.n_edge * L;
    int at[U][4];
    T fx[U], fy[U], tx[U], ty[U];
    Acc<T> ax, ay;
    if constexpr (RS == 1) {
      // no branch between a thread's pairs, the indices clamped: every pair's edge corner is requested
      // before any is used, then every pair's tables, then every pair's grid values (in big launches
      // the SM's other CTAs hide these latencies and the clamped form costs 0.7%: 16 E-ELT systems
      // 1139 -> 1149 us)
      if (tid < kFwdThreads) {
        int c[U], lay[U], x0[U], y0[U], N[U], off[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int pair = min(it.tile * kFwdChunk + u * kFwdThreads + tid, pairs - 1), e = pair / L;
          const T *et = static_cast<const T *>(I.edge_t) + 2 * (W.edge_off + e);
          lay[u] = pair - e * L;
          c[u] = I.edge_idx[W.edge_off + e];
          tx[u] = et[0];
          ty[u] = et[1];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int b = c[u] / nc, a = c[u] - b * nc, po = 2 * lay[u] * nc;
          x0[u] = pi[po + a];
          y0[u] = pi[po + nc + b];
          fx[u] = pf[po + a];
          fy[u] = pf[po + nc + b];
          N[u] = I.layers[lay[u]].N;
          off[u] = I.layers[lay[u]].off;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int x1 = (x0[u] + 1) & (N[u] - 1), y1 = (y0[u] + 1) & (N[u] - 1);
          at[u][0] = off[u] + y0[u] * N[u] + x0[u];
          at[u][1] = off[u] + y0[u] * N[u] + x1;
          at[u][2] = off[u] + y1 * N[u] + x0[u];
          at[u][3] = off[u] + y1 * N[u] + x1;
        }
      }
      pdl_wait();
      if (tid < kFwdThreads) {
        T g[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int q = 0; q < 4; ++q) g[u][q] = phi[at[u][q]];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const T ps = lerp(fy[u], lerp(fx[u], g[u][0], g[u][1]), lerp(fx[u], g[u][2], g[u][3]));
          if (it.tile * kFwdChunk + u * kFwdThreads + tid < pairs) {
            ax.add_prod(tx[u], ps);
            ay.add_prod(ty[u], ps);
          }
        }
      }
    } else {
      bool on[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int pair = it.tile * kFwdChunk + u * kFwdThreads + tid;
        on[u] = pair < pairs;
        if (!on[u]) continue;
        const int e = pair / L, l = pair - e * L;
        const int c = I.edge_idx[W.edge_off + e];
        const int a = c % nc, b = c / nc;
        const T *et = static_cast<const T *>(I.edge_t) + 2 * (W.edge_off + e);
        const int po = 2 * l * nc, N = I.layers[l].N, off = I.layers[l].off;
        const int x0 = pi[po + a], y0 = pi[po + nc + b];
        const int x1 = (x0 + 1) & (N - 1), y1 = (y0 + 1) & (N - 1);
        at[u][0] = off + y0 * N + x0;
        at[u][1] = off + y0 * N + x1;
        at[u][2] = off + y1 * N + x0;
        at[u][3] = off + y1 * N + x1;
        fx[u] = pf[po + a];
        fy[u] = pf[po + nc + b];
        tx[u] = et[0];
        ty[u] = et[1];
      }
      pdl_wait();
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (on[u]) {
          const T v00 = phi[at[u][0]], v01 = phi[at[u][1]];
          const T v10 = phi[at[u][2]], v11 = phi[at[u][3]];
          const T ps = lerp(fy[u], lerp(fx[u], v00, v01), lerp(fx[u], v10, v11));
          ax.add_prod(tx[u], ps);
          ay.add_prod(ty[u], ps);
        }
    }
    store_tile_partial(part + 2 * it.tile, ax, ay);
    return;
  }

  // stage this tile's corner->node tables for every layer (constant data)
  FwdRow<T> *s_row = reinterpret_cast<FwdRow<T> *>(fsm);
  T *s_fx = reinterpret_cast<T *>(s_row + L * kFwdPsi<T>);
  int *s_x0 = reinterpret_cast<int *>(s_fx + L * kFwdLanes);
  int *s_N = s_x0 + L * kFwdLanes;
  int *s_off = s_N + L;
  const int a0 = it.a0, b0 = it.b0;
  if (MODE != 2) {
    for (int idx = tid; idx < L * kFwdLanes; idx += nt) {
      const int l = idx / kFwdLanes, u = idx - l * kFwdLanes;
      const int a = 2 * l * nc + min(max(a0 - 1 + u, 0), nc - 1);
      cp_async_elem(s_x0 + idx, pi + a);
      cp_async_elem(s_fx + idx, pf + a);
    }
    for (int idx = tid; idx < L * kFwdPsi<T>; idx += nt) {
      const int l = idx / kFwdPsi<T>, w = idx - l * kFwdPsi<T>;
      const int b = 2 * l * nc + nc + min(max(b0 - 1 + w, 0), nc - 1);
      cp_async_elem(&s_row[idx].y0, pi + b);
      cp_async_elem(&s_row[idx].f, pf + b);
    }
    cp_async_commit();
    for (int l = tid; l < L; l += nt) {
      s_N[l] = I.layers[l].N;
      s_off[l] = I.layers[l].off;
    }
  }
  const unsigned char *act = I.active + W.act_off;
  const int *sidx = I.sub_idx + W.sub_off;
  const int lane = tid & 31, warp = tid >> 5;
  // the slope indices of step 2 (constant: before the dependency wait)
  constexpr int kSumWarps = kFwdThreads / 32, kSumRounds = (kFwdRows<T> + kSumWarps) / kSumWarps;
  constexpr int kSubWarps = kAllWarps ? kFwdPsi<T> / RS : kSumWarps;
  constexpr int kSubRounds = (kFwdRows<T> + kSubWarps) / kSubWarps;
  int sj[kSubRounds];
#pragma unroll
  for (int q = 0; q < kSubRounds; ++q) {
    const int w = warp + q * kSubWarps, a = a0 - 1 + lane, b = b0 - 1 + w;
    sj[q] = warp < kSubWarps && lane <= kFwdCols && w <= kFwdRows<T> && a >= 0 && b >= 0 && a < n && b < n
                ? sidx[b * n + a]
                : -1;
  }
  // 1. psi on the tile's corners plus a one-corner halo
  {
    const int a = a0 - 1 + lane, w = warp * RS;
    bool on[RS];
#pragma unroll
    for (int j = 0; j < RS; ++j) {
      const int b = b0 - 1 + w + j;
      on[j] = MODE != 2 && a >= 0 && b >= 0 && a < nc && b < nc && act[b * nc + a];
    }
    cp_async_wait_all();
    __syncthreads();
    pdl_wait();
    T val[RS];
    // (a warp without a corner of the pupil traces none)
    bool any = false;
#pragma unroll
    for (int j = 0; j < RS; ++j) any = any || on[j];
    if (MODE != 2 && __any_sync(0xffffffffu, any)) trace_strip<T, RS>(phi, L, w, s_N, s_off, s_x0, s_fx, s_row, val);
#pragma unroll
    for (int j = 0; j < RS; ++j) s_psi[w + j][lane] = on[j] ? val[j] : T(0);
  }
  __syncthreads();
  // 2. weighted slopes of the subapertures the tile's corners touch, one lane per column
  Acc<T> sx_acc, sy_acc, qx_acc, qy_acc;
  const T isg = sizeof(T) == 4 ? T(W.inv_sigma2_f) : T(W.inv_sigma2);   // no FP64 conversion in FP32
  // spot elongation: the block sigma^2 (I + tau g g^T) is inverted in closed
  // form, sigma^-2 (I - c g g^T) with c = tau / (1 + tau |g|^2)
  const bool elong = EL && W.elong != 0;
  const T el_tau = EL ? T(W.el_tau) : T(0), el_eps = EL ? T(W.el_eps) : T(0), el_d = EL ? T(W.d_sub) : T(0);
  const T el_cx = EL ? fma_rn(T(0.5 - 0.5 * n), el_d, -T(W.el_lx)) : T(0);
  const T el_cy = EL ? fma_rn(T(0.5 - 0.5 * n), el_d, -T(W.el_ly)) : T(0);
  const bool four = EL && tile_partials(W) == 4;
  const bool sums = W.kind == kRemoveTT;
  if (warp < kSubWarps && lane <= kFwdCols) {
    const int u = lane, a = a0 - 1 + u;
#pragma unroll
    for (int q = 0; q < kSubRounds; ++q) {
      const int w = warp + q * kSubWarps, b = b0 - 1 + w, j = sj[q];
      if (w > kFwdRows<T>) break;
      T ex = T(0), ey = T(0), zx = T(0), zy = T(0);
      if (j >= 0) {
        const T p00 = s_psi[w][u], p10 = s_psi[w][u + 1];
        const T p01 = s_psi[w + 1][u], p11 = s_psi[w + 1][u + 1];
        T sx = T(0.5) * (p10 + p11 - p00 - p01);
        T sy = T(0.5) * (p01 + p11 - p00 - p10);
        if (MODE == 3) {
          if (u >= 1 && w >= 1) {   // subapertures owned by this tile
            T *so = static_cast<T *>(io.out0[it.inst]);
            so[W.slope_off + j] = sx;
            so[W.slope_off + W.S + j] = sy;
          }
          continue;
        }
        if (MODE == 1) {
          sx = dat[W.slope_off + j] - sx;
          sy = dat[W.slope_off + W.S + j] - sy;
        } else if (MODE == 2) {
          sx = dat[W.slope_off + j];
          sy = dat[W.slope_off + W.S + j];
        }
        if (elong) {
          // (every rounding stated: the compiler contracts products differently from one instance to another)
          const T gx = mul_rn(el_eps, fma_rn(T(a), el_d, el_cx)), gy = mul_rn(el_eps, fma_rn(T(b), el_d, el_cy));
          const T c = el_tau / fma_rn(el_tau, fma_rn(gx, gx, mul_rn(gy, gy)), T(1));
          const T dot = mul_rn(c, fma_rn(gx, sx, mul_rn(gy, sy)));
          ex = mul_rn(isg, fma_rn(-gx, dot, sx));
          ey = mul_rn(isg, fma_rn(-gy, dot, sy));
        } else {
          ex = isg * sx;
          ey = isg * sy;
        }
        if (kAllWarps) {
          zx = sx;
          zy = sy;
        } else if (u >= 1 && w >= 1) {   // subapertures owned by this tile
          sx_acc.add(sx);
          sy_acc.add(sy);
          if (four) {
            qx_acc.add(ex);
            qy_acc.add(ey);
          }
        }
      }
      s_ex[w][u] = ex;
      s_ey[w][u] = ey;
      if (kAllWarps && sums) {
        s_z[0][w][u] = zx;
        s_z[1][w][u] = zy;
      }
    }
  }
  if (MODE == 3) return;
  __syncthreads();
  if (kAllWarps && sums && warp < kSumWarps && lane >= 1 && lane <= kFwdCols) {
    // the owned subapertures' z (zero where there is none) on the four warps, rows in the strips' order
#pragma unroll
    for (int q = 0; q < kSumRounds; ++q) {
      const int w = warp + q * kSumWarps;
      if (w < 1 || w > kFwdRows<T>) continue;
      sx_acc.add(s_z[0][w][lane]);
      sy_acc.add(s_z[1][w][lane]);
    }
  }
  // 3. Gamma^T: each corner gathers its four neighbouring subapertures
  if (lane < kFwdCols) {
    const int u = lane, a = a0 + u;
    for (int w = warp; w < kFwdRows<T>; w += nt >> 5) {
      const int b = b0 + w;
      if (a < nc && b < nc) {
        const T val = T(0.5) * (s_ex[w + 1][u] + s_ex[w][u] - s_ex[w + 1][u + 1] - s_ex[w][u + 1]) +
                      T(0.5) * (-s_ey[w + 1][u] + s_ey[w][u] - s_ey[w + 1][u + 1] + s_ey[w][u + 1]);
        v[b * nc + a] = val;
      }
    }
  }
  if (!sums) return;
  // 4. tip/tilt removal: this tile's sums of z (the consumer forms the means)
  if (four) {
    store_tile_partial(part + 4 * it.tile, sx_acc, sy_acc);
    __syncthreads();   // warp 0 has read the reduction scratch before it is reused
    store_tile_partial(part + 4 * it.tile + 2, qx_acc, qy_acc);
  } else {
    store_tile_partial(part + 2 * it.tile, sx_acc, sy_acc);
  }
}

// ------------------------------------------------------- transform helpers

// Coefficients owned by cluster rank c of one layer, and their place in the
// CTA's shared-memory cache.  Distributed levels k = 1..kd (block side
// M = N/2^(k-1) >= 2S, R = M/C rows per CTA, Rh = R/2, H = M/2): the high-x
// part of the low-y rows c*Rh + jl and the high-y rows H + c*Rh + jl; then the
// CTA's low-low rows of level J (kd == J) or, on rank 0, the coarse pyramid
// block of side S >= C (kd < J).  Levels below cache_kc are read from global memory.
struct CoefMap {
  int N, C, S, J, kd, kc, crank, lgN, lgC, lgS;
  int base[kMaxLevels + 3];
  __device__ void init(int N_, int C_, int S_, int J_, int kc_, int crank_) {
    N = N_;
    C = C_;
    S = S_;
    J = J_;
    crank = crank_;
    lgN = __ffs(N) - 1;
    lgC = __ffs(C) - 1;
    lgS = __ffs(S) - 1;
    kd = 0;
    while (kd < J && (N >> kd) > S) ++kd;
    kc = kc_ < 1 ? 1 : kc_;
    int off = 0;
    for (int k = 1; k <= kd; ++k) {
      base[k] = off;
      if (k >= kc) {
        const int M = N >> (k - 1), Rh = (M / C) >> 1;
        off += Rh * (M >> 1) + Rh * M;
      }
    }
    base[kd + 1] = off;
    if (kd == J) {
      const int M = N >> (J - 1), Rh = (M / C) >> 1;
      off += Rh * (M >> 1);
    } else if (crank == 0) {
      off += S * S;
    }
    base[kd + 2] = off;
  }
  __device__ int total() const { return base[kd + 2]; }
  // sizes of level k as log2: block side M, half H, CTA rows R, half Rh
  __device__ int lgM(int k) const { return lgN - (k - 1); }
  __device__ int hl(int k, int jl, int x) const {
    const int lh = lgM(k) - 1;
    return base[k] + (jl << lh) + (x - (1 << lh));
  }
  __device__ int lh(int k, int jl, int x) const {
    const int lm = lgM(k), lrh = lm - lgC - 1;
    return base[k] + (1 << (lrh + lm - 1)) + (jl << lm) + x;
  }
  __device__ int ll(int jl, int x) const { return base[kd + 1] + (jl << (lgM(J) - 1)) + x; }
  __device__ int coarse(int r, int c) const { return base[kd + 1] + (r << lgS) + c; }
  // pyramid position of cache slot q
  __device__ void pos(int q, int &row, int &col) const {
    if (q >= base[kd + 1]) {
      const int q2 = q - base[kd + 1];
      if (kd == J) {
        const int lh = lgM(J) - 1, lrh = lgM(J) - lgC - 1;
        row = (crank << lrh) + (q2 >> lh);
        col = q2 & ((1 << lh) - 1);
      } else {
        row = q2 >> lgS;
        col = q2 & (S - 1);
      }
      return;
    }
    int k = kd;
    while (base[k] > q) --k;
    const int lm = lgM(k), lh = lm - 1, lrh = lm - lgC - 1;
    int q2 = q - base[k];
    if (q2 < (1 << (lrh + lh))) {
      row = (crank << lrh) + (q2 >> lh);
      col = (1 << lh) + (q2 & ((1 << lh) - 1));
    } else {
      q2 -= 1 << (lrh + lh);
      row = (1 << lh) + (crank << lrh) + (q2 >> lm);
      col = q2 & ((1 << lm) - 1);
    }
  }
};

// Shared-memory copy of the gather tables of one analysis CTA (layer l, rows
// [k0, k0+R0)), laid out by stage_layout: the plan's stage image for the CTA
// (tap records, pupil-edge entries and index, run tables), one bulk copy before
// the dependency wait since the tables are constant, so the copy overlaps the
// previous kernel; after the wait, the corner rows of v that the CTA reads,
// one bulk copy per sensor.
template <typename T>
struct GatherStage {
  unsigned char *base;
  T *xr, *yr, *vs, *tw;
  int *mnc, *vpre, *vsrc, *mslot, *tk;
  const uint16_t *eb;
  int image_bytes;

  __device__ void carve(unsigned char *b, int Md, int N, int R0, const InstDev &I) {
    const StageLayout sl = stage_layout(Md, N, R0, I.rec_stride, static_cast<int>(sizeof(T)), I.max_tt_entries,
                                        I.vstage);
    base = b;
    xr = reinterpret_cast<T *>(b + sl.xr);
    yr = reinterpret_cast<T *>(b + sl.yr);
    tw = reinterpret_cast<T *>(b + sl.tw);
    vs = reinterpret_cast<T *>(b + sl.vs);
    mnc = reinterpret_cast<int *>(b + sl.mnc);
    vpre = reinterpret_cast<int *>(b + sl.vpre);
    vsrc = reinterpret_cast<int *>(b + sl.vsrc);
    mslot = reinterpret_cast<int *>(b + sl.mslot);
    tk = reinterpret_cast<int *>(b + sl.tk);
    eb = reinterpret_cast<const uint16_t *>(b + sl.eb);
    image_bytes = sl.image;
  }

  // One thread: the bulk copy of the CTA's stage image, completing on bar.
  __device__ void issue_image(const InstDev &I, int l, int crank, uint64_t *bar) const {
    const unsigned char *src = static_cast<const unsigned char *>(I.stage_img) + I.img_stride * (l * I.C + crank);
    mbar_arm(bar, static_cast<uint32_t>(image_bytes));
    if (image_bytes > 0) bulk_copy_g2s(base, src, static_cast<uint32_t>(image_bytes), bar);
  }

  // Spot elongation with tip/tilt removal: v += m_x Gx + m_y Gy over the staged
  // corner rows of those sensors (the mean slopes from edge_coefficients).
  __device__ void add_elongation(const InstDev &I, const T *s_coef) const {
    constexpr int vq = 16 / static_cast<int>(sizeof(T));
    const T *gx = static_cast<const T *>(I.gel), *gy = gx + I.v_total;
    for (int md = 0; md < I.n_dense; ++md) {
      const int k = mslot[md];
      if (k < 0) continue;
      const T mx = s_coef[2 * kMaxEdgeSlots + 2 * k], my = s_coef[2 * kMaxEdgeSlots + 2 * k + 1];
      const int e0 = vpre[md] * vq, cnt = (vpre[md + 1] - vpre[md]) * vq, g0 = vsrc[md] * vq;
      for (int i = threadIdx.x; i < cnt; i += blockDim.x) vs[e0 + i] += mx * gx[g0 + i] + my * gy[g0 + i];
    }
  }

  // One thread, after the dependency wait: the bulk copies of the CTA's
  // corner rows of v (one aligned run per sensor, written by the previous
  // kernel), completing on bar.  Needs the stage image in shared memory.
  __device__ void load_v_bulk(const InstDev &I, uint64_t *bar) const {
    const int Md = I.n_dense;
    const uint4 *src = static_cast<const uint4 *>(I.v);
    uint4 *dst = reinterpret_cast<uint4 *>(vs);
    fence_async_global();
    mbar_arm(bar, static_cast<uint32_t>(vpre[Md]) * 16u);
    for (int md = 0; md < Md; ++md) {
      const int n = vpre[md + 1] - vpre[md];
      if (n > 0) bulk_copy_g2s(dst + vpre[md], src + vsrc[md], static_cast<uint32_t>(n) * 16u, bar);
    }
  }
};

// The gather of gather_rows from the staged records and v rows, sensors inner
// with the sums in registers.  A thread takes one column and two adjacent node
// rows: they share the column's tap record, and their windows' corner rows
// overlap, so each corner row's weighted column sum sx is formed once for both
// (rows of the second window d = 0..2 rows below the first's; other offsets
// take the two windows apart).  Each node's sum has window_sum's order.
template <typename T, int KT, int D>
__device__ __forceinline__ void pair_sums(const T *h, const TapRec<T, KT> &y0, const TapRec<T, KT> &y1, T &acc0,
                                          T &acc1) {
  T s0 = T(0), s1 = T(0);
#pragma unroll
  for (int ty = 0; ty < KT; ++ty) s0 += y0.w[ty] * h[ty];
#pragma unroll
  for (int ty = 0; ty < KT; ++ty) s1 += y1.w[ty] * h[D + ty];
  acc0 += s0;
  acc1 += s1;
}

template <typename T, int KT>
__device__ void gather_rows_staged(const InstDev &I, const GatherStage<T> &st, int N, int R0,
                                   T *A, const T *s_coef) {
  constexpr int RS = TapRec<T, KT>::RS;
  const int nt = blockDim.x, tid = threadIdx.x, Md = I.n_dense, lgN = __ffs(N) - 1;
  for (int pr = tid; pr < (R0 >> 1) * N; pr += nt) {
    const int col = pr & (N - 1), k0 = (pr >> lgN) << 1;
    const T *xr = st.xr + col * RS;
    const T *yr = st.yr + k0 * RS;
    T acc0 = T(0), acc1 = T(0);
    for (int md = 0; md < Md; ++md) {
      TapRec<T, KT> x, y0, y1;
      x.load(xr + md * N * RS);
      y0.load(yr + md * R0 * RS);
      y1.load(yr + md * R0 * RS + RS);
      if (x.off < 0) continue;
      const int nc = st.mnc[md];
      const int d = (y0.off >= 0 && y1.off >= 0) ? (y1.off - y0.off) / nc : -1;
      if (d >= 0 && d <= 2 && y1.off - y0.off == d * nc) {
        // the corner rows of both windows, each row's column sum once
        T h[KT + 2];
        const T *p = st.vs + y0.off + x.off;
#pragma unroll
        for (int r = 0; r < KT + 2; ++r) {
          if (r < KT + d) {
            T v[KT];
#pragma unroll
            for (int tx = 0; tx < KT; ++tx) v[tx] = p[r * nc + tx];
            T sx = x.w[0] * v[0];
#pragma unroll
            for (int tx = 1; tx < KT; ++tx) sx += x.w[tx] * v[tx];
            h[r] = sx;
          }
        }
        if (d == 0) pair_sums<T, KT, 0>(h, y0, y1, acc0, acc1);
        else if (d == 1) pair_sums<T, KT, 1>(h, y0, y1, acc0, acc1);
        else pair_sums<T, KT, 2>(h, y0, y1, acc0, acc1);
      } else {
        if (y0.off >= 0) acc0 += window_sum<T, KT, true>(st.vs + y0.off + x.off, nc, x, y0);
        if (y1.off >= 0) acc1 += window_sum<T, KT, true>(st.vs + y1.off + x.off, nc, x, y1);
      }
    }
    if (I.n_edge_wfs > 0) {
      // the nodes' pupil-edge entries (from the dense per-node index), added after the sensors
      const int n0 = k0 * N + col, n1 = n0 + N;
      const int e0 = st.eb[n0], e1 = st.eb[n0 + 1], e2 = st.eb[n1], e3 = st.eb[n1 + 1];
      if (e1 > e0) acc0 += edge_node_sum<T>(e0, e1, st.tk, st.tw, s_coef);
      if (e3 > e2) acc1 += edge_node_sum<T>(e2, e3, st.tk, st.tw, s_coef);
    }
    A[k0 * N + col] = acc0;
    A[(k0 + 1) * N + col] = acc1;
  }
}

// ------------------------------------------------------------ k_analysis
// SRC 0: layer grids from io.in0.  SRC 1: adjoint gather from the plan's v.
// SRC 2: the gather k_gather left in the plan's phi.
// EPI plain: io.out0 = W g.  EPI op: q = W g + alpha D p with p = io.in1 (NULL:
// the plan's p), q = io.out0 (NULL: the plan's q); partial p.q per CTA.
// EPI resid: r = W g - alpha D x (x = io.out0, zeroed when cold), p = z = J^-1 r;
// partials r.z and r.r per CTA.
template <typename T, int SRC, int EPI, int LF>
__global__ void __launch_bounds__(kAnalysisThreadsMax, 1) k_analysis(const InstDev *__restrict__ insts,
                                                      const ClusterItem *__restrict__ items,
                                                      IoArgs io, int flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ InstDev sI;
  __shared__ CoefMap cm;
  __shared__ T s_coef[4 * kMaxEdgeSlots];
  __shared__ T s_dal[kMaxLevels + 1];
  __shared__ uint64_t s_bar[2];   // stage image, corner rows of v (bulk copies)
  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks());
  const int crank = static_cast<int>(cluster.block_rank());
  const ClusterItem it = items[blockIdx.x / C];
  if (io.active && !io.active[it.inst]) return;   // the whole cluster leaves together
  load_inst(&sI, insts + it.inst);
  const InstDev &I = sI;
  const LayerDev &L = I.layers[it.layer];
  const int N = L.N, R0 = N / C, J = I.J, tid = threadIdx.x, nt = blockDim.x;
  T *A = reinterpret_cast<T *>(smem_raw);
  T *B = A + (R0 + kMaxTaps) * N;
  const int S = L.coarse;
  T *cb = S > C ? B : B + (R0 + kMaxTaps) * N;
  T *cb2 = cb + S * S;
  T *cache = reinterpret_cast<T *>(smem_raw) + transform_cache_offset(N, C, S);
  if (tid == 0) cm.init(N, C, S, J, L.cache_kc, crank);
  if (tid <= J) s_dal[tid] = T(L.dalpha[tid]);
  Filt<T, LF> f;
  f.load(I);

  Emit<T, EPI> emit;
  emit.off = L.off;
  emit.N = N;
  emit.dalpha = s_dal;
  emit.precond = I.precond;
  emit.warm = (flags & kFlagWarm) ? 1 : 0;
  emit.jinv = static_cast<const T *>(I.jinv);
  emit.cache = cache;
  emit.out = static_cast<T *>(io.out0[it.inst]);
  emit.P = io.in1[it.inst] ? static_cast<const T *>(io.in1[it.inst]) : static_cast<const T *>(I.p);
  emit.Q = io.out0[it.inst] ? static_cast<T *>(io.out0[it.inst]) : static_cast<T *>(I.q);
  emit.R = static_cast<T *>(I.r);
  emit.Pn = static_cast<T *>(I.p);
  emit.X = static_cast<T *>(io.out0[it.inst]);
  GatherStage<T> st;
  // SRC 1 plans stage their tables (those that cannot run k_gather, SRC 2)
  const bool staged = SRC == 1;
  bool copies_ok = true;
  if (staged) {
    const int off = transform_cache_offset(N, C, S) + transform_cache_size(N, C, S, J, L.cache_kc);
    unsigned char *sb = smem_raw + ((static_cast<size_t>(off) * sizeof(T) + 15) & ~size_t(15));
    st.carve(sb, I.n_dense, N, R0, I);
    if (tid == 0) {
      mbar_init(&s_bar[0]);
      mbar_init(&s_bar[1]);
      st.issue_image(I, it.layer, crank, &s_bar[0]);
    }
    __syncthreads();   // the barriers are initialised
    copies_ok = mbar_wait(&s_bar[0], 0);
  }
  __syncthreads();
  pdl_wait();
  // a new solve starts from the residual: clear the breakdown flag
  if (EPI == kEpiResid && it.layer == 0 && crank == 0 && tid == 0) I.scal[kFlag] = 0.0;

  // asynchronous copies: the gather's corner rows of v, then the epilogue
  // inputs (p, or x for a warm residual) of every owned coefficient into the
  // coefficient cache; both complete before the transform
  if (staged && tid == 0) st.load_v_bulk(I, &s_bar[1]);
  const bool use_cache = (EPI == kEpiOp) || (EPI == kEpiResid && emit.warm);
  if (use_cache) {
    // issued by the warps that the pupil-edge coefficients below leave idle
    // (one warp per edge slot), so the two overlap
    const int w0 = SRC == 1 ? min(I.n_edge_wfs, nt / 32 - 1) : 0, t0 = tid - 32 * w0;
    if (t0 >= 0) {
      const T *srcv = EPI == kEpiOp ? emit.P : emit.X;
      const int total = cm.total();
      for (int q = t0; q < total; q += nt - 32 * w0) {
        int row, col;
        cm.pos(q, row, col);
        cp_async_elem(cache + q, srcv + L.off + row * N + col);
      }
    }
    cp_async_commit();
  }
  // own rows [crank*R0, (crank+1)*R0) of the layer grid
  if (SRC == 0 || SRC == 2) {
    const T *src = (SRC == 0 ? static_cast<const T *>(io.in0[it.inst]) : static_cast<const T *>(I.phi)) +
                   L.off + crank * R0 * N;
    for (int idx = tid; idx < R0 * N; idx += nt) A[idx] = src[idx];
  } else {
    // the tip/tilt-only sensors' measurement term: model (operator), data
    // minus model (warm residual) or data alone (cold residual, right-hand side)
    const int tt_mode = EPI == kEpiOp ? 0 : (EPI == kEpiResid && emit.warm ? 1 : 2);
    if (I.n_edge_wfs > 0)
      edge_coefficients<T>(I, s_coef, tt_mode, static_cast<const T *>(io.in1[it.inst]));
    if (staged) {
      copies_ok = mbar_wait(&s_bar[1], 0) && copies_ok;
      // a copy that never completed (it does not happen with valid tables): the
      // solve reports a breakdown and its iterate stays as it was
      if (!copies_ok) I.scal[kFlag] = 1.0;
      __syncthreads();
      if (I.gel) {
        st.add_elongation(I, s_coef);
        __syncthreads();
      }
      if (I.max_taps <= 2) gather_rows_staged<T, 2>(I, st, N, R0, A, s_coef);
      else if (I.max_taps == 3) gather_rows_staged<T, 3>(I, st, N, R0, A, s_coef);
      else gather_rows_staged<T, 4>(I, st, N, R0, A, s_coef);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  auto slot_hl = [&](int k, int jl, int x) { return (use_cache && k >= cm.kc) ? cm.hl(k, jl, x) : -1; };
  auto slot_lh = [&](int k, int jl, int x) { return (use_cache && k >= cm.kc) ? cm.lh(k, jl, x) : -1; };

  // Distributed levels: one cluster barrier per level (row pass done) before
  // the halo rows are read from the next CTAs; the reads are released with
  // an arrive, and the matching wait comes just before this CTA next
  // overwrites B (the next level's row pass, or the end of the kernel).
  const int lgN = L.log2N, lgC = __ffs(C) - 1;
  int M = N, k = 1;
  for (; k <= J && M > S; ++k, M >>= 1) {
    const int lgM = lgN - (k - 1), lgR = lgM - lgC;
    const int R = M >> lgC, H = M >> 1, Rh = R >> 1;
    if (k > 1) cluster_wait();
    // row pass (x): local
    row_analysis<T, LF>(f, A, B, R, lgM, tid, nt);
    cluster.sync();
    // halo: the LF-2 rows after ours (mod M) from the next CTAs
    for (int idx = tid; idx < (LF - 2) * M; idx += nt) {
      const int j = idx >> lgM, x = idx & (M - 1);
      const int r = ((crank + 1) * R + j) & (M - 1);
      B[(R + j) * M + x] = cluster.map_shared_rank(B, r >> lgR)[(r & (R - 1)) * M + x];
    }
    cluster_arrive();
    __syncthreads();
    // column pass (y), local; the epilogue inputs of kColU outputs per thread
    // are fetched before any of them is written
    constexpr int kColU = SRC == 2 ? 4 : (SRC == 1 ? 1 : 2);
    for (int idx0 = tid; idx0 < Rh * M; idx0 += kColU * nt) {
      T lo[kColU], hi[kColU];
      typename Emit<T, EPI>::Pre fa[kColU], fb[kColU];
#pragma unroll
      for (int u = 0; u < kColU; ++u) {
        const int idx = idx0 + u * nt;
        if (idx < Rh * M) {
          const int il = idx >> lgM, x = idx & (M - 1);
          const int i = crank * Rh + il;
          const T *col = B + 2 * il * M + x;
          T l = T(0), h = T(0);
#pragma unroll
          for (int t = 0; t < LF; ++t) {
            const T val = col[t * M];
            l += f.h[t] * val;
            h += f.g[t] * val;
          }
          lo[u] = l;
          hi[u] = h;
          if (x >= H) fa[u] = emit.fetch(i, x, slot_hl(k, il, x));
          else if (k == J) fa[u] = emit.fetch(i, x, use_cache ? cm.ll(il, x) : -1);
          fb[u] = emit.fetch(H + i, x, slot_lh(k, il, x));
        }
      }
#pragma unroll
      for (int u = 0; u < kColU; ++u) {
        const int idx = idx0 + u * nt;
        if (idx < Rh * M) {
          const int il = idx >> lgM, x = idx & (M - 1);
          const int i = crank * Rh + il;
          if (x < H) {
            if (k == J) emit.put(i, x, J, lo[u], fa[u]);
            else A[il * H + x] = lo[u];
          } else {
            emit.put(i, x, k, lo[u], fa[u]);
          }
          emit.put(H + i, x, k, hi[u], fb[u]);
        }
      }
    }
    __syncthreads();
  }
  if (k > 1) cluster_wait();   // the next CTAs have read this CTA's halo rows
  if (k <= J) {
    // coarse levels: the remaining low-low block (side M = S) in CTA 0
    cluster.sync();   // every CTA's low-low rows are written
    if (crank == 0) {
      const int lgS = __ffs(S) - 1, lgRs = lgS - lgC;   // each CTA holds S / C rows of side S
      for (int idx = tid; idx < M * M; idx += nt) {
        const int r = idx >> lgS, c = idx & (M - 1);
        cb[idx] = cluster.map_shared_rank(A, r >> lgRs)[((r & ((1 << lgRs) - 1)) << lgS) + c];
      }
    }
    cluster.sync();
    if (crank == 0) {
      __syncthreads();
      for (; k <= J; ++k, M >>= 1) {
        const int H = M >> 1, lgMc = __ffs(M) - 1;
        row_analysis<T, LF>(f, cb, cb2, M, lgMc, tid, nt);
        __syncthreads();
        for (int idx = tid; idx < H * M; idx += nt) {
          const int i = idx >> lgMc, x = idx & (M - 1);
          T lo = T(0), hi = T(0);
#pragma unroll
          for (int t = 0; t < LF; ++t) {
            const T val = cb2[((2 * i + t) & (M - 1)) * M + x];
            lo += f.h[t] * val;
            hi += f.g[t] * val;
          }
          if (x < H && k < J) cb[i * H + x] = lo;
          else emit(i, x, (x < H) ? J : k, lo, use_cache ? cm.coarse(i, x) : -1);
          emit(H + i, x, k, hi, use_cache ? cm.coarse(H + i, x) : -1);
        }
        __syncthreads();
      }
    }
  }
  if (EPI == kEpiPlain) return;
  // one FP64 partial per CTA; the next kernel sums them
  const double2 s = block_sum2(emit.acc0, emit.acc1);
  if (tid == 0) {
    const int slot = I.cl_part_off + 2 * (it.layer * C + crank);
    I.part[slot] = s.x;
    I.part[slot + 1] = s.y;
  }
}

// ----------------------------------------------------------- k_synthesis
// SRC 0: coefficients from io.in0.  SRC 1 (PCG iteration it = flags >> 8):
// r.z of this iteration from the previous kernel's partials (the initial
// residual's for it = 0, else the update's), beta = (r.z)_it / (r.z)_(it-1),
// p <- J^-1 r + beta p written back (it = 0: p already holds J^-1 r).
// Output: io.out0 (NULL: the plan's phi).
template <typename T, int SRC, int LF>
__global__ void __launch_bounds__(kSynthThreads, 1) k_synthesis(const InstDev *__restrict__ insts,
                                                       const ClusterItem *__restrict__ items,
                                                       IoArgs io, int flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ InstDev sI;
  __shared__ CoefMap cm;
  __shared__ T s_beta;
  constexpr int HL = LF / 2 - 1;   // halo rows of the column synthesis
  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks());
  const int crank = static_cast<int>(cluster.block_rank());
  const ClusterItem it = items[blockIdx.x / C];
  if (io.active && !io.active[it.inst]) return;   // the whole cluster leaves together
  load_inst(&sI, insts + it.inst);
  const InstDev &I = sI;
  const LayerDev &L = I.layers[it.layer];
  const int N = L.N, R0 = N / C, J = I.J, tid = threadIdx.x, nt = blockDim.x;
  T *buf0 = reinterpret_cast<T *>(smem_raw);
  T *buf1 = buf0 + (R0 + kMaxTaps) * N;
  const int S = L.coarse;
  T *cache = reinterpret_cast<T *>(smem_raw) + transform_cache_offset(N, C, S);
  // low-low of the coarse stage, then its row syntheses (read by the other CTAs while the row
  // buffers are in use: after the cache when the analysis has them in a row buffer)
  T *cb = S > C ? cache + transform_cache_size(N, C, S, J, L.cache_kc) : buf1 + (R0 + kMaxTaps) * N;
  T *cb2 = cb + S * S;
  if (tid == 0) cm.init(N, C, S, J, L.cache_kc, crank);
  Filt<T, LF> f;
  f.load(I);
  T *out = io.out0[it.inst] ? static_cast<T *>(io.out0[it.inst]) : static_cast<T *>(I.phi);
  const T *src = static_cast<const T *>(io.in0[it.inst]);
  T *P = static_cast<T *>(I.p);
  const T *Rv = static_cast<const T *>(I.r);
  const T *Jv = static_cast<const T *>(I.jinv);
  const int iter = flags >> kIterShift;
  const bool first = (flags & kFlagFirst) != 0;
  const bool pre = I.precond != 0;
  pdl_wait();
  if (SRC == 1) {
    // r.z of this iteration; the first CTA of the instance records it
    const double prev = I.scal[kRz0 + ((iter + 1) & 1)];
    const double flag = I.scal[kFlag];
    const double rz = iter == 0 ? sum_partial(I.part + I.cl_part_off, I.n_cl_part, 0)
                                : sum_partial(I.part + I.upd_part_off, I.n_upd_blocks, 0);
    if (tid == 0) {
      double beta = 0.0;
      if (iter > 0) {
        const bool stop = flag != 0.0 || !isfinite(rz) || !(prev != 0.0);
        beta = stop ? 0.0 : rz / prev;
      }
      s_beta = T(beta);
      if (it.layer == 0 && crank == 0) I.scal[kRz0 + (iter & 1)] = rz;
    }
  }
  __syncthreads();
  const T beta = SRC == 1 ? s_beta : T(0);
  // a coefficient of an uncached level: its loads (raw), then the direction
  // update and its store (finish)
  struct Raw {
    T p, r, j;
  };
  auto raw = [&](int row, int col) -> Raw {
    const int idx = L.off + row * N + col;
    Raw v{T(0), T(0), T(1)};
    if (SRC == 0) {
      v.p = src[idx];
    } else {
      v.p = P[idx];
      if (!first) {
        v.r = Rv[idx];
        if (pre) v.j = Jv[idx];
      }
    }
    return v;
  };
  auto finish = [&](const Raw &v, int row, int col) -> T {
    if (SRC == 0 || first) return v.p;
    const T z = pre ? v.j * v.r : v.r;
    const T pn = z + beta * v.p;
    P[L.off + row * N + col] = pn;
    return pn;
  };
  // every owned coefficient of the cached levels, eight in flight per thread
  {
    const int total = cm.total();
    for (int q0 = tid; q0 < total; q0 += 8 * nt) {
      int idx[8];
      T rv[8], jv[8], pv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int q = q0 + u * nt;
        if (q < total) {
          int row, col;
          cm.pos(q, row, col);
          idx[u] = L.off + row * N + col;
          if (SRC == 0) {
            pv[u] = src[idx[u]];
          } else {
            pv[u] = P[idx[u]];
            if (!first) {
              rv[u] = Rv[idx[u]];
              jv[u] = pre ? Jv[idx[u]] : T(1);
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int q = q0 + u * nt;
        if (q < total) {
          T pn = pv[u];
          if (SRC == 1 && !first) {
            const T z = pre ? jv[u] * rv[u] : rv[u];
            pn = z + beta * pv[u];
            P[idx[u]] = pn;
          }
          cache[q] = pn;
        }
      }
    }
  }
  __syncthreads();
  const int kd = cm.kd;

  T *A = buf0, *B = buf1;
  if (kd < J) {
    if (crank == 0) {
      {
        const int HJ = (N >> (J - 1)) >> 1;
        const int lgHJ = __ffs(HJ) - 1;
        for (int idx = tid; idx < HJ * HJ; idx += nt) cb[idx] = cache[cm.coarse(idx >> lgHJ, idx & (HJ - 1))];
      }
      __syncthreads();
      // rows first (x), then columns (y), as at the distributed levels and in
      // the streamed transforms, so every path gives the same bits
      const T *c3 = cache + cm.coarse(0, 0);
      for (int k = J; k > kd; --k) {
        const int M = N >> (k - 1), H = M >> 1, lgMc = __ffs(M) - 1;
        // row r < H: [LL | HL] of low-y row r; r >= H: [LH | HH] of high-y row r - H
        for (int idx = tid; idx < M * M; idx += nt) {
          const int r = idx >> lgMc, j = idx & (M - 1);
          const int q = j & 1;
          T acc = T(0);
#pragma unroll
          for (int s = 0; s < LF / 2; ++s) {
            const int t = q + 2 * s;
            const int jj = ((j - t) & (M - 1)) >> 1;
            const T lo = r < H ? cb[r * H + jj] : c3[r * S + jj];
            const T hi = c3[r * S + H + jj];
            acc += f.hs(q, s) * lo + f.gs(q, s) * hi;
          }
          cb2[r * M + j] = acc;
        }
        __syncthreads();
        for (int idx = tid; idx < M * M; idx += nt) {
          const int y = idx >> lgMc, x = idx & (M - 1);
          const int p = y & 1;
          T acc = T(0);
#pragma unroll
          for (int s = 0; s < LF / 2; ++s) {
            const int t = p + 2 * s;
            const int ii = ((y - t) & (M - 1)) >> 1;
            acc += f.hs(p, s) * cb2[ii * M + x] + f.gs(p, s) * cb2[(H + ii) * M + x];
          }
          cb[y * M + x] = acc;
        }
        __syncthreads();
      }
    }
    cluster.sync();
    // level kd: M = 2S, S / C low-low rows per CTA
    const T *c0 = cluster.map_shared_rank(cb, 0) + crank * (S / C) * S;
    for (int j = tid; j < S / C * S; j += nt) A[j] = c0[j];
  } else {
    const int M = N >> (J - 1), H = M >> 1, Rh = (M / C) >> 1, lgH = __ffs(H) - 1;
    for (int idx = tid; idx < Rh * H; idx += nt) A[idx] = cache[cm.ll(idx >> lgH, idx & (H - 1))];
  }
  __syncthreads();

  // Distributed levels, per level: own coefficient rows (V), their row
  // synthesis (x) into U after HL halo rows, one cluster barrier, the halo
  // rows of the previous CTAs, then the column synthesis (y) into V, which is
  // the next level's low-low block.  The halo reads are released with an
  // arrive; the matching wait comes before this CTA next overwrites U (the
  // next level's first step, or the end of the kernel).
  const int lgN = L.log2N, lgC = __ffs(C) - 1;
  T *U = A, *V = B;   // U holds the low-low block of level kd
  for (int k = kd; k >= 1; --k) {
    const int lgM = lgN - (k - 1), lgRh = lgM - lgC - 1;
    const int M = N >> (k - 1), H = M >> 1, R = M >> lgC, Rh = R >> 1;
    const bool cached = k >= cm.kc;
    if (k < kd) cluster_wait();
    // step 1: own rows, low-y (LL | HL) then high-y (LH | HH), into V; the
    // coefficients of uncached levels (with the fused direction update) are
    // loaded kRowU per thread before any is updated
    if (cached) {
      for (int idx = tid; idx < Rh * M; idx += nt) {
        const int jl = idx >> lgM, x = idx & (M - 1);
        V[jl * M + x] = x < H ? U[jl * H + x] : cache[cm.hl(k, jl, x)];
        V[(Rh + jl) * M + x] = cache[cm.lh(k, jl, x)];
      }
    } else {
      constexpr int kRowU = 4;
      for (int idx0 = tid; idx0 < Rh * M; idx0 += kRowU * nt) {
        Raw ra[kRowU], rb[kRowU];
#pragma unroll
        for (int u = 0; u < kRowU; ++u) {
          const int idx = idx0 + u * nt;
          if (idx < Rh * M) {
            const int jl = idx >> lgM, x = idx & (M - 1);
            const int i = crank * Rh + jl;
            if (x >= H) ra[u] = raw(i, x);
            rb[u] = raw(H + i, x);
          }
        }
#pragma unroll
        for (int u = 0; u < kRowU; ++u) {
          const int idx = idx0 + u * nt;
          if (idx < Rh * M) {
            const int jl = idx >> lgM, x = idx & (M - 1);
            const int i = crank * Rh + jl;
            V[jl * M + x] = x < H ? U[jl * H + x] : finish(ra[u], i, x);
            V[(Rh + jl) * M + x] = finish(rb[u], H + i, x);
          }
        }
      }
    }
    __syncthreads();
    // step 2: row synthesis (x) into U: low-y rows at XL, high-y rows at XH
    T *XL = U;                      // HL halo rows, then Rh own rows
    T *XH = U + (HL + Rh) * M;      // same layout
    for (int idx = tid; idx < 2 * Rh * M; idx += nt) {
      const int r = idx >> lgM, j = idx & (M - 1);
      const int q = j & 1;
      const T *row = V + r * M;
      T acc = T(0);
#pragma unroll
      for (int s = 0; s < LF / 2; ++s) {
        const int jj = ((j >> 1) - s) & (H - 1);
        acc += f.hs(q, s) * row[jj] + f.gs(q, s) * row[H + jj];
      }
      (r < Rh ? XL + (HL + r) * M : XH + (HL + r - Rh) * M)[j] = acc;
    }
    cluster.sync();
    // halo: the HL rows before ours (mod H) from the previous CTAs
    for (int idx = tid; idx < HL * M; idx += nt) {
      const int j = idx >> lgM, x = idx & (M - 1);
      const int ii = (crank * Rh - HL + j) & (H - 1);
      const int owner = ii >> lgRh, li = ii & (Rh - 1);
      const T *oU = cluster.map_shared_rank(U, owner);
      XL[j * M + x] = oU[(HL + li) * M + x];
      XH[j * M + x] = oU[(HL + Rh + HL + li) * M + x];
    }
    cluster_arrive();
    __syncthreads();
    // step 3: column synthesis (y) of own output rows
    for (int idx = tid; idx < R * M; idx += nt) {
      const int yl = idx >> lgM, x = idx & (M - 1);
      const int p = yl & 1;
      const int base = ((yl - p) >> 1) + HL;
      T acc = T(0);
#pragma unroll
      for (int s = 0; s < LF / 2; ++s)
        acc += f.hs(p, s) * XL[(base - s) * M + x] + f.gs(p, s) * XH[(base - s) * M + x];
      if (k == 1) out[L.off + (crank * R + yl) * N + x] = acc;
      else V[yl * M + x] = acc;
    }
    __syncthreads();
    T *tmp = U;
    U = V;
    V = tmp;
  }
  if (kd >= 1) cluster_wait();   // the next CTAs have read this CTA's halo rows
}

// -------------------------------------------------------------- k_update
// alpha = (r.z)_it / (p.Ap) from the analysis partials; x += alpha p,
// r -= alpha q, z = J^-1 r; partials r.z and r.r per CTA.  io.out0: x.
// Four consecutive elements per thread and pass (kUpdChunk = 4 * kThreads);
// a CTA makes it.chunks passes over consecutive chunks.
template <typename T>
__device__ __forceinline__ void upd_load(const T *X, const T *R, const T *P, const T *Q, const T *Jv, int precond,
                                         int n, int i0, bool vec, T *xv, T *rv, T *pv, T *qv, T *jv) {
  if (vec) {
    const float4 x4 = reinterpret_cast<const float4 *>(X)[i0 >> 2];
    const float4 r4 = reinterpret_cast<const float4 *>(R)[i0 >> 2];
    const float4 p4 = reinterpret_cast<const float4 *>(P)[i0 >> 2];
    const float4 q4 = reinterpret_cast<const float4 *>(Q)[i0 >> 2];
    const float4 j4 = precond ? reinterpret_cast<const float4 *>(Jv)[i0 >> 2] : make_float4(1.f, 1.f, 1.f, 1.f);
    xv[0] = x4.x; xv[1] = x4.y; xv[2] = x4.z; xv[3] = x4.w;
    rv[0] = r4.x; rv[1] = r4.y; rv[2] = r4.z; rv[3] = r4.w;
    pv[0] = p4.x; pv[1] = p4.y; pv[2] = p4.z; pv[3] = p4.w;
    qv[0] = q4.x; qv[1] = q4.y; qv[2] = q4.z; qv[3] = q4.w;
    jv[0] = j4.x; jv[1] = j4.y; jv[2] = j4.z; jv[3] = j4.w;
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = i0 + u < n ? i0 + u : n - 1;
      xv[u] = X[idx];
      rv[u] = R[idx];
      pv[u] = P[idx];
      qv[u] = Q[idx];
      jv[u] = precond ? Jv[idx] : T(1);
    }
  }
}

template <typename T>
__device__ __forceinline__ void upd_store(T *X, T *R, int n, int i0, bool vec, const T *xv, const T *rv) {
  if (vec) {
    reinterpret_cast<float4 *>(X)[i0 >> 2] = make_float4(xv[0], xv[1], xv[2], xv[3]);
    reinterpret_cast<float4 *>(R)[i0 >> 2] = make_float4(rv[0], rv[1], rv[2], rv[3]);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < n) {
        X[i0 + u] = xv[u];
        R[i0 + u] = rv[u];
      }
  }
}

//
// The step itself: alpha from the sum p.q of the partials (thread 0 of a CTA).
// A breakdown (p.Ap <= 0 or a value that is not finite) is recorded when `record`.
template <typename T>
__device__ __forceinline__ T step_alpha(const InstDev &I, double pq, double rz, double flag, bool record) {
  // r = 0 (so p = 0 and p.Ap = 0) means the iterate is already exact: step 0
  const bool exact = (pq == 0.0 && rz == 0.0);
  const bool bad = !exact && (!(pq > 0.0) || !isfinite(pq) || !isfinite(rz) || flag != 0.0);
  if (bad && record) {
    I.scal[kFlag] = 1.0;
    if (I.bd_word) *reinterpret_cast<volatile int *>(I.bd_word) = 1;
  }
  return T((bad || exact) ? 0.0 : rz / pq);
}

// alpha of every instance of a big launch, one CTA each, before k_update<T, true>.
// In a launch of many update CTAs the sum and the division, about 60 FP64 warp
// instructions per CTA at 16 cycles of the SM's FP64 pipe each, otherwise cost
// more than the vectors: 64 uneven systems (10332 CTAs), GB300, 90 us an update
// with a sum per CTA, 62 us with this kernel's.  One wave of CTAs (up to
// kUpdAlphaBlocks: one E-ELT or 100 m system) is faster without the extra launch
// (100 m frame 2785 against 2823 us).
template <typename T>
__global__ void __launch_bounds__(128) k_alpha(const InstDev *__restrict__ insts, IoArgs io, int flags) {
  pdl_trigger();
  if (io.active && !io.active[blockIdx.x]) return;
  const InstDev &I = insts[blockIdx.x];
  const int iter = flags >> kIterShift;
  const double *part = I.part + I.cl_part_off;
  const int count = I.n_cl_part;
  double *scal = I.scal;
  pdl_wait();
  const double rz = scal[kRz0 + (iter & 1)], flag = scal[kFlag];
  // the sum of sum_partial, in its order, with eight loads in flight per lane
  __shared__ double s_sp[4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double a = 0.0;
  for (int q0 = threadIdx.x; q0 < count; q0 += 8 * 128) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = q0 + u * 128 < count ? part[2 * (q0 + u * 128)] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (q0 + u * 128 < count) a += v[u];
  }
  a = warp_sum(a);
  if (lane == 0) s_sp[w] = a;
  __syncthreads();
  const double pq = ((s_sp[0] + s_sp[1]) + s_sp[2]) + s_sp[3];
  if (threadIdx.x == 0) *reinterpret_cast<T *>(scal + kAlpha) = step_alpha<T>(I, pq, rz, flag, true);
}

// PRE: k_alpha has stored alpha; otherwise every CTA forms it.
template <typename T, bool PRE>
__global__ void __launch_bounds__(kThreads) k_update(const InstDev *__restrict__ insts,
                                                    const UpdItem *__restrict__ items, IoArgs io,
                                                    int flags) {
  __shared__ T s_alpha;
  pdl_trigger();
  const UpdItem it = items[blockIdx.x];
  if (io.active && !io.active[it.inst]) return;
  const InstDev *I = insts + it.inst;
  T *X = static_cast<T *>(io.out0[it.inst]);
  T *R = static_cast<T *>(I->r);
  const int iter = flags >> kIterShift;
  const T *P = dir_buffer<T>(*I, iter);
  const T *Q = static_cast<const T *>(I->q);
  const T *Jv = static_cast<const T *>(I->jinv);
  const int precond = I->precond;
  const int n = I->n;
  pdl_wait();
  const bool aligned = ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(R) |
                         reinterpret_cast<uintptr_t>(P) | reinterpret_cast<uintptr_t>(Q) |
                         reinterpret_cast<uintptr_t>(Jv)) & 15) == 0;
  // the first pass's vectors do not depend on alpha: their loads go out first
  int i0 = it.start + 4 * threadIdx.x;
  bool vec = sizeof(T) == 4 && i0 + 3 < n && aligned;
  T xv[4], rv[4], pv[4], qv[4], jv[4];
  upd_load(X, R, P, Q, Jv, precond, n, i0, vec, xv, rv, pv, qv, jv);
  T alpha;
  if (PRE) {
    alpha = *reinterpret_cast<const T *>(I->scal + kAlpha);
  } else {
    const double rz = I->scal[kRz0 + (iter & 1)];
    const double flag = I->scal[kFlag];
    const double pq = sum_partial(I->part + I->cl_part_off, I->n_cl_part, 0);
    if (threadIdx.x == 0) s_alpha = step_alpha<T>(*I, pq, rz, flag, it.blk == 0);
    __syncthreads();
    alpha = s_alpha;
  }
  // a step of zero (breakdown, or an exact iterate) leaves x and r as they are,
  // even where p or q is not finite: the iterate is frozen
  const bool step = alpha != T(0);
  Acc<T> rz, rr;
  for (int c = 0;;) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (step) {
        xv[u] += alpha * pv[u];
        rv[u] -= alpha * qv[u];
      }
      const T z = precond ? jv[u] * rv[u] : rv[u];
      if (i0 + u < n) {
        rz.add_prod(rv[u], z);
        rr.add_prod(rv[u], rv[u]);
      }
    }
    upd_store(X, R, n, i0, vec, xv, rv);
    if (++c >= it.chunks) break;
    i0 += kUpdChunk;
    vec = sizeof(T) == 4 && i0 + 3 < n && aligned;
    upd_load(X, R, P, Q, Jv, precond, n, i0, vec, xv, rv, pv, qv, jv);
  }
  const double2 s = block_sum2(rz, rr);
  if (threadIdx.x == 0) {
    I->part[I->upd_part_off + 2 * it.blk] = s.x;
    I->part[I->upd_part_off + 2 * it.blk + 1] = s.y;
  }
}

// --------------------------------------------------------------- k_jacobi
// Modified Jacobi diagonal (Sec. 5.1), exactly, at plan time and when alpha is retuned:
//   J_lambda = sum_{m LGS} sigma_m^-2 ||Gamma_m P_m w_lambda||^2 + alpha D_lambda.
// The basis function is separable, w = u(x) v(y), and so are the traced corner
// coordinates, hence P_m w = U(a) V(b) and the Fried slopes are
// sx = dU(a) mV(b), sy = mU(a) dV(b) (d: forward difference, m: two-point
// mean).  With Td(b), Tm(b) the sums of dU^2 and mU^2 over the valid
// subapertures of row b, the norm is sum_b mV(b)^2 Td(b) + dV(b)^2 Tm(b).
//
// A CTA takes TW columns (basis functions in x) and a group of rows
// (basis functions in y) of one level's block, so that Td, Tm are formed once
// per column and row of subapertures and V once per row, not once per
// coefficient: prefix sums of dU^2, mU^2 per column (a warp scan), then in
// chunks of 32 subaperture rows V^2 per row (lanes = b), Td, Tm per column
// (lanes = columns, the row's runs of valid subapertures) and the products
// (lanes = columns; only the rows b that a basis function reaches, a ballot
// mask, since a Daubechies function has compact support).  FP64 throughout:
// bound by the FP64 pipe, which issues one warp instruction in 16 cycles per
// SM on this GPU.  Measured on GB300, E-ELT system: 377 us a call with its table
// copies; one warp per coefficient with a serial prefix sum, dense over the
// pupil, took 25.4 ms (and 5.4 s on the 100 m system).
constexpr int kJacThreads = 256;
constexpr int kJacRows = 32;    // rows (basis functions in y) per CTA at most
constexpr int kJacChunk = 32;   // subaperture rows per pass

// rows per CTA of a level block of side M: fewer for the coarse blocks, whose
// functions span the whole pupil, so that their CTAs are no longer than the rest
__host__ __device__ inline int jac_rows(int M) { return M >= 64 ? kJacRows : (M >= 32 ? 16 : 8); }

// columns per CTA: 32, or fewer when the prefix sums of that many do not fit
__host__ __device__ inline size_t jac_smem(int tw, int nc_max) {
  const size_t stride = static_cast<size_t>((nc_max + 1) | 1);
  return sizeof(double) * (2 * tw * stride + 2 * kJacChunk * tw + 2 * kJacRows * kJacChunk);
}

template <int TW>
__global__ void __launch_bounds__(kJacThreads) k_jacobi(const InstDev *__restrict__ insts,
                                                        const double *__restrict__ prof,
                                                        const int *__restrict__ prof_off,
                                                        const double *__restrict__ pos_fd,
                                                        double *__restrict__ jdiag, void *jinv, int precision,
                                                        int nc_max, double alpha) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned s_mask[kJacRows];
  __shared__ unsigned s_need;
  constexpr int RW = 32 / TW;                               // rows of one warp's lanes
  constexpr int NA = kJacRows / (kJacThreads / 32) / RW;    // accumulators per lane
  const InstDev &I = insts[0];
  const int J = I.J, k = J - static_cast<int>(blockIdx.y), l = blockIdx.z;   // coarse (longest) levels first
  const LayerDev &L = I.layers[l];
  const int N = L.N, M = N >> (k - 1), H = M >> 1, rows = jac_rows(M);
  const int ntx = (M + TW - 1) / TW, nty = (M + rows - 1) / rows;
  if (static_cast<int>(blockIdx.x) >= ntx * nty) return;
  const int c0 = (static_cast<int>(blockIdx.x) % ntx) * TW, r0 = (static_cast<int>(blockIdx.x) / ntx) * rows;
  if (k < J && c0 + TW <= H && r0 + rows <= H) return;      // all low-low: a coarser level's block
  const int stride = (nc_max + 1) | 1;
  double *Pd = reinterpret_cast<double *>(smem_raw);        // [TW][stride] prefix sums of dU^2
  double *Pm = Pd + TW * stride;                            //   and of mU^2
  double *Td = Pm + TW * stride;                            // [kJacChunk][TW]
  double *Tm = Td + kJacChunk * TW;
  double *Vm = Tm + kJacChunk * TW;                         // [kJacRows][kJacChunk] mV^2
  double *Vd = Vm + kJacRows * kJacChunk;                   //   and dV^2
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kJacThreads / 32;
  // first sample of basis function c of the block on the periodic grid, and its profile
  auto shift = [&](int c) { return (c < H ? c : c - H) << k; };
  auto profile = [&](int c) { return prof + prof_off[(l * (J + 1) + k) * 2 + (c < H ? 0 : 1)]; };
  // samples of a level-k function that are not zero (0: the whole circle)
  const long long sup = ((1LL << k) - 1) * (I.Lf - 1) + 1;
  const int len = sup >= N ? N : static_cast<int>(sup);
  // the function with profile u and shift s at traced corner (x0, f); false: zero there
  auto reaches = [&](int x0, int s) { return ((x0 - s) & (N - 1)) < len || ((x0 + 1 - s) & (N - 1)) < len; };
  auto value = [&](const double *u, int s, int x0, double f) {
    return (1.0 - f) * u[(x0 - s) & (N - 1)] + f * u[(x0 + 1 - s) & (N - 1)];
  };
  double tot[NA];
#pragma unroll
  for (int i = 0; i < NA; ++i) tot[i] = 0.0;
  for (int m = 0; m < I.n_wfs; ++m) {
    const WfsDev &W = I.wfs[m];
    if (!W.is_lgs) continue;
    const int nc = W.nc, n = W.n;
    const int po = I.pos_off[m * I.n_layers + l];
    const int *xi = I.pos_i0 + po, *yi = xi + nc;
    const double *xf = pos_fd + po, *yf = xf + nc;
    __syncthreads();   // the previous sensor's products are done with the prefix sums
    for (int j = warp; j < TW; j += nw) {
      const int c = c0 + j;
      double cd = 0.0, cm = 0.0;   // sums before this chunk of 32 subapertures
      if (lane == 0) Pd[j * stride] = Pm[j * stride] = 0.0;
      const double *u = profile(c < M ? c : 0);
      const int s = shift(c < M ? c : 0);
      for (int a0 = 0; a0 < n; a0 += 32) {
        const int a = a0 + lane;
        const bool on = c < M && a < n && (reaches(xi[a], s) || reaches(xi[a + 1], s));
        double d2 = cd, m2 = cm;
        if (__any_sync(0xffffffffu, on)) {
          d2 = m2 = 0.0;
          if (on) {
            const double u0 = value(u, s, xi[a], xf[a]), u1 = value(u, s, xi[a + 1], xf[a + 1]);
            const double d = u1 - u0, mm = 0.5 * (u0 + u1);
            d2 = d * d;
            m2 = mm * mm;
          }
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double xd = __shfl_up_sync(0xffffffffu, d2, o), xm = __shfl_up_sync(0xffffffffu, m2, o);
            if (lane >= o) {
              d2 += xd;
              m2 += xm;
            }
          }
          d2 += cd;
          m2 += cm;
          cd = __shfl_sync(0xffffffffu, d2, 31);
          cm = __shfl_sync(0xffffffffu, m2, 31);
        }
        if (a < n) {
          Pd[j * stride + a + 1] = d2;
          Pm[j * stride + a + 1] = m2;
        }
      }
    }
    double part[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) part[i] = 0.0;
    const int *runs = I.run_rows + W.run_off;
    for (int b0 = 0; b0 < n; b0 += kJacChunk) {
      if (threadIdx.x == 0) s_need = 0u;
      __syncthreads();   // the prefix sums are written; the previous chunk's products are done
      for (int i = warp; i < rows; i += nw) {
        const int r = r0 + i, b = b0 + lane;
        const int s = shift(r < M ? r : 0);
        const bool on = r < M && b < n && (reaches(yi[b], s) || reaches(yi[b + 1], s));
        const unsigned mask = __ballot_sync(0xffffffffu, on);
        if (on) {
          const double *u = profile(r);
          const double v0 = value(u, s, yi[b], yf[b]), v1 = value(u, s, yi[b + 1], yf[b + 1]);
          const double d = v1 - v0, mm = 0.5 * (v0 + v1);
          Vd[i * kJacChunk + lane] = d * d;
          Vm[i * kJacChunk + lane] = mm * mm;
        }
        if (lane == 0) {
          s_mask[i] = mask;
          if (mask) atomicOr(&s_need, mask);
        }
      }
      __syncthreads();
      const unsigned need = s_need;
      for (int bl = warp; bl < kJacChunk; bl += nw) {
        if (!((need >> bl) & 1u) || lane >= TW) continue;
        double sd = 0.0, sm = 0.0;
        for (int q = runs[b0 + bl]; q < runs[b0 + bl + 1]; ++q) {
          const int2 run = I.run_ab[q];
          sd += Pd[lane * stride + run.y] - Pd[lane * stride + run.x];
          sm += Pm[lane * stride + run.y] - Pm[lane * stride + run.x];
        }
        Td[bl * TW + lane] = sd;
        Tm[bl * TW + lane] = sm;
      }
      __syncthreads();
      const int j = lane & (TW - 1), rl = lane / TW;
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int row = (warp + i * nw) * RW + rl;
        unsigned mask = row < rows ? s_mask[row] : 0u;
        while (mask) {
          const int bl = __ffs(mask) - 1;
          mask &= mask - 1u;
          part[i] += Vm[row * kJacChunk + bl] * Td[bl * TW + j] + Vd[row * kJacChunk + bl] * Tm[bl * TW + j];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NA; ++i) tot[i] += W.inv_sigma2 * part[i];
  }
  // alpha < 0: the plan's own alpha D; otherwise alpha D for the given alpha
  const double ad = alpha < 0.0 ? L.dalpha[k] : alpha * L.dprior[k];
  const int cc = c0 + (lane & (TW - 1)), rl = lane / TW;
#pragma unroll
  for (int i = 0; i < NA; ++i) {
    const int row = (warp + i * nw) * RW + rl, rr = r0 + row;
    if (row >= rows || rr >= M || cc >= M || (k < J && rr < H && cc < H)) continue;
    const int lam = L.off + rr * N + cc;
    const double Jv = tot[i] + ad;
    jdiag[lam] = Jv;
    if (jinv) {
      if (precision) static_cast<double *>(jinv)[lam] = 1.0 / Jv;
      else static_cast<float *>(jinv)[lam] = float(1.0 / Jv);
    }
  }
}

// ------------------------------------------------------------- launchers

namespace {

template <typename K>
cudaError_t allow_cluster(K kernel) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxTransformSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

template <typename T, int LF>
cudaError_t allow_lf() {
  cudaError_t e = cudaSuccess;
#define TOMO_CFG(K) if (e == cudaSuccess) e = allow_cluster(K)
  TOMO_CFG((k_synthesis<T, 0, LF>));
  TOMO_CFG((k_synthesis<T, 1, LF>));
  TOMO_CFG((k_analysis<T, 0, kEpiPlain, LF>));
  TOMO_CFG((k_analysis<T, 1, kEpiPlain, LF>));
  TOMO_CFG((k_analysis<T, 1, kEpiOp, LF>));
  TOMO_CFG((k_analysis<T, 1, kEpiResid, LF>));
  TOMO_CFG((k_analysis<T, 2, kEpiPlain, LF>));
  TOMO_CFG((k_analysis<T, 2, kEpiOp, LF>));
  TOMO_CFG((k_analysis<T, 2, kEpiResid, LF>));
#undef TOMO_CFG
  return e;
}

template <typename T>
cudaError_t allow_type() {
  cudaError_t e = allow_lf<T, 2>();
  if (e == cudaSuccess) e = allow_lf<T, 4>();
  if (e == cudaSuccess) e = allow_lf<T, 6>();
  if (e == cudaSuccess) e = allow_lf<T, 8>();
  const void *fwd[14] = {   // the small launches' forms first
      reinterpret_cast<const void *>(k_forward<T, 0, false, 1>),
      reinterpret_cast<const void *>(k_forward<T, 1, false, 1>),
      reinterpret_cast<const void *>(k_forward<T, 2, false, 1>),
      reinterpret_cast<const void *>(k_forward<T, 0, true, 1>),
      reinterpret_cast<const void *>(k_forward<T, 1, true, 1>),
      reinterpret_cast<const void *>(k_forward<T, 2, true, 1>),
      reinterpret_cast<const void *>(k_forward<T, 3, false, 1>),
      reinterpret_cast<const void *>(k_forward<T, 0, false, kFwdStrip<T>>),
      reinterpret_cast<const void *>(k_forward<T, 1, false, kFwdStrip<T>>),
      reinterpret_cast<const void *>(k_forward<T, 2, false, kFwdStrip<T>>),
      reinterpret_cast<const void *>(k_forward<T, 0, true, kFwdStrip<T>>),
      reinterpret_cast<const void *>(k_forward<T, 1, true, kFwdStrip<T>>),
      reinterpret_cast<const void *>(k_forward<T, 2, true, kFwdStrip<T>>),
      reinterpret_cast<const void *>(k_forward<T, 3, false, kFwdStrip<T>>)};
  for (int i = 0; i < 14 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(fwd[i], cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxForwardSmem);
  for (int i = 0; i < 7 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(fwd[i], cudaFuncAttributePreferredSharedMemoryCarveout, kFwdCarveout);
  return e;
}

template <typename T, int LF>
cudaError_t synth_lf(int src, int flags, const InstDev *insts, const ClusterItem *items, int n_clusters,
                     int C, size_t smem, const IoArgs &io, cudaStream_t s) {
  const dim3 g(n_clusters * C);
  // two CTAs of 256 threads per SM when their shared memory allows (two clusters per GPC),
  // else one CTA of 512
  const int nt = smem <= kTwoPerSmSmem ? kSynthThreads / 2 : kSynthThreads;
  return src ? launch_ex(k_synthesis<T, 1, LF>, g, nt, C, smem, s, insts, items, io, flags)
             : launch_ex(k_synthesis<T, 0, LF>, g, nt, C, smem, s, insts, items, io, flags);
}

template <typename T>
cudaError_t synth_t(int src, int lf, int flags, const InstDev *insts, const ClusterItem *items,
                    int n_clusters, int C, size_t smem, const IoArgs &io, cudaStream_t s) {
  switch (lf) {
    case 2: return synth_lf<T, 2>(src, flags, insts, items, n_clusters, C, smem, io, s);
    case 4: return synth_lf<T, 4>(src, flags, insts, items, n_clusters, C, smem, io, s);
    case 6: return synth_lf<T, 6>(src, flags, insts, items, n_clusters, C, smem, io, s);
    case 8: return synth_lf<T, 8>(src, flags, insts, items, n_clusters, C, smem, io, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, int LF>
cudaError_t anal_lf(int src, int epi, int flags, const InstDev *insts, const ClusterItem *items,
                    int n_clusters, int C, size_t smem, const IoArgs &io, cudaStream_t s) {
  const dim3 g(n_clusters * C);
  // two CTAs of 512 threads per SM when their shared memory allows, else one of 1024
  const int nt = smem <= kTwoPerSmSmem ? kAnalysisThreads : kAnalysisThreadsMax;
#define TOMO_AN(S, E) launch_ex(k_analysis<T, S, E, LF>, g, nt, C, smem, s, insts, items, io, flags)
  if (src == 0) return TOMO_AN(0, kEpiPlain);
  if (src == 2) {
    if (epi == kEpiPlain) return TOMO_AN(2, kEpiPlain);
    if (epi == kEpiOp) return TOMO_AN(2, kEpiOp);
    return TOMO_AN(2, kEpiResid);
  }
  if (epi == kEpiPlain) return TOMO_AN(1, kEpiPlain);
  if (epi == kEpiOp) return TOMO_AN(1, kEpiOp);
  return TOMO_AN(1, kEpiResid);
#undef TOMO_AN
}

template <typename T>
cudaError_t anal_t(int src, int epi, int lf, int flags, const InstDev *insts, const ClusterItem *items,
                   int n_clusters, int C, size_t smem, const IoArgs &io, cudaStream_t s) {
  switch (lf) {
    case 2: return anal_lf<T, 2>(src, epi, flags, insts, items, n_clusters, C, smem, io, s);
    case 4: return anal_lf<T, 4>(src, epi, flags, insts, items, n_clusters, C, smem, io, s);
    case 6: return anal_lf<T, 6>(src, epi, flags, insts, items, n_clusters, C, smem, io, s);
    case 8: return anal_lf<T, 8>(src, epi, flags, insts, items, n_clusters, C, smem, io, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t configure_kernels() {
  cudaError_t e = allow_type<float>();
  if (e == cudaSuccess) e = allow_type<double>();
  if (e == cudaSuccess) e = configure_streamed_kernels();
  if (e == cudaSuccess) e = configure_gather_kernels();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_jacobi<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTransformSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_jacobi<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTransformSmem);
  return e;
}

size_t forward_smem(int n_layers, int precision) {
  return precision ? fwd_table_bytes<double>(n_layers) : fwd_table_bytes<float>(n_layers);
}

cudaError_t launch_synthesis(int precision, int src, int lf, int flags, const InstDev *insts,
                             const ClusterItem *items, int n_clusters, int C, size_t smem,
                             const IoArgs &io, cudaStream_t s) {
  return precision == 0 ? synth_t<float>(src, lf, flags, insts, items, n_clusters, C, smem, io, s)
                        : synth_t<double>(src, lf, flags, insts, items, n_clusters, C, smem, io, s);
}

cudaError_t launch_analysis(int precision, int src, int epi, int lf, int flags, const InstDev *insts,
                             const ClusterItem *items, int n_clusters, int C, size_t smem, const IoArgs &io,
                             cudaStream_t s) {
  return precision == 0 ? anal_t<float>(src, epi, lf, flags, insts, items, n_clusters, C, smem, io, s)
                        : anal_t<double>(src, epi, lf, flags, insts, items, n_clusters, C, smem, io, s);
}

template <typename T, bool EL, int RS>
cudaError_t fwd_rs(int mode, dim3 g, size_t sm, cudaStream_t s, const InstDev *insts, const FwdItem *items,
                   const IoArgs &io) {
  constexpr int nt = 32 * kFwdPsi<T> / RS;
  if (mode == 0) return launch_ex(k_forward<T, 0, EL, RS>, g, nt, 0, sm, s, insts, items, io);
  if (mode == 1) return launch_ex(k_forward<T, 1, EL, RS>, g, nt, 0, sm, s, insts, items, io);
  if (mode == 3) return launch_ex(k_forward<T, 3, false, RS>, g, nt, 0, sm, s, insts, items, io);
  return launch_ex(k_forward<T, 2, EL, RS>, g, nt, 0, sm, s, insts, items, io);
}

template <typename T, bool EL>
cudaError_t fwd_t(int mode, dim3 g, size_t sm, cudaStream_t s, const InstDev *insts, const FwdItem *items,
                  const IoArgs &io) {
  return g.x <= kFwdSmallLaunch ? fwd_rs<T, EL, 1>(mode, g, sm, s, insts, items, io)
                                : fwd_rs<T, EL, kFwdStrip<T>>(mode, g, sm, s, insts, items, io);
}

cudaError_t launch_forward(int precision, int mode, int max_layers, int elong, size_t smem_analysis,
                           const InstDev *insts, const FwdItem *items, int n_items, const IoArgs &io, cudaStream_t s) {
  const dim3 g(n_items);
  const size_t need = forward_smem(max_layers, precision);
  size_t sm = need;
  if (precision == 0 && n_items <= kFwdSmallLaunch && smem_analysis >= kFwdBesideSmem) sm = max(need, kFwdBesideSmem);
  if (precision == 1 && n_items <= kFwdAloneLaunch) sm = max(need, kFwdAloneSmem);
  if (precision == 0)
    return elong ? fwd_t<float, true>(mode, g, sm, s, insts, items, io)
                 : fwd_t<float, false>(mode, g, sm, s, insts, items, io);
  return elong ? fwd_t<double, true>(mode, g, sm, s, insts, items, io)
               : fwd_t<double, false>(mode, g, sm, s, insts, items, io);
}

template <typename T>
cudaError_t update_t(int flags, const InstDev *insts, int count, const UpdItem *items, int n_items, const IoArgs &io,
                     cudaStream_t s) {
  const dim3 g(n_items);
  if (n_items <= kUpdAlphaBlocks) return launch_ex(k_update<T, false>, g, kThreads, 0, 0, s, insts, items, io, flags);
  const cudaError_t e = launch_ex(k_alpha<T>, dim3(count), 128, 0, 0, s, insts, io, flags);
  return e != cudaSuccess ? e : launch_ex(k_update<T, true>, g, kThreads, 0, 0, s, insts, items, io, flags);
}

int update_launches(int n_items) { return n_items <= kUpdAlphaBlocks ? 1 : 2; }

cudaError_t launch_update(int precision, int flags, const InstDev *insts, int count, const UpdItem *items,
                          int n_items, const IoArgs &io, cudaStream_t s) {
  return precision == 0 ? update_t<float>(flags, insts, count, items, n_items, io, s)
                        : update_t<double>(flags, insts, count, items, n_items, io, s);
}

cudaError_t launch_jacobi(const InstDev *insts, int n_layers, int J, int N_max, const double *prof,
                          const int *prof_off, const double *pos_fd, double *jdiag, void *jinv, int precision,
                          int nc_max, double alpha, cudaStream_t s) {
  // 32 columns per CTA while their prefix sums fit (pupils up to about 360 subapertures), else 8
  const int tw = jac_smem(32, nc_max) <= static_cast<size_t>(kMaxTransformSmem) ? 32 : 8;
  const size_t smem = jac_smem(tw, nc_max);
  int tiles = 1;
  for (int k = 1; k <= J; ++k) {
    const int M = N_max >> (k - 1), rows = jac_rows(M);
    tiles = max(tiles, ((M + tw - 1) / tw) * ((M + rows - 1) / rows));
  }
  const dim3 g(tiles, J, n_layers);
  if (tw == 32)
    k_jacobi<32><<<g, kJacThreads, smem, s>>>(insts, prof, prof_off, pos_fd, jdiag, jinv, precision, nc_max, alpha);
  else
    k_jacobi<8><<<g, kJacThreads, smem, s>>>(insts, prof, prof_off, pos_fd, jdiag, jinv, precision, nc_max, alpha);
  return cudaGetLastError();
}

}  // namespace tomo
