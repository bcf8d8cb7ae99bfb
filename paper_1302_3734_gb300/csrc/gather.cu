// The separate gather kernel (sm_103a): g = sum_m P_m^T v_m (Sec. 5.1, the
// transposed ray-trace) for plans whose gather tables do not fit the analysis
// kernel's shared memory, one CTA per (instance, layer, band of rows).
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.h"
#include "device_util.cuh"
#include "launch.h"
#include "transform.cuh"
#include "adjoint.cuh"

namespace tomo {

// Each sensor's term of node (row k, column i) is
//   sum_ty wy_ty(k) * U(b0(k) + ty, i),   U(b, i) = sum_tx wx_tx(i) * v(a0(i) + tx, b),
// the same two nested sums, in the same order, as the window sum of the fused
// gather.  A warp takes 32 of the columns that the sensor's taps reach (one
// per lane) and a run of the band's node rows, and walks down the rows keeping
// the KT column sums U of the last window in registers.  The row records are
// the same for every lane, so the window moves by the same number of corner
// rows in the whole warp: where it moves by one over kWalk node rows (most of
// the time, unless the cone effect skips a row), only its new last row is
// summed, KT products a node instead of KT * KT, and there is no branch in
// between; elsewhere each node sums its own window.  What a sensor needs (the
// corner rows of v that the band reaches, its column records and the band's
// row records) comes by bulk copies into one of two stages while the other is
// used, so the walk reads shared memory only; one barrier per sensor.  Each
// node receives the sensors' terms in sensor order, as the fused gathers do.
//
// Bound by latency (barriers, the stages' copies) at two CTAs per SM.  Against
// one pass for the column sums and one for the nodes, with a barrier after
// each and every corner row summed for every band (GB300, cold launch): 16
// E-ELT systems 49.2 -> 33.5 us, 64 uneven systems 82.9 -> 54.4 us, the 100 m
// system 82.2 -> 55.4 us.
// (Four rows took 16 E-ELT systems 2% longer: one skipped corner row sends the batch to whole windows.)
constexpr int kWalk = 2;

template <typename T, int KT>
__device__ __forceinline__ T col_sum(const T *wx, const T *v) {
  T sx = wx[0] * v[0];
#pragma unroll
  for (int t = 1; t < KT; ++t) sx += wx[t] * v[t];
  return sx;
}

// nrow node rows (records yr) of one lane's column (record at xr): A[r * N] +=
// the sensor's terms, in the lanes that are on.  v: the staged rows, indexed by
// the row records' offsets.
template <typename T, int KT>
__device__ __forceinline__ void gather_column(const T *xr, const T *yr, int nrow, const T *v, int nc, T *A, int N,
                                              bool on) {
  constexpr int RS = TapRec<T, KT>::RS;
  TapRec<T, KT> x;
  x.load(xr);
  on = on && x.off >= 0;   // (every lane walks)
  const T *pv = v + (x.off >= 0 ? x.off : 0);
  T U[KT];
#pragma unroll
  for (int t = 0; t < KT; ++t) U[t] = T(0);
#pragma unroll 1
  for (int b0 = 0; b0 < nrow; b0 += 32) {
    // bit r: row b0 + r has a window one corner row below the one before it
    const int rl = b0 + (threadIdx.x & 31);
    const int ro = rl < nrow ? TapRec<T, KT>::offset(yr + rl * RS) : -1;
    const int rp = rl > 0 && rl < nrow ? TapRec<T, KT>::offset(yr + (rl - 1) * RS) : -1;
    const unsigned steps = __ballot_sync(0xffffffffu, ro >= 0 && rp >= 0 && ro == rp + nc);
#pragma unroll 1
    for (int b = b0; b < min(nrow, b0 + 32); b += kWalk) {
      const T *yb = yr + b * RS;
      T *Ab = A + b * N;
      if (((steps >> (b - b0)) & ((1u << kWalk) - 1u)) == (1u << kWalk) - 1u) {
        TapRec<T, KT> y[kWalk];
#pragma unroll
        for (int u = 0; u < kWalk; ++u) y[u].load(yb + u * RS);
        const T *p = pv + y[0].off + (KT - 1) * nc;
#pragma unroll
        for (int u = 0; u < kWalk; ++u, p += nc) {
          T w[KT];
#pragma unroll
          for (int q = 0; q < KT; ++q) w[q] = p[q];
#pragma unroll
          for (int t = 0; t + 1 < KT; ++t) U[t] = U[t + 1];
          U[KT - 1] = col_sum<T, KT>(x.w, w);
          T s = T(0);
#pragma unroll
          for (int t = 0; t < KT; ++t) s += y[u].w[t] * U[t];
          if (on) Ab[u * N] += s;
        }
      } else {
#pragma unroll 1
        for (int u = 0; u < min(kWalk, nrow - b); ++u) {
          TapRec<T, KT> y;
          y.load(yb + u * RS);
          if (y.off < 0) continue;
          const T *p = pv + y.off;
          T s = T(0);
#pragma unroll
          for (int t = 0; t < KT; ++t, p += nc) {
            T w[KT];
#pragma unroll
            for (int q = 0; q < KT; ++q) w[q] = p[q];
            U[t] = col_sum<T, KT>(x.w, w);
            s += y.w[t] * U[t];
          }
          if (on) Ab[u * N] += s;
        }
      }
    }
  }
}

// ------------------------------------------------------------- k_gather
// g = sum_m P_m^T v_m (Sec. 5.1, the transposed ray-trace) into the plan's phi
// buffer, one CTA per (instance, layer, band of N / gather_bands rows), the
// costliest bands first (the host orders items), for plans whose gather tables
// are not staged in the analysis kernel; k_analysis with SRC 2 or the streamed
// analysis then transforms it.  phi is free here: the forward kernel that read
// it has finished (dependency wait) and the next synthesis rewrites it.
// tt_mode as in edge_coefficients; io.in1: the slopes (tip/tilt-only data).
template <typename T>
__global__ void __launch_bounds__(kGatherThreads, sizeof(T) == 4 ? 2 : 1) k_gather(const InstDev *__restrict__ insts,
                                                           const PassItem *__restrict__ items,
                                                           IoArgs io, int tt_mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ InstDev sI;
  __shared__ T s_coef[4 * kMaxEdgeSlots];
  __shared__ int s_go[kMaxGatherSensors], s_nc[kMaxGatherSensors], s_el[kMaxGatherSensors];
  __shared__ int2 s_cols[kMaxGatherSensors], s_br[kMaxGatherSensors], s_kr[kMaxGatherSensors];
  __shared__ int s_md;
  __shared__ uint64_t s_bar[2];
  constexpr int vq = 16 / static_cast<int>(sizeof(T));   // elements per 16 bytes
  pdl_trigger();
  const PassItem it = items[blockIdx.x];
  const int band = it.row0, tid = threadIdx.x, nt = blockDim.x;
  if (io.active && !io.active[it.inst]) return;
  load_inst(&sI, insts + it.inst);
  const InstDev &I = sI;
  const int Cg = I.gather_bands;
  if (tid < 32) {
    // the dense sensors whose taps reach this band, in sensor order
    int md = 0;
    for (int m0 = 0; m0 < I.n_wfs && md < kMaxGatherSensors; m0 += 32) {
      const int m = m0 + tid, at = m * I.n_layers + it.layer;
      int2 cols = make_int2(0, 0);
      int4 br = make_int4(0, 0, 0, 0);
      if (m < I.n_wfs && I.wfs[m].kind != kTTOnly) {
        cols = I.gt_cols[at];
        br = I.gt_brows[at * Cg + band];
      }
      const bool reach = cols.y != 0 && br.y != 0;
      const unsigned mask = __ballot_sync(0xffffffffu, reach);
      const int j = md + __popc(mask & ((1u << tid) - 1u));
      if (reach && j < kMaxGatherSensors) {
        const WfsDev &W = I.wfs[m];
        s_go[j] = I.gt_off[at];
        s_nc[j] = W.nc;
        s_el[j] = (W.elong && W.kind == kRemoveTT) ? W.tt_idx : -1;
        s_cols[j] = cols;
        s_br[j] = make_int2(br.x, br.y);
        s_kr[j] = make_int2(br.z, br.w);
      }
      md += __popc(mask);
    }
    if (tid == 0) {
      s_md = min(md, kMaxGatherSensors);
      mbar_init(&s_bar[0]);
      mbar_init(&s_bar[1]);
    }
  }
  const LayerDev &L = I.layers[it.layer];
  const int N = L.N, R0 = N / min(Cg, N), KT = I.max_taps, RS = I.rec_stride;
  const GatherSmem gs = gather_smem_layout(R0, N, RS, static_cast<int>(sizeof(T)), I.max_band_v);
  T *A = reinterpret_cast<T *>(smem_raw);
  T *g = static_cast<T *>(I.phi) + L.off + band * R0 * N;
  const int2 seg = I.tt_seg[it.layer * Cg + band];
  const int e0 = I.tt_beg[seg.x], e1 = I.tt_beg[seg.y];
  __syncthreads();
  const int Md = s_md;
  const T *rec = static_cast<const T *>(I.gt_rec), *vv = static_cast<const T *>(I.v);
  // one thread: the copies of sensor md into its stage, completing on its barrier: the constant
  // records, then the band rows [br.x, br.x + nb nc) of v (KT rows at least) and KT more elements
  // (zero-weight taps when nc < KT) from the 16-byte boundary at or below br.x (the plan pads v beyond its last sensor)
  auto stage_records = [&](int md) {
    const int2 br = s_br[md];
    const int nq = (br.x % vq + max(br.y, KT) * s_nc[md] + KT + vq - 1) / vq;
    unsigned char *st = smem_raw + gs.stage + (md & 1) * gs.stage_bytes;
    const uint32_t bx = static_cast<uint32_t>(N * RS * sizeof(T)), by = static_cast<uint32_t>(R0 * RS * sizeof(T));
    mbar_arm(&s_bar[md & 1], bx + by + static_cast<uint32_t>(nq) * 16u);
    bulk_copy_g2s(st + gs.xr, rec + static_cast<size_t>(s_go[md]) * RS, bx, &s_bar[md & 1]);
    bulk_copy_g2s(st + gs.yr, rec + static_cast<size_t>(s_go[md] + N + band * R0) * RS, by, &s_bar[md & 1]);
  };
  auto stage_rows = [&](int md) {
    const int2 br = s_br[md];
    const int nq = (br.x % vq + max(br.y, KT) * s_nc[md] + KT + vq - 1) / vq;
    bulk_copy_g2s(smem_raw + gs.stage + (md & 1) * gs.stage_bytes, vv + br.x / vq * vq,
                  static_cast<uint32_t>(nq) * 16u, &s_bar[md & 1]);
  };
  if (tid == 0)
    for (int md = 0; md < min(2, Md); ++md) stage_records(md);
  for (int node = tid; node < R0 * N; node += nt) A[node] = T(0);
  pdl_wait();
  if (tid == 0) {
    fence_async_global();   // v was written by the previous kernel
    for (int md = 0; md < min(2, Md); ++md) stage_rows(md);
  }
  if (I.n_edge_wfs > 0)
    edge_coefficients<T>(I, s_coef, tt_mode, static_cast<const T *>(io.in1[it.inst]));
  else
    __syncthreads();   // the band buffer is zero
  const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  for (int md = 0; md < Md; ++md) {
    unsigned char *st = smem_raw + gs.stage + (md & 1) * gs.stage_bytes;
    T *V = reinterpret_cast<T *>(st);
    // a copy that never completed (it does not happen with valid tables) makes the solve report a breakdown
    if (!mbar_wait(&s_bar[md & 1], (md >> 1) & 1)) I.scal[kFlag] = 1.0;
    const int2 cols = s_cols[md], br = s_br[md], kr = s_kr[md];
    const int nc = s_nc[md], el = s_el[md], g0 = br.x / vq * vq;
    if (el >= 0) {
      // spot elongation with tip/tilt removal: v + m_x Gx + m_y Gy
      const T mx = s_coef[2 * kMaxEdgeSlots + 2 * el], my = s_coef[2 * kMaxEdgeSlots + 2 * el + 1];
      const T *gx = static_cast<const T *>(I.gel) + br.x, *gy = gx + I.v_total;
      T *vr = V + (br.x - g0);
      for (int i = tid; i < br.y * nc; i += nt) vr[i] += mx * __ldg(gx + i) + my * __ldg(gy + i);
      fence_async_shared();   // before the stage's next bulk copy
      __syncthreads();
    }
    // tiles of 32 columns by rpt of the rows that the sensor reaches, one or more per warp
    const int ntc = (cols.y + 31) >> 5, nts = max(1, nw / ntc), rpt = (kr.y + nts - 1) / nts;
    for (int tile = warp; tile < ntc * nts; tile += nw) {
      const int ts = tile / ntc, c = (tile - ts * ntc) * 32 + lane, k0 = kr.x + ts * rpt;
      const int nrow = min(rpt, kr.x + kr.y - k0);
      if (nrow <= 0) continue;
      const int i = (cols.x + min(c, cols.y - 1)) & (N - 1);
      const T *xr = reinterpret_cast<const T *>(st + gs.xr) + i * RS;
      const T *yr = reinterpret_cast<const T *>(st + gs.yr) + k0 * RS;
      T *At = A + k0 * N + i;
      const bool lane_on = c < cols.y;
      if (KT <= 2) gather_column<T, 2>(xr, yr, nrow, V - g0, nc, At, N, lane_on);
      else if (KT == 3) gather_column<T, 3>(xr, yr, nrow, V - g0, nc, At, N, lane_on);
      else gather_column<T, 4>(xr, yr, nrow, V - g0, nc, At, N, lane_on);
    }
    __syncthreads();   // the stage is free, and the next sensor's tiles may take other columns
    if (tid == 0 && md + 2 < Md) {
      stage_records(md + 2);
      stage_rows(md + 2);
    }
  }
  if (I.n_edge_wfs > 0 && !gather_edges_fit(gs, e1 - e0, static_cast<int>(sizeof(T)))) {
    // more pupil-edge terms than shared memory holds: each node's from global memory, in list order
    for (int j = seg.x + tid; j < seg.y; j += nt)
      A[I.tt_node[j]] += edge_node_sum<T>(I.tt_beg[j], I.tt_beg[j + 1], I.tt_k, static_cast<const T *>(I.tt_w), s_coef);
    __syncthreads();
  } else if (I.n_edge_wfs > 0) {
    // the pupil-edge list, added after the sensors: every entry's term into the free stages
    // (coalesced loads), then each node's terms in list order
    T *C = reinterpret_cast<T *>(smem_raw + gs.stage);
    const int *tk = I.tt_k, *tb = I.tt_beg, *tn = I.tt_node;
    const T *tw = static_cast<const T *>(I.tt_w);
    // (the first nodes' list bounds are requested together with the entries)
    constexpr int kNodes = 3;
    int node[kNodes], beg[kNodes], end[kNodes];
#pragma unroll
    for (int u = 0; u < kNodes; ++u) {
      const int j = seg.x + tid + u * nt;
      node[u] = beg[u] = end[u] = 0;
      if (j < seg.y) {
        node[u] = tn[j];
        beg[u] = tb[j] - e0;
        end[u] = tb[j + 1] - e0;
      }
    }
    for (int e = e0 + tid; e < e1; e += kEdgeBatch * nt) {
      int k[kEdgeBatch];
      T wx[kEdgeBatch], wy[kEdgeBatch];
#pragma unroll
      for (int u = 0; u < kEdgeBatch; ++u) {
        const int q = min(e + u * nt, e1 - 1);
        k[u] = tk[q];
        wx[u] = tw[2 * q];
        wy[u] = tw[2 * q + 1];
      }
#pragma unroll
      for (int u = 0; u < kEdgeBatch; ++u)
        if (e + u * nt < e1) C[e + u * nt - e0] = s_coef[2 * k[u]] * wx[u] + s_coef[2 * k[u] + 1] * wy[u];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kNodes; ++u) {
      T acc = T(0);
      for (int e = beg[u]; e < end[u]; ++e) acc += C[e];
      if (end[u] > beg[u]) A[node[u]] += acc;
    }
    for (int j = seg.x + tid + kNodes * nt; j < seg.y; j += nt) {
      T acc = T(0);
      for (int e = tb[j] - e0; e < tb[j + 1] - e0; ++e) acc += C[e];
      A[tn[j]] += acc;
    }
    __syncthreads();
  }
  const uint4 *A4 = reinterpret_cast<const uint4 *>(A);
  for (int q = tid; q < R0 * N / vq; q += nt) reinterpret_cast<uint4 *>(g)[q] = A4[q];
}

cudaError_t launch_gather(int precision, int tt_mode, const InstDev *insts, const PassItem *items, int n_items,
                          size_t smem, const IoArgs &io, cudaStream_t s) {
  const dim3 g(n_items);
  return precision == 0 ? launch_ex(k_gather<float>, g, kGatherThreads, 0, smem, s, insts, items, io, tt_mode)
                        : launch_ex(k_gather<double>, g, kGatherThreads, 0, smem, s, insts, items, io, tt_mode);
}

cudaError_t configure_gather_kernels() {
  cudaError_t e = cudaFuncSetAttribute(k_gather<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTransformSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_gather<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTransformSmem);
  return e;
}

}  // namespace tomo
