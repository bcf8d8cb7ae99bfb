// Streamed transform kernels (sm_103a): the periodic 2-D Daubechies DWT and its
// inverse of layers too large for the cluster-per-layer kernels to keep more
// than one cluster per GPC resident, level by level over row tiles of the
// whole grid, with the PCG epilogue (Sec. 5.1, eq. eqn_lse) and the fused
// direction update of the cluster kernels.
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.h"
#include "device_util.cuh"
#include "launch.h"
#include "transform.cuh"

namespace tomo {

// ---------------------------------------------------- streamed transforms
// For layers whose transform kernels would hold one cluster per GPC at a time
// (the clusters' rows of the finest level do not fit two CTAs per SM), the
// transforms run level by level over row tiles of the whole grid instead, with
// no cluster: each CTA reads its halo rows from global memory (L2).  Levels
// 1..ks-1 are passes (one launch per level, kPassRows half-rows per CTA); the
// levels from block side N >> (ks-1) <= kCoarseMax on run in one CTA per layer.
// The arithmetic of every output (filter taps, order of the sums) is that of
// the cluster kernels.

// Epilogue setup shared by the streamed analysis kernels (as in k_analysis).
template <typename T, int EPI>
__device__ __forceinline__ void emit_setup(Emit<T, EPI> &emit, const InstDev &I, const LayerDev &L,
                                           const IoArgs &io, int inst, int flags, const T *dal) {
  emit.off = L.off;
  emit.N = L.N;
  emit.dalpha = dal;
  emit.precond = I.precond;
  emit.warm = (flags & kFlagWarm) ? 1 : 0;
  emit.jinv = static_cast<const T *>(I.jinv);
  emit.cache = nullptr;
  emit.out = static_cast<T *>(io.out0[inst]);
  emit.P = io.in1[inst] ? static_cast<const T *>(io.in1[inst]) : dir_buffer<T>(I, flags >> kIterShift);
  emit.Q = io.out0[inst] ? static_cast<T *>(io.out0[inst]) : static_cast<T *>(I.q);
  emit.R = static_cast<T *>(I.r);
  emit.Pn = static_cast<T *>(I.p);
  emit.X = static_cast<T *>(io.out0[inst]);
}

// Asynchronous copy of rows (first + j) & wrap, j < nrows, of M elements each from
// src (row stride `stride` elements) into the dense rows of dst: 16-byte copies
// when the rows are 16-byte aligned, else one element at a time.  Completed by
// cp_async_wait_all() and a barrier.
template <typename T>
__device__ __forceinline__ void stage_rows_async(T *dst, const T *src, int stride, int first, int nrows, int M,
                                                 int wrap) {
  constexpr int V = 16 / static_cast<int>(sizeof(T));
  const int lgM = __ffs(M) - 1;
  const bool vec = M >= V &&
                   ((reinterpret_cast<uintptr_t>(src) | (static_cast<size_t>(stride) * sizeof(T))) & 15) == 0;
  if (vec) {
    const int lgV = __ffs(V) - 1, lgMv = lgM - lgV, mv = M >> lgV;
    for (int idx = threadIdx.x; idx < nrows * mv; idx += blockDim.x) {
      const int j = idx >> lgMv, c = (idx & (mv - 1)) << lgV;
      cp_async16(dst + j * M + c, src + static_cast<size_t>((first + j) & wrap) * stride + c);
    }
  } else {
    for (int idx = threadIdx.x; idx < nrows * M; idx += blockDim.x) {
      const int j = idx >> lgM, x = idx & (M - 1);
      cp_async_elem(dst + idx, src + static_cast<size_t>((first + j) & wrap) * stride + x);
    }
  }
  cp_async_commit();
}

// Outputs of a column pass handled per thread at once: their epilogue inputs
// (p, or x and J^-1) are all requested before any is used.
constexpr int kEmitU = 4;

// One analysis level k over a tile: output half-rows [row0, row0 + kPassRows) of
// the level's M x M block.  SRC 0: level 1 reads io.in0's layer; SRC 2: the
// gathered grid in the plan's phi; levels > 1 read the previous low-low block.
// The low-low part goes to the scratch (or is emitted at k = J); the details
// are emitted.  One partial pair per CTA.
//
// A warp takes 128 input columns (four per lane: two output columns of each
// half) and walks down its share of the tile's half-rows: per half-row two new
// input rows, their row transforms from the lane's window of LF + 2 inputs
// (16-byte loads; the neighbours' overlap hits the L1), then the column sums
// over the last LF row transforms, which stay in registers.  No shared memory
// and no barrier before the partial sums.  Bound by the latency of the row and
// epilogue loads (16 E-ELT systems: DRAM at 14%, SM at 25% of their peaks).  Against staging the tile's rows and
// their row transforms in shared memory for two barrier-separated passes, one
// output column per thread (GB300, cold launch): finest pass of the 100 m system
// 51.2 -> 32 us, of 64 uneven systems 71.6 -> 35 us, of 16 E-ELT systems 25.8 ->
// 14 us.
template <typename T>
struct alignas(16) Quad {
  T v[4];
};

template <typename T, int LF>
struct RowWalk {
  // row transforms of one input row for the lane's four columns: low outputs
  // 2q, 2q + 1 and high outputs 2q, 2q + 1, each sum over t in order
  T l0, l1, h0, h1;
  static constexpr int NV = (LF + 5) / 4;   // vectors of the window of LF + 2 inputs
  __device__ __forceinline__ void sums(const Filt<T, LF> &f, const Quad<T> (&w)[NV]) {
    T lo0 = T(0), hi0 = T(0), lo1 = T(0), hi1 = T(0);
#pragma unroll
    for (int t = 0; t < LF; ++t) {
      lo0 += f.h[t] * w[t >> 2].v[t & 3];
      hi0 += f.g[t] * w[t >> 2].v[t & 3];
      lo1 += f.h[t] * w[(t + 2) >> 2].v[(t + 2) & 3];
      hi1 += f.g[t] * w[(t + 2) >> 2].v[(t + 2) & 3];
    }
    l0 = lo0;
    l1 = lo1;
    h0 = hi0;
    h1 = hi1;
  }
};

template <typename T, int SRC, int EPI, int LF>
__global__ void __launch_bounds__(kDwtThreads) k_dwt_pass(const InstDev *__restrict__ insts,
                                                          const PassItem *__restrict__ items, IoArgs io,
                                                          int k, int flags) {
  __shared__ T s_dal[kMaxLevels + 1];
  pdl_trigger();
  const PassItem it = items[blockIdx.x];
  if (io.active && !io.active[it.inst]) return;
  const InstDev &I = insts[it.inst];
  const LayerDev &L = I.layers[it.layer];
  const int J = I.J, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kDwtThreads / 32;
  const int lgM = L.log2N - (k - 1), M = 1 << lgM, H = M >> 1;
  if (tid <= J) s_dal[tid] = T(L.dalpha[tid]);
  Filt<T, LF> f;
  f.load(I);
  Emit<T, EPI> emit;
  emit_setup<T, EPI>(emit, I, L, io, it.inst, flags, s_dal);
  const T *src = k > 1 ? static_cast<const T *>(I.lls) + L.ll_off[k - 1]
                       : (SRC == 0 ? static_cast<const T *>(io.in0[it.inst]) : static_cast<const T *>(I.phi)) + L.off;
  T *ll = k < J ? static_cast<T *>(I.lls) + L.ll_off[k] : nullptr;
  // columns in groups of 128, the tile's half-rows shared by the warps of a group
  const int groups = M >> 7, per = max(1, nw / groups), rows = kPassRows / per;
  __syncthreads();
  pdl_wait();
  const bool vec = emit.aligned(src);
  constexpr int NV = RowWalk<T, LF>::NV;
  for (int unit = warp; unit < groups * per; unit += nw) {
    const int x0 = (unit % groups) * 128 + 4 * lane, i0 = it.row0 + (unit / groups) * rows;
    RowWalk<T, LF> row[LF];   // the last LF row transforms
    auto load = [&](int r, Quad<T> (&w)[NV]) {
      const T *p = src + static_cast<size_t>(r & (M - 1)) * M;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        const T *q = p + ((x0 + 4 * c) & (M - 1));
        if (vec) {
          w[c] = *reinterpret_cast<const Quad<T> *>(q);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) w[c].v[e] = q[e];
        }
      }
    };
    {
      Quad<T> w[LF - 2 > 0 ? LF - 2 : 1][NV];
#pragma unroll
      for (int t = 0; t < LF - 2; ++t) load(2 * i0 + t, w[t]);
#pragma unroll
      for (int t = 0; t < LF - 2; ++t) row[t].sums(f, w[t]);
    }
#pragma unroll 1
    for (int i = i0; i < i0 + rows; ++i) {
      Quad<T> w[2][NV];
      load(2 * i + LF - 2, w[0]);
      load(2 * i + LF - 1, w[1]);
      const int c = x0 >> 1;   // the lane's output columns c, c + 1 of each half
      const bool top = k == J;
      typename Emit<T, EPI>::Pre fl[2], fa[2], fb[2], fc[2];   // low-low (k = J), high-x, high-y, high-high
      if (top) emit.fetch2(i, c, vec, fl);
      emit.fetch2(i, H + c, vec, fa);
      emit.fetch2(H + i, c, vec, fb);
      emit.fetch2(H + i, H + c, vec, fc);
      row[LF - 2].sums(f, w[0]);
      row[LF - 1].sums(f, w[1]);
      T o[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) o[q] = T(0);
#pragma unroll
      for (int t = 0; t < LF; ++t) {
        o[0] += f.h[t] * row[t].l0;
        o[1] += f.h[t] * row[t].l1;
        o[2] += f.h[t] * row[t].h0;
        o[3] += f.h[t] * row[t].h1;
        o[4] += f.g[t] * row[t].l0;
        o[5] += f.g[t] * row[t].l1;
        o[6] += f.g[t] * row[t].h0;
        o[7] += f.g[t] * row[t].h1;
      }
      if (top) {
        emit.put2(i, c, J, o[0], o[1], fl, vec);
      } else if (vec) {
        store_pair(ll + static_cast<size_t>(i) * H + c, o[0], o[1]);
      } else {
        ll[static_cast<size_t>(i) * H + c] = o[0];
        ll[static_cast<size_t>(i) * H + c + 1] = o[1];
      }
      emit.put2(i, H + c, k, o[2], o[3], fa, vec);
      emit.put2(H + i, c, k, o[4], o[5], fb, vec);
      emit.put2(H + i, H + c, k, o[6], o[7], fc, vec);
#pragma unroll
      for (int t = 0; t + 2 < LF; ++t) row[t] = row[t + 2];
    }
  }
  if (EPI == kEpiPlain) return;
  const double2 s = block_sum2(emit.acc0, emit.acc1);
  if (tid == 0) {
    I.part[I.cl_part_off + 2 * it.slot] = s.x;
    I.part[I.cl_part_off + 2 * it.slot + 1] = s.y;
  }
}

// The coarse analysis levels ks..J of one layer in one CTA: the block of side
// N >> (ks - 1) from the scratch (or, ks = 1, the layer grid); every output emitted,
// its epilogue input from shared memory, where it arrives with the block (GB300,
// cold: 16 E-ELT systems 11.2 us with the inputs read level by level, 9.6 so).
template <typename T, int SRC, int EPI, int LF>
__global__ void __launch_bounds__(kPassThreads) k_dwt_coarse(const InstDev *__restrict__ insts,
                                                             const PassItem *__restrict__ items, IoArgs io,
                                                             int flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ InstDev sI;
  __shared__ T s_dal[kMaxLevels + 1];
  pdl_trigger();
  const PassItem it = items[blockIdx.x];
  if (io.active && !io.active[it.inst]) return;
  load_inst(&sI, insts + it.inst);
  const InstDev &I = sI;
  const LayerDev &L = I.layers[it.layer];
  const int J = I.J, tid = threadIdx.x, nt = blockDim.x, ks = L.ks, N = L.N;
  int lgM = L.log2N - (ks - 1), M = 1 << lgM;
  T *A = reinterpret_cast<T *>(smem_raw);
  T *B = A + M * M;
  T *E = B + M * M;   // the epilogue's p (or x) of the block
  const int lgM0 = lgM;
  if (tid <= J) s_dal[tid] = T(L.dalpha[tid]);
  Filt<T, LF> f;
  f.load(I);
  Emit<T, EPI> emit;
  emit_setup<T, EPI>(emit, I, L, io, it.inst, flags, s_dal);
  const T *src = ks > 1 ? static_cast<const T *>(I.lls) + L.ll_off[ks - 1]
                        : (SRC == 0 ? static_cast<const T *>(io.in0[it.inst]) : static_cast<const T *>(I.phi)) + L.off;
  __syncthreads();
  pdl_wait();
  stage_rows_async<T>(A, src, M, 0, M, M, M - 1);
  const bool staged = EPI == kEpiOp || (EPI == kEpiResid && emit.warm);
  if (staged) {
    stage_rows_async<T>(E, (EPI == kEpiOp ? emit.P : emit.X) + L.off, N, 0, M, M, M - 1);
    emit.cache = E;
  }
  auto slot = [&](int row, int col) { return staged ? (row << lgM0) + col : -1; };
  cp_async_wait_all();
  __syncthreads();
  for (int k = ks; k <= J; ++k, M >>= 1, --lgM) {
    const int H = M >> 1;
    row_analysis<T, LF>(f, A, B, M, lgM, tid, nt);
    __syncthreads();
    for (int idx0 = tid; idx0 < H * M; idx0 += kEmitU * nt) {
      T lo[kEmitU], hi[kEmitU];
      typename Emit<T, EPI>::Pre fa[kEmitU], fb[kEmitU];
#pragma unroll
      for (int u = 0; u < kEmitU; ++u) {
        const int idx = idx0 + u * nt;
        if (idx < H * M) {
          const int i = idx >> lgM, x = idx & (M - 1);
          T l = T(0), h = T(0);
#pragma unroll
          for (int t = 0; t < LF; ++t) {
            const T val = B[((2 * i + t) & (M - 1)) * M + x];
            l += f.h[t] * val;
            h += f.g[t] * val;
          }
          lo[u] = l;
          hi[u] = h;
          if (!(x < H && k < J)) fa[u] = emit.fetch(i, x, slot(i, x));
          fb[u] = emit.fetch(H + i, x, slot(H + i, x));
        }
      }
#pragma unroll
      for (int u = 0; u < kEmitU; ++u) {
        const int idx = idx0 + u * nt;
        if (idx < H * M) {
          const int i = idx >> lgM, x = idx & (M - 1);
          if (x < H && k < J) A[i * H + x] = lo[u];
          else emit.put(i, x, (x < H) ? J : k, lo[u], fa[u]);
          emit.put(H + i, x, k, hi[u], fb[u]);
        }
      }
    }
    __syncthreads();
  }
  if (EPI == kEpiPlain) return;
  const double2 s = block_sum2(emit.acc0, emit.acc1);
  if (tid == 0) {
    I.part[I.cl_part_off + 2 * it.slot] = s.x;
    I.part[I.cl_part_off + 2 * it.slot + 1] = s.y;
  }
}

// beta = (r.z)_iter / (r.z)_(iter-1) from the update's partials, as k_synthesis
// forms it (0 at iteration 0 and after a breakdown); record: store (r.z)_iter
// and beta itself (in the plan's type), which the level passes that follow read.
template <typename T>
__device__ __forceinline__ T streamed_beta(const InstDev &I, int iter, bool record) {
  __shared__ T s_b;
  const double prev = I.scal[kRz0 + ((iter + 1) & 1)];
  const double flag = I.scal[kFlag];
  const double rz = iter == 0 ? sum_partial(I.part + I.cl_part_off, I.n_cl_part, 0)
                              : sum_partial(I.part + I.upd_part_off, I.n_upd_blocks, 0);
  if (threadIdx.x == 0) {
    double beta = 0.0;
    if (iter > 0) {
      const bool stop = flag != 0.0 || !isfinite(rz) || !(prev != 0.0);
      beta = stop ? 0.0 : rz / prev;
    }
    s_b = T(beta);
    if (record) {
      I.scal[kRz0 + (iter & 1)] = rz;
      *reinterpret_cast<T *>(I.scal + kBeta) = T(beta);
    }
  }
  __syncthreads();
  return s_b;
}

// A coefficient of the synthesis input: SRC 0 from io.in0; SRC 1 the PCG direction
// with its update p = J^-1 r + beta p (not at the first iteration), read from the
// previous iteration's buffer and, when `own`, written to this iteration's.
template <typename T, int SRC>
struct SynthCoef {
  const T *src, *Pin, *Rv, *Jv;
  T *Pout;
  T beta;
  bool first, pre;
  struct Raw {
    T p, r, j;
  };
  // the loads of coefficient idx (several are requested before any is used) ...
  __device__ __forceinline__ Raw load(size_t idx) const {
    Raw v{T(0), T(0), T(1)};
    if (SRC == 0) {
      v.p = src[idx];
    } else {
      v.p = Pin[idx];
      if (!first) {
        v.r = Rv[idx];
        if (pre) v.j = Jv[idx];
      }
    }
    return v;
  }
  // ... then its value, with the direction update (stored when owned)
  __device__ __forceinline__ T value(const Raw &v, size_t idx, bool own) const {
    if (SRC == 0 || first) return v.p;
    const T z = pre ? v.j * v.r : v.r;
    const T pn = z + beta * v.p;
    if (own) Pout[idx] = pn;
    return pn;
  }
};

// Coefficients (and low-low values) staged per thread at once by the synthesis kernels; the
// coarse kernel's share of a 64 x 64 block.
constexpr int kCoefU = 4, kCoarseCoefU = 8;

// 16 bytes of T: the unit of the vector loads of the streamed synthesis pass.
template <typename T>
struct Vec16 {
  static constexpr int kN = 16 / static_cast<int>(sizeof(T));
  T v[kN];
  __device__ __forceinline__ void load(const T *p) { *reinterpret_cast<uint4 *>(v) = *reinterpret_cast<const uint4 *>(p); }
  __device__ __forceinline__ void store(T *p) const { *reinterpret_cast<uint4 *>(p) = *reinterpret_cast<const uint4 *>(v); }
};

template <typename T, int SRC>
__device__ __forceinline__ SynthCoef<T, SRC> synth_coef(const InstDev &I, const IoArgs &io, int inst, int flags,
                                                        T beta) {
  const int iter = flags >> kIterShift;
  SynthCoef<T, SRC> c;
  c.src = static_cast<const T *>(io.in0[inst]);
  c.Pin = dir_buffer<T>(I, iter > 0 ? iter - 1 : 0);
  c.Pout = dir_buffer<T>(I, iter);
  c.Rv = static_cast<const T *>(I.r);
  c.Jv = static_cast<const T *>(I.jinv);
  c.beta = beta;
  c.first = (flags & kFlagFirst) != 0;
  c.pre = I.precond != 0;
  return c;
}

// The coarse synthesis levels J..ks of one layer in one CTA: the coefficients of
// the pyramid's block of side N >> (ks - 1) (with the direction update, all owned
// here), the block synthesised level by level (rows, then columns), the result
// to the scratch (the low-low input of level ks - 1) or, ks = 1, the output grid.
// With SRC 1 this kernel records (r.z) and beta of the iteration.
template <typename T, int SRC, int LF>
__global__ void __launch_bounds__(kPassThreads) k_idwt_coarse(const InstDev *__restrict__ insts,
                                                              const PassItem *__restrict__ items, IoArgs io,
                                                              int flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ InstDev sI;
  pdl_trigger();
  const PassItem it = items[blockIdx.x];
  if (io.active && !io.active[it.inst]) return;
  load_inst(&sI, insts + it.inst);
  const InstDev &I = sI;
  const LayerDev &L = I.layers[it.layer];
  const int J = I.J, tid = threadIdx.x, nt = blockDim.x, ks = L.ks, N = L.N;
  const int lgM0 = L.log2N - (ks - 1), M0 = 1 << lgM0;
  T *Cf = reinterpret_cast<T *>(smem_raw);   // the coefficient block, M0 x M0
  T *A = Cf + M0 * M0;                       // the current low-low block
  T *XL = A + M0 * M0;                       // row syntheses of the low-y and high-y rows
  T *XH = XL + (M0 >> 1) * M0;
  Filt<T, LF> f;
  f.load(I);
  pdl_wait();
  SynthCoef<T, SRC> coef = synth_coef<T, SRC>(I, io, it.inst, flags, T(0));
  auto at = [&](int idx) { return static_cast<size_t>(L.off) + static_cast<size_t>(idx >> lgM0) * N + (idx & (M0 - 1)); };
  // the first coefficients of each thread are requested before beta is formed (GB300, cold: 16
  // E-ELT systems 14.2 -> 10.3 us)
  typename SynthCoef<T, SRC>::Raw raw[kCoarseCoefU];
#pragma unroll
  for (int u = 0; u < kCoarseCoefU; ++u)
    if (tid + u * nt < M0 * M0) raw[u] = coef.load(at(tid + u * nt));
  if (SRC == 1) coef.beta = streamed_beta<T>(I, flags >> kIterShift, true);
#pragma unroll
  for (int u = 0; u < kCoarseCoefU; ++u) {
    const int idx = tid + u * nt;
    if (idx < M0 * M0) Cf[idx] = coef.value(raw[u], at(idx), true);
  }
  for (int idx0 = tid + kCoarseCoefU * nt; idx0 < M0 * M0; idx0 += kCoarseCoefU * nt) {
#pragma unroll
    for (int u = 0; u < kCoarseCoefU; ++u)
      if (idx0 + u * nt < M0 * M0) raw[u] = coef.load(at(idx0 + u * nt));
#pragma unroll
    for (int u = 0; u < kCoarseCoefU; ++u) {
      const int idx = idx0 + u * nt;
      if (idx < M0 * M0) Cf[idx] = coef.value(raw[u], at(idx), true);
    }
  }
  __syncthreads();
  {
    const int HJ = (N >> (J - 1)) >> 1;
    for (int idx = tid; idx < HJ * HJ; idx += nt) A[idx] = Cf[(idx / HJ) * M0 + idx % HJ];
  }
  __syncthreads();
  for (int k = J; k >= ks; --k) {
    const int lgM = L.log2N - (k - 1), M = 1 << lgM, H = M >> 1;
    // row synthesis (x) of the low-y rows [LL | HL] into XL and the high-y rows [LH | HH] into XH
    const int lgH = lgM - 1;
    for (int idx = tid; idx < 2 * H * H; idx += nt) {
      const int r = idx >> lgH, m = idx & (H - 1);
      const bool high = r >= H;
      const int ii = high ? r - H : r;
      T even = T(0), odd = T(0);
#pragma unroll
      for (int s = 0; s < LF / 2; ++s) {
        const int jj = (m - s) & (H - 1);
        const T lo = high ? Cf[(H + ii) * M0 + jj] : A[ii * H + jj];
        const T hi = Cf[(high ? H + ii : ii) * M0 + H + jj];
        even += f.h[2 * s] * lo + f.g[2 * s] * hi;
        odd += f.h[2 * s + 1] * lo + f.g[2 * s + 1] * hi;
      }
      T *xr = (high ? XH : XL) + ii * M + 2 * m;
      xr[0] = even;
      xr[1] = odd;
    }
    __syncthreads();
    // column synthesis (y): the block of side M, the next level's low-low block
    for (int idx = tid; idx < H * M; idx += nt) {
      const int b = idx >> lgM, x = idx & (M - 1);
      T even = T(0), odd = T(0);
#pragma unroll
      for (int s = 0; s < LF / 2; ++s) {
        const int ii = (b - s) & (H - 1);
        const T xl = XL[ii * M + x], xh = XH[ii * M + x];
        even += f.h[2 * s] * xl + f.g[2 * s] * xh;
        odd += f.h[2 * s + 1] * xl + f.g[2 * s + 1] * xh;
      }
      A[(2 * b) * M + x] = even;
      A[(2 * b + 1) * M + x] = odd;
    }
    __syncthreads();
  }
  T *out = ks > 1 ? static_cast<T *>(I.lls) + L.ll_off[ks - 1]
                  : (io.out0[it.inst] ? static_cast<T *>(io.out0[it.inst]) : static_cast<T *>(I.phi)) + L.off;
  const int stride = ks > 1 ? M0 : N;
  for (int idx = tid; idx < M0 * M0; idx += nt) out[(idx >> lgM0) * stride + (idx & (M0 - 1))] = A[idx];
}

// One synthesis level k over a tile: output rows [2 row0, 2 row0 + 2 kPassRows) of
// the level's M x M block, from the low-low block of level k (scratch) and the
// level's detail coefficients (with the direction update; the tile owns
// half-rows [row0, row0 + kPassRows) and writes their updated directions).  The
// HL = LF/2 - 1 half-rows before the tile are read too.  Output to the scratch
// (the low-low block of level k - 1) or, k = 1, the output grid.
//
// The CTA stages the tile's coefficients in shared memory, each updated once.
// Then a thread takes four columns of each half of the block (eight output
// columns) and a strip of the half-rows, walked downwards: per half-row the row
// syntheses of the low-y and the high-y row from 16-byte windows, and the column
// synthesis over the last LF/2 half-rows, whose row syntheses stay in registers.
// One barrier; a strip repeats the row syntheses of HL half-rows, so a tile has
// at most four strips.  Bound by the latency of the coefficients' loads (16
// E-ELT systems: DRAM at 19%, SM at 24% of their peaks).  Against writing the row syntheses back to shared
// memory for a second pass (GB300, cold launch): 64 uneven systems 57.7 -> 39 us,
// 16 E-ELT systems 20.1 -> 14 us, the 100 m system's finest pass 45.4 -> 38 us.
// (Without the staging, each thread reading its window from global memory, the
// halo columns are updated twice: 57 us there.)
template <typename T, int SRC, int LF>
__global__ void __launch_bounds__(kIdwtThreads) k_idwt_pass(const InstDev *__restrict__ insts,
                                                            const PassItem *__restrict__ items, IoArgs io,
                                                            int k, int flags) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ InstDev sI;
  constexpr int HL = LF / 2 - 1, NI = kPassRows + HL;
  pdl_trigger();
  const PassItem it = items[blockIdx.x];
  if (io.active && !io.active[it.inst]) return;
  load_inst(&sI, insts + it.inst);
  const InstDev &I = sI;
  const LayerDev &L = I.layers[it.layer];
  const int tid = threadIdx.x, nt = blockDim.x, N = L.N;
  const int lgM = L.log2N - (k - 1), M = 1 << lgM, H = M >> 1;
  T *VL = reinterpret_cast<T *>(smem_raw);   // NI low-y rows [LL | HL], then NI high-y rows [LH | HH]
  T *VH = VL + NI * M;
  Filt<T, LF> f;
  f.load(I);
  const T *ll = static_cast<const T *>(I.lls) + L.ll_off[k];
  pdl_wait();
  const T beta = SRC == 1 ? *reinterpret_cast<const T *>(I.scal + kBeta) : T(0);
  const SynthCoef<T, SRC> coef = synth_coef<T, SRC>(I, io, it.inst, flags, beta);
  // the tile's coefficient rows: 16-byte vectors when every source is aligned (the plan's
  // buffers are; a caller's coefficient vector may not be), else kCoefU positions per
  // thread loaded before any is used
  constexpr int VN = Vec16<T>::kN;
  const bool vec = (((reinterpret_cast<uintptr_t>(SRC == 0 ? coef.src : coef.Pin) |
                      reinterpret_cast<uintptr_t>(coef.Rv) | reinterpret_cast<uintptr_t>(coef.Jv) |
                      reinterpret_cast<uintptr_t>(coef.Pout) | reinterpret_cast<uintptr_t>(ll)) & 15) == 0) &&
                   ((L.off & (VN - 1)) == 0) && H >= VN;
  if (vec) {
    const int lgMv = lgM - (__ffs(VN) - 1), mv = M / VN;
#pragma unroll 4
    for (int q = tid; q < NI * mv; q += nt) {
      const int j = q >> lgMv, x = (q & (mv - 1)) * VN;
      const int ii = (it.row0 - HL + j) & (H - 1);
      const bool own = j >= HL;
      const size_t lo = static_cast<size_t>(L.off) + static_cast<size_t>(ii) * N + x;
      const size_t hi = static_cast<size_t>(L.off) + static_cast<size_t>(H + ii) * N + x;
      Vec16<T> a, b, ar, br, aj, bj;
      // requests first: the low-y row's low-low values or coefficients, the high-y row's coefficients
      if (x < H) {
        a.load(ll + ii * H + x);
      } else if (SRC == 0) {
        a.load(coef.src + lo);
      } else {
        a.load(coef.Pin + lo);
        if (!coef.first) {
          ar.load(coef.Rv + lo);
          if (coef.pre) aj.load(coef.Jv + lo);
        }
      }
      if (SRC == 0) {
        b.load(coef.src + hi);
      } else {
        b.load(coef.Pin + hi);
        if (!coef.first) {
          br.load(coef.Rv + hi);
          if (coef.pre) bj.load(coef.Jv + hi);
        }
      }
      if (SRC == 1 && !coef.first) {
#pragma unroll
        for (int e = 0; e < VN; ++e) {
          if (x >= H) a.v[e] = (coef.pre ? aj.v[e] * ar.v[e] : ar.v[e]) + coef.beta * a.v[e];
          b.v[e] = (coef.pre ? bj.v[e] * br.v[e] : br.v[e]) + coef.beta * b.v[e];
        }
        if (own) {
          if (x >= H) a.store(coef.Pout + lo);
          b.store(coef.Pout + hi);
        }
      }
      a.store(VL + j * M + x);
      b.store(VH + j * M + x);
    }
  } else
  for (int idx0 = tid; idx0 < NI * M; idx0 += kCoefU * nt) {
    typename SynthCoef<T, SRC>::Raw ra[kCoefU], rb[kCoefU];
#pragma unroll
    for (int u = 0; u < kCoefU; ++u) {
      const int idx = idx0 + u * nt;
      if (idx < NI * M) {
        const int j = idx >> lgM, x = idx & (M - 1);
        const int ii = (it.row0 - HL + j) & (H - 1);
        if (x < H) ra[u].p = ll[ii * H + x];
        else ra[u] = coef.load(static_cast<size_t>(L.off) + static_cast<size_t>(ii) * N + x);
        rb[u] = coef.load(static_cast<size_t>(L.off) + static_cast<size_t>(H + ii) * N + x);
      }
    }
#pragma unroll
    for (int u = 0; u < kCoefU; ++u) {
      const int idx = idx0 + u * nt;
      if (idx < NI * M) {
        const int j = idx >> lgM, x = idx & (M - 1);
        const int ii = (it.row0 - HL + j) & (H - 1);
        const bool own = j >= HL;
        VL[idx] = x < H ? ra[u].p : coef.value(ra[u], static_cast<size_t>(L.off) + static_cast<size_t>(ii) * N + x, own);
        VH[idx] = coef.value(rb[u], static_cast<size_t>(L.off) + static_cast<size_t>(H + ii) * N + x, own);
      }
    }
  }
  __syncthreads();
  T *out = k > 1 ? static_cast<T *>(I.lls) + L.ll_off[k - 1]
                 : (io.out0[it.inst] ? static_cast<T *>(io.out0[it.inst]) : static_cast<T *>(I.phi)) + L.off;
  const int stride = k > 1 ? M : N;
  const bool vout = (reinterpret_cast<uintptr_t>(out) & 15) == 0;   // (a caller's grid may not be aligned)
  // threads of a strip (a power of two), strips of the tile, half-rows of a strip
  const int lgLanes = lgM - 3, strips = min(4, max(1, kIdwtThreads >> lgLanes)), rows = kPassRows / strips;
  if ((tid >> lgLanes) >= strips) return;
  constexpr int NS = LF / 2;
  auto load4 = [](const T *p, T *v) {
    const Quad<T> q = *reinterpret_cast<const Quad<T> *>(p);
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = q.v[e];
  };
  // the eight row syntheses of a staged row from its inputs m0 - 4 .. m0 + 3 of both halves (a
  // multiple of four, so a window never straddles the periodic wrap)
  auto row_synth = [&](const T *row, int m0, T *o) {
    T lo[8], hi[8];
    const int mp = (m0 - 4) & (H - 1);
    if (LF > 2) load4(row + mp, lo);
    load4(row + m0, lo + 4);
    if (LF > 2) load4(row + H + mp, hi);
    load4(row + H + m0, hi + 4);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      T even = T(0), odd = T(0);
#pragma unroll
      for (int s = 0; s < LF / 2; ++s) {
        const T l = lo[4 + u - s], h = hi[4 + u - s];
        even += f.h[2 * s] * l + f.g[2 * s] * h;
        odd += f.h[2 * s + 1] * l + f.g[2 * s + 1] * h;
      }
      o[2 * u] = even;
      o[2 * u + 1] = odd;
    }
  };
  auto store8 = [&](T *p, const T *v) {
    if (vout) {
      *reinterpret_cast<Quad<T> *>(p) = {{v[0], v[1], v[2], v[3]}};
      *reinterpret_cast<Quad<T> *>(p + 4) = {{v[4], v[5], v[6], v[7]}};
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) p[e] = v[e];
    }
  };
  for (int m0 = (tid & ((1 << lgLanes) - 1)) << 2; m0 < H; m0 += 4 * kIdwtThreads) {
    const int j0 = (tid >> lgLanes) * rows;   // the strip's first staged half-row (HL before its own)
    T xl[NS][8], xh[NS][8];   // the last NS half-rows' row syntheses, half-row j in slot j mod NS
#pragma unroll 1
    for (int js = 0; js < rows + HL; js += NS) {
#pragma unroll
      for (int u = 0; u < NS; ++u) {
        const int j = js + u;
        if (j >= rows + HL) break;
        row_synth(VL + (j0 + j) * M, m0, xl[u]);
        row_synth(VH + (j0 + j) * M, m0, xh[u]);
        if (j < HL) continue;
        // column synthesis (y): output rows 2b and 2b + 1
        T even[8], odd[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) even[e] = odd[e] = T(0);
#pragma unroll
        for (int s = 0; s < LF / 2; ++s) {
          const int q = (u - s + NS) % NS;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            even[e] += f.h[2 * s] * xl[q][e] + f.g[2 * s] * xh[q][e];
            odd[e] += f.h[2 * s + 1] * xl[q][e] + f.g[2 * s + 1] * xh[q][e];
          }
        }
        T *o = out + static_cast<size_t>(2 * (it.row0 + j0 + j - HL)) * stride + 2 * m0;
        store8(o, even);
        store8(o + stride, odd);
      }
    }
  }
}


namespace {

template <typename T, int LF>
cudaError_t synth_streamed(int src, int flags, const InstDev *insts, const StreamSet &S, const IoArgs &io,
                           cudaStream_t s) {
  const dim3 gc(S.n_coarse);
  cudaError_t e = src == 0
                      ? launch_ex(k_idwt_coarse<T, 0, LF>, gc, kPassThreads, 0, S.smem_coarse, s, insts, S.coarse, io, flags)
                      : launch_ex(k_idwt_coarse<T, 1, LF>, gc, kPassThreads, 0, S.smem_coarse, s, insts, S.coarse, io, flags);
  for (int k = S.kmax; k >= 1 && e == cudaSuccess; --k) {
    if (S.cnt[k] == 0) continue;
    const dim3 g(S.cnt[k]);
    const PassItem *it = S.items + S.off[k];
    const size_t smem = S.smem_pass >> k;   // the staged rows: half of pass_smem_elems at the level's block side
    e = src == 0 ? launch_ex(k_idwt_pass<T, 0, LF>, g, kIdwtThreads, 0, smem, s, insts, it, io, k, flags)
                 : launch_ex(k_idwt_pass<T, 1, LF>, g, kIdwtThreads, 0, smem, s, insts, it, io, k, flags);
  }
  return e;
}

template <typename T, int SRC, int EPI, int LF>
cudaError_t anal_streamed_e(int flags, const InstDev *insts, const StreamSet &S, const IoArgs &io, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (int k = 1; k <= S.kmax && e == cudaSuccess; ++k) {
    if (S.cnt[k] == 0) continue;
    e = launch_ex(k_dwt_pass<T, SRC, EPI, LF>, dim3(S.cnt[k]), kDwtThreads, 0, 0, s, insts,
                  S.items + S.off[k], io, k, flags);
  }
  if (e == cudaSuccess)
    e = launch_ex(k_dwt_coarse<T, SRC, EPI, LF>, dim3(S.n_coarse), kPassThreads, 0, S.smem_coarse, s, insts,
                  S.coarse, io, flags);
  return e;
}

template <typename T, int LF>
cudaError_t anal_streamed(int src, int epi, int flags, const InstDev *insts, const StreamSet &S, const IoArgs &io,
                          cudaStream_t s) {
  if (src == 0) return anal_streamed_e<T, 0, kEpiPlain, LF>(flags, insts, S, io, s);
  if (epi == kEpiPlain) return anal_streamed_e<T, 2, kEpiPlain, LF>(flags, insts, S, io, s);
  if (epi == kEpiOp) return anal_streamed_e<T, 2, kEpiOp, LF>(flags, insts, S, io, s);
  return anal_streamed_e<T, 2, kEpiResid, LF>(flags, insts, S, io, s);
}

template <typename T>
cudaError_t allow_streamed_t() {
  cudaError_t e = cudaSuccess;
#define TOMO_ALLOW(K) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTransformSmem)
#define TOMO_ALLOW_LF(LF)                                     \
  TOMO_ALLOW((k_idwt_coarse<T, 0, LF>));                      \
  TOMO_ALLOW((k_idwt_coarse<T, 1, LF>));                      \
  TOMO_ALLOW((k_idwt_pass<T, 0, LF>));                        \
  TOMO_ALLOW((k_idwt_pass<T, 1, LF>));                        \
  TOMO_ALLOW((k_dwt_coarse<T, 0, kEpiPlain, LF>));            \
  TOMO_ALLOW((k_dwt_coarse<T, 2, kEpiPlain, LF>));            \
  TOMO_ALLOW((k_dwt_coarse<T, 2, kEpiOp, LF>));               \
  TOMO_ALLOW((k_dwt_coarse<T, 2, kEpiResid, LF>))
  TOMO_ALLOW_LF(2);
  TOMO_ALLOW_LF(4);
  TOMO_ALLOW_LF(6);
  TOMO_ALLOW_LF(8);
#undef TOMO_ALLOW_LF
#undef TOMO_ALLOW
  return e;
}

}  // namespace

cudaError_t configure_streamed_kernels() {
  cudaError_t e = allow_streamed_t<float>();
  if (e == cudaSuccess) e = allow_streamed_t<double>();
  return e;
}

int streamed_launches(const StreamSet &S) {
  int n = 1;
  for (int k = 1; k <= S.kmax; ++k) n += S.cnt[k] > 0 ? 1 : 0;
  return n;
}

cudaError_t launch_synthesis_streamed(int precision, int src, int lf, int flags, const InstDev *insts,
                                      const StreamSet &S, const IoArgs &io, cudaStream_t s) {
#define TOMO_S(T, LF) return synth_streamed<T, LF>(src, flags, insts, S, io, s)
  if (precision == 0) {
    switch (lf) { case 2: TOMO_S(float, 2); case 4: TOMO_S(float, 4); case 6: TOMO_S(float, 6); case 8: TOMO_S(float, 8); }
  } else {
    switch (lf) { case 2: TOMO_S(double, 2); case 4: TOMO_S(double, 4); case 6: TOMO_S(double, 6); case 8: TOMO_S(double, 8); }
  }
#undef TOMO_S
  return cudaErrorInvalidValue;
}

cudaError_t launch_analysis_streamed(int precision, int src, int epi, int lf, int flags, const InstDev *insts,
                                     const StreamSet &S, const IoArgs &io, cudaStream_t s) {
#define TOMO_A(T, LF) return anal_streamed<T, LF>(src, epi, flags, insts, S, io, s)
  if (precision == 0) {
    switch (lf) { case 2: TOMO_A(float, 2); case 4: TOMO_A(float, 4); case 6: TOMO_A(float, 6); case 8: TOMO_A(float, 8); }
  } else {
    switch (lf) { case 2: TOMO_A(double, 2); case 4: TOMO_A(double, 4); case 6: TOMO_A(double, 6); case 8: TOMO_A(double, 8); }
  }
#undef TOMO_A
  return cudaErrorInvalidValue;
}

}  // namespace tomo
