// One VTM sweep over all subgraphs (Table 1 steps 3-5; eq. 5.6, 5.8), one CTA per subgraph.
//
// Per subgraph j the CTA
//   1. gathers the incident wave of each line end from its twin, w_in[e] = w_prev[twin(e)]
//      (the N2N exchange), and forms r_j = b̃_j + sum_e w_in[e]/Z_e e_c (eq. 5.8 right side);
//   2. streams the band factor of K_j from HBM in kNB-row slabs with the TMA bulk-copy engine
//      (cp.async.bulk into a ring of shared-memory stages tracked by mbarriers) and runs the
//      forward substitution L y = r on rows of L and the back substitution L^T x = y on rows of
//      U = L^T (both in dot form: 16-byte shared loads, independent FMA chains, 8-lane shuffle
//      reductions) with the diagonal blocks stored as inverses;
//   3. emits w_out[e] = 2 x_c - w_in[e] for every end (u - Z omega of eq. 5.6, written as the
//      single wave that the twin receives next sweep).
// The vector state of the subgraph (y / x: Wp-1 zero rows, n_pad rows, Wp-1 zero rows, x R) stays in
// shared memory.
#include "kernels.h"

namespace vtm {

template <typename T, typename TV, int R>
__global__ void __launch_bounds__(kSweepThreads, 2) k_sweep(const SweepArgs<T, TV> a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int abort_flag;
  const int tid = threadIdx.x;
  const PieceDesc pd = a.pieces[blockIdx.x];
  const int S = a.stages;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
  T* ring = reinterpret_cast<T*>(smem + 128);
  T* ys = ring + (size_t)S * a.slot_elems;
  T* win = ys + a.ys_elems;
  T* tb = win + a.win_elems;

  const int Wp = pd.Wp;
  const int off = Wp - 1;  // ys row of column 0
  const int nblk = pd.n_pad / kNB;
  // unit sources: batch blockIdx.y's columns, rows from the first one that S_j is wanted at
  const int ub = (a.unit_b0 + (int)blockIdx.y) * R;  // first port of the batch
  if (a.unit && ub >= pd.nports) return;
  const int blk0 = a.unit ? a.port_local[pd.port_off + ub / a.unit_gran * a.unit_gran] / kNB : 0;  // first block
  const int row0 = blk0 * kNB;
  const int nfwd = nblk - blk0;
  const int total = 2 * nfwd;
  const uint32_t slab_bytes = (uint32_t)(kNB * Wp * sizeof(T));
  const T* fbase = a.factor + pd.factor_off;
  const T* ubase = a.factor_u + pd.factor_off;

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < S; ++s) mbar_init(&bars[s], 1);
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  __syncthreads();
  auto issue = [&](int s) {
    if (s == a.withhold) return;  // testing hook: this slab's wait can only run out
    const int kb = blk0 + (s < nfwd ? s : total - 1 - s);
    const int slot = s % S;
    mbar_arrive_expect_tx(&bars[slot], slab_bytes);
    bulk_copy_g2s(ring + (size_t)slot * a.slot_elems, (s < nfwd ? fbase : ubase) + (size_t)kb * kNB * Wp, slab_bytes,
                  &bars[slot]);
  };
  if (tid == 0)
    for (int s = 0; s < S && s < total; ++s) issue(s);

  // ---- prologue: r_j = b̃_j + sum_e w_in[e] / Z_e at the port rows
  for (int i = tid; i < off * R; i += kSweepThreads) {
    ys[i] = T(0);
    ys[(size_t)(off + pd.n_pad) * R + i] = T(0);
  }
  const TV* btp = a.bt + (size_t)pd.copy_off * R;
  if (a.unit) {
    // the rows read: from off above row0 (zero: the forward solution starts there)
    for (int i = row0 * R + tid; i < (off + pd.n_pad) * R; i += kSweepThreads) ys[i] = T(0);
  } else {
    for (int i = tid; i < pd.n_pad * R; i += kSweepThreads) ys[(size_t)off * R + i] = (i < pd.n * R) ? (T)btp[i] : T(0);
  }
  __syncthreads();
  if (a.unit && tid < R && ub + tid < pd.nports) ys[(size_t)(off + a.port_local[pd.port_off + ub + tid]) * R + tid] = T(1);
  for (int q = tid; q < pd.nports && !a.unit; q += kSweepThreads) {
    const int l = a.port_local[pd.port_off + q];
    const int e0 = a.port_end_ptr[pd.port_off + q], e1 = a.port_end_ptr[pd.port_off + q + 1];
    T acc[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) acc[rr] = T(0);
    for (int e = e0; e < e1; ++e) {
      const int tw = a.twin[e];
      const T iz = (T)a.invz[e];
#pragma unroll
      for (int rr = 0; rr < R; ++rr) {
        const T w = (T)a.wprev[(size_t)tw * R + rr];
        win[(e - pd.end_off) * R + rr] = w;
        acc[rr] += w * iz;
      }
    }
    if (a.cpl.ptr)
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc[rr] += coupling_current<T, TV>(a.cpl, pd.port_off + q, rr, R, a.wprev);
#pragma unroll
    for (int rr = 0; rr < R; ++rr) ys[(size_t)(off + l) * R + rr] += acc[rr];
  }
  __syncthreads();

  // ---- forward (s < nfwd) then backward (s >= nfwd) over the staged slabs
  const int rg = tid >> 3, g = tid & 7;
  int s = 0;
  for (; s < total; ++s) {
    const int slot = s % S;
    if (!mbar_wait_bounded(&bars[slot], (uint32_t)((s / S) & 1), a.wait_limit)) abort_flag = 1;
    __syncthreads();
    if (abort_flag) break;
    const T* L = ring + (size_t)slot * a.slot_elems;
    if (s < nfwd) {
      const int k0 = row0 + s * kNB;
      // t_r = r_r - sum_{col < k0} L[r][col] y_col   (positions p < off - r of row r)
      const T* Lr = L + rg * Wp;
      const int pend = off - rg;
      const T* yb = ys + (size_t)(k0 + rg) * R;
      T acc[R];
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc[rr] = T(0);
      if constexpr (sizeof(T) == 4 && R == 1) {
        // 16-byte loads of the factor row; four independent FMA chains
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        const float4* L4 = reinterpret_cast<const float4*>(Lr);
        const int nchunk = (pend + 3) >> 2;
        for (int q = g; q < nchunk; q += 8) {
          const float4 l = L4[q];
          const int p = q << 2;
          const float* y = reinterpret_cast<const float*>(yb) + p;
          a0 = fmaf(l.x, y[0], a0);
          if (p + 1 < pend) a1 = fmaf(l.y, y[1], a1);
          if (p + 2 < pend) a2 = fmaf(l.z, y[2], a2);
          if (p + 3 < pend) a3 = fmaf(l.w, y[3], a3);
        }
        acc[0] = (a0 + a1) + (a2 + a3);
      } else {
        for (int p = g; p < pend; p += 8) {
          const T l = Lr[p];
#pragma unroll
          for (int rr = 0; rr < R; ++rr) acc[rr] += l * yb[(size_t)p * R + rr];
        }
      }
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc[rr] = warp_sum_g8(acc[rr]);
      if (g == 0)
#pragma unroll
        for (int rr = 0; rr < R; ++rr) tb[rg * R + rr] = ys[(size_t)(k0 + rg + off) * R + rr] - acc[rr];
      __syncthreads();
      // y_B = inv(L_KK) t
      T acc2[R];
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc2[rr] = T(0);
      for (int c = g; c <= rg; c += 8) {
        const T l = Lr[off - rg + c];
#pragma unroll
        for (int rr = 0; rr < R; ++rr) acc2[rr] += l * tb[c * R + rr];
      }
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc2[rr] = warp_sum_g8(acc2[rr]);
      if (g == 0)
#pragma unroll
        for (int rr = 0; rr < R; ++rr) ys[(size_t)(k0 + rg + off) * R + rr] = acc2[rr];
    } else {
      const int k0 = row0 + (total - 1 - s) * kNB;
      // rows of U = L^T: t_r = y_r - sum_{col > k0+31} U[r][col] x_col  (positions p >= 32 - r)
      const T* Ur = L + rg * Wp;
      const int pbeg = kNB - rg;
      const T* xb = ys + (size_t)(k0 + rg + off) * R;
      T acc[R];
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc[rr] = T(0);
      if constexpr (sizeof(T) == 4 && R == 1) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        const float4* U4 = reinterpret_cast<const float4*>(Ur);
        const int nchunk = Wp >> 2;
        for (int q = (pbeg >> 2) + g; q < nchunk; q += 8) {
          const float4 u = U4[q];
          const int p = q << 2;
          const float* x = reinterpret_cast<const float*>(xb) + p;
          if (p >= pbeg) a0 = fmaf(u.x, x[0], a0);
          if (p + 1 >= pbeg) a1 = fmaf(u.y, x[1], a1);
          if (p + 2 >= pbeg) a2 = fmaf(u.z, x[2], a2);
          a3 = fmaf(u.w, x[3], a3);  // p + 3 >= pbeg always holds for chunks at or after pbeg / 4
        }
        acc[0] = (a0 + a1) + (a2 + a3);
      } else {
        for (int p = pbeg + g; p < Wp; p += 8) {
          const T u = Ur[p];
#pragma unroll
          for (int rr = 0; rr < R; ++rr) acc[rr] += u * xb[(size_t)p * R + rr];
        }
      }
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc[rr] = warp_sum_g8(acc[rr]);
      if (g == 0)
#pragma unroll
        for (int rr = 0; rr < R; ++rr) tb[rg * R + rr] = xb[rr] - acc[rr];
      __syncthreads();
      // x_B = inv(U_KK) t: x_r = sum_{c >= r} inv(U_KK)[r][c] t_c at positions c - r
      T acc2[R];
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc2[rr] = T(0);
      for (int c = rg + g; c < kNB; c += 8) {
        const T u = Ur[c - rg];
#pragma unroll
        for (int rr = 0; rr < R; ++rr) acc2[rr] += u * tb[c * R + rr];
      }
#pragma unroll
      for (int rr = 0; rr < R; ++rr) acc2[rr] = warp_sum_g8(acc2[rr]);
      if (g == 0)
#pragma unroll
        for (int rr = 0; rr < R; ++rr) ys[(size_t)(k0 + rg + off) * R + rr] = acc2[rr];
    }
    __syncthreads();
    if (tid == 0 && s + S < total) {
      fence_proxy_async_smem();
      issue(s + S);
    }
  }
  if (abort_flag) {
    if (tid == 0) {
      atomicExch(a.status, kStatusTimeout);
      // drain the copies still in flight (bounded) before the CTA leaves
      for (int s2 = s; s2 < total && s2 < s + S; ++s2)
        if (s2 != a.withhold) mbar_wait_bounded(&bars[s2 % S], (uint32_t)((s2 / S) & 1), kDrainPolls);
    }
    return;
  }

  // ---- epilogue: w_out[e] = 2 x_c - w_in[e]; local solution
  for (int q = tid; q < pd.nports && !a.unit; q += kSweepThreads) {
    const int l = a.port_local[pd.port_off + q];
    const int e0 = a.port_end_ptr[pd.port_off + q], e1 = a.port_end_ptr[pd.port_off + q + 1];
    for (int e = e0; e < e1; ++e)
#pragma unroll
      for (int rr = 0; rr < R; ++rr)
        a.wnext[(size_t)e * R + rr] = (TV)(T(2) * ys[(size_t)(off + l) * R + rr] - win[(e - pd.end_off) * R + rr]);
  }
  if (a.write_x) {
    TV* xp = a.xc + (size_t)blockIdx.y * a.unit_stride + (size_t)pd.copy_off * R;
    for (int i = row0 * R + tid; i < pd.n * R; i += kSweepThreads) xp[i] = (TV)ys[(size_t)off * R + i];
  }
}

// ------------------------------------------------------------------------------------------------
// Pipelined variant: per 32-row block step the chain warps finish block k -- the 32 columns next to
// the block ("near"), the partial sums prepared one step earlier ("far"), the inverted diagonal
// block -- while the far warps compute the far part of block k + 1.  Forward: near columns
// [k0 - 32, k0), far columns < k0 - 32; backward (rows of U): near columns [k0 + 32, k0 + 64), far
// columns >= k0 + 64.  Both halves read disjoint rows of the vector, and every chain warp keeps its
// own right-hand sides, whose near values it wrote itself, so one CTA barrier per block step is
// enough.  Needs two slabs resident (stages >= 3 keeps one in flight).
//
// A lane owns a row of the block and takes its columns in step with the other lanes: column d of row
// r lies at r (Wp - 1) + d (plus a constant), an odd stride, so the 32 lanes hit 32 banks, and the
// vector entry of a column is one broadcast load for all rows and R right-hand sides.  (With eight
// lanes per row, k_sweep, every product needs its own vector load, and each block step three barriers
// and two chains of shuffles.)
//
// What bounds it: HBM with many subgraphs; with few, the chain of block steps (near part, diagonal
// block, one barrier: about 0.25 us at R = 1 against 0.9 - 1.2 us per step of k_sweep).
constexpr int kChainWarps[9] = {0, 1, 1, 0, 2, 0, 0, 0, 4};

template <int R>
struct Chain {
  static constexpr int NC = kChainWarps[R];              // chain warps
  static constexpr int RP = R / NC;                      // right-hand sides of each
  static constexpr int NF = kSweepThreads / 32 - NC;     // far warps
};

template <typename T, int N>
__device__ __forceinline__ void load_n(const T* p, T (&v)[N]) {
  if constexpr (sizeof(T) == 4 && N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + i);
      v[i] = x.x, v[i + 1] = x.y, v[i + 2] = x.z, v[i + 3] = x.w;
    }
  } else if constexpr (sizeof(T) == 4 && N == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x, v[1] = x.y;
  } else if constexpr (sizeof(T) == 8 && N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const double2 x = *reinterpret_cast<const double2*>(p + i);
      v[i] = x.x, v[i + 1] = x.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = p[i];
  }
}

// acc[q] += sum over columns d0 <= d < d1 (d0, d1 multiples of 4) of l[d] v[d][q], where column d of
// this lane's row counts if keep(d).  v: the entry of column 0, its RP values of the R per row; for
// R = 1 the rows of four columns are one 16-byte load.
template <typename T, int R, int RP, typename K>
__device__ __forceinline__ void dot_columns(const T* l, const T* v, int d0, int d1, K keep, T (&acc)[4][RP]) {
  for (int d = d0; d < d1; d += 4) {
    T x[4][RP];
    if constexpr (R == 1) {
      T y[4];
      load_n<T, 4>(v + d, y);
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j][0] = y[j];
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) load_n<T, RP>(v + (d + j) * R, x[j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const T e = l[d + j];
      const T f = keep(d + j) ? e : T(0);
#pragma unroll
      for (int q = 0; q < RP; ++q) acc[j][q] += f * x[j][q];
    }
  }
}

template <typename T, int R>
__global__ void __launch_bounds__(kSweepThreads, 2) k_sweep_pipe(const SweepArgs<T, T> a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int abort_flag;
  constexpr int NC = Chain<R>::NC, RP = Chain<R>::RP, NF = Chain<R>::NF;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const PieceDesc pd = a.pieces[blockIdx.x];
  const int S = a.stages;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
  T* ring = reinterpret_cast<T*>(smem + 128);
  T* farp = ring + (size_t)S * a.slot_elems;          // [2][NF][kNB][R]
  T* tbuf = farp + 2 * NF * kNB * R;                  // [NC][kNB][RP]
  const int Wp = pd.Wp, w = pd.w;
  const int off = Wp - 1;
  T* ys = tbuf + kNB * R;                             // Wp zero rows, n_pad rows, Wp + 4 zero rows
  constexpr int kFarBuf = NF * kNB * R;

  const int nblk = pd.n_pad / kNB;
  const int total = 2 * nblk;
  const uint32_t slab_bytes = (uint32_t)(kNB * Wp * sizeof(T));
  const T* fbase = a.factor + pd.factor_off;
  const T* ubase = a.factor_u + pd.factor_off;

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < S; ++s) mbar_init(&bars[s], 1);
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  __syncthreads();
  auto issue = [&](int s) {
    if (s == a.withhold) return;  // testing hook: this slab's wait can only run out
    const int kb = s < nblk ? s : total - 1 - s;
    const int slot = s % S;
    mbar_arrive_expect_tx(&bars[slot], slab_bytes);
    bulk_copy_g2s(ring + (size_t)slot * a.slot_elems, (s < nblk ? fbase : ubase) + (size_t)kb * kNB * Wp, slab_bytes,
                  &bars[slot]);
  };
  if (tid == 0)
    for (int s = 0; s < S && s < total; ++s) issue(s);

  // ---- prologue: r_j = b̃_j + sum_e w_in[e] / Z_e at the port rows; far part of block 0 is zero
  for (int i = tid; i < (Wp + 4) * R; i += kSweepThreads) {
    if (i < Wp * R) ys[i] = T(0);
    ys[(size_t)(Wp + pd.n_pad) * R + i] = T(0);  // the last far columns are rounded up to fours
  }
  for (int i = tid; i < kFarBuf; i += kSweepThreads) farp[i] = T(0);
  const T* btp = a.bt + (size_t)pd.copy_off * R;
#pragma unroll 8
  for (int i = tid; i < pd.n_pad * R; i += kSweepThreads) ys[(size_t)Wp * R + i] = (i < pd.n * R) ? btp[i] : T(0);
  __syncthreads();
  for (int q = tid; q < pd.nports; q += kSweepThreads) {
    const int l = a.port_local[pd.port_off + q];
    T acc[R];
    port_inflow<T, R>(a.port_end_ptr, a.twin, a.invz, a.cpl, a.wprev, pd.port_off + q, acc);
#pragma unroll
    for (int rr = 0; rr < R; ++rr) ys[(size_t)(Wp + l) * R + rr] += acc[rr];
  }
  __syncthreads();

  const int r = lane;
  const int nfar = w > kNB ? (w - kNB + 3) / 4 * 4 : 0;  // far columns, in fours
  const bool whole = off >= 2 * kNB - 1;  // the near columns lie inside every row's storage
  int s = 0, slot = 0;                    // slot, phase of item s
  uint32_t phase = 0;
  for (; s < total; ++s) {
    const int par = s & 1;
    const int slot1 = slot + 1 == S ? 0 : slot + 1;  // of item s + 1
    const uint32_t phase1 = slot + 1 == S ? phase ^ 1u : phase;
    if (warp < NC) {
      // ---- chain: finish item s (block k0) for this warp's right-hand sides
      if (!mbar_wait_bounded(&bars[slot], phase, a.wait_limit)) abort_flag = 1;
      const T* L = ring + (size_t)slot * a.slot_elems;
      const bool fwd = s < nblk;
      const int k0 = (fwd ? s : total - 1 - s) * kNB;
      const int q0 = warp * RP;
      T* yk = ys + (size_t)(Wp + k0) * R + q0;  // the block's rows
      const T* Lr = L + r * off + (fwd ? off : 0);  // entry of column d at Lr[d]
      T acc[4][RP];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < RP; ++q) acc[j][q] = T(0);
      const T* fp = farp + par * kFarBuf + r * R + q0;
#pragma unroll
      for (int h = 0; h < NF; ++h) {
        T f[RP];
        load_n<T, RP>(fp + h * kNB * R, f);
#pragma unroll
        for (int q = 0; q < RP; ++q) acc[h & 3][q] += f[q];
      }
      if (whole) {
        const int d0 = fwd ? -kNB : kNB;
        dot_columns<T, R, RP>(Lr + d0, yk + d0 * R, 0, kNB, [](int) { return true; }, acc);
      } else if (fwd) {
        dot_columns<T, R, RP>(Lr, yk, -kNB, 0, [&](int d) { return d + off >= r; }, acc);
      } else {
        dot_columns<T, R, RP>(Lr, yk, kNB, 2 * kNB, [&](int d) { return d - r <= off; }, acc);
      }
      T* tb = tbuf + warp * kNB * RP;
      {
        T y0[RP];
        load_n<T, RP>(yk + r * R, y0);
#pragma unroll
        for (int q = 0; q < RP; ++q) tb[r * RP + q] = y0[q] - ((acc[0][q] + acc[1][q]) + (acc[2][q] + acc[3][q]));
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < RP; ++q) acc[j][q] = T(0);
      // inv(L_KK)[r][c], c <= r (backward: inv(U_KK)[r][c], c >= r)
      if (fwd) dot_columns<T, RP, RP>(Lr, tb, 0, kNB, [&](int c) { return c <= r; }, acc);
      else dot_columns<T, RP, RP>(Lr, tb, 0, kNB, [&](int c) { return c >= r; }, acc);
#pragma unroll
      for (int q = 0; q < RP; ++q) yk[r * R + q] = (acc[0][q] + acc[1][q]) + (acc[2][q] + acc[3][q]);
    } else if (s + 1 < total) {
      // ---- far part of item s + 1 from its slab (values complete at the start of step s)
      const int s1 = s + 1, f = warp - NC;
      if (!mbar_wait_bounded(&bars[slot1], phase1, a.wait_limit)) abort_flag = 1;
      const T* L1 = ring + (size_t)slot1 * a.slot_elems;
      const bool fwd1 = s1 < nblk;
      const int k1 = (fwd1 ? s1 : total - 1 - s1) * kNB;
      const T* yk = ys + (size_t)(Wp + k1) * R;
      const T* Lr = L1 + r * off + (fwd1 ? off : 0);
      T acc[4][R];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < R; ++q) acc[j][q] = T(0);
      // columns in fours, an equal run of them per warp; forward -32 - 4 .. -32 - nfar
      const int c0 = nfar / 4 * f / NF * 4, c1 = nfar / 4 * (f + 1) / NF * 4;
      if (fwd1) {
        dot_columns<T, R, R>(Lr, yk, -kNB - c1, -kNB - c0, [&](int d) { return d + off >= r; }, acc);
      } else {
        dot_columns<T, R, R>(Lr, yk, 2 * kNB + c0, 2 * kNB + c1, [&](int d) { return d - r <= off; }, acc);
      }
      T* fp = farp + (par ^ 1) * kFarBuf + (f * kNB + r) * R;
#pragma unroll
      for (int q = 0; q < R; ++q) fp[q] = (acc[0][q] + acc[1][q]) + (acc[2][q] + acc[3][q]);
    }
    __syncthreads();
    if (abort_flag) break;
    // the last warp issues: the chain warp goes on at once
    if (tid == kSweepThreads - 1 && s + S < total) {
      fence_proxy_async_smem();
      issue(s + S);
    }
    slot = slot1;
    phase = phase1;
  }
  if (abort_flag) {
    if (tid == 0) {
      atomicExch(a.status, kStatusTimeout);
      for (int s2 = s; s2 < total && s2 < s + S; ++s2)
        if (s2 != a.withhold) mbar_wait_bounded(&bars[s2 % S], (uint32_t)((s2 / S) & 1), kDrainPolls);
    }
    return;
  }

  // ---- epilogue: w_out[e] = 2 x_c - w_in[e]; local solution.  The incoming waves are read again (the
  // shared memory they would take holds another slab).
#pragma unroll 4
  for (int q = tid; q < pd.nports; q += kSweepThreads) {
    const int l = a.port_local[pd.port_off + q];
    const int e0 = a.port_end_ptr[pd.port_off + q], e1 = a.port_end_ptr[pd.port_off + q + 1];
    for (int e = e0; e < e1; ++e) {
      const T* wi = a.wprev + (size_t)a.twin[e] * R;
#pragma unroll
      for (int rr = 0; rr < R; ++rr) a.wnext[(size_t)e * R + rr] = T(2) * ys[(size_t)(Wp + l) * R + rr] - wi[rr];
    }
  }
  if (a.write_x) {
    T* xp = a.xc + (size_t)pd.copy_off * R;
#pragma unroll 8
    for (int i = tid; i < pd.n * R; i += kSweepThreads) xp[i] = ys[(size_t)Wp * R + i];
  }
}

size_t sweep_pipe_smem_bytes(size_t elem, int R, int stages, int slot_elems, int ys_elems) {
  // ys: one row more before and five after than the single-block sweep's
  return 128 + elem * ((size_t)stages * slot_elems + ys_elems + 6 * R +
                       (size_t)(2 * (kSweepThreads / 32 - kChainWarps[R]) + 1) * kNB * R);
}

template <typename T>
static const void* pipe_kernel(int R) {
  switch (R) {
    case 1: return (const void*)k_sweep_pipe<T, 1>;
    case 2: return (const void*)k_sweep_pipe<T, 2>;
    case 4: return sizeof(T) == 4 ? (const void*)k_sweep_pipe<float, 4> : nullptr;  // FP64: up to two (sweep_variant 2)
    case 8: return sizeof(T) == 4 ? (const void*)k_sweep_pipe<float, 8> : nullptr;
    default: return nullptr;
  }
}

template <typename T>
cudaError_t sweep_pipe_configure(int R) {
  const void* k = pipe_kernel<T>(R);
  return k ? cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipeSmemMax) : cudaErrorInvalidValue;
}

template <typename T>
cudaError_t sweep_pipe_occupancy(int R, size_t smem, int* n) {
  const void* k = pipe_kernel<T>(R);
  return k ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, kSweepThreads, smem) : cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_sweep_pipe(const SweepArgs<T, T>& a, int R, int npieces, size_t smem, cudaStream_t st) {
  if (npieces <= 0) return cudaSuccess;
  const void* k = pipe_kernel<T>(R);
  if (!k) return cudaErrorInvalidValue;
  SweepArgs<T, T> args = a;
  void* av[] = {&args};
  return cudaLaunchKernel(k, dim3(npieces), dim3(kSweepThreads), av, smem, st);
}

cudaError_t allow_all_smem(const void* kernel) {
  int dev = 0, most = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
}

size_t sweep_smem_bytes(size_t elem, int R, int stages, int slot_elems, int ys_elems, int win_elems) {
  return 128 + elem * ((size_t)stages * slot_elems + ys_elems + win_elems + (size_t)kNB * R);
}

template <typename TF, typename TV>
cudaError_t sweep_configure(int R) {
  switch (R) {
    case 1: return allow_all_smem((const void*)k_sweep<TF, TV, 1>);
    case 2: return allow_all_smem((const void*)k_sweep<TF, TV, 2>);
    case 4: return allow_all_smem((const void*)k_sweep<TF, TV, 4>);
    case 8: return allow_all_smem((const void*)k_sweep<TF, TV, 8>);
    default: return cudaErrorInvalidValue;
  }
}

template <typename TF, typename TV, int R>
static cudaError_t occupancy_one(size_t smem, int* n) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_sweep<TF, TV, R>, kSweepThreads, smem);
}

template <typename TF, typename TV>
cudaError_t sweep_occupancy(int R, size_t smem, int* n) {
  switch (R) {
    case 1: return occupancy_one<TF, TV, 1>(smem, n);
    case 2: return occupancy_one<TF, TV, 2>(smem, n);
    case 4: return occupancy_one<TF, TV, 4>(smem, n);
    case 8: return occupancy_one<TF, TV, 8>(smem, n);
    default: return cudaErrorInvalidValue;
  }
}

template <typename TF, typename TV>
cudaError_t launch_sweep(const SweepArgs<TF, TV>& a, int R, int npieces, size_t smem, cudaStream_t st,
                         int batches) {
  if (npieces <= 0) return cudaSuccess;
  dim3 grid(npieces, batches), block(kSweepThreads);
  switch (R) {
    case 1: k_sweep<TF, TV, 1><<<grid, block, smem, st>>>(a); break;
    case 2: k_sweep<TF, TV, 2><<<grid, block, smem, st>>>(a); break;
    case 4: k_sweep<TF, TV, 4><<<grid, block, smem, st>>>(a); break;
    case 8: k_sweep<TF, TV, 8><<<grid, block, smem, st>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

#define VTM_SWEEP_INST(TF, TV)                                                                    \
  template cudaError_t sweep_configure<TF, TV>(int);                                       \
  template cudaError_t sweep_occupancy<TF, TV>(int, size_t, int*);                                 \
  template cudaError_t launch_sweep<TF, TV>(const SweepArgs<TF, TV>&, int, int, size_t, cudaStream_t, int);
VTM_SWEEP_INST(float, float)
VTM_SWEEP_INST(double, double)
VTM_SWEEP_INST(double, float)

#define VTM_PIPE_INST(T)                                  \
  template cudaError_t sweep_pipe_configure<T>(int);      \
  template cudaError_t sweep_pipe_occupancy<T>(int, size_t, int*); \
  template cudaError_t launch_sweep_pipe<T>(const SweepArgs<T, T>&, int, int, size_t, cudaStream_t);
VTM_PIPE_INST(float)
VTM_PIPE_INST(double)

}  // namespace vtm
