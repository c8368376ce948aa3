// Port-response form of the VTM sweep.
//
// A sweep only needs each subgraph's port values u = P^T x_j, and x_j = K_j^{-1}(b̃_j + P s) with
// s_q = sum_{e at port q} w_in[e] / Z_e (eq. 5.8).  So u = u_base + S_j s with the port response
// S_j = P^T K_j^{-1} P (the open-circuit impedance matrix of Def. 7.1 taken over all ports at once,
// the Schur complement of the interior in K_j^{-1}, cf. eq. A3.3) and u_base = P^T K_j^{-1} b̃_j.
// The outgoing waves are w_out[e] = 2 u_q - w_in[e] (eq. 5.6), exactly as in the band sweep; only
// the way u is obtained differs.  S_j is symmetric, so only its lower block triangle is stored.
//
// Storage of S_j: 32 x 32 tiles (I, J), J <= I, in the order I (I + 1) / 2 + J, from tile s_off on;
// ports beyond n_ports are zero.  Inside a tile the entries lie as the kernel's lanes take them
// (PortLayout), so that the k-th 16-byte load of all lanes reads 512 contiguous bytes:
//  * patches: lane 8 a + b owns the 8 x 4 patch of rows 8a .. +7 and columns 4b .. +3 (R <= 2), or
//    lane 4 a + b the 4 x 8 patch of rows 4a .. +3 and columns 8b .. +7 (R = 4, 8).  The column
//    part T^T s_I leaves the registers with every tile and sums over the lanes of a column group,
//    which few columns per lane make short; the row part T s_J stays in registers along a row of
//    tiles, where few rows per lane take few registers;
//  * fragments: the 16 x 16 blocks of mma.m16n8k16's A operand (FP32 tiles, R = 8).
//
// FP16 storage (FP32 solvers): the same tiles as IEEE half, row by row with the 16-byte chunks of a
// row exchanged for ldmatrix (or as patches), each tile divided by its own largest entry (kept
// per tile in FP32); the tile's products are scaled back before they enter y.  It halves the bytes
// of the sweep; its rounding (2^-11 of each tile's largest entry) is absorbed by the FP64 defect
// correction, and the solver returns to FP32 storage if a correction step stops gaining a digit.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "kernels.h"

namespace vtm {

namespace {

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
  static constexpr int V = 4;
  __device__ static float get(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
};
template <>
struct Vec16<double> {
  using type = double2;
  static constexpr int V = 2;
  __device__ static double get(const double2& v, int i) { return i == 0 ? v.x : v.y; }
};

// Rows of a lane's patch.
__host__ __device__ constexpr int patch_rows(int R) { return R <= 2 ? 8 : 4; }

// Position of element (i, c) of a tile, V entries per 16 bytes.
__host__ __device__ __forceinline__ int tile_pos(int layout, int i, int c, int V) {
  if (layout == kPortFragments) {
    // block (i / 16, c / 16); lane 4 g + t holds rows g, g + 8 and columns 2 t, 2 t + 1 (+ 8): four
    // pairs in register order (row half, then column half)
    const int blk = (i >> 4) * 2 + (c >> 4), lane = (i & 7) * 4 + ((c & 7) >> 1);
    const int pair = ((i >> 3) & 1) + 2 * ((c >> 3) & 1), p = blk * 8 + pair * 2 + (c & 1);
    return ((p / V) * kNB + lane) * V + p % V;
  }
  const int pr = layout == kPortPatch8x4 ? 8 : 4, pc = kNB / pr;
  const int L = (i / pr) * (kNB / pc) + c / pc, p = (i % pr) * pc + (c % pc);
  return ((p / V) * kNB + L) * V + p % V;
}

// Position of element (i, c) of an FP16 tile stored for ldmatrix: rows of 64 bytes whose four 16-byte
// chunks are exchanged by the row pair, so that the eight rows of an 8 x 8 matrix hit 32 banks.
__host__ __device__ __forceinline__ int half_pos(int i, int c) {
  return i * kNB + (((c >> 3) ^ (i >> 1)) & 3) * 8 + (c & 7);
}

// This lane's patch (kNB entries of type TS, in the tile's patch layout) widened to T.
__device__ __forceinline__ void load_patch(const float* tile, int lane, float (&p)[kNB]) {
  const float4* tp = reinterpret_cast<const float4*>(tile);
#pragma unroll
  for (int k = 0; k < kNB / 4; ++k) {
    const float4 v = tp[k * kNB + lane];
    p[4 * k] = v.x, p[4 * k + 1] = v.y, p[4 * k + 2] = v.z, p[4 * k + 3] = v.w;
  }
}

__device__ __forceinline__ void load_patch(const double* tile, int lane, double (&p)[kNB]) {
  const double2* tp = reinterpret_cast<const double2*>(tile);
#pragma unroll
  for (int k = 0; k < kNB / 2; ++k) {
    const double2 v = tp[k * kNB + lane];
    p[2 * k] = v.x, p[2 * k + 1] = v.y;
  }
}

__device__ __forceinline__ void load_patch(const __half* tile, int lane, float (&p)[kNB]) {
  const uint4* tp = reinterpret_cast<const uint4*>(tile);
#pragma unroll
  for (int k = 0; k < kNB / 8; ++k) {
    const uint4 v = tp[k * kNB + lane];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
      p[k * 8 + 2 * j] = f.x;
      p[k * 8 + 2 * j + 1] = f.y;
    }
  }
}

// Shared-memory slot of a tile in flight: its patches and, with FP16 storage, the scale once per lane.
template <typename TS>
__host__ __device__ constexpr int slot_bytes() {
  return kNB * kNB * (int)sizeof(TS) + (sizeof(TS) == 2 ? kNB * 4 : 0);
}

// Tiles in flight per warp.  FP16 tiles with an accumulator per warp: three, which two CTAs per SM
// have room for (96 KB in flight per SM; one tile and three CTAs keep 48 KB, 0.205 ms per sweep of
// 128^3 instead of 0.17).
template <typename TS, bool DEEP>
__host__ __device__ constexpr int port_depth() {
  return sizeof(TS) == 2 && DEEP ? 3 : 1;
}

// This lane's share of a tile on its way to the slot (the caller commits the group).
template <typename TS>
__device__ __forceinline__ void fetch_patch(unsigned char* slot, const TS* tile, const float* scale, int lane, uint64_t policy) {
  const uint32_t d = smem_u32(slot) + lane * 16;
  const unsigned char* g = reinterpret_cast<const unsigned char*>(tile) + lane * 16;
#pragma unroll
  for (int k = 0; k < kNB * (int)sizeof(TS) / 16; ++k)
    asm volatile("cp.async.cg.shared.global.L2::cache_hint.L2::256B [%0], [%1], 16, %2;" ::"r"(d + k * 512), "l"(g + k * 512), "l"(policy)
                 : "memory");
  if constexpr (sizeof(TS) == 2)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(slot) + kNB * kNB * 2 + lane * 4),
                 "l"(scale)
                 : "memory");
}

// Row and column of tile t.
__host__ __device__ __forceinline__ void tile_of(int t, int& I, int& J) {
  I = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((I + 1) * (I + 2) / 2 <= t) ++I;
  while (I * (I + 1) / 2 > t) --I;
  J = t - I * (I + 1) / 2;
}

}  // namespace

__host__ __device__ int64_t port_tiles(int nports) {
  const int64_t nt = (nports + kNB - 1) / kNB;
  return nt * (nt + 1) / 2;
}

// S_j columns from unit-source solves: column cc = b * Rs + r of S_j is x at the ports for the
// unit source at port cc (x0 holds copies x Rs per batch, blockIdx.y: batch b0 + y).  Only tiles with I >= J are written.
template <typename T>
__global__ void k_gather_port_response(const PieceDesc* __restrict__ pieces, const int32_t* __restrict__ port_local,
                                       int Rs, int b0, const T* __restrict__ x0, int64_t stride, T* __restrict__ S,
                                       int layout) {
  const PieceDesc pd = pieces[blockIdx.x];
  const int b = b0 + (int)blockIdx.y;
  const T* xc = x0 + (size_t)blockIdx.y * stride;
  constexpr int V = Vec16<T>::V;
  for (int i = b * Rs / kNB * kNB * Rs + threadIdx.x; i < pd.nports * Rs; i += blockDim.x) {
    const int q = i / Rs, r = i % Rs;
    const int cc = b * Rs + r;
    if (cc >= pd.nports) continue;
    const int I = q / kNB, J = cc / kNB;
    if (I < J) continue;
    const int row = q % kNB, col = cc % kNB;
    const int64_t t = pd.s_off + (int64_t)I * (I + 1) / 2 + J;
    S[t * kNB * kNB + tile_pos(layout, row, col, V)] =
        xc[((size_t)pd.copy_off + port_local[pd.port_off + q]) * Rs + r];
  }
}

// u_base[port][r] = x_j at the port copy (xc from a sweep with zero incident waves).
template <typename T>
__global__ void k_gather_ports(const PieceDesc* __restrict__ pieces, const int32_t* __restrict__ port_local, int R,
                               const T* __restrict__ xc, T* __restrict__ ubase) {
  const PieceDesc pd = pieces[blockIdx.x];
  for (int i = threadIdx.x; i < pd.nports * R; i += blockDim.x) {
    const int q = i / R, r = i % R;
    ubase[(size_t)(pd.port_off + q) * R + r] = xc[((size_t)pd.copy_off + port_local[pd.port_off + q]) * R + r];
  }
}

// Element index of vector entry (port q, column 0) in shared memory.  With pad = 4 (FP32, R >= 4)
// every group of four ports is followed by four unused entries: a lane reads the 16-byte rows of
// its patch's columns (8 ports apart) and rows (4 apart), which without the gap all start in the
// same four banks.
template <int R>
__device__ __forceinline__ int vidx(int q, int pad) {
  return q * R + (q >> 2) * pad;
}

template <typename T, int N>
__device__ __forceinline__ void load_vec(const T* p, T (&v)[N]) {
  if constexpr (N * sizeof(T) == 16 && sizeof(T) == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
  } else if constexpr (N == 2 && sizeof(T) == 4) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x, v[1] = x.y;
  } else if constexpr (N == 2 && sizeof(T) == 8) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    v[0] = x.x, v[1] = x.y;
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = p[i];
  }
}

template <typename T, int N>
__device__ __forceinline__ void store_vec(T* p, const T (&v)[N]) {
  if constexpr (N * sizeof(T) == 16 && sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else if constexpr (N == 2 && sizeof(T) == 4) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else if constexpr (N == 2 && sizeof(T) == 8) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) p[i] = v[i];
  }
}

// Loads that bypass the L1 cache: values that another CTA or the launch before wrote.
template <typename T, int N>
__device__ __forceinline__ void load_cg(const T* p, T (&v)[N]) {
  if constexpr (N == 4 && sizeof(T) == 4) {
    const float4 x = __ldcg(reinterpret_cast<const float4*>(p));
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
  } else if constexpr (N == 2 && sizeof(T) == 4) {
    const float2 x = __ldcg(reinterpret_cast<const float2*>(p));
    v[0] = x.x, v[1] = x.y;
  } else if constexpr (N == 2 && sizeof(T) == 8) {
    const double2 x = __ldcg(reinterpret_cast<const double2*>(p));
    v[0] = x.x, v[1] = x.y;
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = __ldcg(p + i);
  }
}

// Columns that a thread of the port-vector passes takes at once: 16 bytes of them at most.
template <typename T, int R>
__host__ __device__ constexpr int vec_cols() {
  return R < (int)(16 / sizeof(T)) ? R : (int)(16 / sizeof(T));
}

// N consecutive entries, 16-byte aligned, in 16-byte loads.
template <typename T, int N>
__device__ __forceinline__ void load_run(const T* p, T (&v)[N]) {
  constexpr int W = 16 / sizeof(T);
#pragma unroll
  for (int i = 0; i < N; i += W) {
    T w[W];
    load_vec<T, W>(p + i, w);
#pragma unroll
    for (int j = 0; j < W; ++j) v[i + j] = w[j];
  }
}

// Dependent launch (both kernels of a sweep): wait until the launch before has completed and its
// writes are visible; let the next launch's CTAs start as this one's leave.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Sum of N values per lane over the N lanes lane ^ (stride * k): each step halves the values a lane
// keeps; the lane whose position in the group is k ends with the sum of value k in v[0].
template <typename T, int N, int RC, int STRIDE>
__device__ __forceinline__ void reduce_scatter(T (&v)[N][RC], int pos) {
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1) {
    const bool upper = (pos & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i)
#pragma unroll
      for (int q = 0; q < RC; ++q) {
        const T send = upper ? v[i][q] : v[i + h][q];
        const T keep = upper ? v[i + h][q] : v[i][q];
        v[i][q] = keep + __shfl_xor_sync(0xffffffffu, send, STRIDE * h);
      }
  }
}

// The end of a segment, for both sweep kernels: y(q, r, v) gives RV columns of the segment's y.  A
// subgraph of one segment goes straight to its waves; else the partial y goes to scratch and the
// CTA that finishes the subgraph last (a ticket per subgraph) adds the segments' partials in their
// order.  Nothing waits, and the order of arrival does not enter the sums: identical runs agree bit
// for bit.  The waves, w_out[e] = 2 (u_base + y)_q - w_in[e], take kU entries per thread at a time,
// their partials, end ranges, twins and incoming waves loaded in three independent rounds.
template <typename T, int R, int TH, typename Y>
__device__ __forceinline__ void finish_segment(const PortArgs<T>& a, const PortSeg& sg, int si, const PieceDesc& pd,
                                               int rows, int* flag, Y y) {
  constexpr int RV = vec_cols<T, R>();
  constexpr int kU = sizeof(T) * RV >= 8 ? 2 : 4, kP = 4;
  const int tid = threadIdx.x, np = pd.nports;
  const int npad = (np + kNB - 1) / kNB * kNB;
  T* const part = a.part + sg.part;  // [nseg][npad * R]
  if (sg.nseg > 1) {
    for (int i = tid; i < npad * (R / RV); i += TH) {
      T v[RV] = {};
      const int q = i / (R / RV), r = i % (R / RV) * RV;
      if (q < rows) y(q, r, v);
      store_vec<T, RV>(part + (size_t)(si - sg.first) * npad * R + (size_t)i * RV, v);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      const int n = atomicAdd(a.ticket + sg.first, 1);
      *flag = n == sg.nseg - 1;
      if (n == sg.nseg - 1) a.ticket[sg.first] = 0;  // for the next sweep
    }
    __syncthreads();
    const bool last = *flag != 0;
    __syncthreads();
    if (!last) return;
    __threadfence();
  }
  const int nv = np * (R / RV);
  for (int i0 = tid; i0 < nv; i0 += TH * kU) {
    int e0[kU], e1[kU], tw[kU];
    T uu[kU][RV], ub[kU][RV];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * TH;
      e0[u] = e1[u] = 0;
#pragma unroll
      for (int c = 0; c < RV; ++c) uu[u][c] = T(0);
      if (i < nv) {
        const int q = i / (R / RV), r = i % (R / RV) * RV;
        e0[u] = a.port_end_ptr[pd.port_off + q];
        e1[u] = a.port_end_ptr[pd.port_off + q + 1];
        load_cg<T, RV>(a.ubase + (size_t)pd.port_off * R + (size_t)i * RV, ub[u]);
        if (sg.nseg <= 1) y(q, r, uu[u]);
      }
    }
    // the segments' partials, kP of them at a time so that their loads do not wait for each other
    if (sg.nseg > 1)
      for (int k0 = 0; k0 < sg.nseg; k0 += kP) {
        T v[kU][kP][RV];
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
          for (int k = 0; k < kP; ++k) {
            const int i = i0 + u * TH;
#pragma unroll
            for (int c = 0; c < RV; ++c) v[u][k][c] = T(0);
            if (i < nv && k0 + k < sg.nseg) load_cg<T, RV>(part + (size_t)(k0 + k) * npad * R + (size_t)i * RV, v[u][k]);
          }
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
          for (int k = 0; k < kP; ++k)
#pragma unroll
            for (int c = 0; c < RV; ++c) uu[u][c] += v[u][k][c];
      }
#pragma unroll
    for (int u = 0; u < kU; ++u)
#pragma unroll
      for (int c = 0; c < RV; ++c) uu[u][c] += ub[u][c];
#pragma unroll
    for (int u = 0; u < kU; ++u) tw[u] = (e1[u] > e0[u]) ? a.twin[e0[u]] : 0;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = i0 + u * TH;
      if (i >= nv) break;
      const int r = i % (R / RV) * RV;
      T w[RV], o[RV];
      load_cg<T, RV>(a.wprev + (size_t)tw[u] * R + r, w);
#pragma unroll
      for (int c = 0; c < RV; ++c) o[c] = T(2) * uu[u][c] - w[c];
      store_vec<T, RV>(a.wnext + (size_t)e0[u] * R + r, o);
      for (int e = e0[u] + 1; e < e1[u]; ++e) {
        load_cg<T, RV>(a.wprev + (size_t)a.twin[e] * R + r, w);
#pragma unroll
        for (int c = 0; c < RV; ++c) o[c] = T(2) * uu[u][c] - w[c];
        store_vec<T, RV>(a.wnext + (size_t)e * R + r, o);
      }
    }
  }
}

// D += A B, 16 x 8 += 16 x 16 times 16 x 8, FP32 accumulation (HALF: fp16 operands, else bf16).
template <bool HALF>
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if constexpr (HALF)
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  else
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four 8 x 8 matrices of 16-bit entries, lane l giving row l % 8 of matrix l / 8; TR: transposed.
template <bool TR>
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&v)[4]) {
  if constexpr (TR)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ uint32_t movmatrix(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

// Two floats as a bf16 pair, rounded to nearest.
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// Where port p of a strip lies in a row of the vector operand: lane t of a column reads its eight
// entries (k = 2t, 2t + 1, 2t + 8, 2t + 9 of both 16-row halves) in one 16-byte load.
__device__ __forceinline__ int operand_pos(int p) {
  return ((p & 7) >> 1) * 8 + ((p >> 4) * 2 + ((p >> 3) & 1)) * 2 + (p & 1);
}

// Columns of the MMAs' vector operand.
// FP16 tiles: columns 2 r, 2 r + 1 hold the two terms of right-hand side r, x = s_r / sigma_r = t0 + 2^-11 t1, so
// one product takes both and its lane adds them; R = 8 takes two operands.  sigma_r is the power of two
// that puts the segment's max |s_r| just below 2^15, and t1 is what t0 leaves times 2^11: at both ends fp16's
// exponent is used in full, and an entry keeps 2^-23 of itself down to 2^-29 of the largest, 2^-12 to 2^-38.
// (With max |x| = 1 and t1 not scaled an entry kept 2^-25 of the largest: ports whose s was 2^-24 of it
// were lost.)
// FP32 tiles: S and s both as three bf16 terms, columns = right-hand sides.  The first two terms are
// rounded to nearest, so their remainders are at most 2^-8 and 2^-17 of the power of two below the value, of
// either sign, and the third term is exact; six of the nine products count, and what the others (mid lo, lo mid,
// lo lo) leave out is at most 2^-24 of a product and nothing on average.  (Terms cut off instead have
// remainders up to twice as large and of the value's sign: up to 2^-21, always towards zero.)  The
// tensor core cuts its sums off too; the first terms' products of every MMA are therefore added in FP32,
// only the others, 2^-8 of those, accumulate there.  Error of y over |S| |s|, rms, random subgraphs of
// 300 to 1060 ports, signed / positive entries: 1.6e-8 / 9.2e-8; with cut-off terms and one accumulator
// 2.7e-8 / 2.9e-7; an FP32 loop (SIMT products) 1.6e-8 / 7.1e-8.
constexpr float kTerm1 = 4.8828125e-4f;  // 2^-11
template <typename TS, int R>
__host__ __device__ constexpr int operand_rows() {
  return sizeof(TS) == 2 ? 2 * R : 3 * R;
}

// Threads of a CTA: MMA = its warps when the products run on the tensor cores, 0 when they do not.
__host__ __device__ constexpr int sweep_threads(int mma) { return mma ? 32 * mma : kSweepThreads; }

// One sweep in port-response form, R right-hand sides.
//
// Work split.  A CTA works through segments, runs of consecutive 32 x 32 tiles of one subgraph's
// stored lower block triangle (PortSeg).  port_plan cuts the tiles of all subgraphs into as many
// equal shares as CTAs fit on the GPU, so a few large subgraphs fill it as well as many do.  Per
// segment: the port vector s (k_port_vec) of the rows up to the segment's last strip (a strip is one
// row of tiles), y = the tiles' products, then finish_segment.
//
// PRIV (one or two columns, where eight accumulators of a subgraph's ports fit in shared memory):
// each warp takes an equal run of the segment's tiles and adds to its own accumulator; nothing
// couples the warps until the segment's end.  Per tile and lane 64 FMAs per column, 3 shuffles and
// one shared read-modify-write; the row sums of a strip stay in registers along it.
// Otherwise one accumulator serves all warps: tile (I, J) belongs to the warp that owns column J
// (J mod 8 counted forwards and backwards in turn, which gives the warps equally many tiles although
// the columns get shorter), so the column part is a plain addition by its only writer, and the
// warps' row sums of `sb` strips are added in warp order between two barriers.
//
// Each lane copies its own patches one tile ahead into shared-memory slots that only it reads (cp.async, 16 bytes a piece): no registers hold loads in flight, no lane waits for
// another, and a segment's first tile arrives while its vectors are read.
//
// MMA (FP16 tiles; FP32 tiles with R = 8): the tile's products on the tensor cores
// (mma.m16n8k16, FP32 accumulation, each tile's sums added in FP32), the transposed ones from
// ldmatrix.trans or movmatrix.  The SIMT products of an FP16 tile take about 210 instructions per
// lane (32 conversions, 64 FMAs, shuffles), of an FP32 tile at R = 8 about 980: the issue rate, not
// the memory, bound those sweeps.
//
// What bounds it (GB300): HBM at R = 1, 2 and with FP16 tiles, FP64 arithmetic in FP64 (0.9 of its
// pipe), with three-term FP32 tiles the issue rate and the segments' latency.  Measured per sweep, port
// vectors included, against one CTA per subgraph with shared-memory atomics (R > 1, FP64) or an accumulator per
// warp (FP32 / FP16, R = 1): 64^3 in 64 subgraphs 0.116 -> 0.042 ms (FP32, R = 1, 188 MB) and 0.82 -> 0.19 ms (FP64,
// 376 MB); 101 x 67 x 83 in 288 ragged subgraphs, 439 MB: R = 8 0.54 -> 0.144 ms, R = 4 0.108; 128^3 in 512
// subgraphs, FP16, 1.01 GB: 0.199 -> 0.178 ms (0.88 of the copy bandwidth; the tiles are read with an evict-first
// hint, without it 8 % more), R = 2 0.223, R = 4 0.242.
template <typename T, typename TS, int R, bool PRIV, int MMA>
__global__ void __launch_bounds__(sweep_threads(MMA), sizeof(T) == 8 || MMA > 8 ? 1 : 2)
    k_port_sweep(const PortArgs<T> a) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int TH = sweep_threads(MMA), kWarps = TH / 32;
  constexpr int RC = R >= 2 ? 2 : 1;         // columns per pass
  constexpr int PR = patch_rows(R), PC = kNB / PR;  // a lane's patch
  constexpr int RV = vec_cols<T, R>();
  constexpr int kTile = kNB * kNB;
  constexpr int kSlot = slot_bytes<TS>();
  const int pad = PRIV ? 0 : a.pad, sb = a.sb;
  const bool ring = PRIV || MMA || a.ring != 0;
  constexpr bool HALF = sizeof(TS) == 2;
  constexpr int NR = MMA ? operand_rows<TS, R>() : 1;  // rows of the split vector operand
  constexpr int NB = HALF ? (R + 3) / 4 : 3;           // its 8-column operands per strip
  __shared__ int smax[MMA && HALF ? R : 1];            // bits of max |s_r| of the segment
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kDepth = port_depth<TS, PRIV && MMA>();
  unsigned char* const slots = smem + warp * (kDepth * kSlot);
  T* const sv = reinterpret_cast<T*>(smem + (ring ? kWarps * kDepth * kSlot : 0));
  uint16_t* const sop = reinterpret_cast<uint16_t*>(sv);    // MMA: s as [NR][op_stride] 16-bit terms
  T* const yv = MMA ? reinterpret_cast<T*>(sop + NR * a.op_stride) : sv + a.vec_elems;  // PRIV: [kWarps]
  T* const yw = yv + (PRIV ? (size_t)warp * a.vec_elems : 0);
  T* const buf = yv + a.vec_elems;                          // not PRIV: [kWarps][sb strips][kNB * R] row sums
  const int pa = lane / (kNB / PC), pb = lane % (kNB / PC);  // row and column group of the patch
  const TS* Sall;
  if constexpr (sizeof(TS) == 2) Sall = static_cast<const TS*>(a.Sh);
  else Sall = reinterpret_cast<const TS*>(a.S);
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  grid_dep_launch();
  bool waited = false;

  for (int si = a.cta_seg[blockIdx.x]; si < a.cta_seg[blockIdx.x + 1]; ++si) {
    const PortSeg sg = a.segs[si];
    const PieceDesc pd = a.pieces[sg.piece];
    const int np = pd.nports;
    const int I0 = sg.I0, I1 = sg.I1;
    const int rows = (I1 + 1) * kNB;  // the rows that this segment's tiles touch
    const TS* const Sb = Sall + sg.s_off * kTile;
    const float* const tsc = HALF ? a.scale + sg.s_off : nullptr;

    // Walk over this warp's tiles, strip by strip, columns ascending; J < 0 once they are exhausted.
    struct Walk {
      int I, J, step, lim, left;
    };
    // not PRIV: first own column of strip k.I or of a later one (steps 15 - 2 w and 1 + 2 w in turn)
    auto strip = [&](Walk& k) {
      for (;;) {
        if (k.I > I1) {
          k.J = -1;
          return;
        }
        k.lim = (k.I == I1) ? sg.J1 : k.I;
        k.J = warp;
        k.step = kWarps * 2 - 1 - 2 * warp;
        if (k.I == I0)
          while (k.J < sg.J0) {
            k.J += k.step;
            k.step = 2 * kWarps - k.step;
          }
        if (k.J <= k.lim) return;
        ++k.I;
      }
    };
    auto next = [&](Walk& k) {
      if constexpr (PRIV) {
        if (--k.left == 0) {
          k.J = -1;
        } else if (++k.J > k.I) {
          ++k.I;
          k.J = 0;
        }
      } else {
        k.J += k.step;
        k.step = 2 * kWarps - k.step;
        if (k.J > k.lim) {
          ++k.I;
          strip(k);
        }
      }
    };
    Walk cw;  // the tile being multiplied
    if constexpr (PRIV) {
      const int t0 = I0 * (I0 + 1) / 2 + sg.J0, n = I1 * (I1 + 1) / 2 + sg.J1 + 1 - t0;
      const int f = n * warp / kWarps;
      cw.left = n * (warp + 1) / kWarps - f;
      tile_of(t0 + f, cw.I, cw.J);
      if (cw.left == 0) cw.J = -1;
    } else {
      cw.I = I0;
      strip(cw);
    }
    Walk fw = cw;  // the next tile to fetch
    int slot = 0;  // of the tile being multiplied; its slot takes the tile kDepth ahead
    auto fetch = [&](int to) {
      if (fw.J >= 0) {
        const int64_t t = fw.I * (fw.I + 1) / 2 + fw.J;
        fetch_patch<TS>(slots + to * kSlot, Sb + t * kTile, HALF ? tsc + t : nullptr, lane, policy);
        next(fw);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (ring)
#pragma unroll
      for (int d = 0; d < kDepth; ++d) fetch(d);
    if (!waited) grid_dep_wait();  // everything above is constant between sweeps
    waited = true;
    float sigma[RV], inv[RV];  // MMA, FP16 tiles: the scale of s in the columns this thread writes out, its inverse
    if constexpr (MMA) {
      // s as 16-bit terms, through an FP32 copy in the accumulators' place; then y = 0
      const T* sp = a.s + (size_t)pd.port_off * R;
      const int r = tid % (R / RV) * RV;
      float m[RV] = {};
      if (HALF && tid < R) smax[tid] = 0;
#pragma unroll 4
      for (int i = tid; i < rows * (R / RV); i += TH) {
        T v[RV] = {};
        if (i / (R / RV) < np) load_cg<T, RV>(sp + (size_t)i * RV, v);
        store_vec<T, RV>(yv + i * RV, v);
        if constexpr (HALF)
#pragma unroll
          for (int c = 0; c < RV; ++c) m[c] = fmaxf(m[c], fabsf(v[c]));
      }
      __syncthreads();
      if constexpr (HALF) {
#pragma unroll
        for (int c = 0; c < RV; ++c) {
#pragma unroll
          for (int o = R / RV; o < 32; o <<= 1) m[c] = fmaxf(m[c], __shfl_xor_sync(0xffffffffu, m[c], o));
          if (lane < R / RV) atomicMax(&smax[r + c], __float_as_int(m[c]));
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < RV; ++c) {
          int e = 0;
          const float mm = __int_as_float(smax[r + c]);
          if (mm > 0.f && isfinite(mm)) frexpf(mm, &e);
          e = max(-110, e) - 15;
          sigma[c] = ldexpf(1.f, e);
          inv[c] = ldexpf(1.f, -e);
        }
      }
      for (int i = tid; i < rows * (R / RV); i += TH) {
        const int q = i / (R / RV);
        uint16_t* o = sop + (q & ~(kNB - 1)) + operand_pos(q & (kNB - 1));
        T v[RV];
        load_vec<T, RV>(yv + i * RV, v);
#pragma unroll
        for (int c = 0; c < RV; ++c) {
          if constexpr (HALF) {
            const float x = v[c] * inv[c];
            const __half t0 = __float2half_rn(x);
            o[(2 * (r + c)) * a.op_stride] = __half_as_ushort(t0);
            o[(2 * (r + c) + 1) * a.op_stride] = __half_as_ushort(__float2half_rn((x - __half2float(t0)) / kTerm1));
          } else {
            float x = v[c];
#pragma unroll
            for (int term = 0; term < 3; ++term) {
              const uint32_t t = bf16_pair(x, 0.f);
              o[(term * R + r + c) * a.op_stride] = (uint16_t)t;
              x -= __uint_as_float(t << 16);
            }
          }
        }
      }
      __syncthreads();
      constexpr int W = 16 / sizeof(T);
      const T z4[W] = {};
      if constexpr (PRIV) {
        for (int i = lane; i < rows * R / W; i += 32) store_vec<T, W>(yw + i * W, z4);
      } else {
        for (int i = tid; i < rows * R / W; i += TH) store_vec<T, W>(yv + i * W, z4);
      }
    } else {
      // s and y = 0, RV columns at a time; padding ports are zero
      const T* sp = a.s + (size_t)pd.port_off * R;
      const T zero[RV] = {};
#pragma unroll 4
      for (int i = tid; i < rows * (R / RV); i += TH) {
        const int q = i / (R / RV), r = i % (R / RV) * RV;
        T v[RV] = {};
        if (q < np) load_cg<T, RV>(sp + (size_t)q * R + r, v);
        store_vec<T, RV>(sv + vidx<R>(q, pad) + r, v);
        if constexpr (!PRIV) store_vec<T, RV>(yv + vidx<R>(q, pad) + r, zero);
      }
      if constexpr (PRIV) {
        constexpr int W = 16 / sizeof(T);
        const T z4[W] = {};
        for (int i = lane; i < rows * R / W; i += 32) store_vec<T, W>(yw + i * W, z4);
      }
    }
    __syncthreads();

    // ---- tensor-core products.  Lane 4 g + t: rows g, g + 8 of a 16-row block, columns 2 t, 2 t + 1.
    const int fg = lane >> 2, ft = lane & 3;
    // the vector operand of strip K: registers (k half, k + 8) of both 16-row halves per operand
    auto operand = [&](int K, uint32_t (&b)[NB][4]) {
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        const int row = HALF ? 8 * n + fg : n * R + fg;
        const bool on = HALF ? row < NR : fg < R;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (on) v = *reinterpret_cast<const uint4*>(sop + (size_t)row * a.op_stride + K * kNB + ft * 8);
        b[n][0] = v.x, b[n][1] = v.y, b[n][2] = v.z, b[n][3] = v.w;
      }
    };
    constexpr int ND = HALF ? NB : 1;    // accumulators per 16-row block
    constexpr int NV = HALF ? ND : 2;    // sums per row that this lane holds
    // column of the k-th sum of this lane
    auto out_col = [&](int k) { return HALF ? 4 * k + ft : 2 * ft + k; };
    // products of the current tile: row sums added to rp[row g, + 8, + 16, + 24], column sums into
    // the accumulator
    auto mma_tile = [&](int I, int J, const uint32_t (&bI)[NB][4], float (&rp)[4][NV]) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
      unsigned char* const tile = slots + slot * kSlot;
      uint32_t bJ[NB][4];
      operand(J, bJ);
      float dr[2][ND][4], dc[2][ND][4];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int n = 0; n < ND; ++n)
#pragma unroll
          for (int k = 0; k < 4; ++k) dr[h][n][k] = dc[h][n][k] = 0.f;
      float sc = 1.f;
      if constexpr (HALF) {
        sc = reinterpret_cast<const float*>(tile + kNB * kNB * 2)[lane];
        __syncwarp();  // the other lanes' copies
        const int row = ((lane >> 3) & 1) * 8 + (lane & 7);
        const uint32_t base = smem_u32(tile) + row * 64;
        uint32_t A[4][4], At[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int mi = k >> 1, chunk = (k & 1) * 2 + (lane >> 4);
          const uint32_t ad = base + mi * 1024 + (((chunk ^ (row >> 1)) & 3) << 4);
          ldmatrix4<false>(ad, A[k]);
          ldmatrix4<true>(ad, At[k]);
        }
        __syncwarp();  // every lane is through with the slot
        fetch(slot);
        slot = slot + 1 == kDepth ? 0 : slot + 1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int mi = k >> 1, ki = k & 1;
          const uint32_t At2[4] = {At[k][0], At[k][2], At[k][1], At[k][3]};
#pragma unroll
          for (int n = 0; n < ND; ++n) {
            mma16816<true>(dr[mi][n], A[k], bJ[n][2 * ki], bJ[n][2 * ki + 1]);
            if (I != J) mma16816<true>(dc[ki][n], At2, bI[n][2 * mi], bI[n][2 * mi + 1]);
          }
        }
      } else {
        float x[kNB];
        load_patch(reinterpret_cast<const float*>(tile), lane, x);
        fetch(slot);
        slot = slot + 1 == kDepth ? 0 : slot + 1;
        float lr[2][4], lc[2][4];  // the products of all but the first terms
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int u = 0; u < 4; ++u) lr[h][u] = lc[h][u] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int mi = k >> 1, ki = k & 1;
#pragma unroll
          for (int term = 0; term < 3; ++term) {
            uint32_t A[4], At[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              A[u] = bf16_pair(x[8 * k + 2 * u], x[8 * k + 2 * u + 1]);
              x[8 * k + 2 * u] -= __uint_as_float(A[u] << 16);
              x[8 * k + 2 * u + 1] -= __uint_as_float(A[u] & 0xFFFF0000u);
            }
            At[0] = movmatrix(A[0]), At[1] = movmatrix(A[2]), At[2] = movmatrix(A[1]), At[3] = movmatrix(A[3]);
#pragma unroll
            for (int n = 0; n < 3 - term; ++n) {
              if (term + n > 0) {
                mma16816<false>(lr[mi], A, bJ[n][2 * ki], bJ[n][2 * ki + 1]);
                if (I != J) mma16816<false>(lc[ki], At, bI[n][2 * mi], bI[n][2 * mi + 1]);
              } else {
                float hr[4] = {0.f, 0.f, 0.f, 0.f};
                mma16816<false>(hr, A, bJ[0][2 * ki], bJ[0][2 * ki + 1]);
#pragma unroll
                for (int u = 0; u < 4; ++u) dr[mi][0][u] += hr[u];
                if (I != J) {
                  float hc[4] = {0.f, 0.f, 0.f, 0.f};
                  mma16816<false>(hc, At, bI[0][2 * mi], bI[0][2 * mi + 1]);
#pragma unroll
                  for (int u = 0; u < 4; ++u) dc[ki][0][u] += hc[u];
                }
              }
            }
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int u = 0; u < 4; ++u) dr[h][0][u] += lr[h][u], dc[h][0][u] += lc[h][u];
      }
#pragma unroll
      for (int h = 0; h < 4; ++h)
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          if constexpr (HALF) {
            const float* d = &dr[h >> 1][k][2 * (h & 1)];
            rp[h][k] += fmaf(d[1], kTerm1, d[0]) * sc;
          } else {
            rp[h][k] += dr[h >> 1][0][2 * (h & 1) + k];
          }
        }
      if (I != J) {
        if constexpr (HALF) {
#pragma unroll
          for (int k = 0; k < NV; ++k)
            if (out_col(k) < R)
#pragma unroll
              for (int h = 0; h < 4; ++h) {
                const float* d = &dc[h >> 1][k][2 * (h & 1)];
                yw[(J * kNB + 8 * h + fg) * R + out_col(k)] += fmaf(d[1], kTerm1, d[0]) * sc;
              }
        } else if (2 * ft < R) {
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            float2* at = reinterpret_cast<float2*>(yw + (J * kNB + 8 * h + fg) * R + 2 * ft);
            const float* d = &dc[h >> 1][0][2 * (h & 1)];
            float2 v = *at;
            v.x += d[0], v.y += d[1];
            *at = v;
          }
        }
      }
    };

    auto wait_patch = [&](int I, int J, T (&pt)[kNB], T& sc) {
      if (ring) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        load_patch(reinterpret_cast<const TS*>(slots), lane, pt);
        if constexpr (sizeof(TS) == 2) sc = reinterpret_cast<const float*>(slots + kNB * kNB * 2)[lane];
        fetch(0);
      } else {
        const TS* t = Sb + (int64_t)(I * (I + 1) / 2 + J) * kTile;
        load_patch(t, lane, pt);
        if constexpr (sizeof(TS) == 2) sc = tsc[I * (I + 1) / 2 + J];
      }
    };
    // T s_J into the lane's row sums rp, T^T s_I (off the diagonal) into the accumulator at column J
    auto multiply = [&](int I, int J, const T (&pt)[kNB], T sc, T (&rp)[PR][R]) {
#pragma unroll
      for (int rc = 0; rc < R; rc += RC) {
        T sI[PR][RC], sJ[PC][RC];
        if constexpr (R == 1) {
          load_run(sv + I * kNB + PR * pa, *reinterpret_cast<T(*)[PR]>(&sI[0][0]));
          load_run(sv + J * kNB + PC * pb, *reinterpret_cast<T(*)[PC]>(&sJ[0][0]));
        } else {
#pragma unroll
          for (int ii = 0; ii < PR; ++ii) load_vec<T, RC>(sv + vidx<R>(I * kNB + PR * pa + ii, pad) + rc, sI[ii]);
#pragma unroll
          for (int jj = 0; jj < PC; ++jj) load_vec<T, RC>(sv + vidx<R>(J * kNB + PC * pb + jj, pad) + rc, sJ[jj]);
        }
        // FP16 storage: the tile was divided by sc
        if constexpr (sizeof(TS) == 2) {
#pragma unroll
          for (int jj = 0; jj < PC; ++jj)
#pragma unroll
            for (int q = 0; q < RC; ++q) sJ[jj][q] *= sc;
        }
        T cp[PC][RC];
#pragma unroll
        for (int jj = 0; jj < PC; ++jj)
#pragma unroll
          for (int q = 0; q < RC; ++q) cp[jj][q] = T(0);
#pragma unroll
        for (int ii = 0; ii < PR; ++ii)
#pragma unroll
          for (int jj = 0; jj < PC; ++jj)
#pragma unroll
            for (int q = 0; q < RC; ++q) {
              rp[ii][rc + q] += pt[ii * PC + jj] * sJ[jj][q];
              cp[jj][q] += pt[ii * PC + jj] * sI[ii][q];
            }
        if (I != J) {
          reduce_scatter<T, PC, RC, kNB / PC>(cp, pa);  // lane (pa, pb) ends with column PC pb + pa
          T* at = yw + vidx<R>(J * kNB + PC * pb + pa, pad) + rc;
#pragma unroll
          for (int q = 0; q < RC; ++q) at[q] += (sizeof(TS) == 2) ? cp[0][q] * sc : cp[0][q];
        }
      }
    };

    if constexpr (PRIV) {
      while (MMA && cw.J >= 0) {
        const int I = cw.I;
        uint32_t bI[NB][4];
        operand(I, bI);
        float rp[4][NV] = {};
        do {
          const int J = cw.J;
          next(cw);
          mma_tile(I, J, bI, rp);
        } while (cw.J >= 0 && cw.I == I);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NV; ++k)
          if (out_col(k) < R)
#pragma unroll
            for (int h = 0; h < 4; ++h) yw[(I * kNB + 8 * h + fg) * R + out_col(k)] += rp[h][k];
        __syncwarp();
      }
      while (!MMA && cw.J >= 0) {
        const int I = cw.I;
        T rp[PR][R];
#pragma unroll
        for (int ii = 0; ii < PR; ++ii)
#pragma unroll
          for (int r = 0; r < R; ++r) rp[ii][r] = T(0);
        do {
          const int J = cw.J;
          T pt[kNB], sc = T(1);
          wait_patch(I, J, pt, sc);
          next(cw);
          multiply(I, J, pt, sc, rp);
        } while (cw.J >= 0 && cw.I == I);
        reduce_scatter<T, PR, R, 1>(rp, pb);  // lane (pa, pb) ends with row PR pa + pb
        __syncwarp();
        T* at = yw + (I * kNB + PR * pa + pb) * R;
#pragma unroll
        for (int r = 0; r < R; ++r) at[r] += rp[0][r];
        __syncwarp();
      }
      __syncthreads();
      finish_segment<T, R, TH>(a, sg, si, pd, rows, reinterpret_cast<int*>(sv), [&](int q, int r, T(&v)[RV]) {
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
          T x[RV];
          load_vec<T, RV>(yv + (size_t)w * a.vec_elems + q * R + r, x);
#pragma unroll
          for (int c = 0; c < RV; ++c) v[c] += x[c];
        }
        if constexpr (MMA && HALF)
#pragma unroll
          for (int c = 0; c < RV; ++c) v[c] *= sigma[c];
      });
    } else {
      for (int Ib = I0; Ib <= I1; Ib += sb) {
        const int Ie = min(Ib + sb, I1 + 1);
        for (int I = Ib; MMA && I < Ie; ++I) {
          uint32_t bI[NB][4];
          operand(I, bI);
          float rp[4][NV] = {};
          while (cw.I == I && cw.J >= 0) {
            const int J = cw.J;
            next(cw);
            mma_tile(I, J, bI, rp);
          }
          T* o = buf + (size_t)(warp * sb + (I - Ib)) * kNB * R;
#pragma unroll
          for (int k = 0; k < NV; ++k)
            if (out_col(k) < R)
#pragma unroll
              for (int h = 0; h < 4; ++h) o[(8 * h + fg) * R + out_col(k)] = rp[h][k];
        }
        for (int I = Ib; !MMA && I < Ie; ++I) {
          T rp[PR][R];
#pragma unroll
          for (int ii = 0; ii < PR; ++ii)
#pragma unroll
            for (int r = 0; r < R; ++r) rp[ii][r] = T(0);
          while (cw.I == I && cw.J >= 0) {
            const int J = cw.J;
            T pt[kNB], sc = T(1);
            wait_patch(I, J, pt, sc);
            next(cw);
            multiply(I, J, pt, sc, rp);
          }
          reduce_scatter<T, PR, R, 1>(rp, pb);  // lane (pa, pb) ends with row PR pa + pb
          T* o = buf + ((size_t)(warp * sb + (I - Ib)) * kNB + PR * pa + pb) * R;
#pragma unroll
          for (int r = 0; r < R; ++r) o[r] = rp[0][r];
        }
        __syncthreads();
        for (int i = tid; i < (Ie - Ib) * kNB * R; i += TH) {
          T v = T(0);
#pragma unroll
          for (int w = 0; w < kWarps; ++w) v += buf[(size_t)w * sb * kNB * R + i];
          yv[vidx<R>(Ib * kNB + i / R, pad) + i % R] += v;
        }
        __syncthreads();
      }
      finish_segment<T, R, TH>(a, sg, si, pd, rows, reinterpret_cast<int*>(sv),
                           [&](int q, int r, T(&v)[RV]) {
                             load_vec<T, RV>(yv + vidx<R>(q, pad) + r, v);
                             if constexpr (MMA && HALF)
#pragma unroll
                               for (int c = 0; c < RV; ++c) v[c] *= sigma[c];
                           });
    }
    __syncthreads();
  }
  if (!waited) grid_dep_wait();
}

// The port vectors of a sweep: s_q = sum_e w_in[e] / Z_e (w_in[e] = w_prev[twin[e]], the N2N
// exchange) plus the coupling currents, one thread per port and RV columns.  Its loads depend on
// each other in three steps (list ranges, list entries, waves); a kernel of its own has every port
// of every subgraph in flight at once, and a subgraph that several CTAs work on gathers once.
template <typename T, int R>
__global__ void __launch_bounds__(256) k_port_vec(const PortArgs<T> a, int nports) {
  constexpr int RV = vec_cols<T, R>();
  grid_dep_launch();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = i < nports * (R / RV);
  const int q = i / (R / RV), r = i % (R / RV) * RV;
  int e0 = 0, e1 = 0, k0 = 0, k1 = 0;
  if (live) {
    e0 = a.port_end_ptr[q], e1 = a.port_end_ptr[q + 1];
    if (a.cpl.ptr) k0 = a.cpl.ptr[q], k1 = a.cpl.ptr[q + 1];
  }
  T acc[RV] = {}, cc[RV] = {};
  bool waited = false;  // the lists are constant: only the waves come from the sweep before
  constexpr int kB = 4;  // list entries loaded together
  auto list = [&](int lo, int hi, const int32_t* row, const T* coef, T (&sum)[RV]) {
    for (int k = lo; k < hi; k += kB) {
      int at[kB];
      T c[kB], w[kB][RV];
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        at[j] = k + j < hi ? row[k + j] : -1;
        c[j] = k + j < hi ? coef[k + j] : T(0);
      }
      if (!waited) grid_dep_wait();
      waited = true;
#pragma unroll
      for (int j = 0; j < kB; ++j)
        if (at[j] >= 0) load_cg<T, RV>(a.wprev + (size_t)at[j] * R + r, w[j]);
#pragma unroll
      for (int j = 0; j < kB; ++j)
        if (at[j] >= 0)
#pragma unroll
          for (int v = 0; v < RV; ++v) sum[v] += w[j][v] * c[j];
    }
  };
  list(e0, e1, a.twin, a.invz, acc);
  if (k1 > k0) {
    list(k0, k1, a.cpl.oth, a.cpl.y, cc);
#pragma unroll
    for (int v = 0; v < RV; ++v) acc[v] += cc[v];
  }
  if (!waited) grid_dep_wait();
  if (live) store_vec<T, RV>(a.s + (size_t)q * R + r, acc);
}

// Shared memory of a sweep and the kernel that goes with it.  Accumulators per warp (R <= 2) if they
// leave room for two CTAs per SM (one in FP64); the tensor cores for FP16 tiles and for FP32 tiles with
// R = 8 wherever their operands and slots fit.  FP32 tiles, SIMT and tensor-core products: R = 4, 288
// subgraphs of 300 to 1060 ports 0.076 and 0.088 ms, 512 of 600 to 1360 0.221 and 0.250, 2500 of 40 to 130
// 0.046 and 0.058; R = 8 0.164 and 0.108, 0.486 and 0.325, 0.073 and 0.060.  Vectors too long for that many
// CTAs take one, then the SIMT products, then give up the gaps and the slots.
PortShape port_shape(size_t elem, size_t stored, int R, int max_ports) {
  const size_t npad = (size_t)((max_ports + kNB - 1) / kNB) * kNB;
  const size_t sum1 = (size_t)kNB * R * elem;  // a warp's row sums of one strip
  const size_t slot1 = (stored == 2 ? slot_bytes<__half>() : stored == 4 ? slot_bytes<float>() : slot_bytes<double>());
  const size_t kSmemMax = 226 * 1024;  // the tensor-core kernels have a static part
  const int per_sm = elem == 8 ? 1 : 2;
  const size_t all = (228 * 1024) / per_sm - 1024;  // an SM's shared memory, 1 KB per CTA reserved
  const size_t share = all < kSmemMax ? all : kSmemMax;
  PortShape p{};
  auto fit = [&](int mma, bool priv, int pad, bool ring, int sb, size_t most) {
    const int warps = sweep_threads(mma) / 32;
    p.mma = mma;
    p.priv = priv;
    p.pad = pad;
    p.ring = ring;
    p.sb = sb;
    p.vec_elems = (int)(npad * R + npad / 4 * pad);
    // rows of the vector operand start half a bank row apart (an odd number of 64-byte strips)
    p.op_stride = (int)(npad / kNB % 2 ? npad : npad + kNB);
    const size_t op = (size_t)(stored == 2 ? operand_rows<__half, 1>() : operand_rows<float, 1>()) * R * p.op_stride * 2;
    const size_t depth = stored == 2 && mma && priv ? port_depth<__half, true>() : 1;
    p.smem = (ring ? warps * slot1 * depth : 0) + (mma ? op : p.vec_elems * elem) + (size_t)p.vec_elems * elem * (priv ? warps : 1) +
             sb * warps * sum1;
    p.layout = mma && stored == 4 ? kPortFragments : R <= 2 ? kPortPatch8x4 : kPortPatch4x8;
    return p.smem <= most;
  };
  const bool mma = stored == 2 || (stored == 4 && R >= 8);
  if (R <= 2 && fit(mma ? 8 : 0, true, 0, true, 0, share)) return p;
  // tensor cores: two CTAs of 8 warps per SM where they fit, else FP32 one of 16 warps (439 MB, one CTA
  // per SM: 260 k cycles with 16 warps, 283 k with 8), else one of 8
  if (mma)
    for (int sb : {8, 4, 2, 1})
      if (fit(8, false, 0, true, sb, share)) return p;
  if (mma && stored == 4)
    for (int sb : {8, 4, 2, 1})
      if (fit(16, false, 0, true, sb, kSmemMax)) return p;
  if (mma)
    for (int sb : {8, 4, 2, 1})
      if (fit(8, false, 0, true, sb, kSmemMax)) return p;
  const int pad = (elem == 4 && R >= 4) ? 4 : 0;
  for (size_t most : {share, kSmemMax})
    for (int sb : {8, 4, 2, 1})
      if (fit(0, false, pad, true, sb, most)) return p;
  const size_t all_smem = 227 * 1024;
  if (fit(0, false, 0, true, 1, all_smem)) return p;
  fit(0, false, 0, false, 1, all_smem);  // with more ports than this has room for the band sweep has none either
  return p;
}

// Cuts the tiles of all subgraphs, in order, into shares for `ctas` CTAs, as equal as whole tiles and
// pieces of at least kMinSeg tiles allow: the smallest share for which the last CTA has no more than the
// others, by bisection.  Besides its tiles a segment costs the latency of its vectors, its partial sums
// and its waves, and a little per strip of them.  In tiles of the same kernel, from the cycles of every
// CTA of a sweep over 288 ragged subgraphs of 1 to 33 strips (least squares):
//   FP64 8 + 0.3 per strip (R = 1), 5 + 0.3 (R = 2); FP32 27 + 0.6 (R = 1, 2); FP16 41 + 1.2 (R = 1);
//   tensor cores, 8 warps: FP32 48 + 1.0 (R = 8), FP16 54 + 1.9 (R = 4), 67 + 2.6 (R = 8); 16 warps: FP32 71 + 0.1.
// FP32 at R = 4: 20 (five sets of 64 to 2500 subgraphs: 10 is up to 24 % slower, 30 and 40 within 1 % but
// 10 % slower with 2500 small ones).
PortPlan port_plan(const PieceDesc* pd, int npieces, size_t elem, size_t stored, int R, int ctas, int mma) {
  constexpr int kMinSeg = 32;
  double seg = 20, strip = 0;  // SIMT products, R >= 4
  if (elem == 8) seg = 7, strip = 0.3;
  else if (R <= 2) seg = stored == 2 ? 41 : 27, strip = stored == 2 ? 1.2 : 0.6;
  else if (mma == 16) seg = 71, strip = 0.1;
  else if (mma) seg = stored == 2 ? 60 : 46, strip = stored == 2 ? 2.3 : 0.9;
  auto strips = [](int t) {  // of the rows up to tile t's
    int I, J;
    tile_of(t, I, J);
    return I + 1;
  };
  // shares of `share` each, the last CTA takes the rest; returns what it has got
  auto cut = [&](double share, PortPlan* pl) {
    int cta = 0, nseg_all = 0;
    double load = 0;
    auto close = [&]() {
      ++cta;
      load = 0;
      if (pl) pl->cta_seg.push_back(nseg_all);
    };
    if (pl) pl->cta_seg.push_back(0);
    for (int j = 0; j < npieces; ++j) {
      if (pd[j].nports <= 0) continue;
      const int n = (int)port_tiles(pd[j].nports), first = nseg_all;
      int t = 0;
      while (t < n) {
        int take = n - t;
        const double room = share - load - seg;
        if (cta + 1 < ctas && take + strip * strips(n - 1) > room) {
          take = (int)room;
          if (take > 0) take = (int)(room - strip * strips(std::min(n, t + take) - 1));
          if (n - t - take < kMinSeg) take = n - t - kMinSeg;
          if (take < kMinSeg) {
            if (load > 0) {
              close();
              continue;
            }
            take = n - t < 2 * kMinSeg ? n - t : kMinSeg;
          }
        }
        if (pl) {
          PortSeg sg{};
          sg.piece = j;
          sg.s_off = pd[j].s_off;
          tile_of(t, sg.I0, sg.J0);
          tile_of(t + take - 1, sg.I1, sg.J1);
          sg.first = first;
          pl->segs.push_back(sg);
        }
        ++nseg_all;
        load += seg + take + strip * strips(t + take - 1);
        t += take;
        if (t < n && cta + 1 < ctas) close();
      }
      if (!pl) continue;
      const int nseg = nseg_all - first;
      for (int k = first; k < nseg_all; ++k) {
        pl->segs[k].nseg = nseg;
        pl->segs[k].part = pl->part_elems;
      }
      if (nseg > 1) pl->part_elems += (int64_t)nseg * ((pd[j].nports + kNB - 1) / kNB) * kNB * R;
    }
    if (pl && pl->cta_seg.back() != nseg_all) pl->cta_seg.push_back(nseg_all);
    return load;
  };
  double lo = 0, hi = 1;
  for (int j = 0; j < npieces; ++j)
    if (pd[j].nports > 0) {
      const int n = (int)port_tiles(pd[j].nports);
      lo += n + seg + strip * strips(n - 1);
    }
  lo = std::max(1.0, lo / std::max(1, ctas));
  hi = 2 * lo + seg + 2 * kMinSeg;
  while (cut(hi, nullptr) > hi) hi *= 2;
  for (int k = 0; k < 12; ++k) {
    const double mid = (lo + hi) / 2;
    (cut(mid, nullptr) > mid ? lo : hi) = mid;
  }
  PortPlan pl;
  cut(hi, &pl);
  return pl;
}

template <typename T, typename TS, int R>
static const void* port_kernel_r(bool priv, int mma) {
  constexpr bool can_mma = sizeof(TS) == 2 || (sizeof(TS) == 4 && R >= 8);
  if constexpr (can_mma) {
    if constexpr (R <= 2) {
      if (mma && priv) return (const void*)k_port_sweep<T, TS, R, true, 8>;
    } else if constexpr (sizeof(TS) == 4) {
      if (mma == 16) return (const void*)k_port_sweep<T, TS, R, false, 16>;
    }
    if (mma) return (const void*)k_port_sweep<T, TS, R, false, 8>;
  } else if constexpr (R <= 2) {
    if (priv) return (const void*)k_port_sweep<T, TS, R, true, 0>;
  }
  return (const void*)k_port_sweep<T, TS, R, false, 0>;
}

template <typename T, typename TS>
static const void* port_kernel(int R, bool priv, int mma) {
  switch (R) {
    case 1: return port_kernel_r<T, TS, 1>(priv, mma);
    case 2: return port_kernel_r<T, TS, 2>(priv, mma);
    case 4: return port_kernel_r<T, TS, 4>(priv, mma);
    case 8: return port_kernel_r<T, TS, 8>(priv, mma);
    default: return nullptr;
  }
}

template <typename T>
static const void* port_kernel_of(int R, bool priv, int mma, bool half) {
  if constexpr (sizeof(T) == 4)
    if (half) return port_kernel<T, __half>(R, priv, mma);
  return port_kernel<T, T>(R, priv, mma);
}

template <typename T>
cudaError_t port_sweep_configure(int R, const PortShape& sh, bool half, int* ctas_per_sm) {
  const void* k = port_kernel_of<T>(R, sh.priv, sh.mma, half);
  if (!k) return cudaErrorInvalidValue;
  // the limit is the kernel's, not the solver's: the device maximum, whatever solver came last
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (sh.mma ? 226 : 227) * 1024);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, sweep_threads(sh.mma), sh.smem);
  return e;
}

// A launch whose CTAs may start while the launch before it on the stream still runs (the kernel
// waits for its results itself, grid_dep_wait).
template <typename T>
static cudaError_t launch_dependent(const void* k, int grid, int block, size_t smem, void** args, cudaStream_t st) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, k, args);
}

template <typename T>
cudaError_t launch_port_sweep(const PortArgs<T>& a, int R, int nports, int grid, size_t smem, cudaStream_t st) {
  if (grid <= 0 || nports <= 0) return cudaSuccess;
  const void* k = port_kernel_of<T>(R, a.priv != 0, a.mma, sizeof(T) == 4 && a.Sh);
  const void* v = R == 1   ? (const void*)k_port_vec<T, 1>
                  : R == 2 ? (const void*)k_port_vec<T, 2>
                  : R == 4 ? (const void*)k_port_vec<T, 4>
                           : (const void*)k_port_vec<T, 8>;
  if (!k) return cudaErrorInvalidValue;
  PortArgs<T> args = a;
  const int n = nports * std::max(1, R * (int)sizeof(T) / 16);
  void* av[] = {&args, &nports};
  cudaError_t e = launch_dependent<T>(v, (n + 255) / 256, 256, 0, av, st);
  if (e != cudaSuccess) return e;
  return launch_dependent<T>(k, grid, sweep_threads(a.mma), smem, av, st);
}

// FP16 copy of the FP32 tiles of one subgraph per CTA, one warp per tile: each tile is divided by
// its largest |entry| (1 if all zero), kept in scale[], and re-laid out (for ldmatrix, or as patches).  A scale per tile keeps the small far-field blocks of S_j at full FP16 precision.
__global__ void k_port_to_half(const PieceDesc* __restrict__ pieces, const float* __restrict__ S,
                               __half* __restrict__ Sh, float* __restrict__ scale, int from, int to, int mma) {
  const PieceDesc pd = pieces[blockIdx.x];
  const int64_t nt = port_tiles(pd.nports);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t t = warp; t < nt; t += blockDim.x >> 5) {
    const float* src = S + (pd.s_off + t) * kNB * kNB;
    __half* dst = Sh + (pd.s_off + t) * kNB * kNB;
    float m = 0.f;
    for (int k = lane; k < kNB * kNB; k += 32) m = fmaxf(m, fabsf(src[k]));
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float sc = m > 0.f ? m : 1.f;
    if (lane == 0) scale[pd.s_off + t] = sc;
    const float inv = 1.f / sc;
    for (int k = lane; k < kNB * kNB; k += 32) {
      const int i = k / kNB, c = k % kNB;
      dst[mma ? half_pos(i, c) : tile_pos(to, i, c, 8)] = __float2half_rn(src[tile_pos(from, i, c, 4)] * inv);
    }
  }
}

cudaError_t launch_port_to_half(const PieceDesc* pieces, int npieces, const float* S, __half* Sh, float* scale,
                                const PortShape& from, const PortShape& to, cudaStream_t st) {
  if (npieces <= 0) return cudaSuccess;
  k_port_to_half<<<npieces, kSweepThreads, 0, st>>>(pieces, S, Sh, scale, from.layout, to.layout, to.mma);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gather_port_response(const PieceDesc* pieces, int npieces, const int32_t* port_local, int Rs, int b,
                                        const T* xc, T* S, int layout, cudaStream_t st, int batches, int64_t stride) {
  if (npieces <= 0) return cudaSuccess;
  k_gather_port_response<T><<<dim3(npieces, batches), 256, 0, st>>>(pieces, port_local, Rs, b, xc, stride, S, layout);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gather_ports(const PieceDesc* pieces, int npieces, const int32_t* port_local, int R, const T* xc,
                                T* ubase, cudaStream_t st) {
  if (npieces <= 0) return cudaSuccess;
  k_gather_ports<T><<<npieces, 256, 0, st>>>(pieces, port_local, R, xc, ubase);
  return cudaGetLastError();
}

#define VTM_PORT_INST(T)                                                                                       \
  template cudaError_t port_sweep_configure<T>(int, const PortShape&, bool, int*);                             \
  template cudaError_t launch_port_sweep<T>(const PortArgs<T>&, int, int, int, size_t, cudaStream_t);          \
  template cudaError_t launch_gather_port_response<T>(const PieceDesc*, int, const int32_t*, int, int, const T*, \
                                                      T*, int, cudaStream_t, int, int64_t);                        \
  template cudaError_t launch_gather_ports<T>(const PieceDesc*, int, const int32_t*, int, const T*, T*, cudaStream_t);
VTM_PORT_INST(float)
VTM_PORT_INST(double)

}  // namespace vtm
