// Port-response sweeps of small systems in one launch: the port responses stay in shared memory and
// the waves go from subgraph to subgraph without leaving the kernel.
//
// The method's own exchange (Table 1 steps 3 and 5, Neighbor-To-Neighbor): a subgraph's next sweep
// needs the waves of its neighbours and nothing else, so no barrier over the whole GPU stands
// between two sweeps.  Every CTA holds the dense S_j of its subgraphs (res_plan packs them) and per
// sweep
//   1. reads each incoming wave from the exchange buffer of the sweep before, waiting until it is
//      there, and forms s = sum_e w_in[e] / Z_e plus the coupling currents;
//   2. computes y = S_j s from shared memory;
//   3. publishes w_out[e] = 2 (u_base + y) - w_in[e].
// A published value is a 64-bit word with the sweep's number in its upper half (FP64: two words, one
// per half of the value), stored and read as a whole, so that the value and the news of its arrival
// are one access and no fence stands between them.  The two exchange buffers alternate: a CTA
// writes its word of sweep k + 2 only after it has read its twins' words of sweep k + 1, which they
// publish after reading its word of sweep k (every subgraph that reads a wave of another also sends
// it one: lines and coupled lines join the same two subgraphs).
//
// All CTAs must run at the same time: the launch is cooperative, with at most one CTA per SM.  Every
// wait is bounded; a CTA whose wait runs out records VTM_ERR_TIMEOUT and goes on without waiting, so
// that the launch ends.
//
// What bounds it: the latency of the exchange (a store, a load that sees it) and of the product's three
// block-wide steps, about 2 us together; S is not read from memory at all.  Measured per sweep in batches of 160
// (of 20), launch and clearing included, against one launch per sweep: 32^2 in 4 subgraphs, FP64 8.9 -> 2.2
// (2.5) us; 256^2 in 64 subgraphs, FP32, coupled lines 6.8 -> 2.0 (2.3) us; 100 finite-element subgraphs of about
// 100 ports, 16 right-hand sides (tensor-core sweep before) 13 -> 7.0 (7.3) us.
#include <algorithm>
#include <numeric>

#include "kernels.h"

namespace vtm {

namespace {

constexpr int kResThreads = 256;
constexpr int kResWarps = kResThreads / 32;
constexpr int kParts = 4;  // lanes of a warp that share a group of rows, each with every fourth column

template <typename T>
__host__ __device__ constexpr int res_vr() {  // rows per lane: 16 bytes of a column of S
  return 16 / (int)sizeof(T);
}
template <typename T>
__host__ __device__ constexpr int res_group() {  // rows per unit of work
  return 8 * res_vr<T>();
}

// Columns that a thread of the wave passes takes at once (their words are contiguous): enough that
// the ports of a subgraph of about a hundred ports take one round of the block, because every round
// waits for its own loads.  And list entries whose loads it keeps in flight together.
template <typename T, int R>
__host__ __device__ constexpr int res_cols() {
  return sizeof(T) == 8 ? (R < 4 ? R : 4) : (R <= 4 ? R : R / 2);
}
template <typename T, int R>
__host__ __device__ constexpr int res_batch() {
  return res_cols<T, R>() * (int)(sizeof(T) / 4) <= 4 ? 4 : res_cols<T, R>() <= 8 ? 2 : 1;
}

template <int N>
__device__ __forceinline__ void store_words(unsigned long long* p, const unsigned long long (&w)[N]) {
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2)
      asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p + i), "l"(w[i]), "l"(w[i + 1]) : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p + i), "l"(w[i]) : "memory");
  }
}

template <int N>
__device__ __forceinline__ void load_words(const unsigned long long* p, unsigned long long (&w)[N]) {
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2)
      asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w[i]), "=l"(w[i + 1]) : "l"(p + i) : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w[i]) : "l"(p + i) : "memory");
  }
}

// Values k .. k + C - 1 of a buffer as tagged words.
template <typename T, int C>
__device__ __forceinline__ void publish(unsigned long long* buf, size_t k, const T (&v)[C], uint32_t tag) {
  constexpr int W = sizeof(T) / 4;
  unsigned long long w[C * W];
  const unsigned long long hi = (unsigned long long)tag << 32;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    if constexpr (W == 1) {
      w[c] = hi | __float_as_uint(v[c]);
    } else {
      const unsigned long long b = (unsigned long long)__double_as_longlong(v[c]);
      w[2 * c] = hi | (b & 0xffffffffull);
      w[2 * c + 1] = hi | (b >> 32);
    }
  }
  store_words<C * W>(buf + k * W, w);
}

// The C values from each of N places at[j] of a buffer (skipped where at[j] < 0) once all of them
// carry the tag, their loads in flight together.  False if the wait ran out.
template <typename T, int C, int N>
__device__ __forceinline__ bool receive(const unsigned long long* buf, const int64_t (&at)[N], uint32_t tag, long limit,
                                        T (&v)[N][C]) {
  constexpr int W = sizeof(T) / 4;
  unsigned long long w[N][C * W];
  for (long it = 0;; ++it) {
    bool all = true;
#pragma unroll
    for (int j = 0; j < N; ++j)
      if (at[j] >= 0) load_words<C * W>(buf + at[j] * W, w[j]);
#pragma unroll
    for (int j = 0; j < N; ++j)
      if (at[j] >= 0)
#pragma unroll
        for (int h = 0; h < C * W; ++h) all = all && (uint32_t)(w[j][h] >> 32) == tag;
    if (all) break;
    if (it >= limit) return false;
  }
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (at[j] >= 0)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if constexpr (W == 1) v[j][c] = __uint_as_float((uint32_t)w[j][c]);
        else v[j][c] = __longlong_as_double((long long)((w[j][2 * c + 1] << 32) | (w[j][2 * c] & 0xffffffffull)));
      }
  return true;
}

}  // namespace

// Sweeps 1 .. k of the subgraphs' ports from the waves wprev (ends x R); the last one writes wout.
template <typename T, int R>
__global__ void __launch_bounds__(kResThreads, 1) k_port_resident(const ResArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int VR = res_vr<T>(), C = res_cols<T, R>(), kB = res_batch<T, R>();
  const ResCta ct = a.ctas[blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T* const Ss = reinterpret_cast<T*>(smem);
  T* const ss = Ss + ct.s_elems;                        // [ports][R], subgraph after subgraph
  T* const yp = ss + (size_t)ct.vec * R;                // [splits][ports][R]
  T* const win = yp + (size_t)ct.splits * ct.vec * R;   // [ends][R]
  const ResUnit* const units = a.units + ct.unit0;
  // S into shared memory (contiguous for the CTA), zero rows for the padding of s
  for (int64_t i = tid; i < ct.s_elems / VR; i += kResThreads)
    reinterpret_cast<uint4*>(Ss)[i] = reinterpret_cast<const uint4*>(a.S + ct.s_off)[i];
  for (int i = tid; i < ct.vec * R; i += kResThreads) ss[i] = T(0);
  __syncthreads();
  bool ok = true;
  for (int k = 1; k <= a.sweeps; ++k) {
    const unsigned long long* in = a.xch[k & 1];  // sweep k - 1 wrote buffer (k - 1 + 1) & 1
    // ---- incoming waves, port vectors
    // entries lo .. hi - 1 of a list (place of the wave, coefficient): sum of coefficient times wave;
    // keep: the waves themselves to win
    auto gather = [&](int lo, int hi, const int32_t* place, const T* coef, int r, T* keep, T(&sum)[C]) {
      for (int q0 = lo; q0 < hi; q0 += kB) {
        int64_t at[kB];
        T y[kB], w[kB][C];
#pragma unroll
        for (int j = 0; j < kB; ++j) {
          at[j] = q0 + j < hi ? (int64_t)place[q0 + j] * R + r : -1;
          y[j] = q0 + j < hi ? coef[q0 + j] : T(0);
#pragma unroll
          for (int c = 0; c < C; ++c) w[j][c] = T(0);
        }
        if (k == 1) {
#pragma unroll
          for (int j = 0; j < kB; ++j)
            if (at[j] >= 0)
#pragma unroll
              for (int c = 0; c < C; ++c) w[j][c] = a.wprev[at[j] + c];
        } else if (ok) {
          ok = receive<T, C, kB>(in, at, (uint32_t)(k - 1), a.wait_limit, w);
        }
#pragma unroll
        for (int j = 0; j < kB; ++j)
          if (at[j] >= 0)
#pragma unroll
            for (int c = 0; c < C; ++c) {
              sum[c] += y[j] * w[j][c];
              if (keep) keep[(size_t)(q0 + j - lo) * R + c] = w[j][c];
            }
      }
    };
    for (int i = tid; i < ct.nports * (R / C); i += kResThreads) {
      const int p = i / (R / C), r = i % (R / C) * C;
      const ResPort pt = a.ports[ct.port0 + p];
      T acc[C] = {}, cc[C] = {};
      gather(pt.e0, pt.e1, a.twin, a.invz, r, win + (size_t)pt.w0 * R + r, acc);
      if (a.cpl.ptr) gather(a.cpl.ptr[pt.port], a.cpl.ptr[pt.port + 1], a.cpl.oth, a.cpl.y, r, nullptr, cc);
#pragma unroll
      for (int c = 0; c < C; ++c) ss[(size_t)pt.vec * R + r + c] = acc[c] + cc[c];
    }
    __syncthreads();
    // ---- y = S_j s: a warp per unit (G rows of one subgraph, a run of its columns)
    for (int u = warp; u < ct.nunits; u += kResWarps) {
      const ResUnit un = units[u];
      const int quad = lane & 7, part = lane >> 3;
      const T* Sc = Ss + un.s + quad * VR;
      const T* sc = ss + (size_t)un.vec * R;
      T acc[VR][R];
#pragma unroll
      for (int v = 0; v < VR; ++v)
#pragma unroll
        for (int r = 0; r < R; ++r) acc[v][r] = T(0);
#pragma unroll 4
      for (int c = un.c0 + part; c < un.c1; c += kParts) {
        T col[VR];
        if constexpr (sizeof(T) == 4) {
          const float4 x = *reinterpret_cast<const float4*>(Sc + (size_t)c * un.stride);
          col[0] = x.x, col[1] = x.y, col[2] = x.z, col[3] = x.w;
        } else {
          const double2 x = *reinterpret_cast<const double2*>(Sc + (size_t)c * un.stride);
          col[0] = x.x, col[1] = x.y;
        }
        const T* sp = sc + (size_t)c * R;
        T sr[R];
        if constexpr (sizeof(T) == 4 && R % 4 == 0) {
#pragma unroll
          for (int q = 0; q < R / 4; ++q) {
            const float4 x = reinterpret_cast<const float4*>(sp)[q];
            sr[4 * q] = x.x, sr[4 * q + 1] = x.y, sr[4 * q + 2] = x.z, sr[4 * q + 3] = x.w;
          }
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) sr[r] = sp[r];
        }
#pragma unroll
        for (int v = 0; v < VR; ++v)
#pragma unroll
          for (int r = 0; r < R; ++r) acc[v][r] += col[v] * sr[r];
      }
#pragma unroll
      for (int v = 0; v < VR; ++v)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          T x = acc[v][r];
          x += __shfl_xor_sync(0xffffffffu, x, 8);
          x += __shfl_xor_sync(0xffffffffu, x, 16);
          acc[v][r] = x;
        }
      // lane of part q writes rows q, q + kParts, ... of its quad
      T* o = yp + ((size_t)un.split * ct.vec + un.vec + un.row0 + quad * VR) * R;
#pragma unroll
      for (int v = 0; v < VR; ++v)
        if (v % kParts == part && un.row0 + quad * VR + v < un.n)
#pragma unroll
          for (int r = 0; r < R; ++r) o[(size_t)v * R + r] = acc[v][r];
    }
    __syncthreads();
    // ---- outgoing waves
    const bool lastk = k == a.sweeps;
    unsigned long long* out = a.xch[(k + 1) & 1];
    for (int i = tid; i < ct.nports * (R / C); i += kResThreads) {
      const int p = i / (R / C), r = i % (R / C) * C;
      const ResPort pt = a.ports[ct.port0 + p];
      T u[C];
#pragma unroll
      for (int c = 0; c < C; ++c) u[c] = a.ubase[(size_t)pt.port * R + r + c];
      for (int q = 0; q < ct.splits; ++q)
#pragma unroll
        for (int c = 0; c < C; ++c) u[c] += yp[((size_t)q * ct.vec + pt.vec) * R + r + c];
      for (int e = pt.e0; e < pt.e1; ++e) {
        T w[C];
#pragma unroll
        for (int c = 0; c < C; ++c) w[c] = T(2) * u[c] - win[(size_t)(pt.w0 + e - pt.e0) * R + r + c];
        if (lastk) {
#pragma unroll
          for (int c = 0; c < C; ++c) a.wout[(size_t)e * R + r + c] = w[c];
        } else {
          publish<T, C>(out, (size_t)e * R + r, w, (uint32_t)k);
        }
      }
    }
    // the next sweep writes s after the barrier above and each thread its own entries of win
  }
  if (!ok) atomicExch(a.status, kStatusTimeout);
}

// Packs the subgraphs onto at most `nsm` CTAs: largest first, each onto the CTA with the least work so
// far that has room for it.  Not ok when they do not fit into the CTAs' shared memory.
ResPlan res_plan(const PieceDesc* pd, int npieces, size_t elem, int R, int nsm) {
  ResPlan pl;
  const int vr = 16 / (int)elem, group = 8 * vr;
  const size_t kSmemMax = 227 * 1024;
  std::vector<int> order;
  for (int j = 0; j < npieces; ++j)
    if (pd[j].nports > 0) order.push_back(j);
  if (order.empty()) return pl;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return pd[x].nports > pd[y].nports; });
  struct Bin {
    std::vector<int> pieces;
    int64_t s = 0, vec = 0, ends = 0;
    int groups = 0;
  };
  auto stride = [&](int n) { return (n + group - 1) / group * group; };
  auto bytes = [&](const Bin& b, int splits) { return elem * (size_t)(b.s + (b.vec * (1 + splits) + b.ends) * R); };
  std::vector<Bin> bins(std::min<size_t>(nsm, order.size()));
  for (int j : order) {
    const int n = pd[j].nports;
    int best = -1;
    for (int b = 0; b < (int)bins.size(); ++b) {
      Bin t = bins[b];
      t.s += (int64_t)n * stride(n);
      t.vec += n;
      t.ends += pd[j].nends;
      if (bytes(t, 1) > kSmemMax) continue;
      if (best < 0 || bins[b].s < bins[best].s) best = b;
    }
    if (best < 0) return pl;
    Bin& b = bins[best];
    b.pieces.push_back(j);
    b.s += (int64_t)n * stride(n);
    b.vec += n;
    b.ends += pd[j].nends;
    b.groups += (n + group - 1) / group;
  }
  for (const Bin& b : bins) {
    // columns of a group in `splits` units where that fills the warps better
    int splits = 1;
    double best = 1e30;
    for (int c = 1; c <= 4; ++c) {
      const double t = (double)((b.groups * c + kResWarps - 1) / kResWarps) / c + 0.03 * c;
      if (t < best - 1e-9 && bytes(b, c) <= kSmemMax) best = t, splits = c;
    }
    ResCta ct{};
    ct.s_off = pl.s_elems;
    ct.s_elems = (int32_t)b.s;
    ct.vec = (int32_t)b.vec;
    ct.splits = splits;
    ct.port0 = (int32_t)pl.ports.size();
    ct.unit0 = (int32_t)pl.units.size();
    int64_t s = 0;
    int vec = 0;
    for (int j : b.pieces) {
      const int n = pd[j].nports, st = stride(n);
      pl.piece_s.push_back({pd[j].port_off, n, st, ct.s_off + s, j});
      for (int p = 0; p < n; ++p) {
        ResPort rp{};
        rp.port = pd[j].port_off + p;
        rp.vec = vec + p;
        pl.ports.push_back(rp);  // e0, e1, w0 from the end lists (res_plan_ends)
      }
      for (int row0 = 0; row0 < n; row0 += group)
        for (int c = 0; c < splits; ++c) {
          ResUnit u{};
          u.s = (int32_t)(s + row0);
          u.stride = st;
          u.n = n;
          u.row0 = row0;
          u.vec = vec;
          u.c0 = (int)((int64_t)n * c / splits);
          u.c1 = (int)((int64_t)n * (c + 1) / splits);
          u.split = c;
          pl.units.push_back(u);
        }
      s += (int64_t)n * st;
      vec += n;
    }
    ct.nports = (int32_t)pl.ports.size() - ct.port0;
    ct.nunits = (int32_t)pl.units.size() - ct.unit0;
    pl.s_elems += b.s;
    pl.smem = std::max(pl.smem, bytes(b, splits));
    pl.ctas.push_back(ct);
  }
  pl.ok = true;
  return pl;
}

void res_plan_ends(ResPlan& pl, const int32_t* port_end_ptr) {
  for (const ResCta& ct : pl.ctas) {
    int w0 = 0;
    for (int i = ct.port0; i < ct.port0 + ct.nports; ++i) {
      ResPort& p = pl.ports[i];
      p.e0 = port_end_ptr[p.port];
      p.e1 = port_end_ptr[p.port + 1];
      p.w0 = w0;
      w0 += p.e1 - p.e0;
    }
  }
}

// Columns cc = b * Rs + r of S_j from unit-source solves (xc: copies x Rs) into the dense storage,
// column by column.  As in the tiled storage the entry of the lower tile triangle counts for both
// (i, c) and (c, i): S_j is symmetric up to the rounding of those solves.
template <typename T>
__global__ void k_gather_port_dense(const ResPieceS* __restrict__ ps, const PieceDesc* __restrict__ pieces,
                                    const int32_t* __restrict__ port_local, int Rs, int b0, const T* __restrict__ x0,
                                    int64_t stride, T* __restrict__ S) {
  const ResPieceS p = ps[blockIdx.x];
  const int b = b0 + (int)blockIdx.y;
  const T* xc = x0 + (size_t)blockIdx.y * stride;
  const int64_t copy0 = pieces[p.piece].copy_off;
  for (int i = b * Rs / kNB * kNB * Rs + threadIdx.x; i < p.n * Rs; i += blockDim.x) {
    const int q = i / Rs, r = i % Rs;
    const int cc = b * Rs + r;
    if (cc >= p.n || q / kNB < cc / kNB) continue;
    const T v = xc[(size_t)(copy0 + port_local[p.port_off + q]) * Rs + r];
    S[p.s + (int64_t)cc * p.stride + q] = v;
    if (q / kNB > cc / kNB) S[p.s + (int64_t)q * p.stride + cc] = v;
  }
}

template <typename T>
cudaError_t launch_gather_port_dense(const ResPieceS* ps, int n, const PieceDesc* pieces, const int32_t* port_local,
                                     int Rs, int b, const T* xc, T* S, cudaStream_t st, int batches, int64_t stride) {
  if (n <= 0) return cudaSuccess;
  k_gather_port_dense<T><<<dim3(n, batches), 256, 0, st>>>(ps, pieces, port_local, Rs, b, xc, stride, S);
  return cudaGetLastError();
}

template <typename T>
static const void* resident_kernel(int R) {
  switch (R) {
    case 1: return (const void*)k_port_resident<T, 1>;
    case 2: return (const void*)k_port_resident<T, 2>;
    case 4: return (const void*)k_port_resident<T, 4>;
    case 8: return (const void*)k_port_resident<T, 8>;
    case 16: return sizeof(T) == 4 ? (const void*)k_port_resident<float, 16> : nullptr;
    case 32: return sizeof(T) == 4 ? (const void*)k_port_resident<float, 32> : nullptr;
    default: return nullptr;
  }
}

template <typename T>
cudaError_t port_resident_configure(int R, size_t smem, int* ctas_per_sm) {
  const void* k = resident_kernel<T>(R);
  if (!k) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, kResThreads, smem);
  return e;
}

template <typename T>
cudaError_t launch_port_resident(const ResArgs<T>& a, int R, int grid, size_t smem, size_t xch_bytes, cudaStream_t st) {
  if (grid <= 0 || a.sweeps <= 0) return cudaSuccess;
  const void* k = resident_kernel<T>(R);
  if (!k) return cudaErrorInvalidValue;
  if (a.sweeps > 1) {  // no word of an earlier launch may carry one of this launch's numbers
    cudaError_t e = cudaMemsetAsync(a.xch[0], 0, xch_bytes, st);
    if (e != cudaSuccess) return e;
  }
  ResArgs<T> args = a;
  void* av[] = {&args};
  return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kResThreads), av, smem, st);
}

#define VTM_RES_INST(T)                                                                                           \
  template cudaError_t launch_gather_port_dense<T>(const ResPieceS*, int, const PieceDesc*, const int32_t*, int, int, \
                                                   const T*, T*, cudaStream_t, int, int64_t);                     \
  template cudaError_t port_resident_configure<T>(int, size_t, int*);                                             \
  template cudaError_t launch_port_resident<T>(const ResArgs<T>&, int, int, size_t, size_t, cudaStream_t);
VTM_RES_INST(float)
VTM_RES_INST(double)

}  // namespace vtm
