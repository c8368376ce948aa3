// Port-response sweep for 16 or 32 right-hand sides on the 5th-generation tensor cores.
//
// Per subgraph the sweep needs y = S_j s (then u = u_base + y, w_out = 2u - w_in; see port.cu for
// the method).  With R = 16/32 columns this is a dense product, run as tcgen05.mma (kind::f16,
// FP32 accumulation in tensor memory).
//
// Storage of S_j.  S_j is symmetric (the open-circuit impedance matrix of Def. 7.1 over all ports,
// the S of eq. A3.3), so only its lower block triangle is kept: 128 x 128 blocks (I, J), J <= I,
// row by row.  Block (I, J) serves two products: y_I += S_IJ s_J reads it K-major and
// y_J += S_IJ^T s_I reads the same bytes as an MN-major (transposed) operand.  Each block is four
// 128-byte-swizzled panels [hi, cols 0-63][hi, cols 64-127][lo, 0-63][lo, 64-127] of h_I rows
// (rows of 128 bytes, 16-byte units XOR-ed with the row mod 8, 8-row groups 1024 bytes apart);
// h_I = 128 except for the last super-row, whose height is its port count rounded up to 16.  The
// values are those of the diagonally balanced S'_j = G^-1 S_j G^-1 (G = diag(sqrt(S_pp)), so that
// S'_pp = 1 and |S'_pq| <= 1 even across coefficient jumps of many decades) divided by sigma_j, the
// power of two at or above max |S'_j|; hi = fp16(x) and lo = fp16(x - hi), so hi + lo keeps about
// 22 significant bits.  The port vector is balanced the other way (s' = G s) and y = G^-1 S' s'.  Transposed fp16 operands work on
// this tensor core; kind::tf32 with the same MN-major descriptor returns zeros, which is why the
// storage is fp16 pairs and not FP32.
//
// Products.  The port vector s = sum_e w_in[e] / Z_e (plus coupling currents) is split the same
// way per subgraph and column: s / sigma_r = s_hi + s_lo (sigma_r a power of two).  Per block and
// K step: hi(S) s_hi + hi(S) s_lo (+ lo(S) s_hi when the lo half is used), FP32 accumulation.
// With the lo half the products keep about 2^-21 of |S||s| (the dropped lo(S) s_lo term and the
// fp16 roundings); without it (FP16 storage, half the bytes) S carries fp16 rounding, 2^-11 of
// sigma_j, and the FP64 defect correction absorbs it as for the FP16 tiles of port.cu.
//
// Work split.  A CTA takes items, each a run of super-rows hi .. lo of one subgraph (tc_plan): whole
// subgraphs where they are many, cut ones where a subgraph is more than a CTA's share, the items
// dealt out largest first to the CTA with the least work so far.  An item that is a whole subgraph
// writes its waves itself; the others leave the rows y_0 .. y_hi they added to as partial sums, and
// k_port_finish_tc adds a row's partials in the items' order and writes the waves.  (Every CTA
// taking subgraphs c, c + grid, ... : 64 subgraphs left 88 of 152 SMs idle, 512 uneven ones kept the
// unluckiest CTA busy 1.3 times the average.)
//
// One persistent kernel per sweep, one CTA per SM looping over its items, 448 threads:
//  * warp 0 streams the blocks (and the s_J tile of off-diagonal blocks) through a ring of 16 KB
//    shared-memory slots by bulk copies (mbarrier complete_tx).  A block's panels go out one pair
//    at a time, each as soon as its slots are free, so that the next blocks stream in while the
//    current one is multiplied; the s_I tile of each super-row goes into a 2-slot row buffer a few
//    blocks before its row starts;
//  * warp 1 issues the MMAs: y_I at tensor-memory columns I R .. I R + R - 1, lane = port, all
//    super-rows of a subgraph held at once (n4 R <= 512 columns); tcgen05.commit releases stages
//    and row buffers and hands each finished y_I to the epilogue;
//  * epilogue warps, four at a time (one per tensor-memory lane quadrant): tcgen05.ld of each y_I
//    (released at once for the next item's MMAs), u = u_base + sigma_j sigma_r y, w_out[e] = 2u - w_in[e].
// The port vectors come one of two ways:
//  * FUSED (many items per CTA): warps 6-13 compute the next item's s: a gather pass driven by per-port
//    records (FP32 values to a staging area), a coalesced pass over that area for the column maxima,
//    then the split values written to a per-CTA global scratch slot that stays in L2.  With the next
//    items' blocks to stream meanwhile the gathers cost nothing (256^3: 27 subgraphs per CTA, 0.955 of
//    the copy bandwidth).
//  * else (few items per CTA) in a launch of their own before it (k_port_vec_tc), which has every
//    subgraph's gathers in flight at once, and warps 6-13 are two more sets of epilogue warps: super-row
//    I belongs to set I mod 3.  Fused, eight warps waiting for 1.4 MB of scattered rows per subgraph
//    were what such a sweep waited for.  Measured per sweep, 32 right-hand sides: 64^3 (1.2 items per
//    CTA) 0.193 -> 0.083 ms, 128^3 (3.4) 0.557 -> 0.521 ms.
// Every wait is bounded; a CTA that gives up records VTM_ERR_TIMEOUT, lets its copies and MMAs
// finish, frees its tensor memory and returns.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "kernels.h"
#include "tc.cuh"

namespace vtm {

using namespace tc;

namespace {

constexpr int kSB = 128;                // ports per super-block (MMA M; K extent of a block)
constexpr int kEpiWarps = 4;            // a set of epilogue warps: one per tensor-memory lane quadrant
constexpr int kEpiSets = 3;             // sets, not FUSED
constexpr int kVecWarps = 8;            // port vectors, FUSED (the place of two sets)
constexpr int kTcThreads = 32 * (2 + kEpiWarps + kVecWarps);  // warp 0 copies, warp 1 MMA
static_assert(kEpiSets * kEpiWarps == kEpiWarps + kVecWarps, "warps");
constexpr int kVecThreads = 32 * kVecWarps;
constexpr int kEpiBar = 1;              // named barriers of the epilogue sets: 1, 2, 3
constexpr int kVecBar = 4;              // named barrier of the vector warps
constexpr int kMaxSuper = kTcMaxSuper;  // super-rows per subgraph (and tensor memory: n4 R <= 512)

__host__ __device__ __forceinline__ int n_super(int nports) { return (nports + kSB - 1) / kSB; }

// Stored rows of super-row I (a multiple of 16).
__host__ __device__ __forceinline__ int sb_rows(int nports, int I) {
  const int n4 = n_super(nports);
  if (I < n4 - 1) return kSB;
  return ((nports - kSB * I) + 15) & ~15;
}

// Byte offset of block (I, J) from the subgraph's first block (hi + lo: 512 bytes per row).
__host__ __device__ __forceinline__ int64_t blk_off(int nports, int I, int J) {
  return (int64_t)I * (I + 1) / 2 * (kSB * 512) + (int64_t)J * sb_rows(nports, I) * 512;
}

__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void vec_sync() { asm volatile("bar.sync %0, %1;" ::"n"(kVecBar), "n"(kVecThreads) : "memory"); }
__device__ __forceinline__ void epi_sync(int set) {
  asm volatile("bar.sync %0, %1;" ::"r"(kEpiBar + set), "n"(32 * kEpiWarps) : "memory");
}

// Header offsets (bytes from the aligned start).
constexpr uint32_t kOffFull = 0, kOffEmpty = 64, kOffRowFull = 128, kOffRowEmpty = 144, kOffSReady = 160,
                   kOffSlotFree = 176, kOffRReady = 192, kOffRowRead = 320, kOffDone = 448, kOffTslot = 456,
                   kOffFlags = 464, kOffSsig = 512, kOffOwner = 896, kOffRed = 1024;
static_assert(kOffRReady + 8 * kMaxSuper <= kOffRowRead && kOffRowRead + 8 * kMaxSuper <= kOffDone, "header");

// Shared-memory plan.  The kernel has no static shared memory: up to 1008 bytes to align the start
// to 1024, a 2 KB header (mbarriers, flags, the column scales sigma_r, the copy warp's slot owners,
// the vector warps' reduction scratch), a ring of 10 slots of 16 KB that carries the S panels and
// s_J tiles, then two s_I row tiles.  Ten slots hold two stages of an off-diagonal block with its
// lo half (four panels and the s_J tile) at once; every further slot is taken from the L1 cache that
// the gathers of the vector and epilogue warps hit in, which costs more than the extra bytes in
// flight gain (measured: 9, 10, 11, 12 slots run one sweep in 1.12, 1, 1.08, 1.10 times the time).
template <int R>
struct Plan {
  static constexpr uint32_t kSlot = 16384;              // one panel of a full-height block
  static constexpr uint32_t kVec = (uint32_t)R * 512u;  // s tile: hi / lo x 2 panels of R rows
  static constexpr uint32_t kHead = 2048;
  static constexpr int kSlots = 10;
  static constexpr uint32_t kRow = kHead + kSlots * kSlot;  // the two row tiles, from the aligned start
  static constexpr uint32_t kAlloc = 1008 + kRow + 2 * kVec;
  static_assert(kAlloc <= 227 * 1024, "shared-memory plan");
  static_assert(kOffSsig + 4 * kEpiSets * R <= kOffOwner && kOffOwner + 4 * kSlots <= kOffRed &&
                    kOffRed + 4 * kVecWarps * R <= kHead,
                "header");
};
constexpr int kStg = 8;  // stage barriers (full / empty) in use round robin

// Ring slots of one block (stage).  The hi panels (and, with the lo half, the lo panels) take two
// adjacent slots each: the transposed product reads a pair as one MN-major operand whose halves are
// one slot apart, so a pair never wraps around the end of the ring.  The s_J tile of an off-diagonal
// block takes one slot, the ring's last one when a pair would otherwise start there (else that slot
// is skipped).  Copy warp and MMA issuer place the same sequence of blocks and so agree on every
// position; `a` counts slots from the start of the launch.
struct StagePos {
  int hi, lo, s;
};
template <int NS>
__device__ __forceinline__ StagePos place_stage(int64_t& a, bool lo, bool has_s) {
  StagePos p{-1, -1, -1};
  bool s_open = has_s;
  auto pair = [&]() {
    if ((int)(a % NS) == NS - 1) {
      if (s_open) {
        p.s = NS - 1;
        s_open = false;
      }
      ++a;
    }
    const int r = (int)(a % NS);
    a += 2;
    return r;
  };
  p.hi = pair();
  if (lo) p.lo = pair();
  if (s_open) {
    p.s = (int)(a % NS);
    ++a;
  }
  return p;
}

// The MMAs of one block (I, J) of height h: y_I += S_IJ s_J (A K-major: the block's two panels
// along K; B = the s tile bv) and, off the diagonal, y_J += S_IJ^T s_I (A MN-major: M over the two
// panels of a pair, one ring slot apart; K = the block's rows in steps of 16; B = the row tile si).
// Products per K step: hi(S) s_hi, hi(S) s_lo and, with LO, lo(S) s_hi.  first / first_t: the
// product overwrites y_I / y_J instead of adding.  Descriptors are formed once and advanced by
// address offsets (16-byte units in the low bits).
template <int R, bool LO>
__device__ __forceinline__ void block_mmas(uint32_t hiA, uint32_t loA, uint32_t bv, uint32_t si, int h, uint32_t dI,
                                           uint32_t dJ, bool first, bool first_t, bool transposed) {
  constexpr uint32_t idK = idesc_f16(false, R), idT = idesc_f16(true, R);
  constexpr uint32_t vpan = (uint32_t)R * 128 / 16;  // s tile panel, 16-byte units
  constexpr uint32_t pan = Plan<R>::kSlot / 16;      // ring slot, 16-byte units
  const uint64_t aK = sdesc(hiA, 16, 1024), aKl = sdesc(loA, 16, 1024);
  const uint64_t bB = sdesc(bv, 16, 1024), bR = sdesc(si, 16, 1024);
#pragma unroll
  for (int kk = 0; kk < kSB / 16; ++kk) {
    const uint32_t p = kk >> 2, o = (kk & 3) * 2;  // panel, 32-byte step in 16-byte units
    const uint64_t aH = aK + p * pan + o, bH = bB + p * vpan + o, bL = bB + (2 + p) * vpan + o;
    if (kk == 0) mma_f16(dI, aH, bH, idK, first ? 0u : 1u);
    else mma_f16_acc(dI, aH, bH, idK);
    mma_f16_acc(dI, aH, bL, idK);
    if constexpr (LO) mma_f16_acc(dI, aKl + p * pan + o, bH, idK);
  }
  if (!transposed) return;
  const uint64_t aT = sdesc(hiA, Plan<R>::kSlot, 1024), aTl = sdesc(loA, Plan<R>::kSlot, 1024);
  const int nk = h / 16;
#pragma unroll
  for (int kk = 0; kk < kSB / 16; ++kk) {
    if (kk >= nk) break;
    const uint32_t p = kk >> 2, o = (kk & 3) * 2;
    const uint64_t aH = aT + kk * 128, bH = bR + p * vpan + o, bL = bR + (2 + p) * vpan + o;  // 2048 B per kk
    if (kk == 0) mma_f16(dJ, aH, bH, idT, first_t ? 0u : 1u);
    else mma_f16_acc(dJ, aH, bH, idT);
    mma_f16_acc(dJ, aH, bL, idT);
    if constexpr (LO) mma_f16_acc(dJ, aTl + kk * 128, bH, idT);
  }
}

// s_p for one port and all R columns: sum over its ends of w_in / Z_e plus the coupling currents.
// The loads wait on a busy HBM, so they come in few dependent steps: the port's gather record
// (loaded one port ahead by the caller) gives the wave rows and coefficients of its first four
// entries, whose rows are read two at a time; entries past the fourth (rare) follow the per-port
// lists.  The additions keep the order ends-then-coupling.
template <int R>
__device__ __forceinline__ void port_vector(const PortTCArgs& a, const int4 (&rec)[3], float (&v)[R]) {
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = 0.f;
  const int row[4] = {rec[0].x, rec[0].y, rec[0].z, rec[0].w};
  const float c[4] = {__int_as_float(rec[1].x), __int_as_float(rec[1].y), __int_as_float(rec[1].z),
                      __int_as_float(rec[1].w)};
#pragma unroll
  for (int j = 0; j < 4; j += 2) {
    if (row[j] < 0) break;  // entries are packed, absent ones at the end
    const bool two = row[j + 1] >= 0;
    const float4* w0 = reinterpret_cast<const float4*>(a.wprev + (size_t)row[j] * R);
    const float4* w1 = reinterpret_cast<const float4*>(a.wprev + (size_t)(two ? row[j + 1] : row[j]) * R);
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
      const float4 x = w0[q], y = w1[q];
      v[4 * q] += x.x * c[j];
      v[4 * q + 1] += x.y * c[j];
      v[4 * q + 2] += x.z * c[j];
      v[4 * q + 3] += x.w * c[j];
      if (two) {
        v[4 * q] += y.x * c[j + 1];
        v[4 * q + 1] += y.y * c[j + 1];
        v[4 * q + 2] += y.z * c[j + 1];
        v[4 * q + 3] += y.w * c[j + 1];
      }
    }
  }
  for (int e = rec[2].x; e < rec[2].y; ++e) {
    const float4* w = reinterpret_cast<const float4*>(a.wprev + (size_t)a.twin[e] * R);
    const float iz = a.invz[e];
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
      const float4 x = w[q];
      v[4 * q] += x.x * iz;
      v[4 * q + 1] += x.y * iz;
      v[4 * q + 2] += x.z * iz;
      v[4 * q + 3] += x.w * iz;
    }
  }
  for (int k = rec[2].z; k < rec[2].w; ++k) {
    const float yk = a.cpl.y[k];
    const float4* w = reinterpret_cast<const float4*>(a.wprev + (size_t)a.cpl.oth[k] * R);
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
      const float4 x = w[q];
      v[4 * q] += yk * x.x;
      v[4 * q + 1] += yk * x.y;
      v[4 * q + 2] += yk * x.z;
      v[4 * q + 3] += yk * x.w;
    }
  }
}

}  // namespace

int64_t port_f16_bytes(int nports) {
  if (nports <= 0) return 0;
  const int n4 = n_super(nports);
  const int64_t b = blk_off(nports, n4 - 1, 0) + (int64_t)n4 * sb_rows(nports, n4 - 1) * 512;
  return (b + 1023) & ~int64_t(1023);
}

int64_t port_f32_blocks(int nports) {
  const int64_t n4 = n_super(nports);
  return n4 * (n4 + 1) / 2;
}

size_t port_tc_smem_bytes(int R, bool) { return R == 16 ? Plan<16>::kAlloc : Plan<32>::kAlloc; }

// S_j columns cc = b * Rs + r from unit-source solves into FP32 128 x 128 row-major blocks of the
// lower block triangle (block (I, J) at s_off + I (I + 1) / 2 + J; diagonal blocks whole).
__global__ void k_gather_port_blocks(const PieceDesc* __restrict__ pieces, const int32_t* __restrict__ port_local,
                                     int Rs, int b0, const float* __restrict__ x0, int64_t stride,
                                     float* __restrict__ S32) {
  const PieceDesc pd = pieces[blockIdx.x];
  const int b = b0 + (int)blockIdx.y;
  const float* xc = x0 + (size_t)blockIdx.y * stride;
  for (int i = b * Rs / kSB * kSB * Rs + threadIdx.x; i < pd.nports * Rs; i += blockDim.x) {
    const int q = i / Rs, r = i % Rs;
    const int cc = b * Rs + r;
    if (cc >= pd.nports) continue;
    const int I = q / kSB, J = cc / kSB;
    if (J > I) continue;
    const int64_t blk = pd.s_off + (int64_t)I * (I + 1) / 2 + J;
    S32[blk * (kSB * kSB) + (q % kSB) * kSB + cc % kSB] =
        xc[((size_t)pd.copy_off + port_local[pd.port_off + q]) * Rs + r];
  }
}

// FP32 blocks -> fp16 hi / lo panels of the sweep's layout.  S_j is first balanced by its diagonal,
// S'_pq = S_pq / (g_p g_q) with g_p = sqrt(S_pp) (so S'_pp = 1 and |S'_pq| <= 1, S_j being SPD):
// across a coefficient jump the entries of S_j span many decades (a soft region's input impedances
// are orders of magnitude above a stiff one's), which one scale per subgraph would push below the
// fp16 range.  g_p goes to gscale[port]; sigma_j = 2^e >= max |S'| (about 1) to sig.
__global__ void k_port_blocks_to_f16(const PieceDesc* __restrict__ pieces, const float* __restrict__ S32,
                                     unsigned char* __restrict__ S16, float* __restrict__ sig,
                                     float* __restrict__ gscale) {
  const PieceDesc pd = pieces[blockIdx.x];
  const int P = pd.nports;
  if (P == 0) return;
  const int n4 = n_super(P);
  const float* src = S32 + pd.s_off * (kSB * kSB);
  __shared__ float g[kMaxSuper * kSB];  // 1 / g_p, zero-padded
  __shared__ float red[32];
  for (int p = threadIdx.x; p < n4 * kSB; p += blockDim.x) {
    float gi = 0.f;
    if (p < P) {
      const int I = p / kSB, r = p % kSB;
      const float d = src[((int64_t)I * (I + 1) / 2 + I) * (kSB * kSB) + r * kSB + r];
      const float gp = d > 0.f ? sqrtf(d) : 1.f;
      gscale[pd.port_off + p] = gp;
      gi = 1.f / gp;
    }
    g[p] = gi;
  }
  __syncthreads();
  float m = 0.f;
  for (int I = 0; I < n4; ++I)
    for (int J = 0; J <= I; ++J) {
      const float* blk = src + ((int64_t)I * (I + 1) / 2 + J) * (kSB * kSB);
      for (int k = threadIdx.x; k < kSB * kSB; k += blockDim.x)
        m = fmaxf(m, fabsf(blk[k] * g[I * kSB + k / kSB] * g[J * kSB + k % kSB]));
    }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float mm = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mm = fmaxf(mm, red[w]);
    int e = 0;
    if (mm > 0.f) frexpf(mm, &e);
    red[0] = ldexpf(1.f, e);  // power of two >= mm (1 for an all-zero matrix)
    sig[blockIdx.x] = red[0];
  }
  __syncthreads();
  const float inv = 1.f / red[0];
  unsigned char* dst = S16 + pd.h_off;
  for (int I = 0; I < n4; ++I) {
    const int h = sb_rows(P, I);
    for (int J = 0; J <= I; ++J) {
      const float* blk = src + ((int64_t)I * (I + 1) / 2 + J) * (kSB * kSB);
      unsigned char* o = dst + blk_off(P, I, J);
      const uint32_t panel = (uint32_t)h * 128;
      for (int k = threadIdx.x; k < h * kSB; k += blockDim.x) {
        const int row = k / kSB, col = k % kSB;
        const float x = blk[k] * g[I * kSB + row] * g[J * kSB + col] * inv;
        const __half hi = __float2half_rn(x);
        const __half lo = __float2half_rn(x - __half2float(hi));
        const uint32_t off = (uint32_t)(col / 64) * panel + swz16(row, col % 64);
        *reinterpret_cast<__half*>(o + off) = hi;
        *reinterpret_cast<__half*>(o + 2 * panel + off) = lo;
      }
    }
  }
}

// The port vectors of every subgraph as operand tiles: s = sum_e w_in[e] / Z_e plus the coupling
// currents, s' = G s, split per subgraph and column as s' / sigma_r = hi + lo (sigma_r the power of two
// at or above max |s'_r|).  A CTA takes sixteen columns of a subgraph: their incoming waves go to shared
// memory once (a row of 64 bytes per end, all ends' loads independent) and the sums, which read every
// wave about five times, are formed from there, a port's terms from one list (launch_port_entries); the
// maxima stay inside the CTA.  Four lanes share a port, each with four columns: a row's four 16-byte
// pieces come from four lanes of one load, so two ports' rows meet in a bank half the time (a port per
// lane: eight lanes, four bank groups).  Bound by the latency of its phases and the issue rate of the sums,
// one CTA of 32 warps per SM: 64^3 with 32 right-hand sides 19 us, 128^3 115 us (22 and 150 with a port
// per lane and its lists read from global memory).
constexpr int kVecTcThreads = 1024;
constexpr int kVecCols = 16;

template <int R>
__global__ void __launch_bounds__(kVecTcThreads, 1) k_port_vec_tc(const PortTCArgs a) {
  constexpr int kStep = kVecTcThreads / 4;                // ports per pass
  constexpr int kPass = kMaxSuper * kSB / kStep;          // passes, at most
  extern __shared__ __align__(16) float win[];            // [ends][kVecCols]
  __shared__ float red[kVecTcThreads / 32][kVecCols];
  __shared__ float inv[kVecCols];
  grid_dep_launch();
  const int piece = blockIdx.x, q0 = blockIdx.y * kVecCols;
  const PieceDesc pd = a.pieces[piece];
  const int Pn = pd.nports, np = n_super(Pn) * kSB;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, c4 = tid & 3, p0 = tid >> 2;
  // before the wait, what no sweep changes: the lists into the shared memory that the waves leave (read
  // in place where they do not fit), their bounds and the first twins into registers
  const int first = Pn > 0 ? a.ent_ptr[pd.port_off] : 0, nent = Pn > 0 ? a.ent_ptr[pd.port_off + Pn] - first : 0;
  int2* const list = reinterpret_cast<int2*>(win + (size_t)pd.nends * kVecCols);
  const bool staged = ((size_t)pd.nends * kVecCols + 2 * (size_t)nent) * sizeof(float) <= kVecTcSmemMax;
  if (staged)
    for (int k = tid; k < nent; k += kVecTcThreads)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(list + k)), "l"(a.ent + first + k));
  const int2* const ent = staged ? list : a.ent + first;
  int k0[kPass], k1[kPass];
#pragma unroll
  for (int i = 0; i < kPass; ++i) {
    const int p = i * kStep + p0;
    k0[i] = k1[i] = 0;
    if (p < Pn) {
      k0[i] = a.ent_ptr[pd.port_off + p] - first;
      k1[i] = a.ent_ptr[pd.port_off + p + 1] - first;
    }
  }
  constexpr int kTwins = 8;
  int tw[kTwins];
#pragma unroll
  for (int u = 0; u < kTwins; ++u) {
    const int i = tid + u * kVecTcThreads;
    tw[u] = i < 4 * pd.nends ? a.twin[pd.end_off + (i >> 2)] : 0;
  }
  grid_dep_wait();
  auto wave = [&](int i, int t) {  // 16 bytes of the incoming wave of end i / 4
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(win + 4 * i)),
                 "l"(a.wprev + (size_t)t * R + q0 + 4 * c4));
  };
#pragma unroll
  for (int u = 0; u < kTwins; ++u)
    if (tid + u * kVecTcThreads < 4 * pd.nends) wave(tid + u * kVecTcThreads, tw[u]);
  for (int i = tid + kTwins * kVecTcThreads; i < 4 * pd.nends; i += kVecTcThreads)
    wave(i, a.twin[pd.end_off + (i >> 2)]);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  float v[kPass][4];
#pragma unroll
  for (int i = 0; i < kPass; ++i) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int k = k0[i]; k < k1[i]; ++k) {
      const int2 en = ent[k];
      const float4 x = reinterpret_cast<const float4*>(win)[4 * en.x + c4];
      const float y = __int_as_float(en.y);
      s[0] += x.x * y, s[1] += x.y * y, s[2] += x.z * y, s[3] += x.w * y;
    }
    const int p = i * kStep + p0;
    const float gp = p < Pn ? a.gscale[pd.port_off + p] : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[i][q] = s[q] * gp;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < kPass; ++i) m = fmaxf(m, fabsf(v[i][q]));
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane < 4) red[warp][4 * lane + q] = m;
  }
  __syncthreads();
  if (warp < kVecCols / 2) {  // two columns per warp, sixteen lanes each
    const int c = 2 * warp + (lane >> 4);
    float m = fmaxf(red[lane & 15][c], red[16 + (lane & 15)][c]);
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((lane & 15) == 0) {
      int e = 0;
      if (m > 0.f && isfinite(m)) frexpf(m, &e);
      e = e < -120 ? -120 : e;
      inv[c] = ldexpf(1.f, -e);
      a.ssig[(size_t)piece * R + q0 + c] = ldexpf(1.f, e);  // power of two >= max |s_r|
    }
  }
  __syncthreads();
  // tile: [hi, ports 0-63][hi, 64-127][lo, 0-63][lo, 64-127] of R rows (columns of s) each.  The lanes of
  // ports p and p + 1 exchange half their columns, so that each writes both ports of two columns at once.
  unsigned char* const tiles = a.stiles + (size_t)a.tile_off[piece] * ((size_t)R * 512);
  const bool odd = lane & 4;
#pragma unroll
  for (int i = 0; i < kPass; ++i) {
    const int p = (i * kStep + p0) & ~1;
    if (p >= np) continue;  // the same for both lanes of a pair: np is a multiple of 128, and for the warp
    unsigned char* const panel = tiles + (size_t)(p / kSB) * R * 512 + (size_t)((p % kSB) / 64) * R * 128;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float got = __shfl_xor_sync(0xffffffffu, odd ? v[i][h] : v[i][2 + h], 4);
      const int c = 4 * c4 + (odd ? 2 : 0) + h;
      const float x0 = (odd ? got : v[i][h]) * inv[c], x1 = (odd ? v[i][2 + h] : got) * inv[c];
      const __half2 hi = __floats2half2_rn(x0, x1);
      const uint32_t off = swz16(q0 + c, p % 64);
      *reinterpret_cast<__half2*>(panel + off) = hi;
      *reinterpret_cast<__half2*>(panel + 2 * R * 128 + off) =
          __floats2half2_rn(x0 - __low2float(hi), x1 - __high2float(hi));
    }
  }
}

// The terms of a port's sum as one list, (place of the wave among the subgraph's ends, coefficient): its
// ends with 1 / Z_e, then its coupling entries (the incoming wave of end e' is the twin's, whose own twin
// is e').  The lists of the ports follow each other in port order.
__global__ void k_port_entries(const PieceDesc* __restrict__ pieces, const int32_t* __restrict__ port_end_ptr,
                               const int32_t* __restrict__ twin, const float* __restrict__ invz, CoupleRef<float> cpl,
                               int32_t* __restrict__ ent_ptr, int2* __restrict__ ent) {
  const PieceDesc pd = pieces[blockIdx.x];
  for (int q = pd.port_off + threadIdx.x; q < pd.port_off + pd.nports; q += blockDim.x) {
    const int e0 = port_end_ptr[q], e1 = port_end_ptr[q + 1];
    const int k0 = cpl.ptr ? cpl.ptr[q] : 0, k1 = cpl.ptr ? cpl.ptr[q + 1] : 0;
    int at = e0 + k0;
    ent_ptr[q] = at;
    ent_ptr[q + 1] = e1 + k1;  // the next port's thread writes the same
    for (int e = e0; e < e1; ++e) ent[at++] = make_int2(e - pd.end_off, __float_as_int(invz[e]));
    for (int k = k0; k < k1; ++k) ent[at++] = make_int2(twin[cpl.oth[k]] - pd.end_off, __float_as_int(cpl.y[k]));
  }
}

cudaError_t launch_port_entries(const PieceDesc* pieces, int npieces, const int32_t* port_end_ptr, const int32_t* twin,
                                const float* invz, CoupleRef<float> cpl, int32_t* ent_ptr, int2* ent, cudaStream_t st) {
  if (npieces <= 0) return cudaSuccess;
  k_port_entries<<<npieces, 256, 0, st>>>(pieces, port_end_ptr, twin, invz, cpl, ent_ptr, ent);
  return cudaGetLastError();
}

size_t port_vec_tc_smem_bytes(int max_ends) { return (size_t)std::max(1, max_ends) * kVecCols * sizeof(float); }

template <int R, bool LO, bool FUSED>
__global__ void __launch_bounds__(kTcThreads, 1) k_port_sweep_tc(const PortTCArgs a) {
  using P = Plan<R>;
  constexpr int NS = P::kSlots;
  static_assert(kVecThreads % (R / 4) == 0 && 32 % (R / 4) == 0, "column groups of the maxima pass");
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kOffFull);          // [kStg] stage landed
  uint64_t* empty = reinterpret_cast<uint64_t*>(sm + kOffEmpty);        // [kStg] MMAs done with the stage
  uint64_t* rowfull = reinterpret_cast<uint64_t*>(sm + kOffRowFull);    // [2] s_I tile landed
  uint64_t* rowempty = reinterpret_cast<uint64_t*>(sm + kOffRowEmpty);  // [2] MMAs done with the s_I tile
  uint64_t* sready = reinterpret_cast<uint64_t*>(sm + kOffSReady);      // FUSED: [2] scratch slot written
  uint64_t* slotfree = reinterpret_cast<uint64_t*>(sm + kOffSlotFree);  // FUSED: [2] epilogue of the slot's last item done
  uint64_t* rready = reinterpret_cast<uint64_t*>(sm + kOffRReady);      // [kMaxSuper] accumulator y_I complete
  uint64_t* rowread = reinterpret_cast<uint64_t*>(sm + kOffRowRead);    // [kMaxSuper] y_I read by the epilogue
  uint64_t* done = reinterpret_cast<uint64_t*>(sm + kOffDone);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kOffTslot);
  volatile int* flags = reinterpret_cast<volatile int*>(sm + kOffFlags);  // abort, epilogue stops, vector stop
  float (*ssig)[R] = reinterpret_cast<float (*)[R]>(sm + kOffSsig);        // sigma_r: [2] per scratch slot (FUSED), or per set
  float (*red)[R] = reinterpret_cast<float (*)[R]>(sm + kOffRed);          // FUSED: [kVecWarps][R]
  const uint32_t ring = base + P::kHead;
  const uint32_t row0 = base + P::kRow;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const TcItem* const items = a.items + a.cta_item[blockIdx.x];
  const int npc = a.cta_item[blockIdx.x + 1] - a.cta_item[blockIdx.x];  // items of this CTA
  const size_t slot_bytes = (size_t)a.n4max * P::kVec;  // FUSED
  unsigned char* scratch = a.scratch + (size_t)blockIdx.x * (2 * slot_bytes + (size_t)a.n4max * kSB * R * 4);
  float* stage32 = reinterpret_cast<float*>(scratch + 2 * slot_bytes);  // FP32 port vectors, ports x R

  if (tid == 0) {
    for (int i = 0; i < 5; ++i) flags[i] = 0;
    for (int s = 0; s < kStg; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&rowfull[s], 1);
      mbar_init(&rowempty[s], 1);
      mbar_init(&sready[s], 1);
      mbar_init(&slotfree[s], 1);
    }
    for (int s = 0; s < kMaxSuper; ++s) {
      mbar_init(&rready[s], 1);
      mbar_init(&rowread[s], kEpiWarps);
    }
    mbar_init(done, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  volatile int& abort_flag = flags[0];
  grid_dep_launch();

  if (warp == 0) {
    // ---- copies: super-rows in descending order; per block (I, J), J = I .. 0, its panels and
    // (off the diagonal) the s_J tile; the s_I tile of the next super-row a few blocks ahead.  Each piece goes out as soon as
    // its slots are free (the MMAs of the stage that last filled them are complete), so the next
    // blocks stream in while the current one is multiplied; the stage's full barrier counts the
    // bytes of every piece and completes after the last piece has been issued and has landed.
    // The blocks are read once per sweep: evict first.
    if (lane == 0) {
      uint64_t policy;
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
      // stage that last filled each slot, in shared memory: a local array would sit in a cache that
      // the ring leaves small, and this one thread issues every copy
      int* owner = reinterpret_cast<int*>(sm + kOffOwner);
      for (int i = 0; i < NS; ++i) owner[i] = -1;
      grid_dep_wait();  // the operand tiles
      asm volatile("fence.proxy.async.global;" ::: "memory");  // written by generic stores, read by bulk copies
      int gblk = 0, rel = -1;  // rel: stages 0 .. rel known released
      int64_t grow = 0, aslot = 0;
      auto release_upto = [&](int j) -> bool {
        while (rel < j) {
          ++rel;
          if (!mbar_wait_bounded(&empty[rel % kStg], (uint32_t)((rel / kStg) & 1), a.wait_limit)) return false;
        }
        return true;
      };
      for (int k = 0; k < npc && !abort_flag; ++k) {
        const TcItem it = items[k];
        const PieceDesc pd = a.pieces[it.piece];
        const int Pn = pd.nports, n4 = it.hi + 1;
        if (FUSED && !mbar_wait_bounded(&sready[k & 1], (uint32_t)((k >> 1) & 1), a.wait_limit)) {
          abort_flag = 1;
          break;
        }
        const unsigned char* slot =
            FUSED ? scratch + (size_t)(k & 1) * slot_bytes : a.stiles + (size_t)a.tile_off[it.piece] * P::kVec;
        const unsigned char* Sp = a.S16 + pd.h_off;
        // s_I tile of super-row I into the row buffer grow & 1, once the MMAs of the row two
        // before it (same buffer) are done
        auto issue_row = [&](int I) -> bool {
          const int rb = (int)(grow & 1);
          if (grow >= 2 && !mbar_wait_bounded(&rowempty[rb], (uint32_t)(((grow >> 1) - 1) & 1), a.wait_limit))
            return false;
          mbar_arrive_expect_tx(&rowfull[rb], P::kVec);
          bulk_g2s(row0 + rb * P::kVec, slot + (size_t)I * P::kVec, P::kVec, &rowfull[rb]);
          ++grow;
          return true;
        };
        if (n4 > 0 && !issue_row(n4 - 1)) {
          abort_flag = 1;
          break;
        }
        for (int I = n4 - 1; I >= it.lo && !abort_flag; --I) {
          const int h = sb_rows(Pn, I);
          const uint32_t pbytes = (uint32_t)h * 128;  // one panel
          for (int J = I; J >= 0; --J) {
            const int st = (int)(gblk % kStg);
            // full[st] and empty[st] were last used by stage gblk - kStg
            bool ok = release_upto(gblk - kStg);
            const StagePos ps = place_stage<NS>(aslot, LO, J < I);
            const unsigned char* blk = Sp + blk_off(Pn, I, J);
            // one pair: two panels of the block into two adjacent slots
            auto pair = [&](int s0, const unsigned char* src) {
              ok = ok && release_upto(owner[s0] > owner[s0 + 1] ? owner[s0] : owner[s0 + 1]);
              if (!ok) return;
              owner[s0] = owner[s0 + 1] = gblk;
              const uint32_t dst = ring + (uint32_t)s0 * P::kSlot;
              mbar_expect_tx(&full[st], 2 * pbytes);
              if (h == kSB) {
                bulk_g2s_hint(dst, src, 2 * pbytes, &full[st], policy);
              } else {
                bulk_g2s_hint(dst, src, pbytes, &full[st], policy);
                bulk_g2s_hint(dst + P::kSlot, src + pbytes, pbytes, &full[st], policy);
              }
            };
            pair(ps.hi, blk);
            if (LO) pair(ps.lo, blk + 2 * pbytes);
            if (ps.s >= 0) {
              ok = ok && release_upto(owner[ps.s]);
              if (ok) {
                owner[ps.s] = gblk;
                mbar_expect_tx(&full[st], P::kVec);
                bulk_g2s(ring + (uint32_t)ps.s * P::kSlot, slot + (size_t)J * P::kVec, P::kVec, &full[st]);
              }
            }
            mbar_arrive(&full[st]);  // completes once what was issued has landed
            ++gblk;
            // the next row's tile goes out a few blocks ahead: by the third block of this row the
            // MMAs have finished the row before it, whose buffer it takes
            if (ok && I > it.lo && J == (I >= 2 ? I - 2 : 0)) ok = issue_row(I - 1);
            if (!ok) {
              abort_flag = 1;
              break;
            }
          }
        }
      }
      // copies still in flight must land before the shared memory can go away
      for (int g = (gblk > kStg ? gblk - kStg : 0); g < gblk; ++g)
        mbar_wait_bounded(&full[g % kStg], (uint32_t)((g / kStg) & 1), kDrainPolls);
      for (int64_t g = (grow > 2 ? grow - 2 : 0); g < grow; ++g)
        mbar_wait_bounded(&rowfull[g & 1], (uint32_t)((g >> 1) & 1), kDrainPolls);
    }
  } else if (warp == 1) {
    // ---- MMA issuer.  In descending row order y_I is complete once row I is done (the rows
    // below only add to y_J, J < I), so its epilogue runs while the MMAs go on.  The first row
    // processed (n4 - 1) initialises every accumulator: y_{n4-1} through the direct product of the
    // diagonal block, every other y_J through the transposed product of block (n4 - 1, J).  Before
    // it overwrites y_J it waits until the epilogue has read y_J of the subgraph before (rowread);
    // that subgraph's epilogue reads its rows in the same descending order, so the MMAs of the
    // next subgraph start while the last rows of this one are still being written out.
    if (lane == 0) {
      int64_t gblk = 0, grow = 0, aslot = 0;
      uint32_t pend = 0, wpar = 0;  // rows handed to the epilogue and not yet waited for; parity of the next wait
      for (int k = 0; k < npc && !abort_flag; ++k) {
        const TcItem it = items[k];
        const int Pn = a.pieces[it.piece].nports, n4 = it.hi + 1;
        for (int I = n4 - 1; I >= it.lo && !abort_flag; --I) {
          const int rb = (int)(grow & 1);
          if (!mbar_wait_bounded(&rowfull[rb], (uint32_t)((grow >> 1) & 1), a.wait_limit)) {
            abort_flag = 1;
            break;
          }
          const uint32_t si = row0 + rb * P::kVec;
          const int h = sb_rows(Pn, I);
          const bool top = (I == n4 - 1);
          for (int J = I; J >= 0; --J) {
            const int st = (int)(gblk % kStg);
            const StagePos ps = place_stage<NS>(aslot, LO, J < I);
            if (top && ((pend >> J) & 1u)) {  // first write into y_J (y_I on the diagonal) this subgraph
              if (!mbar_wait_bounded(&rowread[J], (wpar >> J) & 1u, a.wait_limit)) {
                abort_flag = 1;
                break;
              }
              wpar ^= 1u << J;
              pend &= ~(1u << J);
            }
            if (!mbar_wait_bounded(&full[st], (uint32_t)((gblk / kStg) & 1), a.wait_limit)) {
              abort_flag = 1;
              break;
            }
            tc_fence_after();
            const uint32_t hiA = ring + (uint32_t)ps.hi * P::kSlot;
            const uint32_t loA = LO ? ring + (uint32_t)ps.lo * P::kSlot : hiA;
            const uint32_t bv = (J == I) ? si : ring + (uint32_t)ps.s * P::kSlot;
            const uint32_t dI = tmem + (uint32_t)(I * R), dJ = tmem + (uint32_t)(J * R);
            block_mmas<R, LO>(hiA, loA, bv, si, h, dI, dJ, top && J == I, top, J < I);
            mma_commit(&empty[st]);
            ++gblk;
          }
          mma_commit(&rowempty[rb]);
          mma_commit(&rready[I]);  // y_I is final (of this item)
          ++grow;
        }
        for (int J = it.lo - 1; J >= 0; --J) mma_commit(&rready[J]);
        pend |= (n4 >= 32 ? ~0u : (1u << n4) - 1u);
      }
      mma_commit(done);  // arrives once every MMA issued above has completed
    }
  } else if (!FUSED || warp < 2 + kEpiWarps) {
    // ---- epilogue warps (a set: one per tensor-memory lane quadrant): u = u_base + sigma_j sigma_r y_I,
    // w_out[e] = 2 u - w_in[e], super-row by super-row as the MMA issuer completes them, super-row I by
    // set I mod kSets (a row's loads depend on each other in three steps; other sets' rows go on
    // meanwhile).  rready[I] completes once per item that has a super-row I, so its phases are counted
    // per barrier; one set waits for all of them, so none is missed or taken for the next.  A warp releases y_I (rowread[I]) as soon as its tcgen05.ld has completed.
    constexpr int kSets = FUSED ? 1 : kEpiSets;
    const int set = FUSED ? 0 : (warp - 2) / kEpiWarps, q = warp & 3;
    const int lead = 64 + 32 * kEpiWarps * set;  // the set's first thread
    uint32_t uses = 0;  // lead: parity of the next phase of each row barrier, one bit per super-row
    bool stop = false;
    grid_dep_wait();  // the waves, sigma_r
    for (int k = 0; k < npc && !stop; ++k) {
      const TcItem it = items[k];
      const PieceDesc pd = a.pieces[it.piece];
      const int Pn = pd.nports, n4 = it.hi + 1;
      const float sj = a.sig_s[it.piece];
      float* const sg = ssig[FUSED ? (k & 1) : set];
      if constexpr (FUSED) {
        // sready[k & 1] also orders the sigma_r written with the item's port vectors
        if (tid == lead)
          flags[1] = mbar_wait_bounded(&sready[k & 1], (uint32_t)((k >> 1) & 1), a.wait_limit) ? 0 : 1;
        epi_sync(set);
        stop = flags[1] != 0;
        epi_sync(set);
      } else {
        epi_sync(set);  // the set is through with the item before
        if (tid - lead < R) sg[tid - lead] = __ldcg(a.ssig + (size_t)it.piece * R + tid - lead);
      }
      for (int I = n4 - 1; I >= 0 && !stop; --I) {
        if (I % kSets != set) continue;
        // the set decides together: one lane waits, the named barrier publishes the outcome
        if (tid == lead) flags[1 + set] = mbar_wait_bounded(&rready[I], (uses >> I) & 1u, a.wait_limit) ? 0 : 1;
        uses ^= 1u << I;
        epi_sync(set);
        stop = flags[1 + set] != 0;
        epi_sync(set);
        if (stop) break;
        tc_fence_after();
        uint32_t v[R];
        tmem_ld<R>(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(I * R), v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowread[I]);
        const int p = I * kSB + 32 * q + lane;
        if (p < Pn) {
          const int port = pd.port_off + p;
          const float gs = sj * a.gscale[port];  // y = D^-1 (sigma_j S'') (sigma_r s'')
#pragma unroll
          for (int c = 0; c < R; ++c) v[c] = __float_as_uint(gs * sg[c] * __uint_as_float(v[c]));
          if (it.part >= 0) {
            // part of a subgraph: this item's share of y
            uint4* o = reinterpret_cast<uint4*>(a.part + it.part + (size_t)p * R);
#pragma unroll
            for (int k4 = 0; k4 < R / 4; ++k4) o[k4] = make_uint4(v[4 * k4], v[4 * k4 + 1], v[4 * k4 + 2], v[4 * k4 + 3]);
          } else {
            const float4* ub = reinterpret_cast<const float4*>(a.ubase + (size_t)port * R);
            const int e0 = a.port_end_ptr[port], e1 = a.port_end_ptr[port + 1];
#pragma unroll
            for (int k4 = 0; k4 < R / 4; ++k4) {
              const float4 b4 = __ldg(ub + k4);
              v[4 * k4] = __float_as_uint(b4.x + __uint_as_float(v[4 * k4]));
              v[4 * k4 + 1] = __float_as_uint(b4.y + __uint_as_float(v[4 * k4 + 1]));
              v[4 * k4 + 2] = __float_as_uint(b4.z + __uint_as_float(v[4 * k4 + 2]));
              v[4 * k4 + 3] = __float_as_uint(b4.w + __uint_as_float(v[4 * k4 + 3]));
            }
            for (int e = e0; e < e1; ++e) {
              const float4* wi = reinterpret_cast<const float4*>(a.wprev + (size_t)a.twin[e] * R);
              float4* wo = reinterpret_cast<float4*>(a.wnext + (size_t)e * R);
#pragma unroll
              for (int k4 = 0; k4 < R / 4; ++k4) {
                const float4 w = __ldg(wi + k4);
                wo[k4] = make_float4(2.f * __uint_as_float(v[4 * k4]) - w.x, 2.f * __uint_as_float(v[4 * k4 + 1]) - w.y,
                                     2.f * __uint_as_float(v[4 * k4 + 2]) - w.z,
                                     2.f * __uint_as_float(v[4 * k4 + 3]) - w.w);
              }
            }
          }
        }
        __syncwarp();
      }
      if (stop) {
        if (tid == lead) abort_flag = 1;
        break;
      }
      if constexpr (FUSED) {
        epi_sync(set);
        if (tid == lead) mbar_arrive(&slotfree[k & 1]);
      }
    }
  } else if constexpr (FUSED) {
    // ---- vector warps: the port vectors s of subgraph k, one gather pass (FP32 values to a
    // staging area and the column maxima), then the fp16 split into the scratch slot k & 1.  Slot
    // and sigma_r of subgraph k are free again once the epilogue of subgraph k - 2 is done
    // (slotfree[k & 1] completes once per subgraph of that slot).
    const int vt = tid - 32 * (2 + kEpiWarps);
    const int vw = vt >> 5;
    grid_dep_wait();  // the waves
    for (int k = 0; k < npc; ++k) {
      if (k >= 2) {
        if (vt == 0) flags[4] = mbar_wait_bounded(&slotfree[k & 1], (uint32_t)(((k >> 1) - 1) & 1), a.wait_limit) ? 0 : 1;
        vec_sync();
        const bool stop = flags[4] != 0;
        vec_sync();
        if (stop) {
          if (vt == 0) abort_flag = 1;
          break;
        }
      }
      const PieceDesc pd = a.pieces[items[k].piece];
      const int np = (items[k].hi + 1) * kSB;         // rows that the item's products read
      const int Pn = pd.nports < np ? pd.nports : np;
      // gather: s' = D^-1 s per port into the FP32 staging area; the next port's record is
      // loaded before this port's wave rows
      int4 rec[3];
      if (vt < Pn)
#pragma unroll
        for (int i = 0; i < 3; ++i) rec[i] = a.prec[3 * (size_t)(pd.port_off + vt) + i];
      for (int p = vt; p < Pn; p += kVecThreads) {
        int4 nrec[3];
        if (p + kVecThreads < Pn)
#pragma unroll
          for (int i = 0; i < 3; ++i) nrec[i] = a.prec[3 * (size_t)(pd.port_off + p + kVecThreads) + i];
        float v[R];
        port_vector<R>(a, rec, v);
        const float gp = a.gscale[pd.port_off + p];  // s' = D^-1 s, D = diag(1 / g)
        float4* o = reinterpret_cast<float4*>(stage32 + (size_t)p * R);
#pragma unroll
        for (int k4 = 0; k4 < R / 4; ++k4)
          o[k4] = make_float4(v[4 * k4] * gp, v[4 * k4 + 1] * gp, v[4 * k4 + 2] * gp, v[4 * k4 + 3] * gp);
#pragma unroll
        for (int i = 0; i < 3; ++i) rec[i] = nrec[i];
      }
      vec_sync();
      // column maxima in a coalesced pass over the staged values: the thread stride is a multiple
      // of R / 4, so every float4 a thread reads holds the same four columns
      {
        float4 m4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4* s4 = reinterpret_cast<const float4*>(stage32);
        for (int i = vt; i < Pn * (R / 4); i += kVecThreads) {
          const float4 x = s4[i];
          m4 = make_float4(fmaxf(m4.x, fabsf(x.x)), fmaxf(m4.y, fabsf(x.y)), fmaxf(m4.z, fabsf(x.z)),
                           fmaxf(m4.w, fabsf(x.w)));
        }
#pragma unroll
        for (int o = R / 4; o < 32; o <<= 1) {
          m4.x = fmaxf(m4.x, __shfl_xor_sync(0xffffffffu, m4.x, o));
          m4.y = fmaxf(m4.y, __shfl_xor_sync(0xffffffffu, m4.y, o));
          m4.z = fmaxf(m4.z, __shfl_xor_sync(0xffffffffu, m4.z, o));
          m4.w = fmaxf(m4.w, __shfl_xor_sync(0xffffffffu, m4.w, o));
        }
        if (lane < R / 4) {
          red[vw][4 * lane] = m4.x;
          red[vw][4 * lane + 1] = m4.y;
          red[vw][4 * lane + 2] = m4.z;
          red[vw][4 * lane + 3] = m4.w;
        }
      }
      vec_sync();
      if (vt < R) {
        float m = 0.f;
        for (int w = 0; w < kVecWarps; ++w) m = fmaxf(m, red[w][vt]);
        int e = 0;
        if (m > 0.f) frexpf(m, &e);
        ssig[k & 1][vt] = ldexpf(1.f, e);  // power of two >= max |s_r|
      }
      vec_sync();
      unsigned char* slot = scratch + (size_t)(k & 1) * slot_bytes;
      for (int p = vt; p < np; p += kVecThreads) {
        unsigned char* tile = slot + (size_t)(p / kSB) * P::kVec;
        const int c = p % kSB;
        const uint32_t pn = (uint32_t)(c / 64) * R * 128;
        const float4* src = reinterpret_cast<const float4*>(stage32 + (size_t)p * R);
#pragma unroll
        for (int k4 = 0; k4 < R / 4; ++k4) {
          const float4 x4 = (p < Pn) ? src[k4] : make_float4(0.f, 0.f, 0.f, 0.f);
          const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 4 * k4 + i;
            const float x = xs[i] / ssig[k & 1][r];
            const __half hi = __float2half_rn(x);
            const __half lo = __float2half_rn(x - __half2float(hi));
            const uint32_t off = pn + swz16(r, c % 64);
            *reinterpret_cast<__half*>(tile + off) = hi;
            *reinterpret_cast<__half*>(tile + 2 * R * 128 + off) = lo;
          }
        }
      }
      // the bulk copies (async proxy) read what these generic stores wrote
      asm volatile("fence.proxy.async.global;" ::: "memory");
      vec_sync();
      if (vt == 0) mbar_arrive(&sready[k & 1]);
    }
  }
  __syncthreads();
  const bool ok = mbar_wait_bounded(done, 0, kDrainPolls) && !abort_flag;
  if (!ok && tid == 0) atomicExch(a.status, kStatusTimeout);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
  }
}

// Waves of the subgraphs whose rows several items added to: u = u_base + the items' shares in their
// order, w_out[e] = 2u - w_in[e]; thread = (port, four columns).
template <int R>
__global__ void __launch_bounds__(256) k_port_finish_tc(const PortTCArgs a) {
  grid_dep_launch();
  const TcSplit sp = a.splits[blockIdx.y];
  const PieceDesc pd = a.pieces[sp.piece];
  grid_dep_wait();
  const int i = blockIdx.x * 256 + threadIdx.x;
  const int p = i / (R / 4), k4 = i % (R / 4);
  if (p >= pd.nports) return;
  const int port = pd.port_off + p, I = p / kSB;
  const int e0 = a.port_end_ptr[port], e1 = a.port_end_ptr[port + 1];
  float4 u = __ldcg(reinterpret_cast<const float4*>(a.ubase + (size_t)port * R) + k4);
  float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int q = 0; q < kTcMaxSplit; ++q) {
    if (q < sp.nitems && sp.hi[q] >= I) {
      const float4 x = __ldcg(reinterpret_cast<const float4*>(a.part + sp.part + ((size_t)q * pd.nports + p) * R) + k4);
      y.x += x.x, y.y += x.y, y.z += x.z, y.w += x.w;
    }
  }
  u.x += y.x, u.y += y.y, u.z += y.z, u.w += y.w;
  for (int e = e0; e < e1; ++e) {
    const float4 w = __ldcg(reinterpret_cast<const float4*>(a.wprev + (size_t)a.twin[e] * R) + k4);
    reinterpret_cast<float4*>(a.wnext + (size_t)e * R)[k4] =
        make_float4(2.f * u.x - w.x, 2.f * u.y - w.y, 2.f * u.z - w.z, 2.f * u.w - w.w);
  }
}

// Items of the subgraphs for `ctas` CTAs.  A subgraph of more than 1.1 CTA shares (in blocks) is cut
// between super-rows into up to kTcMaxSplit items of about a share each.
TcPlan tc_plan(const PieceDesc* pd, int npieces, int R, int ctas) {
  constexpr double kItemCost = 3.0;  // what an item costs besides its blocks, in blocks
  TcPlan pl;
  double total = 0;
  for (int j = 0; j < npieces; ++j) {
    const int n4 = n_super(pd[j].nports);
    total += n4 * (n4 + 1) / 2 + (n4 > 0 ? kItemCost : 0.0);
  }
  for (int j = 0; j < npieces; ++j) {
    pl.tile_off.push_back((int32_t)pl.tiles);
    pl.tiles += n_super(pd[j].nports);
  }
  const double share = total / std::max(1, ctas);
  std::vector<std::pair<double, TcItem>> items;
  for (int j = 0; j < npieces; ++j) {
    const int n4 = n_super(pd[j].nports);
    if (n4 == 0) continue;
    const int blocks = n4 * (n4 + 1) / 2;
    int c = 1;
    if (blocks + kItemCost > 1.1 * share)
      c = std::min({kTcMaxSplit, n4, (int)std::ceil(blocks / std::max(1.0, share - kItemCost))});
    TcSplit sp{};
    sp.piece = j;
    sp.part = pl.part_elems;
    int row = n4 - 1, left = blocks;
    for (int q = 0; q < c && row >= 0; ++q) {
      // rows until the item has its share of what is left (the last one takes the rest)
      const double want = (double)left / (c - q);
      int lo = row, got = row + 1;
      while (lo > 0 && (q == c - 1 || got + lo / 2.0 < want)) got += lo--;
      TcItem it{};
      it.piece = j;
      it.hi = row;
      it.lo = lo;
      it.part = c > 1 ? sp.part + (int64_t)q * pd[j].nports * R : -1;
      items.push_back({got + kItemCost, it});
      sp.hi[q] = row;
      sp.nitems = q + 1;
      left -= got;
      row = lo - 1;
    }
    if (sp.nitems == 1) items.back().second.part = -1;
    if (sp.nitems > 1) {
      pl.splits.push_back(sp);
      pl.part_elems += (int64_t)sp.nitems * pd[j].nports * R;
      pl.max_split_ports = std::max(pl.max_split_ports, (int)pd[j].nports);
    }
  }
  std::stable_sort(items.begin(), items.end(), [](const auto& x, const auto& y) { return x.first > y.first; });
  const int n = std::max(1, std::min<int>(ctas, (int)items.size()));
  std::vector<std::vector<TcItem>> of(n);
  std::vector<std::pair<double, int>> heap;  // least loaded CTA on top
  for (int c = 0; c < n; ++c) heap.push_back({0.0, c});
  auto later = [](const std::pair<double, int>& x, const std::pair<double, int>& y) { return x > y; };
  std::make_heap(heap.begin(), heap.end(), later);
  for (const auto& it : items) {
    std::pop_heap(heap.begin(), heap.end(), later);
    of[heap.back().second].push_back(it.second);
    heap.back().first += it.first;
    std::push_heap(heap.begin(), heap.end(), later);
  }
  pl.cta_item.push_back(0);
  for (const auto& v : of) {
    pl.items.insert(pl.items.end(), v.begin(), v.end());
    pl.cta_item.push_back((int32_t)pl.items.size());
  }
  return pl;
}

// Gather record of port q: the wave rows and coefficients of its first four entries in the order
// the sweep adds them (ends e0 .. e1 - 1 with 1 / Z_e, then coupling entries k0 .. k1 - 1 with y;
// row -1 and coefficient 0 past the last one), and where the remaining entries resume.
__global__ void k_port_records(int nports, const int32_t* __restrict__ port_end_ptr, const int32_t* __restrict__ twin,
                               const float* __restrict__ invz, CoupleRef<float> cpl, int4* __restrict__ rec) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nports) return;
  const int e0 = port_end_ptr[q], e1 = port_end_ptr[q + 1];
  const int k0 = cpl.ptr ? cpl.ptr[q] : 0, k1 = cpl.ptr ? cpl.ptr[q + 1] : 0;
  int row[4] = {-1, -1, -1, -1};
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  int n = 0, e = e0, k = k0;
  for (; e < e1 && n < 4; ++e, ++n) {
    row[n] = twin[e];
    c[n] = invz[e];
  }
  for (; e == e1 && k < k1 && n < 4; ++k, ++n) {
    row[n] = cpl.oth[k];
    c[n] = cpl.y[k];
  }
  rec[3 * (size_t)q] = make_int4(row[0], row[1], row[2], row[3]);
  rec[3 * (size_t)q + 1] = make_int4(__float_as_int(c[0]), __float_as_int(c[1]), __float_as_int(c[2]), __float_as_int(c[3]));
  rec[3 * (size_t)q + 2] = make_int4(e, e1, k, k1);
}

cudaError_t launch_port_records(int nports, const int32_t* port_end_ptr, const int32_t* twin, const float* invz,
                                CoupleRef<float> cpl, int4* rec, cudaStream_t st) {
  if (nports <= 0) return cudaSuccess;
  k_port_records<<<(nports + 255) / 256, 256, 0, st>>>(nports, port_end_ptr, twin, invz, cpl, rec);
  return cudaGetLastError();
}

template <int R>
static const void* tc_kernel(bool lo, bool fused) {
  return lo ? (fused ? (const void*)k_port_sweep_tc<R, true, true> : (const void*)k_port_sweep_tc<R, true, false>)
            : (fused ? (const void*)k_port_sweep_tc<R, false, true> : (const void*)k_port_sweep_tc<R, false, false>);
}

cudaError_t port_tc_configure(int R) {
  if (R != 16 && R != 32) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
    const void* k = R == 16 ? tc_kernel<16>(i & 1, i & 2) : tc_kernel<32>(i & 1, i & 2);
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)port_tc_smem_bytes(R, true));
  }
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(R == 16 ? (const void*)k_port_vec_tc<16> : (const void*)k_port_vec_tc<32>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVecTcSmemMax);
  return e;
}

cudaError_t launch_port_sweep_tc(const PortTCArgs& a, int R, bool lo, int npieces, int grid, int nsplits,
                                 int max_split_ports, cudaStream_t st) {
  if (grid <= 0) return cudaSuccess;
  if (R != 16 && R != 32) return cudaErrorInvalidValue;
  PortTCArgs args = a;
  void* av[] = {&args};
  const bool fused = a.stiles == nullptr;
  // early: the kernel's CTAs may start while the launch before still runs; they wait for its results
  // themselves, and read them past the L1 cache.  Not the sweep proper: its epilogue reads a row of
  // waves per lane, in 16-byte pieces that need the L1 cache.
  auto launch = [&](const void* k, dim3 g, int threads, size_t smem, bool early) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelExC(&cfg, k, av);
  };
  cudaError_t e = cudaSuccess;
  if (!fused)
    e = launch(R == 16 ? (const void*)k_port_vec_tc<16> : (const void*)k_port_vec_tc<32>, dim3(npieces, R / kVecCols),
               kVecTcThreads, kVecTcSmemMax, true);
  if (e != cudaSuccess) return e;
  const void* k = R == 16 ? tc_kernel<16>(lo, fused) : tc_kernel<32>(lo, fused);
  e = launch(k, dim3(grid), kTcThreads, port_tc_smem_bytes(R, lo), false);
  if (e != cudaSuccess || nsplits == 0) return e;
  return launch(R == 16 ? (const void*)k_port_finish_tc<16> : (const void*)k_port_finish_tc<32>,
                dim3((max_split_ports * (R / 4) + 255) / 256, nsplits), 256, 0, true);
}

cudaError_t launch_gather_port_blocks(const PieceDesc* pieces, int npieces, const int32_t* port_local, int Rs, int b,
                                      const float* xc, float* S32, cudaStream_t st, int batches, int64_t stride) {
  if (npieces <= 0) return cudaSuccess;
  k_gather_port_blocks<<<dim3(npieces, batches), 256, 0, st>>>(pieces, port_local, Rs, b, xc, stride, S32);
  return cudaGetLastError();
}

cudaError_t launch_port_blocks_to_f16(const PieceDesc* pieces, int npieces, const float* S32, unsigned char* S16,
                                      float* sig, float* gscale, cudaStream_t st) {
  if (npieces <= 0) return cudaSuccess;
  k_port_blocks_to_f16<<<npieces, 256, 0, st>>>(pieces, S32, S16, sig, gscale);
  return cudaGetLastError();
}

}  // namespace vtm
