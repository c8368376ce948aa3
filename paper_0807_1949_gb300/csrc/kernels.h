// Host-callable launchers of the libvtm CUDA kernels (internal).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <cuda_fp16.h>

#include <vector>

#include "device.cuh"

namespace vtm {

// Lets a kernel take all the dynamic shared memory that an SM has for it.  The limit belongs to the kernel and
// not to a solver: set to what the solver at hand needs, the next one's setup would lower it for solvers
// that are still in use, whose launches would then be refused.
cudaError_t allow_all_smem(const void* kernel);

// Arguments of one VTM sweep (Table 1 steps 3-5) over a set of subgraphs.  TF: factor and
// substitution type; TV: type of the sources, local solutions, waves and 1/Z in global memory.
template <typename TF, typename TV = TF>
struct SweepArgs {
  const PieceDesc* pieces;     // the subgraphs of this launch, one CTA each
  const TF* factor;            // band factors (see device.cuh)
  const TF* factor_u;          // transposed band (rows of U = L^T, left-aligned), R <= 8 kernel
  const TV* bt;                // b̃: copies x R, R contiguous
  TV* xc;                      // local solutions: copies x R (written when write_x)
  const TV* wprev;             // outgoing waves of the previous sweep: ends x R
  TV* wnext;                   // outgoing waves of this sweep
  const int32_t* port_local;   // per port: local row of the port copy
  const int32_t* port_end_ptr; // per port: first (sorted) end; nports_total + 1 entries
  const int32_t* twin;         // per end: the twin end of the same line
  const TV* invz;              // per end: 1 / Z_e
  int* status;                 // kernel status word (0 = ok)
  int write_x;
  int stages;                  // staged slabs in flight (>= 2)
  int slot_elems;              // ring slot stride in elements (kNB * max Wp)
  int ys_elems;                // (2 (max Wp - 1) + max n_pad) * R
  int win_elems;               // (max ends per piece) * R
  long wait_limit;             // bounded mbarrier polls before a timeout is recorded
  int withhold;                // testing: slab index whose copy is never issued (-1 = none)
  int cap;                     // wide kernel: window rows (power of two >= max Wp - 1 + kNB)
  TF* yspill;                  // wide kernel: forward result y in factor precision, n_pad x R per
                               // piece at row_off (nullptr: y goes through xc, TF == TV)
  CoupleRef<TV> cpl;           // coupled lines: per-port coupling lists (cpl.ptr == nullptr: none)
  const unsigned char* wt;     // tensor-core factor of sweep_wide_tc.cu (nullptr: not built)
  // Unit sources (all kernels but the pipelined one) at the ports instead of b̃ and waves (the columns of S_j): CTA (j, y)
  // solves for the R ports from (unit_b0 + y) R on, for the rows from port
  // floor((unit_b0 + y) R / unit_gran) unit_gran on, into xc + y unit_stride; no waves are read or written.
  int unit = 0;
  int unit_b0 = 0;
  int unit_gran = 1;
  int64_t unit_stride = 0;
};

size_t sweep_smem_bytes(size_t elem, int R, int stages, int slot_elems, int ys_elems, int win_elems);
template <typename TF, typename TV>
cudaError_t sweep_configure(int R);
template <typename TF, typename TV>
cudaError_t sweep_occupancy(int R, size_t smem, int* ctas_per_sm);
template <typename TF, typename TV>
cudaError_t launch_sweep(const SweepArgs<TF, TV>& a, int R, int npieces, size_t smem, cudaStream_t st, int batches = 1);

// Pipelined variant: chain warps finish block k while the others prepare block k+1.
constexpr size_t kPipeSmemMax = 226 * 1024;  // dynamic shared memory the kernel may take
size_t sweep_pipe_smem_bytes(size_t elem, int R, int stages, int slot_elems, int ys_elems);
template <typename T>
cudaError_t sweep_pipe_configure(int R);
template <typename T>
cudaError_t sweep_pipe_occupancy(int R, size_t smem, int* ctas_per_sm);
template <typename T>
cudaError_t launch_sweep_pipe(const SweepArgs<T, T>& a, int R, int npieces, size_t smem, cudaStream_t st);

// Multi-RHS sweep with the band products on the tensor cores (R = 16, 32; FP32 solvers): the factor
// of each subgraph, balanced and split into fp16 hi / lo panels of 128-row groups, built once from
// the FP32 band factor (sweep_wide_tc.cu).  Half-bandwidths up to 128 kWideTcMaxTiles.
constexpr int kWideTcMaxTiles = 3;
int64_t wide_tc_bytes(int n, int w);
int64_t wide_tc_zero_bytes();  // the zero panel the factor buffer starts with
bool wide_tc_fits(int w);
int wide_tc_groups(int n);
size_t wide_tc_smem_bytes(int R);
cudaError_t wide_tc_configure(int R);
cudaError_t launch_wide_tc_factor(const PieceDesc* pieces, int npieces, int max_groups, const float* band,
                                  unsigned char* wt, cudaStream_t st);
cudaError_t launch_sweep_wide_tc(const SweepArgs<float, float>& a, int R, int npieces, cudaStream_t st,
                                 int batches = 1);

// Wide variant (R = 16, 32): vectors spill to xc, a circular window of 512 rows stays in shared memory.
size_t sweep_wide_smem_bytes(size_t elem, int R, int stages, int slot_elems, int cap);
template <typename TF, typename TV>
cudaError_t sweep_wide_configure(int R);
template <typename TF, typename TV>
cudaError_t launch_sweep_wide(const SweepArgs<TF, TV>& a, int R, int npieces, size_t smem, cudaStream_t st,
                              int batches = 1);
// One segment of a port sweep (port.cu): the tiles (I0, J0) .. (I1, J1) of a subgraph's lower block
// triangle, row by row.
struct PortSeg {
  int64_t s_off;   // the subgraph's first tile
  int32_t piece;   // index into PortArgs::pieces
  int32_t I0, J0, I1, J1;
  int32_t first;   // index of the subgraph's first segment (its segments are consecutive)
  int32_t nseg;    // segments of the subgraph
  int64_t part;    // nseg > 1: element offset of the subgraph's partial vectors y, one per segment
};

// Order of the entries inside a tile of S_j (port.cu).
enum { kPortPatch8x4 = 0, kPortPatch4x8 = 1, kPortFragments = 2 };

// Shared-memory shape of the port sweep kernel, and which kernel.
struct PortShape {
  int vec_elems;   // elements of a padded port vector
  int pad;         // unused entries after every four ports
  int op_stride;   // tensor cores: 16-bit entries of a row of the vector operand
  int layout;      // of S_j's tiles (kPort...)
  int mma;         // warps of a CTA with its products on the tensor cores (0: SIMT products)
  int priv;        // 1: an accumulator per warp (R <= 2), 0: one for all
  int ring;        // 1: shared-memory slots for the tiles in flight (0: no room)
  int sb;          // strips whose row sums the warps keep between barriers (priv: 0)
  size_t smem;
};

// Division of a sweep's tiles among CTAs: CTA c takes the segments cta_seg[c] .. cta_seg[c + 1] - 1.
struct PortPlan {
  std::vector<PortSeg> segs;
  std::vector<int32_t> cta_seg;
  int64_t part_elems = 0;
};

// Arguments of one sweep in port-response form (port.cu): u = u_base + S_j s per subgraph.
template <typename T>
struct PortArgs {
  const PieceDesc* pieces;
  const PortSeg* segs;
  const int32_t* cta_seg;      // grid + 1
  T* s;                        // port vectors of the sweep: ports x R
  T* part;                     // partial y of the subgraphs with several segments
  int* ticket;                 // one per segment, zero between sweeps
  int vec_elems, op_stride, mma, pad, priv, ring, sb;  // PortShape
  const T* S;                  // port responses, lower block triangle of 32 x 32 tiles
  const void* Sh;              // FP32 solvers: the same tiles in IEEE half (nullptr: use S)
  const float* scale;          // FP16 storage: per stored tile, the factor it was divided by
  const T* ubase;              // P^T K_j^{-1} b̃_j: ports x R
  const T* wprev;              // outgoing waves of the previous sweep: ends x R
  T* wnext;                    // outgoing waves of this sweep
  const int32_t* port_end_ptr;
  const int32_t* twin;
  const T* invz;
  CoupleRef<T> cpl;            // coupled lines (cpl.ptr == nullptr: none)
};

__host__ __device__ int64_t port_tiles(int nports);
PortShape port_shape(size_t elem, size_t stored, int R, int max_ports);
PortPlan port_plan(const PieceDesc* pieces, int npieces, size_t elem, size_t stored, int R, int ctas,
                   int mma);
template <typename T>
cudaError_t port_sweep_configure(int R, const PortShape& sh, bool half, int* ctas_per_sm);
// Two launches: the port vectors of all nports ports, then the sweep proper.
template <typename T>
cudaError_t launch_port_sweep(const PortArgs<T>& a, int R, int nports, int grid, size_t smem, cudaStream_t st);
template <typename T>
cudaError_t launch_gather_port_response(const PieceDesc* pieces, int npieces, const int32_t* port_local, int Rs, int b,
                                        const T* xc, T* S, int layout, cudaStream_t st, int batches = 1,
                                        int64_t stride = 0);
template <typename T>
cudaError_t launch_gather_ports(const PieceDesc* pieces, int npieces, const int32_t* port_local, int R, const T* xc,
                                T* ubase, cudaStream_t st);
// FP16 copy (and per-tile scale) of the FP32 port-response tiles.
cudaError_t launch_port_to_half(const PieceDesc* pieces, int npieces, const float* S, __half* Sh, float* scale,
                                const PortShape& from, const PortShape& to, cudaStream_t st);

// Port sweeps of small systems in one launch, S_j resident in shared memory (port_resident.cu).
struct ResCta {
  int64_t s_off;               // the CTA's subgraphs' S_j in the dense storage
  int32_t s_elems;
  int32_t vec;                 // ports of the CTA
  int32_t splits;              // units that share a group of rows
  int32_t port0, nports;       // into ResPlan::ports
  int32_t unit0, nunits;       // into ResPlan::units
};
struct ResUnit {
  int32_t s;                   // first row of the unit in the CTA's S (column 0)
  int32_t stride, n, row0;     // column stride, the subgraph's ports, first row
  int32_t vec;                 // the subgraph's first port in the CTA's vectors
  int32_t c0, c1, split;       // columns of the unit
};
struct ResPort {
  int32_t port, vec;           // port (global), its place in the CTA's vectors
  int32_t e0, e1, w0;          // its ends, the first one's place among the CTA's ends
};
struct ResPieceS {
  int32_t port_off, n, stride;
  int64_t s;                   // element offset of its dense S_j: entry (i, c) at s + c stride + i
  int32_t piece;               // index into the subgraphs the plan was made of
};
struct ResPlan {
  bool ok = false;
  std::vector<ResCta> ctas;
  std::vector<ResUnit> units;
  std::vector<ResPort> ports;
  std::vector<ResPieceS> piece_s;
  int64_t s_elems = 0;
  size_t smem = 0;
};
template <typename T>
struct ResArgs {
  const ResCta* ctas;
  const ResUnit* units;
  const ResPort* ports;
  const T* S;
  const T* ubase;
  const T* wprev;              // ends x R: incoming waves of the first sweep
  T* wout;                     // outgoing waves of the last sweep
  unsigned long long* xch[2];  // exchange buffers, ends x R words each (FP64: two words), contiguous
  const int32_t* twin;
  const T* invz;
  CoupleRef<T> cpl;
  int sweeps;
  int* status;
  long wait_limit;
};
ResPlan res_plan(const PieceDesc* pd, int npieces, size_t elem, int R, int nsm);
void res_plan_ends(ResPlan& pl, const int32_t* port_end_ptr);  // host copy of the end lists
template <typename T>
cudaError_t launch_gather_port_dense(const ResPieceS* ps, int n, const PieceDesc* pieces, const int32_t* port_local,
                                     int Rs, int b, const T* xc, T* S, cudaStream_t st, int batches = 1,
                                     int64_t stride = 0);
template <typename T>
cudaError_t port_resident_configure(int R, size_t smem, int* ctas_per_sm);
// a.sweeps sweeps in one cooperative launch (after clearing the exchange buffers, xch_bytes in all).
template <typename T>
cudaError_t launch_port_resident(const ResArgs<T>& a, int R, int grid, size_t smem, size_t xch_bytes, cudaStream_t st);

// Tensor-core port-response sweep for 16 / 32 right-hand sides (port_tc.cu), FP32 solvers.
constexpr int kTcMaxSplit = 8;        // items that a subgraph is cut into at most
struct TcItem {
  int32_t piece;               // index into PortTCArgs::pieces
  int32_t hi, lo;              // super-rows hi .. lo
  int64_t part;                // element offset of its share of y (ports x R); -1: the whole subgraph
};
struct TcSplit {               // a subgraph of several items
  int32_t piece, nitems;
  int32_t hi[kTcMaxSplit];     // first super-row of each item
  int64_t part;                // the items' shares, one after the other
};
struct TcPlan {
  std::vector<TcItem> items;
  std::vector<int32_t> cta_item;  // CTA c takes the items cta_item[c] .. cta_item[c + 1] - 1
  std::vector<TcSplit> splits;
  std::vector<int32_t> tile_off;  // per subgraph, its first operand tile
  int64_t part_elems = 0, tiles = 0;
  int max_split_ports = 0;
};
TcPlan tc_plan(const PieceDesc* pieces, int npieces, int R, int ctas);

struct PortTCArgs {
  const PieceDesc* pieces;     // subgraphs of the launch
  const TcItem* items;
  const int32_t* cta_item;
  const TcSplit* splits;
  float* part;
  const unsigned char* S16;    // lower block triangle of S_j / sigma_j as fp16 hi / lo panels (h_off)
  const float* sig_s;          // sigma_j per subgraph of the launch
  const float* gscale;         // g_p = sqrt(S_pp) per port (diagonal balance of S_j)
  unsigned char* scratch;      // FUSED: per CTA two slots of n4max s^T tiles (R x 512 bytes each)
  int n4max;                   // most 128-port super-rows of a subgraph
  const int4* prec;            // FUSED: per port 3 x int4: first four entries' wave rows, their coefficients
                               // (float bits), {next end, e1, next coupling, k1} (launch_port_records)
  unsigned char* stiles;       // not FUSED: the port vectors' operand tiles (R x 512 bytes per super-row)
  const int32_t* tile_off;     // per subgraph, its first tile
  float* ssig;                 // sigma_r per subgraph and column
  const int32_t* ent_ptr;      // not FUSED: per port, first entry of its sum's terms
  const int2* ent;             // (the wave's place among the subgraph's ends, coefficient)
  int tmem_cols;               // tensor-memory columns per CTA (power of two >= n4max R)
  const float* ubase;          // ports x R
  const float* wprev;          // ends x R
  float* wnext;
  const int32_t* port_end_ptr;
  const int32_t* twin;
  const float* invz;
  CoupleRef<float> cpl;        // coupled lines (cpl.ptr == nullptr: none)
  int* status;
  long wait_limit;
};

constexpr int kTcMaxSuper = 16;       // 128-port super-rows per subgraph on the tensor cores
int64_t port_f16_bytes(int nports);   // fp16 hi / lo blocks of one subgraph (1 KB multiple)
int64_t port_f32_blocks(int nports);  // 128 x 128 FP32 blocks of the lower triangle (setup)
size_t port_tc_smem_bytes(int R, bool lo);
// Per-port gather records of the fused sweep (3 int4 per port, nports of them).
cudaError_t launch_port_records(int nports, const int32_t* port_end_ptr, const int32_t* twin, const float* invz,
                                CoupleRef<float> cpl, int4* rec, cudaStream_t st);
// Places of the coupling entries' waves for the separate port vectors.
cudaError_t launch_port_entries(const PieceDesc* pieces, int npieces, const int32_t* port_end_ptr, const int32_t* twin,
                                const float* invz, CoupleRef<float> cpl, int32_t* ent_ptr, int2* ent, cudaStream_t st);
constexpr size_t kVecTcSmemMax = 220 * 1024;
size_t port_vec_tc_smem_bytes(int max_ends);
cudaError_t port_tc_configure(int R);
// The port vectors (unless fused: a.stiles == nullptr), one persistent launch for the sweep (grid <=
// SMs), and one for the cut subgraphs' waves if there are any; lo = use the lo half of S_j
// (FP32-accurate).
cudaError_t launch_port_sweep_tc(const PortTCArgs& a, int R, bool lo, int npieces, int grid, int nsplits,
                                 int max_split_ports, cudaStream_t st);
cudaError_t launch_gather_port_blocks(const PieceDesc* pieces, int npieces, const int32_t* port_local, int Rs, int b,
                                      const float* xc, float* S32, cudaStream_t st, int batches = 1,
                                      int64_t stride = 0);
cudaError_t launch_port_blocks_to_f16(const PieceDesc* pieces, int npieces, const float* S32, unsigned char* S16,
                                      float* sig, float* gscale, cudaStream_t st);

constexpr int kWideWindow = 512;
constexpr int kMaxRhs = 32;

// Assemble K_j = Ã_j + sum_e Z_e^{-1} e_c e_c^T into the (zeroed) band storage (eq. 5.8).
template <typename T>
cudaError_t launch_build_band(int64_t ncopies, const int32_t* copy_piece, const PieceDesc* pieces,
                              const int64_t* l_rowptr, const int32_t* l_col, const double* l_val,
                              const int32_t* port_of_copy, const int32_t* port_end_ptr, const double* invz,
                              int npieces, int max_pad_rows, T* band, int* status, cudaStream_t st);
// U = L^T (left-aligned rows, transposed inverse diagonal blocks) for the dot-form back substitution.
template <typename T>
cudaError_t launch_transpose_band(const PieceDesc* pieces, int npieces, const T* L, T* U, cudaStream_t st);
// Banded Cholesky of every K_j in place; each diagonal block replaced by its inverse.
// piece_flag[j] (may be NULL): 1 = non-positive pivot, 2 = pivot^2 < kFlagRatio K_ii (precision
// lost); the global status gets kStatusNotSpd only when piece_flag is NULL.  diag0 (may be NULL):
// per-row scratch (sum of n_pad entries) holding the original diagonal.
// FP32 factorisation with the trailing update on the tensor cores (factor_tc.cu), 64 <= max_w <= 384.
size_t factor_tc_smem_bytes(int max_w);
cudaError_t launch_factor_tc(const PieceDesc* pieces, int npieces, int max_w, float* band, int* status,
                             int* piece_flag, float* diag0, long wait_limit, cudaStream_t st);
template <typename T>
cudaError_t launch_factor(const PieceDesc* pieces, int npieces, int max_w, T* band, int* status, int* piece_flag,
                          T* diag0, cudaStream_t st);

// Unit right-hand sides for batch b of every subgraph's ports (b̃ of port b*R + r = e_c in column r).
template <typename T>
cudaError_t launch_unit_rhs(const PieceDesc* pieces, int npieces, const int32_t* port_local, int R, int b, T* bt,
                            cudaStream_t st);
// g[port] = x_c of column r for the ports of batch b (diagonal of K_j^{-1}).
template <typename T>
cudaError_t launch_gather_diag(const PieceDesc* pieces, int npieces, const int32_t* port_local, int R, int b,
                               const T* xc, double* g, cudaStream_t st);
// b̃_c = share_c * src[vertex(c)]  (§4 step 3), into T precision, R contiguous.
template <typename T>
cudaError_t launch_split(int64_t ncopies, int R, const int64_t* copy_vertex, const double* share,
                         const double* src, int64_t ld, T* bt, cudaStream_t st);
// xt[i] = xbase[i] + mean over the copies of i of xc (xbase may be NULL).
template <typename T>
cudaError_t launch_assemble(int64_t n, int R, const int64_t* vc_ptr, const int64_t* vc_copy, const T* xc,
                            const double* xbase, double* xt, int64_t ld, cudaStream_t st);
// sums_r[q] += ||b_q - A x_q||^2, sums_b[q] += ||b_q||^2 (R <= 8) on a device of nsm SMs.
cudaError_t launch_residual_norms(int nsm, int64_t n, int R, const int64_t* rowptr, const int32_t* col, const double* val,
                                  const double* b, int64_t ldb, const double* x, int64_t ldx, double* sums_r,
                                  double* sums_b, cudaStream_t st);
// res = b - A x (res may be NULL) and squared norms with fixed-order sums (identical inputs give
// identical norms): norms[r] = ||res_r||^2 (resp. ||v_r||^2), through the scratch part of
// norm_parts(n) * R doubles.
int64_t norm_parts(int64_t n);
cudaError_t launch_residual_det(int64_t n, int R, const int64_t* rowptr, const int32_t* col, const double* val,
                                const double* b, int64_t ldb, const double* x, int64_t ldx, double* res, int64_t ldr,
                                double* part, double* norms, cudaStream_t st);
cudaError_t launch_sqnorm_det(int64_t n, int R, const double* v, int64_t ld, double* part, double* norms,
                              cudaStream_t st);
// dst[i + r*ldd] = src[i + r*lds]
cudaError_t launch_copy2d(int64_t n, int R, const double* src, int64_t lds, double* dst, int64_t ldd, cudaStream_t st);

}  // namespace vtm
