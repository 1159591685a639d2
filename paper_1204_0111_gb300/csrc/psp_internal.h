// Internal declarations shared by the translation units of libpsp.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "psp.h"

struct psp_ctx_s;

namespace psp {

// sweep with caller-provided work vectors (defined in psp_api.cu)
size_t apply_workspace_bytes(const psp_ctx_s* X, int nrhs);
psp_status apply_with_workspace(psp_ctx_s* X, double2* u, int nrhs, void* ws, cudaStream_t st);
int64_t handle_points(const psp_ctx_s* X);   // N, or -1 when the handle has no factorisation
int handle_device(const psp_ctx_s* X);       // CUDA device the handle was set up on
psp_status set_error(psp_status s, const char* msg);

// ---------------------------------------------------------------------------
// Symbolic analysis of one auxiliary-problem box (nx x ny x depth): the
// supernodal nested-dissection tree of §2.1 (separator-tree figure), postorder.
// ---------------------------------------------------------------------------
struct Shape {
  int nx = 0, ny = 0, nz = 0;  // box extents (nz = depth of the auxiliary problem)
  int leaf = 0;
  int nsn = 0;
  std::vector<int32_t> order;       // elimination index -> box node id
  std::vector<int32_t> elim;        // box node id -> elimination index
  std::vector<int32_t> first;       // nsn + 1: elimination index of each supernode's first node
  std::vector<int32_t> s, u;        // supernode size, |struct(S)|
  std::vector<int32_t> parent;      // -1 for the root
  std::vector<int32_t> child_ptr, child_idx;
  std::vector<int64_t> struct_ptr;  // nsn + 1 offsets into struct_elim / rel
  std::vector<int32_t> struct_elim; // struct(S) as sorted elimination indices
  std::vector<int32_t> rel;         // position of each struct entry in the parent's front rows
  std::vector<int32_t> height;      // leaves 0, parent = 1 + max(children)
  int nlevels = 0;
  std::vector<std::vector<int32_t>> level_sns;
  std::vector<int32_t> depth;       // root 0, child = parent + 1
  int ndepths = 0;
  // solve-side pull map: for each front row position p of S u struct(S), up to two
  // offsets (within the per-panel update-vector slab) of children's update entries
  std::vector<int64_t> pull_ptr;    // nsn + 1, = sum (s + u)
  std::vector<int32_t> pull;        // 2 per position, -1 = none
  // per-panel layouts
  std::vector<int64_t> g_off;       // G block offset within a panel's factor slab (elements)
  int64_t g_total = 0;
  std::vector<int64_t> upd_off;     // update-vector offset within the panel's update slab
  int64_t upd_total = 0;
};

void build_shape(Shape& sh, int nx, int ny, int nz, int leaf);

// ---------------------------------------------------------------------------
// Device views
// ---------------------------------------------------------------------------
struct ShapeDev {
  int nx, ny, nz, nsn;
  const int32_t* order;
  const int32_t* elim;
  const int32_t* first;
  const int32_t* s;
  const int32_t* u;
  const int32_t* child_ptr;
  const int32_t* child_idx;
  const int64_t* struct_ptr;
  const int32_t* struct_elim;
  const int32_t* rel;
  const int64_t* pull_ptr;
  const int32_t* pull;
};

// 7-point operator on a box: -sum_j d_j(a_j d_j u) - k2num / c^2 * s1 s2 s3 u (Eq. (1.1)/(1.5),
// s1 s2 s3-scaled).  Stretch tables are complex; half[k] sits between node k-1 and node k.
struct BoxOp {
  int nx, ny, nz;
  double inv_h2;
  double2 k2num;            // omega^2 (A) or (omega + i alpha)^2 (J)
  const double* ic2;        // 1 / c^2 of the global wave speed, nx*ny*nz_global
  const int32_t* cplane;    // box plane -> global plane whose c is used
  const double2* s1n;
  const double2* s1h;
  const double2* s2n;
  const double2* s2h;
  const double2* s3n;
  const double2* s3h;
};

enum GemmFlags : int {
  GF_BETA0 = 1,           // C = alpha * A B^T (do not read C)
  GF_C_LOWER = 2,         // write only local row >= local col (diagonal tiles)
  GF_B_NN = 4,            // B(n,k) = B[k + n ldb]   (default NT: B[n + k ldb])
  GF_B_UNIT_LOWER_NT = 8, // B(n,k) is T[n,k] of a unit lower T stored with D on its diagonal
  GF_B_UNIT_LOWER_NN = 16,// B(n,k) is T[k,n] of a unit lower T stored with D on its diagonal
  GF_D_MUL = 32,          // scale A(:,k) by d(k)
  GF_D_DIV = 64,          // scale A(:,k) by 1/d(k)
  GF_NEG = 128,           // alpha = -1 (else +1)
  GF_SI = 256,            // selective-inversion work (inv(L_TL), M_BL): host accounting only, kernels ignore it
  GF_TEST_STALL = 512     // tests: a tensor-core tile whose first operand block is never copied
};

// C(m x n) (+)= alpha * A(m x k) * diag(d)^{+-1} * B(n x k)^T ; pointers already offset.
template <typename T>
struct GemmTask {
  T* C;
  const T* A;
  const T* B;
  const T* d;
  int ldc, lda, ldb, ldd;
  int m, n, k;
  int kg0, ng0;   // global k / n index of the first element (for the unit-lower masks)
  int flags;
  int pad_;
};

// Update matrices F_BR (u x u, symmetric) keep only their lower tiles: tiles of ut x ut (ut = 64 for
// fronts whose products run on CUDA cores, 128 for tensor-core fronts), tile (I, J), I >= J, stored
// column of tiles after column of tiles, each tile column-major with leading dimension ut.
__host__ __device__ __forceinline__ int64_t upd_tile_offset(int64_t I, int64_t J, int64_t ntiles, int ut) {
  return (J * ntiles - J * (J - 1) / 2 + (I - J)) * (int64_t)ut * ut;
}
__host__ __device__ __forceinline__ int64_t upd_index(int r, int c, int u, int ut) {   // r >= c; ut 64 or 128
  const int sh = ut == 128 ? 7 : 6;
  const int nt = (u + ut - 1) >> sh;
  return upd_tile_offset(r >> sh, c >> sh, nt, ut) + ((int64_t)(c & (ut - 1)) << sh) + (r & (ut - 1));
}
// column c of that matrix, for many r
struct UpdColumn {
  int64_t tile0, within;   // tiles before tile row 0 of the column's tiles; the column's start in a tile
  int sh;
  __host__ __device__ __forceinline__ UpdColumn(int c, int u, int ut) {
    sh = ut == 128 ? 7 : 6;
    const int64_t nt = (u + ut - 1) >> sh, J = c >> sh;
    tile0 = J * nt - J * (J - 1) / 2 - J;
    within = (int64_t)(c & (ut - 1)) << sh;
  }
  __host__ __device__ __forceinline__ int64_t at(int r) const {
    return ((tile0 + (r >> sh)) << (2 * sh)) + within + (r & ((1 << sh) - 1));
  }
};
__host__ __device__ __forceinline__ int64_t upd_packed_elems(int u, int ut) {
  const int64_t nt = (u + ut - 1) / ut;
  return nt * (nt + 1) / 2 * (int64_t)ut * ut;
}

// A front in a level batch.
template <typename T>
struct FrontTask {
  T* G;        // (s+u) x s, ld = s+u
  T* U;        // u x u update (F_BR) in lower tiles of ut x ut (upd_index); nullptr for the root
  T* W;        // s x s work: inv(L_TL) under construction
  T* Z;        // u x s work: F_BL L^{-T}
  T* ZD;       // u x s: Z D^{-1}, leading dimension ldzd (a work block for the extended selective
               // inversion of CUDA-core fronts, G's bottom block when L_BL itself is stored; else nullptr)
  T* dinv;     // the front's reciprocal pivots (for the sweep)
  T* W2;       // s x s work: the second inverse of L_TL under construction (two-inverse form), else nullptr
  int s, u;
  int panel, sn;
  int64_t gfid;
  int ut, ldzd;   // tile size of U; leading dimension of ZD
};

// elements from a front's G block to its second inverse of L_TL (two-inverse form): G padded to 16
__host__ __device__ __forceinline__ int64_t second_inverse_offset(int64_t s, int64_t u) {
  return ((s + u) * s + 15) / 16 * 16;
}

constexpr int kAssembleCols = 32;   // columns of a front per assembly CTA

struct ColTask {   // a chunk of columns / rows of one front
  int front;       // index into the level's FrontTask array
  int c0, c1;
};

// ---------------------------------------------------------------------------
// Launchers (defined in the .cu files)
// ---------------------------------------------------------------------------
void launch_matvec(const BoxOp& op, const double2* x, double2* y, int nrhs, int64_t N, cudaStream_t st);
void launch_inverse_square(double* c, int64_t N, cudaStream_t st);   // c := 1 / c^2
void launch_scale_rhs(const BoxOp& op, const double2* f, double2* b, int nrhs, int64_t N, cudaStream_t st);

template <typename T>
void launch_assemble_impl(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, const ShapeDev* shapes,
                          const BoxOp* boxops, T* const* upd_ptr, const int32_t* upd_tile, const int32_t* panel_shape,
                          cudaStream_t st);
template <typename T>
void launch_diag_ldlt(const FrontTask<T>* fronts, const int* list, int nlist, int kb, double tiny, int* status, bool wide,
                      cudaStream_t st);
template <typename T>
void launch_panel_right(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, int kb, bool wide, cudaStream_t st);
template <typename T>
void launch_panel_left(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, int kb, bool wide, cudaStream_t st);
template <typename T>
void launch_panel_rsolve(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, int kb, bool wide, cudaStream_t st);
template <typename T>
void launch_gemm(const GemmTask<T>* tasks, int ntasks, cudaStream_t st);
// tensor-core path (complex64): operands packed once per front into TF32 planes, then tiles
enum TcPackMode { TC_PACK_PLAIN = 0, TC_PACK_UNIT_LOWER = 1, TC_PACK_UNIT_LOWER_T = 2, TC_PACK_TRANSPOSED = 3 };
struct TcPackTask {        // one 128-row x 16-k block of a packed operand
  const float2* src;       // column-major source, ld
  const float2* d;         // PLAIN only: divide column k by d[k * ldd] (nullptr: no scaling)
  void* dst;               // 48 KB destination block
  int ld, ldd;
  int r0, k0;              // first row / k of the block
  int R, K;                // source extents (rows, k); outside -> 0
  int mode;                // TcPackMode: PLAIN X[r, k]; UNIT_LOWER T[r, k]; UNIT_LOWER_T T[k, r]
  int pad_;
};
struct TcGemmTask {        // one 128 x 128 tile of C (+)= +-A B^T from packed blocks
  const unsigned char* A;  // packed A row block (k-blocks contiguous)
  const unsigned char* B;  // packed B row block
  float2* C;
  int ldc, m, n;
  int kb0, nkb;            // k-blocks [kb0, kb0 + nkb)
  int flags;               // GF_NEG, GF_BETA0, GF_C_LOWER
};
void launch_tc_pack(const TcPackTask* tasks, int ntasks, cudaStream_t st);
void launch_tc_gemm(const TcGemmTask* tasks, int ntasks, int* status, cudaStream_t st);
// tensor-core path of complex128 fronts: operands written once as eight base-256 digits, then 128 x 32 tiles
struct OzShape { int tile_m, tile_n, k, kc; int64_t a_block, b_block; };   // tile, k per block and per row scale, bytes per block
constexpr OzShape kOz{128, 32, 16, 128, 65536, 24576};
struct OzPackTask {        // 128 rows x 128 k of an operand
  const double2* src;      // column-major source, ld
  const double2* scale;    // PLAIN only: column k times scale[k * lds] (nullptr: no scaling)
  unsigned char* dst;      // first block (16 k) of these rows; the following ones adjacent
  int* exps;               // row exponents of this block of k
  int64_t sub_stride;      // B operands: bytes between the blocks of 32 rows ...
  int64_t exp_stride;      // ... and entries between their exponents
  int ld, lds, r0, k0, R, K;   // first row / k, source extents (outside -> 0)
  int mode;                // TcPackMode (TRANSPOSED: X[k, r])
  int rows_b;              // 0: A operand (128-row blocks), 1: B operand (32-row blocks)
  const int* ka;           // balance of the product's columns k (k_oz_pack): exponents of A's columns before its scale ...
  const int* kb;           // ... and of B's (both nullptr: taken as equal)
  const double2* kd;       // A's scale, stride ldk (nullptr: none)
  int ldk;
  int near;                // OZ_NEAR: the scale's balance alone serves 128 k where it is close to the whole one; OZ_KEEP: and
                           // then this operand's digits in that balance are in place already
};
enum OzNear { OZ_NEAR = 1, OZ_KEEP = 2 };
struct OzColTask {         // 32 columns k of an operand: exponents of their largest entries
  const double2* src;
  int* out;                // out[k]
  int ld, k0, R, K, mode;  // as in OzPackTask
  int pad_;
};
struct OzGemmTask {        // one 128 x 32 tile of C (+)= +-A B^T
  const unsigned char* A;  // block of 16 k number 0 of its 128 rows
  const unsigned char* B;  // block of 16 k number 0 of its 32 rows
  const int* ea;           // row exponents, 128 per 128 k
  const int* eb;           // 32 per 128 k
  double2* C;
  int ldc, m, n;
  int kb0, nkb;            // blocks of 16 k [kb0, kb0 + nkb)
  int doff;                // entries with row + doff < column are not written
  int flags;               // GF_NEG, GF_BETA0
  int pad_;
};
void launch_oz_colmax(const OzColTask* tasks, int ntasks, cudaStream_t st);
void launch_oz_pack(const OzPackTask* tasks, int ntasks, cudaStream_t st);
void launch_oz_gemm(const OzGemmTask* tasks, int ntasks, int* status, cudaStream_t st);
int tc_block_k();
int64_t tc_block_bytes();
int tc_gemm_tile();
template <typename T>
void launch_copy_linv(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, cudaStream_t st);
template <typename T>
void launch_scale_zd(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, cudaStream_t st);

// ---- the whole sweep (Alg. 1.5, each panel's multifrontal solve as in Alg. 1.3) in one cooperative launch ----
struct SolveTask {  // rows [r0, r1) of front sn (up the tree) or columns [r0, r1) of S (down)
  int sn, r0, r1;
};

// one front as a task reads it
struct FrontRec {
  int s, u, first, pad_;
  int64_t g_off;      // its G block within the panel's factor slab (elements)
  int64_t row_off;    // its rows' index words within the shape's
  int64_t sel_off;    // its struct indices within the shape's
  int64_t upd_off;    // its update vector within the panel's update vectors
  int64_t pad2_[2];
};
static_assert(sizeof(FrontRec) == 64, "records are copied word by word");

// one panel solve of Alg. 1.5: its panel, its problem's vectors and coupling tables
struct StepRec {
  int64_t gbase;         // factor slab offset (elements)
  int64_t dbase;         // offset of the panel's reciprocal pivots
  int64_t off1;          // offset of the problem's block in a batched vector, per right-hand side
  int64_t N;             // points of the problem
  const double2* s1n;    // global stretch tables for the plane coupling J_{i+1,i}: s1 s2 (1 / s3 at the plane boundary)
  const double2* s2n;
  const double2* s3c;
  double cz;             // +- 1 / h^2
  const int4* rows;      // the shape's index words per front row: {node, child update entry, child update entry, 0}
  const int32_t* sel;    // the shape's struct indices (elimination order)
  int z0, z1, lead;      // panel planes, pad planes
  int nx, plane;         // nx, nx * ny
  int mode;              // 0: forward sweep (u_i := T_i(u_i - J_{i,i-1} u_{i-1})); 1: backward (u_i -= T_i J^T u_{i+1})
  int couple;            // there is a previous (mode 0) / next (mode 1) panel
  int prob;              // problem of a batch (0 for a single problem)
  int pad_[4];
};
static_assert(sizeof(StepRec) == 128, "records are copied word by word");

// one task of the sweep's queue (topological order: panel solves in Alg. 1.5 order; inside
// one, the up-the-tree tasks level by level, then the down-the-tree tasks from the root).  An entry
// carries its one dependency and the counters it signals.  Counters are words of the sweep's counter array
// (zeroed before every sweep):
//   [0] dequeue head, [1, 5) status, then per step the tasks completed, then per step and front the
//   up tasks completed, the down tasks completed and the up tasks of the front's children completed.
struct QueueEntry {
  int step, front;              // panel solve index, front record
  int r0, r1;                   // rows (up) or columns (down) [r0, r1) of the front
  int wait;                     // counter the task waits for (-1: none) ...
  unsigned target;              // ... until it reaches this count
  int done;                     // counter of the front's own completed tasks (this direction)
  int kids;                     // counter of the parent's children's completed up tasks (-1: none)
  int step_done;                // counter of the step's completed tasks (-1: nothing waits for it)
  short dir;                    // 0 up the tree, 1 down the tree; 2 / 3 the second phase up / down of a front
                                // whose factor keeps L_BL (the first phase is then 0 / 1)
  short pad0_;
  int pad_[2];
};
static_assert(sizeof(QueueEntry) == 48, "queue entries are copied word by word");
// second phases of a front (factors that keep L_BL rather than L_BL inv(L_TL))
constexpr int kDirUpB = 2, kDirDownB = 3;
constexpr int kSweepStepCounters = 5;   // first word of the per-step counters
template <typename T>
struct SweepArgs {
  T* xf;                        // box vectors after L^{-1} and D^{-1} (elimination order), n_loc x nrhs per problem
  T* xb;                        // box vectors after L^{-T}
  T* upd;                       // fronts' update vectors, upd_ld x nrhs per problem
  double2* u;                   // global vector block
  int64_t n_loc, upd_ld;
  int nrhs;
  int si;                       // psp_si_mode of the factors (what G keeps)
  const StepRec* steps;
  const FrontRec* fronts;
  const T* factor;
  const T* dinv;                // reciprocal pivots, per panel in elimination order
  const QueueEntry* queue;
  int nqueue;
  unsigned* ctr;                // counter array (layout above)
  int* status;                  // status[2] set when a wait gave up (= ctr + 1)
  int* sticky;                  // also set then; kept until the host reads it (psp_check_status)
  int chunk;                    // vector entries a task stages in shared memory at a time (set by launch_sweep)
  int tri_global;               // substitution tasks keep their vector in xb: too wide for shared memory (set by launch_sweep)
  int claim_ahead;              // 2: a CTA holds the two tasks after the one it runs; 1: the next one only
};
void launch_build_rows(const ShapeDev& sh, int4* rows, cudaStream_t st);
// returns 0 on success, -1 when the kernel does not fit the device, else a cudaError_t; smax / ldmax:
// the widest front's s and s + u
template <typename T>
int launch_sweep(const SweepArgs<T>& args, int smax, int ldmax, int max_per_sm, int rhs_group, cudaStream_t st);
// what that launch would take: columns a CTA carries through a pass, resident CTAs per SM
struct SweepFit { int rg = 0, per_sm = 0; };
template <typename T>
SweepFit sweep_fit(int nrhs, int si, int smax, int ldmax, int max_per_sm, int rhs_group);

// ---- GMRES helpers (complex128) ----
// A block of vectors holds ncol columns (right-hand sides, and problems of a batch); column c of
// every vector of the block is the span [off, off + len).
struct ColSpan {
  int64_t off, len;
};
// out[i * ncol + c] = sum_g conj(V_i[c][g]) w[c][g], V_i = V + i * ldv_vec; fixed two-stage order
void launch_multidot(const double2* V, int64_t ldv_vec, int nvec, const double2* w, const ColSpan* cols, int ncol,
                     int64_t maxlen, double2* partial, double2* out, cudaStream_t st);
int multidot_blocks(int64_t maxlen);   // partial blocks per column (size partial as blocks * nvec * ncol)
// w[c] += sign * sum_i h[i * ncol + c] V_i[c]
void launch_multiaxpy(const double2* V, int64_t ldv_vec, int nvec, const double2* h, double2* w, const ColSpan* cols,
                      int ncol, int64_t maxlen, double sign, cudaStream_t st);
// y[c] = alpha_c x[c] (mode 0), y[c] = x[c] - y[c] (mode 1), y[c] += alpha_c x[c] (mode 2)
void launch_axpby_batch(const double2* x, double2* y, const ColSpan* cols, int ncol, int64_t maxlen,
                        const double2* alpha, int alpha_mode, cudaStream_t st);

// Hessenberg least-squares state, one column block per right-hand side
struct LsqState {
  double2* H;        // (k+1) x k per rhs, column-major, ld = k+1
  double* cs;        // k per rhs
  double2* sn;       // k per rhs
  double2* g;        // k+1 per rhs
  double* resid;     // |g_{j+1}| per rhs
  double2* scl;      // scale of the next basis vector per rhs (0 when inactive)
  const int* active; // 1 while the rhs iterates
  int k, nrhs;
};
void launch_arnoldi_step(const LsqState& L, int j, const double2* h1, const double2* h2, const double2* nrm2,
                         cudaStream_t st);
void launch_backsolve(const LsqState& L, const int* jr, double2* y, cudaStream_t st);
void launch_cycle_start(const LsqState& L, const double2* nrm2, cudaStream_t st);

}  // namespace psp
