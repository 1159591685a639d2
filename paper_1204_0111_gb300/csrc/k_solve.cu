// Multifrontal solve with selectively inverted fronts (§2.2) as the T_i of Alg. 1.3 inside the sweep
// of Alg. 1.5: the whole sweep in one persistent launch.
//
// Each front stores G = [inv(L_TL) (unit lower, D on the diagonal); M_BL = L_BL inv(L_TL)], so
//   up the tree:   v_S = inv(L_TL) w_S,  x_S = D^{-1} v_S,  update_U = w_U - M_BL w_S
//   down the tree: x_S = inv(L_TL)^T x_S - M_BL^T x_U
// which are matrix-vector products (the point of selective inversion): every task reads its
// block of G once, column segments contiguous, and no task depends on another task of the same
// level.  Children's update vectors are pulled (at most two per row), never scattered, so the
// summation order is fixed.  Extension by zero over the pad, the plane coupling J_{i+1,i} of
// the previous / next panel and the extraction of the panel's planes are fused into the
// gathers and the final write.
//
// Work vectors (xf, xb, upd) are kept per right-hand-side group of RG columns, entry after entry
// with the group's columns adjacent: a gathered entry is one contiguous read for the whole group.
#include "cplx.cuh"
#include "psp_internal.h"

namespace psp {

constexpr int kComputeThreads = 256;                    // product threads of a sweep CTA
constexpr int kComputeWarps = kComputeThreads / 32;
constexpr int kSweepThreads = kComputeThreads + 64;     // + the scheduling warp and the signalling warp
constexpr int kGatherIdx = 256;   // index words (16 bytes) of front rows a slot holds; the rest are read from global memory
constexpr int kOwnIdx = 256;      // index words of a task's own rows (sweep_max_rows at most)

// named barriers: 1 among the product warps; per task slot, ready (scheduler -> product warps), done
// (product warps -> signaller) and free (signaller -> scheduler)
enum SweepBarrier { kBarCompute = 1, kBarReady = 2, kBarDone = 4, kBarFree = 6 };
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void compute_sync() { bar_sync(kBarCompute, kComputeThreads); }

// one task as the product warps see it, filled by the scheduling warp.  The product warps read a field where they
// need it (a broadcast from shared memory) rather than keep it in a register across their loops.
template <typename T>
struct TaskSlot {
  int ok;                 // 0: stop
  int tr_log;             // up: 2^tr_log threads along the rows
  int splits;             // down: warps that share a block of columns
  int pad_;
  const T* G;             // the front's block
  const T* dinv;          // its reciprocal pivots
  const int4* rows_g;     // its rows' index words in global memory
  const int32_t* sel_g;   // its struct indices in global memory
  T* xf;                  // the problem's work vectors and vector block
  T* xb;
  T* upd;                 // at the front's update vector: own_upd; children's entries are relative to upd
  double2* u;
  StepRec st;
  QueueEntry e;
  FrontRec fr;
  int4 rows[kGatherIdx];  // up: index words of the S rows; down: struct indices (int32)
  int4 own[kOwnIdx];      // up: index words of the task's rows r >= s
};

// shared-memory elements per vector entry: RG columns, padded by 16 bytes where the lanes of a quarter
// warp reading consecutive entries with 128-bit loads would meet in the same banks
template <typename T, int RG>
__host__ __device__ constexpr int entry_stride() {
  return RG * (int)sizeof(T) <= 16 ? RG : RG + 16 / (int)sizeof(T);
}

// RG adjacent entries from shared memory
template <typename T, int RG>
__device__ __forceinline__ void load_shared(const T* p, T (&v)[RG]) {
  if constexpr (sizeof(T) == 8 && RG >= 2) {
#pragma unroll
    for (int q = 0; q < RG; q += 2) {
      const float4 f = *reinterpret_cast<const float4*>(p + q);
      v[q] = make_float2(f.x, f.y);
      v[q + 1] = make_float2(f.z, f.w);
    }
  } else {
#pragma unroll
    for (int q = 0; q < RG; ++q) v[q] = p[q];
  }
}

// right-hand-side group g of the sweep: its columns [g RG, g RG + w); vec: the group is full and its vectors are
// 16-byte aligned
struct Group {
  int g, w;
  bool vec;
};

// the group's columns of one work-vector entry from global memory (L2: other SMs wrote them); base: group 0's
// vector of ld entries
template <typename T, int RG>
__device__ __forceinline__ void load_entry(const T* base, const int64_t ld, const int64_t entry, const Group gr, T (&v)[RG]) {
  if constexpr (RG == 1) {
    v[0] = __ldcg(base + gr.g * ld + entry);
  } else {
    const T* p = base + gr.g * RG * ld + entry * gr.w;
    if (sizeof(T) == 8 && gr.vec) {
#pragma unroll
      for (int q = 0; q < RG; q += 2) {
        const float4 f = __ldcg(reinterpret_cast<const float4*>(p + q));
        v[q].x = f.x;
        v[q].y = f.y;
        v[q + 1].x = f.z;
        v[q + 1].y = f.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < RG; ++q) v[q] = q < gr.w ? __ldcg(p + q) : CplxTraits<T>::zero();
    }
  }
}
template <typename T, int RG>
__device__ __forceinline__ T* entry_ptr(T* base, const int64_t ld, const int64_t entry, const Group gr) {
  if constexpr (RG == 1) return base + gr.g * ld + entry;
  else return base + gr.g * RG * ld + entry * gr.w;
}

// children's update entries a and b (-1: none): both reads are issued before either is used
template <typename T, int RG>
__device__ __forceinline__ void pull_entries(const TaskSlot<T>& sl, const int64_t ld, const Group gr, const int a, const int b,
                                             T (&v)[RG]) {
  T t[RG];
#pragma unroll
  for (int q = 0; q < RG; ++q) v[q] = t[q] = CplxTraits<T>::zero();
  if (a >= 0) load_entry<T, RG>(sl.upd, ld, a, gr, v);
  if (b >= 0) load_entry<T, RG>(sl.upd, ld, b, gr, t);
#pragma unroll
  for (int q = 0; q < RG; ++q) v[q] = cadd(v[q], t[q]);
}

// The panel's input at a box node: forward u_i - J_{i,i-1} u_{i-1}, backward J_{i+1,i}^T u_{i+1} (supported on the
// panel's last plane); zero over the pad (Alg. 1.3).  J's coupling entry is -s1 s2 / s3 / h^2.
template <typename T, int RG>
__device__ __forceinline__ void input_entry(const TaskSlot<T>& sl, const Group gr, const int node, T (&v)[RG]) {
  const StepRec& st = sl.st;
  const int own = node - st.lead * st.plane;   // index within the panel's planes
  const int at = st.mode == 0 ? own : own - (st.z1 - st.z0 - 1) * st.plane;   // index within the coupled plane
  const bool coupled = st.couple && own >= 0 && (st.mode == 0 ? own < st.plane : at >= 0);
  double2 x[RG];
#pragma unroll
  for (int q = 0; q < RG; ++q) x[q] = make_double2(0.0, 0.0);
  const double2* u = sl.u + gr.g * RG * st.N + ((int64_t)st.plane * st.z0 + own);
  if (st.mode == 0 && own >= 0) {
#pragma unroll
    for (int q = 0; q < RG; ++q)
      if (RG == 1 || q < gr.w) x[q] = __ldcg(u + q * st.N);
  }
  if (coupled) {
    u += st.mode == 0 ? -(int64_t)st.plane : (int64_t)st.plane;
    const double2 a = cscale(cmul(cmul(__ldg(st.s1n + at % st.nx), __ldg(st.s2n + at / st.nx)), __ldg(st.s3c)), st.cz);
#pragma unroll
    for (int q = 0; q < RG; ++q)
      if (RG == 1 || q < gr.w) cfma(x[q], a, __ldcg(u + q * st.N));
  }
#pragma unroll
  for (int q = 0; q < RG; ++q) v[q] = CplxTraits<T>::from(x[q]);
}

// Sums NV per-lane scalars over the warp with halving exchanges: after the exchange over `off` each lane keeps
// half of its values, so NV values cost about NV + 5 shuffles instead of 5 NV.  Lane l ends with the totals of
// indices base .. base + max(1, NV / 32) - 1; `lead` marks the one lane of each total that stores it.
template <typename R, int NV>
__device__ __forceinline__ void warp_sum(R (&v)[NV], const int lane, int& base, bool& lead) {
  base = 0;
  lead = true;
  int off = 16;
#pragma unroll
  for (int n = NV; n > 1 && off > 0; n >>= 1, off >>= 1) {
    const int half = n >> 1;
    const bool up = lane & off;
#pragma unroll
    for (int k = 0; k < NV / 2; ++k)
      if (k < half) {
        const R send = up ? v[k] : v[k + half];
        const R keep = up ? v[k + half] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
    if (up) base += half;
  }
  for (; off > 0; off >>= 1) {
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    if (lane & off) lead = false;
  }
}

// factor entries in flight: columns per thread (up), blocks of `cols` columns times 32-row steps per warp (down).
// Bounded by the 96 registers of a thread with two CTAs per SM: one more step spills.  Complex64 groups with eight
// columns in flight instead of four: salt body 128^3 x 8 46.6 -> 44.8 ms, 88^3 x 8 18.3 -> 18.2 ms.
template <typename T, int RG>
struct Tile {
  static constexpr bool wide = sizeof(T) == 16;
  static constexpr int up = wide ? (RG == 1 ? 2 : 4) : 8;
  static constexpr int cols = RG == 8 ? 2 : 4;
  static constexpr int down = RG >= 2 ? 1 : (wide ? 1 : 2);
};

// up-the-tree task: rows [r0, r1) of one front, one right-hand-side group.
// phase 0 gathers w_S (zero-extended input + children's updates) and, for rows r < s, writes
// x_r = D^{-1} y_r with y_S = inv(L_TL) w_S (and y_r itself into xb when the second phase needs it);
// for rows r >= s it writes the update w_U - M_BL w_S (extended selective inversion).
// phase 1 (factors keeping L_BL) takes y_S from xb and writes the update w_U - L_BL y_S of rows r >= s.
//
// Thread (i, grp) sums row r0 + i over the columns grp, grp + ngrp, ...
template <typename T, int RG, int PHASE, bool EXT>
__device__ __forceinline__ void fwd_task(const TaskSlot<T>& sl, const SweepArgs<T>& a, const Group gr, unsigned char* smem) {
  constexpr int SP = entry_stride<T, RG>(), U = Tile<T, RG>::up;
  const int tid = threadIdx.x;
  T* own = reinterpret_cast<T*>(smem);            // the task's rows' own entries: w_r, r < s, or w_U
  T* part = own + kComputeThreads * RG;           // partial sums, (group, row, right-hand side)
  T* w = part + kComputeThreads * RG;             // chunk x SP: w_S (or y_S)
  const int trl = sl.tr_log, ngrp = kComputeThreads >> trl, grp = tid >> trl;
  const int s = sl.fr.s, r0 = sl.e.r0, jend = min(sl.e.r1, s);   // jend: entries of w_S this task needs
  const int r = r0 + (tid & ((1 << trl) - 1));
  for (int p = max(r0, s) + tid; p < sl.e.r1; p += kComputeThreads) {
    const int4 ix = sl.own[p - r0];
    T v[RG];
    pull_entries<T, RG>(sl, a.upd_ld, gr, ix.y, ix.z, v);
#pragma unroll
    for (int q = 0; q < RG; ++q) own[(p - r0) * RG + q] = v[q];
  }
  T acc[RG];
#pragma unroll
  for (int q = 0; q < RG; ++q) acc[q] = CplxTraits<T>::zero();
  const int jmax = r < sl.e.r1 ? min(r, s) : 0;   // strictly lower part of inv(L_TL), all of the bottom block
  for (int j0 = 0; j0 < jend; j0 += a.chunk) {
    const int j1 = min(j0 + a.chunk, jend);
    if (j0 > 0) compute_sync();   // the previous chunk is consumed
    for (int p = j0 + tid; p < j1; p += kComputeThreads) {
      T v[RG];
      if constexpr (PHASE == 0) {
        const int4 ix = p < kGatherIdx ? sl.rows[p] : __ldg(sl.rows_g + p);
        T t[RG];
        input_entry<T, RG>(sl, gr, ix.x, t);
        pull_entries<T, RG>(sl, a.upd_ld, gr, ix.y, ix.z, v);
#pragma unroll
        for (int q = 0; q < RG; ++q) v[q] = cadd(v[q], t[q]);
      } else {
        load_entry<T, RG>(sl.xb, a.n_loc, sl.fr.first + p, gr, v);
      }
#pragma unroll
      for (int q = 0; q < RG; ++q) w[(p - j0) * SP + q] = v[q];
      if (p >= r0)
#pragma unroll
        for (int q = 0; q < RG; ++q) own[(p - r0) * RG + q] = v[q];
    }
    compute_sync();
    const int jm = min(jmax, j1), ld = s + sl.fr.u;
    int j = j0 + grp;
    const T* Gp = sl.G + (int64_t)j * ld + r;
    const T* wp = w + (j - j0) * SP;
    for (; j < jm; j += U * ngrp, Gp += (int64_t)U * ngrp * ld, wp += U * ngrp * SP) {
      T g[U];
#pragma unroll
      for (int t = 0; t < U; ++t)
        if (j + t * ngrp < jm) g[t] = __ldg(Gp + t * ngrp * ld);
#pragma unroll
      for (int t = 0; t < U; ++t)
        if (j + t * ngrp < jm) {
          T x[RG];
          load_shared<T, RG>(wp + t * ngrp * SP, x);
#pragma unroll
          for (int q = 0; q < RG; ++q) cfma(acc[q], g[t], x[q]);
        }
    }
  }
  // rows of a warp that several of its lanes share are summed over the lanes first
  const int tr = 1 << trl;
  if (tr < 32) {
#pragma unroll
    for (int q = 0; q < RG; ++q)
      for (int off = tr; off < 32; off <<= 1) {
        acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, off);
        acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, off);
      }
  }
  if (tr >= 32 || (tid & 31) < tr) {
    T* out = part + ((tr < 32 ? (tid >> 5) * tr + (tid & 31) : tid) * RG);
#pragma unroll
    for (int q = 0; q < RG; ++q) out[q] = acc[q];
  }
  const int nparts = tr < 32 ? kComputeWarps : ngrp;
  compute_sync();
  const int rows = sl.e.r1 - sl.e.r0;
  for (int o = tid; o < rows * RG; o += kComputeThreads) {
    const int ro = sl.e.r0 + o / RG, q = o % RG;
    T sum = part[o];
    for (int g2 = 1; g2 < nparts; ++g2) sum = cadd(sum, part[(g2 << trl) * RG + o]);
    if (RG > 1 && q >= gr.w) continue;
    if (ro < sl.fr.s) {
      const T y = cadd(sum, own[o]);
      const T d = __ldg(sl.dinv + ro);
      entry_ptr<T, RG>(sl.xf, a.n_loc, sl.fr.first + ro, gr)[q] = cmul(y, d);
      if (!EXT) entry_ptr<T, RG>(sl.xb, a.n_loc, sl.fr.first + ro, gr)[q] = y;
    } else {
      entry_ptr<T, RG>(sl.upd, a.upd_ld, sl.fr.upd_off + (ro - sl.fr.s), gr)[q] = csub(own[o], sum);
    }
  }
}

__device__ __forceinline__ float2 from_lane(const float2 v, const int l) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
__device__ __forceinline__ double2 from_lane(const double2 v, const int l) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}

// Substitution through a 32 x 32 diagonal block by one warp, lane k holding row (up) or column (down) b + k of the vector in
// registers.  The block's entries are read tri_cols columns at a time before they are used: read one by one, each is a trip
// to L2 in the chain of 32, and with two CTAs per SM too few other fronts hide it.  One application without inversion, lens
// models, read one by one -> so (before the warps had roles, with four CTAs per SM): 48^3 complex64 28.1 -> 14.6 ms (22.6),
// 100^3 complex64 179.6 -> 97.9 (128.5), 100^3 complex128 364.6 -> 268.5 (339.0).  Complex128 leaves out columns that no lane
// needs, whose operations the FP64 pipe would run all the same (14^3 x 8 8.57 -> 7.62 ms, 72^3 x 8 772 -> 742); in
// complex64 the branches cost more than they save (72^3 x 8 74.1 -> 79.2).
template <typename T>
constexpr int tri_cols() { return sizeof(T) == 8 ? 16 : 8; }

// Without inversion (G keeps L_TL): the first phase up the tree of front sn by one CTA: w_S gathered
// as above, then forward substitution y_S = L_TL^{-1} w_S in blocks of 32 columns (one warp solves
// the diagonal block, all threads update the rows below it), x_S = D^{-1} y_S into xf, y_S into xb.
// The vector, RG x s entries (right-hand side major), is in shared memory or, for a front too wide for it (WIDE), in the
// front's own entries of xb, which no other task reads or writes before this one is done.
template <typename T, int RG, bool WIDE>
__device__ __noinline__ void fwd_tri_task(const TaskSlot<T>& sl, const SweepArgs<T>& a, const Group gr) {
  extern __shared__ __align__(16) unsigned char smem[];
  T* const w = WIDE ? entry_ptr<T, RG>(sl.xb, a.n_loc, sl.fr.first, gr) : reinterpret_cast<T*>(smem);
  const int s = sl.fr.s, ld = s + sl.fr.u;
  const T* G = sl.G;
  const int tid = threadIdx.x;
  for (int p = tid; p < s; p += kComputeThreads) {
    const int4 ix = p < kGatherIdx ? sl.rows[p] : __ldg(sl.rows_g + p);
    T v[RG], t[RG];
    input_entry<T, RG>(sl, gr, ix.x, t);
    pull_entries<T, RG>(sl, a.upd_ld, gr, ix.y, ix.z, v);
#pragma unroll
    for (int q = 0; q < RG; ++q) w[q * s + p] = cadd(v[q], t[q]);
  }
  compute_sync();
  const int lane = tid & 31, warp = tid >> 5;
  for (int b = 0; b < s; b += 32) {
    const int be = min(b + 32, s);
    if (warp == 0) {
      // diagonal block: y_j final, then w_k -= L[k, j] y_j for b <= j < k < be
      constexpr int JB = tri_cols<T>();
      const int k = b + lane;
      T v[RG];
#pragma unroll
      for (int q = 0; q < RG; ++q) v[q] = k < be ? w[q * s + k] : CplxTraits<T>::zero();
      for (int j0 = b; j0 < be; j0 += JB) {
        T l[JB];
#pragma unroll
        for (int t = 0; t < JB; ++t)
          l[t] = (k > j0 + t && k < be) ? __ldg(G + (int64_t)(j0 + t) * ld + k) : CplxTraits<T>::zero();
#pragma unroll
        for (int t = 0; t < JB; ++t) {
          if (sizeof(T) == 16 && j0 + t >= be - 1) break;   // no row below it
#pragma unroll
          for (int q = 0; q < RG; ++q) {
            const T y = from_lane(v[q], j0 + t - b);
            if (k > j0 + t && k < be) cfms(v[q], l[t], y);
          }
        }
      }
      if (k < be)
#pragma unroll
        for (int q = 0; q < RG; ++q) w[q * s + k] = v[q];
    }
    compute_sync();
    // rows below the block: w_i -= sum_{j in block} L[i, j] y_j
    for (int i = be + tid; i < s; i += kComputeThreads) {
      T acc[RG];
#pragma unroll
      for (int q = 0; q < RG; ++q) acc[q] = CplxTraits<T>::zero();
#pragma unroll 8
      for (int j = b; j < be; ++j) {
        const T l = __ldg(G + (int64_t)j * ld + i);
#pragma unroll
        for (int q = 0; q < RG; ++q) cfma(acc[q], l, w[q * s + j]);
      }
#pragma unroll
      for (int q = 0; q < RG; ++q) w[q * s + i] = csub(w[q * s + i], acc[q]);
    }
    compute_sync();
  }
  for (int r = tid; r < s; r += kComputeThreads) {
    const T dinv = __ldg(sl.dinv + r);
#pragma unroll
    for (int q = 0; q < RG; ++q)
      if (q < gr.w) {
        entry_ptr<T, RG>(sl.xb, a.n_loc, sl.fr.first + r, gr)[q] = w[q * s + r];
        entry_ptr<T, RG>(sl.xf, a.n_loc, sl.fr.first + r, gr)[q] = cmul(w[q * s + r], dinv);
      }
  }
}

// position of a box node in the problem's vector block, -1 over the pad (Alg. 1.3 extraction)
__device__ __forceinline__ int64_t extracted(const StepRec& st, const int node) {
  const int own = node - st.lead * st.plane;
  return own < 0 ? -1 : (int64_t)st.plane * st.z0 + own;
}

// the final write of column q of x_S entry c of a front: xb (elimination order) and, for the panel's own planes,
// the global vector at g (assigned in the forward sweep, subtracted from `old` in the backward sweep)
template <typename T, int RG>
__device__ __forceinline__ void write_solution(const TaskSlot<T>& sl, const SweepArgs<T>& a, const Group gr, const int entry,
                                               const int q, const int64_t g, const double2 old, const T out) {
  entry_ptr<T, RG>(sl.xb, a.n_loc, entry, gr)[q] = out;
  if (g >= 0) {
    const double2 o = to_c128(out);
    sl.u[(int64_t)(gr.g * RG + q) * sl.st.N + g] = sl.st.mode == 0 ? o : csub(old, o);
  }
}
template <typename T, int RG>
__device__ __forceinline__ double2 old_solution(const TaskSlot<T>& sl, const Group gr, const int q, const int64_t g) {
  return g >= 0 && sl.st.mode != 0 ? __ldcg(sl.u + (int64_t)(gr.g * RG + q) * sl.st.N + g) : make_double2(0.0, 0.0);
}

// down-the-tree task: columns [r0, r1) of S of front sn.
//   extended factors (phase 0): x_c = xf_c + sum_{r > c} G[r, c] y_r over all s + u rows, with
//     y = xf on S and -x_U on the struct rows; writes the solution.
//   factors keeping L_BL, phase 0: t_c = xf_c - sum_{r >= s} L_BL[r, c] x_U[r] into xf.
//   paper's factors, phase 1: x_c = t_c + sum_{c < r < s} inv(L_TL)[r, c] t_r; writes the solution.
//
// A warp carries blocks of four adjacent columns, its lanes over the rows, so an entry of y serves four columns;
// tasks of few columns split their rows over the warps instead.  Which rows a lane sums depends on the task alone
// (quads of columns, steps of 32 rows) where a front's vector is staged in one chunk, and then every RG gives a column the
// same bits, as up the tree.  A front wider than a chunk (384 entries at eight complex64 columns, 7,680 at one) is summed
// chunk by chunk, so there the groups differ by the rounding of another order.
template <typename T, int RG, int PHASE, bool EXT>
__device__ __forceinline__ void bwd_task(const TaskSlot<T>& sl, const SweepArgs<T>& a, const Group gr, unsigned char* smem) {
  using Real = typename CplxTraits<T>::real;
  constexpr int SP = entry_stride<T, RG>(), CB = Tile<T, RG>::cols, U = Tile<T, RG>::down;
  constexpr bool writes = EXT || PHASE == 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int s = sl.fr.s, c0 = sl.e.r0, nc = sl.e.r1 - c0;
  // rows of the inner sums: [lo, hi), passed through shared memory in chunks of a.chunk rows
  const int lo = writes ? c0 : s, hi = (EXT || PHASE == 0) ? s + sl.fr.u : s;
  T* part = reinterpret_cast<T*>(smem);         // column sums, (split, column, right-hand side)
  T* y = part + 2 * kComputeThreads * RG;       // chunk x SP
  const int nb = (nc + CB - 1) / CB, splits = sl.splits;   // blocks of CB columns, warps that share a block's rows
  // this thread's first output: its own entry and, where the solution is written, its place and (backward sweep) the
  // old value there are read before the products
  T own0 = CplxTraits<T>::zero();
  int64_t g0 = -1;
  double2 old0 = make_double2(0.0, 0.0);
  if (tid < nc * RG && (RG == 1 || tid % RG < gr.w)) {
    own0 = __ldcg(entry_ptr<T, RG>(sl.xf, a.n_loc, sl.fr.first + c0 + tid / RG, gr) + tid % RG);
    if (writes) {
      g0 = extracted(sl.st, __ldg(sl.rows_g + c0 + tid / RG).x);
      old0 = old_solution<T, RG>(sl, gr, tid % RG, g0);
    }
  }
  for (int rb = lo; rb < hi; rb += a.chunk) {
    const int re = min(rb + a.chunk, hi);
    if (rb > lo) compute_sync();   // the previous chunk is consumed
    constexpr int GU = RG >= 2 ? 1 : 2;
    for (int p0 = rb + tid; p0 < re; p0 += GU * kComputeThreads) {
      T v[GU][RG];
#pragma unroll
      for (int t = 0; t < GU; ++t) {
        const int r = p0 + t * kComputeThreads;
        if (r < re) {
          const int k = r - s;
          const int e = k < 0 ? sl.fr.first + r
                              : (k < 4 * kGatherIdx ? reinterpret_cast<const int32_t*>(sl.rows)[k] : __ldg(sl.sel_g + k));
          load_entry<T, RG>(k < 0 ? sl.xf : sl.xb, a.n_loc, e, gr, v[t]);
        }
      }
#pragma unroll
      for (int t = 0; t < GU; ++t) {
        const int r = p0 + t * kComputeThreads;
        if (r < re)
#pragma unroll
          for (int q = 0; q < RG; ++q) y[(r - rb) * SP + q] = r < s ? v[t][q] : cneg(v[t][q]);
      }
    }
    compute_sync();
    // the columns the inner sums read: G's, or in the two-inverse form's second phase the second inverse of L_TL
    // (s x s after G), which was built row by row for this direction
    const bool second = PHASE == 1 && a.si == PSP_SI_TWO;
    const T* Gs = second ? sl.G + second_inverse_offset(s, sl.fr.u) : sl.G;
    const int lds = second ? s : s + sl.fr.u;
    const int step = 32 * splits;
    for (int wb = warp; wb < nb * splits; wb += kComputeWarps) {
      const int b = splits > 1 ? wb % nb : wb, sp = splits > 1 ? wb / nb : 0;
      const int c = c0 + b * CB, ncb = min(CB, c0 + nc - c);
      Real acc[CB * RG * 2];
#pragma unroll
      for (int k = 0; k < CB * RG * 2; ++k) acc[k] = Real(0);
      int r = max(rb, c0 + ((c - c0) & ~3) + 1) + sp * 32 + lane;
      const T* Gp = Gs + (int64_t)c * lds + r;
      const T* yp = y + (r - rb) * SP;
      for (; r < re; r += U * step, Gp += U * step, yp += U * step * SP) {
        T g[U][CB];
#pragma unroll
        for (int t = 0; t < U; ++t)
#pragma unroll
          for (int k = 0; k < CB; ++k)   // rows below each column's diagonal
            if (k < ncb && r + step * t < re && r + step * t > c + k) g[t][k] = __ldg(Gp + k * lds + step * t);
#pragma unroll
        for (int t = 0; t < U; ++t)
          if (r + step * t < re) {
            T x[RG];
            load_shared<T, RG>(yp + step * t * SP, x);
#pragma unroll
            for (int k = 0; k < CB; ++k)
              if (k < ncb && r + step * t > c + k)
#pragma unroll
                for (int q = 0; q < RG; ++q) {
                  T s2;
                  s2.x = acc[(k * RG + q) * 2];
                  s2.y = acc[(k * RG + q) * 2 + 1];
                  cfma(s2, g[t][k], x[q]);
                  acc[(k * RG + q) * 2] = s2.x;
                  acc[(k * RG + q) * 2 + 1] = s2.y;
                }
          }
      }
      int base;
      bool lead;
      warp_sum<Real, CB * RG * 2>(acc, lane, base, lead);
      if (lead) {
        constexpr int per = CB * RG * 2 > 32 ? CB * RG * 2 / 32 : 1;
        Real* out = reinterpret_cast<Real*>(part + (sp * nb * CB + b * CB) * RG);
#pragma unroll
        for (int k = 0; k < per; ++k) out[base + k] = rb == lo ? acc[k] : out[base + k] + acc[k];
      }
    }
  }
  compute_sync();
  for (int o = tid; o < nc * RG; o += kComputeThreads) {
    const int c = o / RG, q = o % RG;
    if (RG > 1 && q >= gr.w) continue;
    const int entry = sl.fr.first + c0 + c;
    T v = o == tid ? own0 : __ldcg(entry_ptr<T, RG>(sl.xf, a.n_loc, entry, gr) + q);
    if (hi > lo)
      for (int sp = 0; sp < splits; ++sp) v = cadd(v, part[sp * nb * CB * RG + o]);
    if constexpr (!writes) {   // t_c
      entry_ptr<T, RG>(sl.xf, a.n_loc, entry, gr)[q] = v;
    } else {
      int64_t g = g0;
      double2 old = old0;
      if (o != tid) {
        g = extracted(sl.st, __ldg(sl.rows_g + c0 + c).x);
        old = old_solution<T, RG>(sl, gr, q, g);
      }
      write_solution<T, RG>(sl, a, gr, entry, q, g, old, v);
    }
  }
}

// Without inversion: the second phase down the tree of front sn by one CTA: back substitution
// L_TL^T x_S = t (t in xf) in blocks of 32 columns from the last, each block first takes the
// products with the solved rows below it (one warp per column), then one warp solves the block.
template <typename T, int RG, bool WIDE>
__device__ __noinline__ void bwd_tri_task(const TaskSlot<T>& sl, const SweepArgs<T>& a, const Group gr) {
  extern __shared__ __align__(16) unsigned char smem[];
  // RG x s entries (right-hand side major) as in fwd_tri_task: t, overwritten by x block by block
  T* const x = WIDE ? entry_ptr<T, RG>(sl.xb, a.n_loc, sl.fr.first, gr) : reinterpret_cast<T*>(smem);
  const int s = sl.fr.s, ld = s + sl.fr.u;
  const T* G = sl.G;
  const int tid = threadIdx.x;
  for (int r = tid; r < s; r += kComputeThreads) {
    T v[RG];
    load_entry<T, RG>(sl.xf, a.n_loc, sl.fr.first + r, gr, v);
#pragma unroll
    for (int q = 0; q < RG; ++q) x[q * s + r] = v[q];
  }
  compute_sync();
  const int lane = tid & 31, warp = tid >> 5;
  const int nblk = (s + 31) / 32;
  for (int bi = nblk - 1; bi >= 0; --bi) {
    const int b = bi * 32, be = min(b + 32, s);
    // x_c -= sum_{r >= be} L[r, c] x_r for the block's columns
    for (int c = b + warp; c < be; c += kComputeWarps) {
      T acc[RG];
#pragma unroll
      for (int q = 0; q < RG; ++q) acc[q] = CplxTraits<T>::zero();
      for (int r = be + lane; r < s; r += 32) {
        const T l = __ldg(G + (int64_t)c * ld + r);
#pragma unroll
        for (int q = 0; q < RG; ++q) cfma(acc[q], l, x[q * s + r]);
      }
#pragma unroll
      for (int q = 0; q < RG; ++q) {
        for (int off = 16; off > 0; off >>= 1) {
          acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, off);
          acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, off);
        }
        if (lane == 0) x[q * s + c] = csub(x[q * s + c], acc[q]);
      }
    }
    compute_sync();
    if (warp == 0) {
      // the block, from its last column: x_c final, then x_k -= L[c, k] x_c for b <= k < c
      constexpr int JB = tri_cols<T>();
      const int k = b + lane;
      T v[RG];
#pragma unroll
      for (int q = 0; q < RG; ++q) v[q] = k < be ? x[q * s + k] : CplxTraits<T>::zero();
      for (int c0 = b + 32 - JB; c0 >= b; c0 -= JB) {
        T l[JB];
#pragma unroll
        for (int t = 0; t < JB; ++t)
          l[t] = (k < c0 + t && c0 + t < be) ? __ldg(G + (int64_t)k * ld + c0 + t) : CplxTraits<T>::zero();
#pragma unroll
        for (int t = JB - 1; t >= 0; --t) {
          if (sizeof(T) == 16 && (c0 + t >= be || c0 + t == b)) continue;   // beyond the block, or no column before it
#pragma unroll
          for (int q = 0; q < RG; ++q) {
            const T y = from_lane(v[q], c0 + t - b);
            if (k < c0 + t && c0 + t < be) cfms(v[q], l[t], y);
          }
        }
      }
      if (k < be)
#pragma unroll
        for (int q = 0; q < RG; ++q) x[q * s + k] = v[q];
    }
    compute_sync();
  }
  for (int c = tid; c < s; c += kComputeThreads) {
    const int64_t g = extracted(sl.st, __ldg(sl.rows_g + c).x);
#pragma unroll
    for (int q = 0; q < RG; ++q)
      if (q < gr.w) write_solution<T, RG>(sl, a, gr, sl.fr.first + c, q, g, old_solution<T, RG>(sl, gr, q, g), x[q * s + c]);
  }
}

// ---------------------------------------------------------------------------
// The whole sweep of Alg. 1.5 in one cooperative launch, as a dataflow over the elimination trees.
// CTAs take tasks from one queue in topological order.  An up-the-tree task of a front waits until
// every task of its children has finished (one counter per front, which its children's tasks
// increment); a front without children waits for the previous panel solve of its problem's chain: for the
// same front's down tasks there when both boxes have the same tree (its input is read at its own (x, y) only,
// and every work entry it overwrites has then been read), else for the whole solve.  (The chains of a batch of
// independent problems are interleaved in the queue and run side by side.)  A down-the-tree task waits for its
// parent (the root: for its own up-the-tree tasks).  A task only waits on tasks earlier in the queue.  A
// CTA claims its tasks in queue order, a few ahead of the task it runs; the earliest unfinished
// task is therefore the one some CTA runs (a CTA holding it only as a later task would be running an
// earlier unfinished one), every task it waits for has finished, and since every CTA of a
// cooperative launch is resident, the sweep progresses.  Each wait is bounded anyway: a CTA that
// gives up sets status[2] and stops; the others then give up at their next wait.
//
// A CTA's warps have three roles, so that the latencies around a task's products overlap with the products of
// the task before it.  A scheduling warp claims the next task, reads its records, copies the index words its
// gathers need into shared memory, warms L2 with its factor block and waits for its dependency; eight product
// warps gather, multiply and write; a signalling warp makes a finished task's writes visible and counts it.
// Tasks alternate between two slots.
//
// What bounds it: in complex128 the FP64 pipe (2 FMAs per clock and SM, 4 per factor entry and column) together with
// the chain of levels; in complex64 the chain, about 3 us of gather and reduction per task around its products, and
// with many columns the shared-memory reads of the gathered vector.  With all of a CTA's warps doing every role in
// turn a task took about 8 us for 2.6 us of products.  Two CTAs of 320 threads per SM (96 registers); three with
// 64 registers spill.  One application, all roles in turn -> as it is: 100^3 lens complex128 51.6 -> 33.9 ms (25.4 ms
// of FP64), complex64 15.2 -> 11.5 ms (4.1 ms of HBM), 88^3 complex64 x 8 40.3 -> 18.2 ms, salt body 128^3 x 8
// 65.7 -> 44.8 ms, 20^3 complex128 1.07 -> 0.70 ms.
// ---------------------------------------------------------------------------
constexpr long long kWaitCycles = 4000000000LL;   // SM clock cycles: about two seconds at 2 GHz
constexpr long long kWaitSpins = 400000000LL;     // and a hard cap on polls, whatever the clock does

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// a wait that gives up sets status[2] (cleared before every sweep) and the handle's sticky flag
// (cleared only when the host reads it)
__device__ __forceinline__ bool wait_count(const unsigned* p, unsigned target, int* status, int* sticky) {
  if (load_acquire(p) >= target) return true;
  const long long t0 = clock64();
  long long it = 0;
  for (;;) {
    if (load_acquire(p) >= target) return true;
    if ((++it & 15) == 0) {
      if (*(volatile int*)(status + 2) != 0) return false;
      if (it > kWaitSpins || clock64() - t0 > kWaitCycles) {
        atomicExch(status + 2, 1);
        if (sticky) atomicExch(sticky, 1);
        return false;
      }
    }
    __nanosleep(20);
  }
}

// Warm L2 with the factor lines a task will stream, while its dependencies are still being
// waited for (the lines do not depend on them): up the tree rows [r0, r1) of the columns
// j < min(r1, s), down the tree columns [c0, c1) from below their diagonal to the end.  One warp, at most
// kPrefetchLines lines (the product reads the rest itself).  1024 lines: 40 MB over 304 CTAs; with 2048 those of large tasks
// push each other out of L2 before they are read (one complex64 column, layered models: 176^3 85.4 / 83.3 ms, 200^3 134.4 /
// 128.1; salt body 128^3 x 8 45.3 / 44.7; no difference up to 160^3), with 512 smaller ones arrive late (100^3 14.5 / 14.9)
constexpr int kPrefetchLines = 1024;

template <typename T>
__device__ __forceinline__ void prefetch_task(const TaskSlot<T>& sl, const SweepArgs<T>& a, const int lane) {
  const int s = sl.fr.s, u = sl.fr.u, ld = s + u, dir = sl.e.dir, r0 = sl.e.r0, r1 = sl.e.r1;
  const char* G = reinterpret_cast<const char*>(sl.G);
  constexpr int kLine = 128;
  if (dir == 0 || dir == kDirUpB) {
    const int ncol = min(r1, s);
    const int seg = (r1 - r0) * (int)sizeof(T);
    const int lines = (seg + kLine - 1) / kLine + 1;   // the segment may straddle one more line
    const int total = min(ncol * lines, kPrefetchLines);
    for (int w = lane; w < total; w += 32) {
      const int j = w / lines, l = w - j * lines;
      const char* col = G + ((int64_t)j * ld + r0) * sizeof(T);
      if (l * kLine < seg) asm volatile("prefetch.global.L2 [%0];" ::"l"(col + (int64_t)l * kLine));
    }
  } else {
    const bool second = dir == kDirDownB && a.si == PSP_SI_TWO;   // the second inverse after G
    const char* Gs = second ? G + second_inverse_offset(s, u) * sizeof(T) : G;
    const int lds = second ? s : ld;
    int left = kPrefetchLines;
    for (int c = r0; c < r1 && left > 0; ++c) {
      const char* col = Gs + ((int64_t)c * lds + c + 1) * sizeof(T);
      const int64_t seg = (int64_t)(lds - c - 1) * sizeof(T);
      for (int64_t off = (int64_t)lane * kLine; off < seg; off += 32 * kLine)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(col + off));
      left -= (int)(seg / kLine) + 1;
    }
  }
}

// asynchronous copies global -> shared (completed by cp_async_wait_all of the same thread)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// the scheduling warp: task after task into alternating slots
template <typename T>
__device__ __forceinline__ void schedule(TaskSlot<T>* slots, const SweepArgs<T>& a, const int lane) {
  constexpr int kEntryWords = sizeof(QueueEntry) / 4, kStepWords = sizeof(StepRec) / 4, kFrontWords = sizeof(FrontRec) / 4;
  static_assert(kEntryWords <= 32 && kStepWords <= 32 && kFrontWords <= 32, "records are copied one word per lane");
  const bool early = a.claim_ahead > 1;   // claim the next task before the slot it will use is free
  auto claim = [&] {
    int v = 0;
    if (lane == 0) v = (int)atomicAdd(a.ctr, 1u);
    return __shfl_sync(0xffffffffu, v, 0);
  };
  int next = early ? claim() : 0;
  for (int n = 0;; ++n) {
    TaskSlot<T>& sl = slots[n & 1];
    int idx = next;
    int ew = 0;
    if (early && idx < a.nqueue && lane < kEntryWords) ew = __ldg(reinterpret_cast<const int*>(a.queue + idx) + lane);
    if (n >= 2) bar_sync(kBarFree + (n & 1), 64);   // the slot's last task has been signalled
    if (!early) {
      idx = claim();
      if (idx < a.nqueue && lane < kEntryWords) ew = __ldg(reinterpret_cast<const int*>(a.queue + idx) + lane);
    }
    bool ok = idx < a.nqueue;
    if (ok) {
      if (lane < kEntryWords) reinterpret_cast<int*>(&sl.e)[lane] = ew;
      __syncwarp();
      int sw = 0, fw = 0;
      if (lane < kStepWords) sw = __ldg(reinterpret_cast<const int*>(a.steps + sl.e.step) + lane);
      if (lane < kFrontWords) fw = __ldg(reinterpret_cast<const int*>(a.fronts + sl.e.front) + lane);
      if (early) next = claim();
      if (lane < kStepWords) reinterpret_cast<int*>(&sl.st)[lane] = sw;
      if (lane < kFrontWords) reinterpret_cast<int*>(&sl.fr)[lane] = fw;
      __syncwarp();
      const int dir = sl.e.dir, r0 = sl.e.r0, r1 = sl.e.r1, s = sl.fr.s, u = sl.fr.u;
      const int4* rows = sl.st.rows + sl.fr.row_off;
      const int32_t* sel = sl.st.sel + sl.fr.sel_off;
      if (lane == 0) {
        int tl = 1;
        while ((1 << tl) < r1 - r0 && (1 << tl) < kComputeThreads) ++tl;
        sl.tr_log = tl;
        int sp = 1;
        while (2 * sp * ((r1 - r0 + 3) / 4) <= kComputeWarps) sp <<= 1;
        sl.splits = sp;
        sl.G = a.factor + sl.st.gbase + sl.fr.g_off;
        sl.dinv = a.dinv + sl.st.dbase + sl.fr.first;
        sl.rows_g = rows;
        sl.sel_g = sel;
        const int64_t box = (int64_t)sl.st.prob * a.n_loc * a.nrhs;
        sl.xf = a.xf + box;
        sl.xb = a.xb + box;
        sl.upd = a.upd + (int64_t)sl.st.prob * a.upd_ld * a.nrhs;
        sl.u = a.u + sl.st.off1 * a.nrhs;
      }
      __syncwarp();
      const bool up = dir == 0 || dir == kDirUpB, tri = a.si == PSP_SI_NONE && (dir == 0 || dir == kDirDownB);
      if (dir == 0) {
        for (int p = lane; p < min(min(r1, s), kGatherIdx); p += 32) cp_async16(&sl.rows[p], rows + p);
      } else if (dir == 1) {
        int32_t* dst = reinterpret_cast<int32_t*>(sl.rows);
        for (int p = lane; p < min(u, 4 * kGatherIdx); p += 32) cp_async4(dst + p, sel + p);
      }
      if (up && !tri)
        for (int p = max(r0, s) + lane; p < r1; p += 32) cp_async16(&sl.own[p - r0], rows + p);
      prefetch_task<T>(sl, a, lane);
      int got = 1;
      if (lane == 0 && sl.e.wait >= 0) got = wait_count(a.ctr + sl.e.wait, sl.e.target, a.status, a.sticky);
      ok = __shfl_sync(0xffffffffu, got, 0) != 0;
      __threadfence();
      cp_async_wait_all();
    }
    if (lane == 0) sl.ok = ok;
    __syncwarp();
    bar_arrive(kBarReady + (n & 1), kComputeThreads + 32);
    if (!ok) break;
  }
}

// the signalling warp: a finished task's completion counters
template <typename T>
__device__ __forceinline__ void signal_done(TaskSlot<T>* slots, const SweepArgs<T>& a, const int lane) {
  for (int n = 0;; ++n) {
    TaskSlot<T>& sl = slots[n & 1];
    bar_sync(kBarDone + (n & 1), kComputeThreads + 32);
    if (!sl.ok) break;
    if (lane < 3) {
      __threadfence();   // the product warps' writes, ordered before this by the barrier, become visible first
      const int c = lane == 0 ? sl.e.done : (lane == 1 ? sl.e.kids : sl.e.step_done);
      if (c >= 0) atomicAdd(a.ctr + c, 1u);
    }
    __syncwarp();
    bar_arrive(kBarFree + (n & 1), 64);
  }
}

// FORM: extended selective inversion (one task per front and direction), the forms that keep L_BL and inverses of L_TL, or no
// inversion.  A kernel for each, so that none holds registers for another's tasks.
// The registers are held to sweep_ctas CTAs per SM (65,536 / (320 threads x CTAs)).
template <typename T, int RG>
constexpr int sweep_ctas() { return 2; }

enum SweepForm { kFormExtended, kFormInverse, kFormNone };

template <typename T, int RG, int FORM>
__global__ void __launch_bounds__(kSweepThreads, (sweep_ctas<T, RG>())) k_sweep(const __grid_constant__ SweepArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(16) TaskSlot<T> slots[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == kComputeWarps) {
    schedule<T>(slots, a, lane);
    return;
  }
  if (warp == kComputeWarps + 1) {
    signal_done<T>(slots, a, lane);
    return;
  }
  const int nrg = (a.nrhs + RG - 1) / RG;
  for (int n = 0;; ++n) {
    const TaskSlot<T>& sl = slots[n & 1];
    bar_sync(kBarReady + (n & 1), kComputeThreads + 32);
    const bool ok = sl.ok;
    if (ok) {
      for (int g = 0; g < nrg; ++g) {
        Group gr{g, min(RG, a.nrhs - g * RG), false};
        if (RG > 1)
          gr.vec = gr.w == RG && ((reinterpret_cast<uintptr_t>(sl.xf + g * RG * a.n_loc) |
                                   reinterpret_cast<uintptr_t>(sl.xb + g * RG * a.n_loc) |
                                   reinterpret_cast<uintptr_t>(sl.upd + g * RG * a.upd_ld)) & 15) == 0;
        if (g > 0) compute_sync();
        const int dir = sl.e.dir;
        if constexpr (FORM == kFormExtended) {
          if (dir == 0) fwd_task<T, RG, 0, true>(sl, a, gr, smem);
          else bwd_task<T, RG, 0, true>(sl, a, gr, smem);
        } else {
          if (dir == 0) {
            if constexpr (FORM == kFormInverse) fwd_task<T, RG, 0, false>(sl, a, gr, smem);
            else if (RG == 1 && a.tri_global) fwd_tri_task<T, 1, true>(sl, a, gr);
            else fwd_tri_task<T, RG, false>(sl, a, gr);
          } else if (dir == kDirUpB) {
            fwd_task<T, RG, 1, false>(sl, a, gr, smem);
          } else if (dir == 1) {
            bwd_task<T, RG, 0, false>(sl, a, gr, smem);
          } else {
            if constexpr (FORM == kFormInverse) bwd_task<T, RG, 1, false>(sl, a, gr, smem);
            else if (RG == 1 && a.tri_global) bwd_tri_task<T, 1, true>(sl, a, gr);
            else bwd_tri_task<T, RG, false>(sl, a, gr);
          }
        }
      }
    }
    bar_arrive(kBarDone + (n & 1), kComputeThreads + 32);
    if (!ok) break;
  }
}

template <typename T, int RG, int FORM>
static int sweep_rg(const SweepArgs<T>& args, size_t smem, int max_per_sm, SweepFit* fit, cudaStream_t st) {
  if (cudaFuncSetAttribute(k_sweep<T, RG, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  int dev = 0, sms = 0, per_sm = 0, coop = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep<T, RG, FORM>, kSweepThreads, smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return -1;
  }
  per_sm = per_sm > max_per_sm ? max_per_sm : per_sm;
  if (fit) {
    *fit = SweepFit{RG, per_sm};
    return 0;
  }
  SweepArgs<T> a = args;
  void* kargs[] = {&a};
  cudaError_t e;
  if (coop) {
    e = cudaLaunchCooperativeKernel((const void*)k_sweep<T, RG, FORM>, dim3(sms * per_sm), dim3(kSweepThreads), kargs, smem, st);
  } else {   // one CTA alone takes the queue in order and never waits
    k_sweep<T, RG, FORM><<<1, kSweepThreads, smem, st>>>(a);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? 0 : (int)e;
}

// A CTA carries RG right-hand sides through each pass over a factor block (as many as nrhs, at most 8 in complex64
// and 4 in complex128, where the FP64 pipe and not the factor's bytes is the bound; or rhs_group when > 0), and the
// vectors of a task pass through shared memory in chunks sized so that two CTAs stay resident per SM (a CTA that
// waits on a dependency leaves the SM to the other).  Substitution tasks (fronts keeping L_TL) hold a front's
// whole vector, so for them RG shrinks until that fits; one column of a front wider than shared memory (13,400 rows in
// complex128) stays in its work vector.
template <typename T, int RG>
constexpr size_t sweep_smem() { return (sizeof(T) == 16 && RG == 4 ? 84 : 64) * 1024; }

template <typename T, int RG>
static int sweep_sized(const SweepArgs<T>& args, int smax, int ldmax, int max_per_sm, SweepFit* fit, cudaStream_t st) {
  constexpr size_t es = sizeof(T), entry = entry_stride<T, RG>() * es, fixed = 2 * (size_t)kComputeThreads * RG * es;
  const int full = ldmax > smax ? ldmax : smax;
  int chunk = (int)((sweep_smem<T, RG>() - fixed) / entry / 64 * 64);
  if (chunk >= full) chunk = full > 0 ? full : 1;   // one chunk: every task's vector at once
  SweepArgs<T> a = args;
  a.chunk = chunk;
  size_t smem = fixed + chunk * entry;
  if (a.si == PSP_SI_NONE) {
    const size_t whole = (size_t)smax * RG * es;
    a.tri_global = RG == 1 && whole + 2 * sizeof(TaskSlot<T>) > 226 * 1024;
    if (!a.tri_global && smem < whole) smem = whole;
  }
  if (a.si == PSP_SI_EXTENDED) return sweep_rg<T, RG, kFormExtended>(a, smem, max_per_sm, fit, st);
  if (a.si == PSP_SI_NONE) return sweep_rg<T, RG, kFormNone>(a, smem, max_per_sm, fit, st);
  return sweep_rg<T, RG, kFormInverse>(a, smem, max_per_sm, fit, st);
}

template <typename T>
static int sweep(const SweepArgs<T>& a, int smax, int ldmax, int max_per_sm, int rhs_group, SweepFit* fit, cudaStream_t st) {
  int rg = sizeof(T) == 8 ? 8 : 4;
  while (rg > 1 && rg >= 2 * a.nrhs) rg >>= 1;
  if (rhs_group > 0)
    while (rg > 1 && rg > rhs_group) rg >>= 1;
  if (a.si == PSP_SI_NONE)
    while (rg > 1 && (size_t)smax * rg * sizeof(T) > 180 * 1024) rg >>= 1;
  switch (rg) {
    case 8:
      if constexpr (sizeof(T) == 8) return sweep_sized<T, 8>(a, smax, ldmax, max_per_sm, fit, st);
    case 4: return sweep_sized<T, 4>(a, smax, ldmax, max_per_sm, fit, st);
    case 2: return sweep_sized<T, 2>(a, smax, ldmax, max_per_sm, fit, st);
    default: return sweep_sized<T, 1>(a, smax, ldmax, max_per_sm, fit, st);
  }
}

template <typename T>
int launch_sweep(const SweepArgs<T>& a, int smax, int ldmax, int max_per_sm, int rhs_group, cudaStream_t st) {
  return sweep<T>(a, smax, ldmax, max_per_sm, rhs_group, nullptr, st);
}
template <typename T>
SweepFit sweep_fit(int nrhs, int si, int smax, int ldmax, int max_per_sm, int rhs_group) {
  SweepArgs<T> a{};
  a.nrhs = nrhs;
  a.si = si;
  SweepFit f;
  sweep<T>(a, smax, ldmax, max_per_sm, rhs_group, &f, nullptr);
  return f;
}

template int launch_sweep<double2>(const SweepArgs<double2>&, int, int, int, int, cudaStream_t);
template int launch_sweep<float2>(const SweepArgs<float2>&, int, int, int, int, cudaStream_t);
template SweepFit sweep_fit<double2>(int, int, int, int, int, int);
template SweepFit sweep_fit<float2>(int, int, int, int, int, int);

// index words of a shape's front rows: row p of front f gets {its box node (p < s, else -1), the two update-vector
// entries its children add to it, 0}, so that a gather reads one 16-byte word per row
__global__ void __launch_bounds__(128) k_build_rows(ShapeDev sh, int4* rows) {
  const int f = blockIdx.x;
  const int s = sh.s[f], n = s + sh.u[f], first = sh.first[f];
  const int64_t o = sh.pull_ptr[f];
  for (int p = threadIdx.x; p < n; p += blockDim.x)
    rows[o + p] = make_int4(p < s ? sh.order[first + p] : -1, sh.pull[2 * (o + p)], sh.pull[2 * (o + p) + 1], 0);
}

void launch_build_rows(const ShapeDev& sh, int4* rows, cudaStream_t st) {
  if (sh.nsn > 0) k_build_rows<<<sh.nsn, 128, 0, st>>>(sh, rows);
}

}  // namespace psp
