// 7-point Helmholtz operators with PML (Eq. (1.1), Eq. (1.5), §1.1): coefficients, the
// complex128 stencil matvec used by GMRES, and batched front assembly + extend-add (§2.2).
#include "cplx.cuh"
#include "psp_internal.h"

namespace psp {

// Row of the s1 s2 s3-scaled operator at box node (x, y, z):
//   a_1(x -+ 1/2) = s2 s3 / s1(x -+ 1/2), a_2, a_3 alike; off-diagonals -a/h^2,
//   diagonal sum(a)/h^2 - k2num / c^2 * s1 s2 s3.
// The BoxOp stores the reciprocal stretches at half-points (s?h fields hold 1/s there).
struct Row7 {
  double2 d, xm, xp, ym, yp, zm, zp;
};

__device__ __forceinline__ Row7 row7(const BoxOp& op, int x, int y, int z) {
  const double2 s1 = op.s1n[x], s2 = op.s2n[y], s3 = op.s3n[z];
  const double2 s23 = cmul(s2, s3), s13 = cmul(s1, s3), s12 = cmul(s1, s2);
  const double2 axm = cmul(s23, op.s1h[x]), axp = cmul(s23, op.s1h[x + 1]);
  const double2 aym = cmul(s13, op.s2h[y]), ayp = cmul(s13, op.s2h[y + 1]);
  const double2 azm = cmul(s12, op.s3h[z]), azp = cmul(s12, op.s3h[z + 1]);
  const double ic2 = op.ic2[((int64_t)op.cplane[z] * op.ny + y) * op.nx + x];
  const double2 mass = cmul(cscale(op.k2num, ic2), cmul(s12, s3));
  Row7 r;
  double2 sum = cadd(cadd(cadd(axm, axp), cadd(aym, ayp)), cadd(azm, azp));
  r.d = csub(cscale(sum, op.inv_h2), mass);
  r.xm = cscale(axm, -op.inv_h2);
  r.xp = cscale(axp, -op.inv_h2);
  r.ym = cscale(aym, -op.inv_h2);
  r.yp = cscale(ayp, -op.inv_h2);
  r.zm = cscale(azm, -op.inv_h2);
  r.zp = cscale(azp, -op.inv_h2);
  return r;
}

// bitwise tests: a floating-point comparison takes the FP64 pipe
__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }
__device__ __forceinline__ bool is_one(double2 v) { return __double_as_longlong(v.x) == 0x3ff0000000000000ll && is_zero(v.y); }

// y = Op x for nrhs vectors (column-major, ld = N); one thread per node.
//
// Bound by the FP64 pipe, not by its 40 bytes per node: the seven complex coefficients of a row and their products took
// about 110 FP64 operations.  Outside an axis' PML its stretches are exactly one; a warp leaves out what that makes
// trivial for all its nodes: with no PML a row needs 15 operations (17 for J), in one axis' PML about 46, and with
// several vectors a PML node 32 more per vector.  The same operations whatever nrhs, so every vector keeps its bits.
// 100^3, one vector: 189 -> 83 us; 61 x 83 x 47, three vectors: 80 -> 56 us.
//
// matvec_rows<ONE1, ONE2, ONE3>: the nodes of a warp, ONEj: axis j's stretches are one for all of them.  A function per
// combination, so that what it leaves out is not computed and then discarded.
template <bool ONE1, bool ONE2, bool ONE3>
__device__ __forceinline__ void matvec_rows(const BoxOp& op, const double2* __restrict__ x, double2* __restrict__ y, int nrhs,
                                            int64_t N, int64_t g, bool in, int xx, int yy, int zz) {
  const int plane = op.nx * op.ny;
  const bool xl = xx > 0, xh = xx + 1 < op.nx, yl = yy > 0, yh = yy + 1 < op.ny, zl = zz > 0, zh = zz + 1 < op.nz;
  const double2 zero = make_double2(0.0, 0.0);
  const double ic2 = op.ic2[(int64_t)op.cplane[zz] * plane + yy * op.nx + xx];
  const bool real_k = is_zero(op.k2num.y);
  constexpr bool kAll = ONE1 && ONE2 && ONE3;
  double2 d;                                    // the diagonal
  double2 m1 = zero, m2 = zero, m3 = zero;      // s2 s3, s1 s3, s1 s2
  double2 a1 = zero, b1 = zero, a2 = zero, b2 = zero, a3 = zero, b3 = zero;   // minus the couplings, times h^2
  if constexpr (kAll) {
    d = make_double2(fma(6.0, op.inv_h2, -op.k2num.x * ic2), -op.k2num.y * ic2);
  } else {
    const double2 one = make_double2(1.0, 0.0);
    const double2 s1 = ONE1 ? one : op.s1n[xx], s2 = ONE2 ? one : op.s2n[yy], s3 = ONE3 ? one : op.s3n[zz];
    m1 = ONE2 ? s3 : (ONE3 ? s2 : cmul(s2, s3));
    m2 = ONE1 ? s3 : (ONE3 ? s1 : cmul(s1, s3));
    m3 = ONE1 ? s2 : (ONE2 ? s1 : cmul(s1, s2));
    double2 sum = zero;
    if constexpr (ONE1) {
      sum = cscale(m1, 2.0);
    } else {
      a1 = op.s1h[xx];
      b1 = op.s1h[xx + 1];
      if constexpr (!(ONE2 && ONE3)) {
        a1 = cmul(m1, a1);
        b1 = cmul(m1, b1);
      }
      sum = cadd(a1, b1);
    }
    if constexpr (ONE2) {
      sum = make_double2(fma(2.0, m2.x, sum.x), fma(2.0, m2.y, sum.y));
    } else {
      a2 = op.s2h[yy];
      b2 = op.s2h[yy + 1];
      if constexpr (!(ONE1 && ONE3)) {
        a2 = cmul(m2, a2);
        b2 = cmul(m2, b2);
      }
      sum = cadd(sum, cadd(a2, b2));
    }
    if constexpr (ONE3) {
      sum = make_double2(fma(2.0, m3.x, sum.x), fma(2.0, m3.y, sum.y));
    } else {
      a3 = op.s3h[zz];
      b3 = op.s3h[zz + 1];
      if constexpr (!(ONE1 && ONE2)) {
        a3 = cmul(m3, a3);
        b3 = cmul(m3, b3);
      }
      sum = cadd(sum, cadd(a3, b3));
    }
    const double2 s123 = ONE1 ? m1 : (ONE2 && ONE3 ? s1 : cmul(s1, m1));
    d = cscale(sum, op.inv_h2);
    if (real_k) {
      const double k = op.k2num.x * ic2;
      d = make_double2(fma(-k, s123.x, d.x), fma(-k, s123.y, d.y));
    } else {
      cfms(d, cscale(op.k2num, ic2), s123);
    }
  }
  for (int q = 0; q < nrhs; ++q) {
    const double2* xv = x + q * N + g;
    const double2 c = xv[0];
    const double2 xm = xl ? xv[-1] : zero, xp = xh ? xv[1] : zero, ym = yl ? xv[-op.nx] : zero, yp = yh ? xv[op.nx] : zero;
    const double2 zm = zl ? xv[-plane] : zero, zp = zh ? xv[plane] : zero;
    double2 v;
    if constexpr (kAll) {
      const double2 n = cadd(cadd(cadd(xm, xp), cadd(ym, yp)), cadd(zm, zp));
      v = make_double2(fma(-op.inv_h2, n.x, d.x * c.x), fma(-op.inv_h2, n.y, d.x * c.y));
      if (!real_k) {
        v.x = fma(-d.y, c.y, v.x);
        v.y = fma(d.y, c.x, v.y);
      }
    } else {
      // the axes outside their PML have one coefficient for both neighbours, and two of them share it
      double2 n;
      if constexpr (ONE2 && ONE3) n = cmul(m2, cadd(cadd(ym, yp), cadd(zm, zp)));
      else if constexpr (ONE1 && ONE3) n = cmul(m1, cadd(cadd(xm, xp), cadd(zm, zp)));
      else if constexpr (ONE1 && ONE2) n = cmul(m1, cadd(cadd(xm, xp), cadd(ym, yp)));
      else if constexpr (ONE1) n = cmul(m1, cadd(xm, xp));
      else if constexpr (ONE2) n = cmul(m2, cadd(ym, yp));
      else if constexpr (ONE3) n = cmul(m3, cadd(zm, zp));
      else n = zero;
      if constexpr (!ONE1) {
        cfma(n, a1, xm);
        cfma(n, b1, xp);
      }
      if constexpr (!ONE2) {
        cfma(n, a2, ym);
        cfma(n, b2, yp);
      }
      if constexpr (!ONE3) {
        cfma(n, a3, zm);
        cfma(n, b3, zp);
      }
      v = cmul(d, c);
      v = make_double2(fma(-op.inv_h2, n.x, v.x), fma(-op.inv_h2, n.y, v.y));
    }
    if (in) y[q * N + g] = v;
  }
}

__global__ void __launch_bounds__(256) k_matvec(BoxOp op, const double2* __restrict__ x, double2* __restrict__ y, int nrhs,
                                                int64_t N) {
  const int64_t g0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool in = g0 < N;
  const int64_t g = in ? g0 : N - 1;   // every lane takes part in the votes
  const unsigned gu = (unsigned)g, plane = (unsigned)op.nx * op.ny;   // grids have at most 2^31 points
  const int zz = (int)(gu / plane), p = (int)(gu - (unsigned)zz * plane), yy = p / op.nx, xx = p - yy * op.nx;
  // axis by axis: the stretches at the node and at both half-points are one
  const bool o1 = __all_sync(0xffffffffu, is_one(op.s1n[xx]) && is_one(op.s1h[xx]) && is_one(op.s1h[xx + 1]));
  const bool o2 = __all_sync(0xffffffffu, is_one(op.s2n[yy]) && is_one(op.s2h[yy]) && is_one(op.s2h[yy + 1]));
  const bool o3 = __all_sync(0xffffffffu, is_one(op.s3n[zz]) && is_one(op.s3h[zz]) && is_one(op.s3h[zz + 1]));
  switch ((o1 ? 1 : 0) | (o2 ? 2 : 0) | (o3 ? 4 : 0)) {
    case 7: matvec_rows<true, true, true>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    case 6: matvec_rows<false, true, true>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    case 5: matvec_rows<true, false, true>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    case 3: matvec_rows<true, true, false>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    case 4: matvec_rows<false, false, true>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    case 2: matvec_rows<false, true, false>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    case 1: matvec_rows<true, false, false>(op, x, y, nrhs, N, g, in, xx, yy, zz); break;
    default: matvec_rows<false, false, false>(op, x, y, nrhs, N, g, in, xx, yy, zz);
  }
}

// b = s1 s2 s3 f (the right-hand side of the symmetrised system)
__global__ void k_scale_rhs(BoxOp op, const double2* __restrict__ f, double2* __restrict__ b, int nrhs, int64_t N) {
  const int64_t plane = (int64_t)op.nx * op.ny;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < N; g += (int64_t)gridDim.x * blockDim.x) {
    const int xx = (int)(g % op.nx);
    const int yy = (int)((g / op.nx) % op.ny);
    const int zz = (int)(g / plane);
    const double2 s = cmul(cmul(op.s1n[xx], op.s2n[yy]), op.s3n[zz]);
    for (int q = 0; q < nrhs; ++q) b[q * N + g] = cmul(s, f[q * N + g]);
  }
}

static int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 64) b = 152 * 64;
  return (int)(b < 1 ? 1 : b);
}

void launch_matvec(const BoxOp& op, const double2* x, double2* y, int nrhs, int64_t N, cudaStream_t st) {
  k_matvec<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(op, x, y, nrhs, N);
}

// 1 / c^2 once per handle: every row of every operator divides by c^2
__global__ void k_inverse_square(double* c, int64_t N) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < N; g += (int64_t)gridDim.x * blockDim.x)
    c[g] = 1.0 / (c[g] * c[g]);
}
void launch_inverse_square(double* c, int64_t N, cudaStream_t st) {
  k_inverse_square<<<grid_for(N, 256), 256, 0, st>>>(c, N);
}
void launch_scale_rhs(const BoxOp& op, const double2* f, double2* b, int nrhs, int64_t N, cudaStream_t st) {
  k_scale_rhs<<<grid_for(N, 256), 256, 0, st>>>(op, f, b, nrhs, N);
}

// ---------------------------------------------------------------------------
// Front assembly (§2.2): F_TL = H[S,S], F_BL = H[U,S], F_BR = 0, then the children's update
// matrices are added through the relative index maps (extend-add).  One CTA owns a chunk of
// the front's (s+u) columns, so no two CTAs touch the same entry; children are added one after
// the other, which fixes the summation order.  The same pass initialises W = I (s x s).
//
// Bound by latency and instructions rather than by its bytes (it took the same 29 ms for complex64 and complex128 fronts).  A column's seven coefficients (about 110 FP64 operations)
// are computed once by one warp while the others zero, not by each entry's thread; G's and W's columns are one contiguous
// range, zeroed 16 bytes at a time; a warp searches a child's rows 32 probes at a time.  100^3 layered complex64 setup:
// 22.8 -> 11.8 ms (3.0 TB/s), 80^3 lens complex128 13.4 -> 11.9 ms (3.5 TB/s).
// ---------------------------------------------------------------------------
constexpr int kZeroWarps = 7;   // zeroing warps of an assembly CTA, before the warp that computes coefficients
static_assert(kAssembleCols <= 32, "one lane per owned column");

// n elements from p by the zeroing warps, 16 bytes at a time between an unaligned head and tail
template <typename T>
__device__ __forceinline__ void zero_range(T* p, int64_t n) {
  if constexpr (sizeof(T) == 16) {
    for (int64_t i = threadIdx.x; i < n; i += kZeroWarps * 32) p[i] = CplxTraits<T>::zero();
  } else {
    if ((reinterpret_cast<uintptr_t>(p) & 8) && n > 0) {
      if (threadIdx.x == 0) *p = CplxTraits<T>::zero();
      ++p;
      --n;
    }
    float4* q = reinterpret_cast<float4*>(p);
    for (int64_t i = threadIdx.x; i < n / 2; i += kZeroWarps * 32) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((n & 1) && threadIdx.x == 0) p[n - 1] = CplxTraits<T>::zero();
  }
}

// first i in [0, n) with v[i] >= key (n: none), v ascending; one warp, 32 probes at a time
__device__ __forceinline__ int lower_bound_warp(const int32_t* __restrict__ v, int n, int key) {
  const int lane = threadIdx.x & 31;
  int lo = 0;
  while (n > 0) {
    const int step = (n + 31) >> 5, i = lane * step;
    const int below = __popc(__ballot_sync(0xffffffffu, i < n && v[lo + i] < key));   // probes below key: the first ones
    if (below == 0) break;
    const int skip = (below - 1) * step + 1;   // elements known to be below
    lo += skip;
    n = min(step - 1, n - skip);
  }
  return lo;
}

template <typename T>
__global__ void __launch_bounds__(256) k_assemble(const FrontTask<T>* __restrict__ fronts,
                                                  const ColTask* __restrict__ tasks, const ShapeDev* __restrict__ shapes,
                                                  const BoxOp* __restrict__ boxops, T* const* __restrict__ upd_ptr,
                                                  const int32_t* __restrict__ upd_tile,
                                                  const int32_t* __restrict__ panel_shape) {
  const ColTask tk = tasks[blockIdx.x];
  const FrontTask<T> ft = fronts[tk.front];
  const ShapeDev sh = shapes[panel_shape[ft.panel]];
  const BoxOp op = boxops[ft.panel];
  const int s = ft.s, u = ft.u, ld = s + u;
  const int c0 = tk.c0, c1 = tk.c1;
  const int first = sh.first[ft.sn];
  const int32_t* sel = sh.struct_elim + sh.struct_ptr[ft.sn];
  const T zero = CplxTraits<T>::zero();
  __shared__ double2 coef[7][kAssembleCols];   // the owned columns' rows of H
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cs1 = c1 < s ? c1 : s;

  // 1. the last warp: the owned columns' coefficients of H; the others zero the owned columns, and W, W2
  if (warp == kZeroWarps) {
    if (c0 + lane < cs1) {
      const int node = sh.order[first + c0 + lane];
      const Row7 r7 = row7(op, node % sh.nx, (node / sh.nx) % sh.ny, node / (sh.nx * sh.ny));
      coef[0][lane] = r7.d;
      coef[1][lane] = r7.xm;
      coef[2][lane] = r7.xp;
      coef[3][lane] = r7.ym;
      coef[4][lane] = r7.yp;
      coef[5][lane] = r7.zm;
      coef[6][lane] = r7.zp;
    }
  } else {
    if (c0 < s) {
      zero_range(ft.G + (int64_t)c0 * ld, (int64_t)(cs1 - c0) * ld);
      if (ft.W) zero_range(ft.W + (int64_t)c0 * s, (int64_t)(cs1 - c0) * s);
      if (ft.W2) zero_range(ft.W2 + (int64_t)c0 * s, (int64_t)(cs1 - c0) * s);
    }
    // the lower part of column c - s of the packed update matrix
    for (int c = max(c0, s) + warp; c < c1; c += kZeroWarps) {
      const UpdColumn uc(c - s, u, ft.ut);
      for (int r = c - s + lane; r < u; r += 32) ft.U[uc.at(r)] = zero;
    }
  }
  __syncthreads();

  // the identity of W and W2
  if (c0 + (int)threadIdx.x < cs1) {
    const int64_t dd = (int64_t)(c0 + threadIdx.x) * s + c0 + threadIdx.x;
    if (ft.W) ft.W[dd] = CplxTraits<T>::one();
    if (ft.W2) ft.W2[dd] = CplxTraits<T>::one();
  }

  // 2. original entries H[r, j], j in S (column), elim(r) >= elim(j)
  for (int w = threadIdx.x; w < (cs1 - c0) * 7; w += blockDim.x) {
    const int c = c0 + w / 7, which = w % 7;
    const int node = sh.order[first + c];
    const int x = node % sh.nx, y = (node / sh.nx) % sh.ny, z = node / (sh.nx * sh.ny);
    int nx = x, ny = y, nz = z;
    switch (which) {
      case 1: nx = x - 1; break;
      case 2: nx = x + 1; break;
      case 3: ny = y - 1; break;
      case 4: ny = y + 1; break;
      case 5: nz = z - 1; break;
      case 6: nz = z + 1; break;
      default: break;
    }
    if (nx < 0 || nx >= sh.nx || ny < 0 || ny >= sh.ny || nz < 0 || nz >= sh.nz) continue;
    const int rnode = nx + sh.nx * (ny + sh.ny * nz);
    const int e = sh.elim[rnode];
    if (e < first + c) continue;
    int pos;
    if (e < first + s) {
      pos = e - first;
    } else {
      int lo = 0, hi = u;  // lower_bound in struct(S)
      while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (sel[mid] < e) lo = mid + 1; else hi = mid;
      }
      pos = s + lo;
    }
    ft.G[(int64_t)c * ld + pos] = CplxTraits<T>::from(coef[which][c - c0]);
  }
  __syncthreads();

  // 3. extend-add of each child's update matrix (lower triangle), child by child
  for (int ci = sh.child_ptr[ft.sn]; ci < sh.child_ptr[ft.sn + 1]; ++ci) {
    const int ch = sh.child_idx[ci];
    const int uc = sh.u[ch];
    const int32_t* rel = sh.rel + sh.struct_ptr[ch];
    const T* Uc = upd_ptr[ft.gfid - ft.sn + ch];
    const int utc = upd_tile[ft.gfid - ft.sn + ch];
    // child columns b whose target column rel[b] lies in [c0, c1): a contiguous range
    const int b0 = lower_bound_warp(rel, uc, c0), b1 = b0 + lower_bound_warp(rel + b0, uc - b0, c1);
    // one warp per child column (the columns land in distinct target columns, so the warps never
    // touch the same entry), four independent entries in flight per lane
    for (int b = b0 + warp; b < b1; b += kZeroWarps + 1) {
      const int tc = rel[b];
      const UpdColumn from(b, uc, utc), to(max(tc - s, 0), u, ft.ut);
      for (int a0 = b + lane; a0 < uc; a0 += 4 * 32) {
        T* dst[4];
        T val[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int a = a0 + 32 * t;
          dst[t] = nullptr;
          if (a < uc) {
            const int ra = rel[a];
            dst[t] = tc < s ? ft.G + (int64_t)tc * ld + ra : ft.U + to.at(ra - s);
            val[t] = Uc[from.at(a)];
          }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (dst[t]) *dst[t] = cadd(*dst[t], val[t]);
      }
    }
    __syncthreads();
  }
}

template <typename T>
void launch_assemble_impl(const FrontTask<T>* fronts, const ColTask* tasks, int ntasks, const ShapeDev* shapes,
                          const BoxOp* boxops, T* const* upd_ptr, const int32_t* upd_tile, const int32_t* panel_shape,
                          cudaStream_t st) {
  if (ntasks <= 0) return;
  k_assemble<T><<<ntasks, 256, 0, st>>>(fronts, tasks, shapes, boxops, upd_ptr, upd_tile, panel_shape);
}

template void launch_assemble_impl<double2>(const FrontTask<double2>*, const ColTask*, int, const ShapeDev*,
                                            const BoxOp*, double2* const*, const int32_t*, const int32_t*,
                                            cudaStream_t);
template void launch_assemble_impl<float2>(const FrontTask<float2>*, const ColTask*, int, const ShapeDev*,
                                           const BoxOp*, float2* const*, const int32_t*, const int32_t*,
                                           cudaStream_t);

}  // namespace psp
