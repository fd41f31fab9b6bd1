// Kernels of one Liouvillian application and of the two Lanczos recursions (sm_103a).
//
// Layouts (all complex interleaved, C order):
//   batch vector      x[vec][k][v][npw_pad]          one orbital per (vec, k, v) on sphere(k+Q)
//   column buffer     cbuf[o][j3][ncol_max]          per orbital o: the sphere's (m1, m2)
//                                                    columns after the 1D FFT along axis 3
//   real-space grids  g[j3][j2][j1]                  (j1 fastest)
//   orbital grids     ur[k][v][j3][j2][j1]           u_{vk}(r) sqrt(Omega), sphere(k)
// A 3D transform of a sphere is split as: 1D FFTs of the occupied columns (axis 3), then for
// every plane j3 a 2D transform over (axis 2, axis 1) restricted to the sphere's rows and
// columns; the full N^3 grid of one orbital is never materialised.
#pragma once
#include "fft.cuh"
#include "sums.cuh"

namespace ll {

// Plane-wave sphere tables of one family (spheres of k, or of k+Q) on the device.
struct SphereDev {
  int nks, npw_pad, ncol_max, nrow_max;
  const int* npw;       // [nks]
  const int* ncol;      // [nks]
  const int* nrow;      // [nks]
  const int4* col;      // [nks][ncol_max]  (m1, m2, m3 of the first point, point count),
                        //                  ordered by (m2, m1)
  const int* colstart;  // [nks][ncol_max]  first point of the column in the sphere order
  const int4* row;      // [nks][nrow_max]  (m2, first column, m1 of the first column, columns),
                        //                  consecutive m2, each row's m1 consecutive
};

// m mod N for m >= -N (a mask when N is a power of two)
template <int N>
__device__ __forceinline__ int wrapn(int m) { return (int)((unsigned)(m + N) % (unsigned)N); }

// Pruned lines: with PR > 0 every sphere of the system has |m| <= PR on all three axes, so only the
// points p <= PR and p >= N - PR of a line are kept; with the stores of the other points gone at
// compile time, the compiler drops the butterflies that only feed them.  PR = N/2 - 1 keeps the whole
// line (line_hi): m = -N/2 or N/2 too, whichever lies in a sphere's run of indices that starts at
// lo (line_m).  PR = 0: every point, of any indices.
__host__ __device__ constexpr int line_hi(int n, int pr) { return pr == n / 2 - 1 ? n / 2 : pr; }
template <int N, int PR>
__device__ __forceinline__ int line_m(int p, int lo) {
  if (PR == N / 2 - 1 && p == N / 2) return lo > -N / 2 ? N / 2 : -N / 2;
  return p <= PR ? p : p - N;
}
template <int N, int PR>
__device__ __forceinline__ constexpr bool line_kept(int p) {
  return PR == 0 || p <= PR || p >= N - line_hi(N, PR);
}

// ---------------------------------------------------------------------------------------
// Sphere -> columns: scatter each column's points and inverse-FFT along axis 3.
// grid (nks, nvec, split), block 128; item = (v, column), the k block's items spread over
// the split CTAs.  PR > 0: every point of the spheres has |m| <= PR (PR < N/2), so a point's
// offset is a compile-time constant and the zeros outside are known (PR = 0: any indices).
// FP64 through fixed point (line_transform): KB workload 107 -> 58 us per launch, k_zfwd 146 -> 71.
template <typename T, int N, int PR = 0>
__global__ void __launch_bounds__(128) k_zinv(SphereDev s, const cplx<T>* __restrict__ x, int nbnd,
                                              cplx<T>* __restrict__ cbuf, int cb_ncol) {
  const int k = blockIdx.x, vec = blockIdx.y;
  const int nc = s.ncol[k];
  for (int it = blockIdx.z * blockDim.x + threadIdx.x; it < nbnd * nc; it += blockDim.x * gridDim.z) {
    const int v = it / nc, c = it - v * nc;
    const long o = ((long)vec * s.nks + k) * nbnd + v;
    const int4 cl = s.col[k * s.ncol_max + c];
    const int st = s.colstart[k * s.ncol_max + c];
    const cplx<T>* src = x + o * s.npw_pad + st;
    cplx<T> a[N];
#pragma unroll
    for (int p = 0; p < N; ++p) {
      a[p] = czero<T>();
      if (line_kept<N, PR>(p)) {
        const int i = PR > 0 ? line_m<N, PR>(p, cl.z) - cl.z : wrapn<N>(p - cl.z);
        if ((unsigned)i < (unsigned)cl.w && LL_INB(st >= 0 && st + i < s.npw_pad)) a[p] = src[i];
      }
    }
    if constexpr (PR > 0) line_transform<T, N, +1, PR, line_hi(N, PR)>(a);
    else line_transform<T, N, +1>(a);
    if (!LL_INB(c < cb_ncol)) continue;
    cplx<T>* dst = cbuf + o * (long)N * cb_ncol + c;
#pragma unroll
    for (int p = 0; p < N; ++p) dst[(long)p * cb_ncol] = a[p];
  }
}

// ---------------------------------------------------------------------------------------
// Bulk prefetch of a contiguous global range into L2 (no data returned to the SM): address
// 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

// ---------------------------------------------------------------------------------------
// Per-plane pass of one operator application, for any Miller indices that fit the grid (the
// orbital grids at set-up, and spheres that no index shift brings within -N/2 .. N/2, fold_index;
// every other application takes k_plane, plane.cuh, with the same modes).  grid (N planes, groups),
// block 128.
// The sphere's columns are ordered by (m2, m1) and grouped in rows of equal m2 (consecutive
// m1).  For every orbital of the group (BO at a time), at plane j3 = blockIdx.x:
//   rows     1D FFT along axis 1 (m1 <-> j1) of every sphere row, between the column buffer
//            Cs and the row buffer Ys[row][j1];
//   lines    one thread per (orbital, j1): 1D FFT along axis 2 (m2 <-> j2) of the line
//            x(j2, j1), j2 = 0..N-1, held in registers.  Thread t = s N + j1 (s < S = 128/N)
//            always takes column j1, for the batch's orbitals b = s, s + S, ...; consecutive
//            threads take consecutive j1, so every real-space plane (V, v', u, the density)
//            is read and written with unit stride across a warp straight from HBM.
// Modes:
//   XY_PASS1       inverse 2D FFT of the plane's columns, t(r) = V(r) x(r), forward 2D FFT
//                  back to the columns (in place);
//   XY_PASS1_DENS  the same plus the response-density partial sum_o conj(u_o(r)) x_o(r) of the
//                  orbitals of vector dens_vec, written per (group, plane) to nprt.  Each
//                  thread adds its lines' products into its own column of its slot's plane
//                  Pb[s] (no other thread touches it: no barrier, a fixed order); the S slots
//                  are summed in order once, at the end;
//   XY_PASS2       t(r) = v'(r) u(r) from the orbital grid, forward 2D FFT, added into the
//                  columns (linearity: one axis-3 transform serves both passes);
//   XY_STORE       inverse 2D FFT only, x(r) stored to grid_out (orbital grids at set-up).
enum XYMode { XY_PASS1 = 0, XY_PASS1_DENS = 1, XY_PASS2 = 2, XY_STORE = 3 };

struct XYArgs {
  SphereDev s;
  int nbnd, norb;              // orbitals handled by this launch
  int cb_ncol;
  int per_group;               // orbitals per group
  int o_off;                   // first orbital of this launch (orbital o = o_off + local index)
  int dens_vec;                // vector whose orbitals feed the density (XY_PASS1_DENS)
  int bo;                      // orbitals per batch (as many as shared memory allows, <= the mode's default)
  FastDiv f_ncol, f_nrow;      // divisions by cb_ncol and by the sphere table's nrow_max
  FastDiv f_nbnd, f_nks;       // orbital -> k: (o / nbnd) mod nks
  FastDiv f_pervec;            // orbital -> vector: o / (nks nbnd)
  int polls;                   // of a wait on a copy before it gives up (plane.cuh)
};

template <typename T, int N, int MODE>
__global__ void __launch_bounds__(128, N > 36 ? 2 : (MODE == XY_PASS1_DENS ? 3 : 4)) k_xy(XYArgs a, cplx<T>* __restrict__ cbuf, const T* __restrict__ vloc,
                                               const cplx<T>* __restrict__ vpr, const cplx<T>* __restrict__ ur,
                                               cplx<T>* __restrict__ nprt, cplx<T>* __restrict__ grid_out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NP = N + 1;
  constexpr int NN = N * N;
  const int iz = blockIdx.x, g = blockIdx.y;
  const int BO = a.bo;
  const SphereDev& s = a.s;
  cplx<T>* Cs = reinterpret_cast<cplx<T>*>(smem_raw);                 // [BO][cb_ncol]
  cplx<T>* Ys = Cs + BO * a.cb_ncol;                                    // [BO][nrow_max][NP]
  constexpr int S = 128 / N;                                           // line slots
  cplx<T>* Pl = Ys + BO * s.nrow_max * NP;                              // [N][N] v' (pass 2)
  cplx<T>* Pb = Pl + (MODE == XY_PASS2 ? NN : 0);                       // [S][N][N] density
  T* Pv = reinterpret_cast<T*>(Pb + (MODE == XY_PASS1_DENS ? S * NN : 0));  // [N][N] V (real)
  const long plane = (long)NN;
  const int ls = threadIdx.x / N, lj1 = threadIdx.x - ls * N;           // line slot, column

  if (MODE == XY_PASS1 || MODE == XY_PASS1_DENS) {
    for (int i = threadIdx.x; i < NN; i += blockDim.x) Pv[i] = vloc[iz * plane + i];
  } else if (MODE == XY_PASS2) {
    for (int i = threadIdx.x; i < NN; i += blockDim.x) Pl[i] = vpr[iz * plane + i];
  }
  if (MODE == XY_PASS1_DENS)
    for (int i = threadIdx.x; i < S * NN; i += blockDim.x) Pb[i] = czero<T>();

  const int o_begin = a.o_off + g * a.per_group;
  const int o_end = a.o_off + min(a.norb, g * a.per_group + a.per_group);
  // The next batch's column-buffer rows of this plane (cb_ncol is even: 16-byte multiples)
  // are prefetched into L2 while this batch is transformed; the density pass also prefetches
  // the current batch's orbital-grid planes before its row transforms, which then hide the
  // HBM latency.  (Prefetching the next batch's grid planes a whole batch ahead was
  // measured: their lines were evicted before use and re-read, +20 % DRAM.)
  auto prefetch_batch = [&](int obatch) {
    const int t = threadIdx.x;
    if (t < BO && obatch + t < o_end)
      prefetch_l2(cbuf + (long)(obatch + t) * N * a.cb_ncol + (long)iz * a.cb_ncol,
                  (unsigned)(a.cb_ncol * sizeof(cplx<T>)));
  };
  prefetch_batch(o_begin);
  for (int ob = o_begin; ob < o_end; ob += BO) {
    const int nb = min(BO, o_end - ob);
    __syncthreads();
    if (ob + BO < o_end) prefetch_batch(ob + BO);
    if (MODE == XY_PASS1_DENS && threadIdx.x < nb) {
      const int o = ob + threadIdx.x;
      if (a.f_pervec.div(o) == a.dens_vec)
        prefetch_l2(ur + (long)a.f_pervec.mod(o) * N * plane + iz * plane, (unsigned)(NN * sizeof(cplx<T>)));
    }
    if (MODE != XY_PASS2) {
      for (int i = threadIdx.x; i < nb * a.cb_ncol; i += blockDim.x) {
        const int b = a.f_ncol.div(i), c = i - b * a.cb_ncol;
        const int o = ob + b, k = a.f_nks.mod(a.f_nbnd.div(o));
        Cs[i] = (c < s.ncol[k]) ? cbuf[(long)o * N * a.cb_ncol + (long)iz * a.cb_ncol + c] : czero<T>();
      }
      __syncthreads();
      // inverse FFT along axis 1 of every sphere row (fixed m2)
      for (int i = threadIdx.x; i < nb * s.nrow_max; i += blockDim.x) {
        const int b = a.f_nrow.div(i), r = i - b * s.nrow_max;
        const int o = ob + b, k = a.f_nks.mod(a.f_nbnd.div(o));
        if (r >= s.nrow[k]) continue;
        const int4 rw = s.row[k * s.nrow_max + r];
        cplx<T> l[N];
        const cplx<T>* cs = Cs + b * a.cb_ncol + rw.y;
#pragma unroll
        for (int p = 0; p < N; ++p) {
          const int j = wrapn<N>(p - rw.z);
          l[p] = (j < rw.w && LL_INB(rw.y >= 0 && rw.y + j < a.cb_ncol)) ? cs[j] : czero<T>();
        }
        fft_line<T, N, +1>(l);
        cplx<T>* ys = Ys + (b * s.nrow_max + r) * NP;
#pragma unroll
        for (int p = 0; p < N; ++p) ys[p] = l[p];
      }
      __syncthreads();
    }
    // axis 2: one line per (orbital, j1), element p of the line at grid point (j2 = p, j1)
#pragma unroll 1
    for (int b = ls; ls < S && b < nb; b += S) {
      const int j1 = lj1;
      const int o = ob + b, k = a.f_nks.mod(a.f_nbnd.div(o));
      const int nr = s.nrow[k];
      const int m2min = s.row[k * s.nrow_max].x;
      cplx<T> l[N];
      if (MODE == XY_PASS2) {
        const cplx<T>* u = ur + (long)a.f_pervec.mod(o) * N * plane + iz * plane + j1;
#pragma unroll
        for (int p = 0; p < N; ++p) l[p] = cmul(Pl[p * N + j1], u[p * N]);
      } else {
#pragma unroll
        for (int p = 0; p < N; ++p) {
          const int r = wrapn<N>(p - m2min);
          l[p] = (r < nr && LL_INB(r < s.nrow_max)) ? Ys[(b * s.nrow_max + r) * NP + j1] : czero<T>();
        }
        fft_line<T, N, +1>(l);
        if (MODE == XY_STORE) {
          cplx<T>* dst = grid_out + (long)o * N * plane + iz * plane + j1;
#pragma unroll
          for (int p = 0; p < N; ++p) dst[p * N] = l[p];
          continue;
        }
        if (MODE == XY_PASS1_DENS && a.f_pervec.div(o) == a.dens_vec) {
          // conj(u) x of this line into this thread's own column of its slot
          const cplx<T>* u = ur + (long)a.f_pervec.mod(o) * N * plane + iz * plane + j1;
          cplx<T>* pb = Pb + ls * NN + j1;
#pragma unroll
          for (int p = 0; p < N; ++p) pb[p * N] = pb[p * N] + cjmul(u[p * N], l[p]);
        }
#pragma unroll
        for (int p = 0; p < N; ++p) l[p] = l[p] * Pv[p * N + j1];
      }
      fft_line<T, N, -1>(l);
#pragma unroll
      for (int p = 0; p < N; ++p) {
        const int r = wrapn<N>(p - m2min);
        if (r < nr && LL_INB(r < s.nrow_max)) Ys[(b * s.nrow_max + r) * NP + j1] = l[p];
      }
    }
    __syncthreads();
    if (MODE == XY_STORE) continue;
    // forward FFT along axis 1 of every row, keep the row's columns
    for (int i = threadIdx.x; i < nb * s.nrow_max; i += blockDim.x) {
      const int b = a.f_nrow.div(i), r = i - b * s.nrow_max;
      const int o = ob + b, k = a.f_nks.mod(a.f_nbnd.div(o));
      if (r >= s.nrow[k]) continue;
      const int4 rw = s.row[k * s.nrow_max + r];
      cplx<T> l[N];
      const cplx<T>* ys = Ys + (b * s.nrow_max + r) * NP;
#pragma unroll
      for (int p = 0; p < N; ++p) l[p] = ys[p];
      fft_line<T, N, -1>(l);
      cplx<T>* cs = Cs + b * a.cb_ncol + rw.y;
#pragma unroll
      for (int p = 0; p < N; ++p) {
        const int j = wrapn<N>(p - rw.z);
        if (j < rw.w && LL_INB(rw.y >= 0 && rw.y + j < a.cb_ncol)) cs[j] = l[p];
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb * a.cb_ncol; i += blockDim.x) {
      const int b = a.f_ncol.div(i), c = i - b * a.cb_ncol;
      const int o = ob + b, k = a.f_nks.mod(a.f_nbnd.div(o));
      if (c >= s.ncol[k]) continue;
      cplx<T>* dst = cbuf + (long)o * N * a.cb_ncol + (long)iz * a.cb_ncol + c;
      *dst = (MODE == XY_PASS2) ? *dst + Cs[i] : Cs[i];
    }
  }
  if (MODE == XY_PASS1_DENS) {  // the slots summed in order
    __syncthreads();
    for (int i = threadIdx.x; i < NN; i += blockDim.x) {
      cplx<T> acc = Pb[i];
      for (int q = 1; q < S; ++q) acc = acc + Pb[q * NN + i];
      nprt[(long)g * N * plane + iz * plane + i] = acc;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Response potential of one density (Eqs. 12-13): n'(r) from the group partials, 3D FFT,
// Hartree 4 pi/|Q+G|^2, inverse FFT, plus f_xc(n0) n'.  Three launches over the grid.
template <typename T, int N>
__global__ void __launch_bounds__(256) k_hxc_fwd(const cplx<T>* __restrict__ nprt, int ngroups, T scale,
                                                cplx<T>* __restrict__ nr, cplx<T>* __restrict__ ng) {
  __shared__ cplx<T> P[N][N + 1];
  const int iz = blockIdx.x;
  const long plane = (long)N * N;
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) {
    cplx<T> acc = czero<T>();
    for (int gi = 0; gi < ngroups; ++gi) acc = acc + nprt[(long)gi * N * plane + iz * plane + i];
    acc = acc * scale;
    nr[iz * plane + i] = acc;
    P[i / N][i % N] = acc;
  }
  __syncthreads();
  if (threadIdx.x < N) {  // axis 1, row j2
    const int j2 = threadIdx.x;
    cplx<T> l[N];
#pragma unroll
    for (int p = 0; p < N; ++p) l[p] = P[j2][p];
    fft_line<T, N, -1>(l);
#pragma unroll
    for (int p = 0; p < N; ++p) P[j2][p] = l[p];
  }
  __syncthreads();
  if (threadIdx.x < N) {  // axis 2, column m1
    const int m1 = threadIdx.x;
    cplx<T> l[N];
#pragma unroll
    for (int p = 0; p < N; ++p) l[p] = P[p][m1];
    fft_line<T, N, -1>(l);
#pragma unroll
    for (int p = 0; p < N; ++p) ng[iz * plane + p * N + m1] = l[p];
  }
}

// The response density averaged over the small group of Q (Sec. 2.6): out(r_j) = (1/nsym)
// sum_S scale n~(r_{M_S j}), n~ = the sum of the density groups (the order of k_hxc_fwd),
// M_S the integer matrices sym[S] on the grid indices (j1, j2, j3), mod N.  Grid layout
// [j3][j2][j1]; grid-stride loop over the N^3 points.
template <typename T>
__global__ void k_dens_sym(const cplx<T>* __restrict__ nprt, int ngroups, int n, T scale, int nsym,
                           const int* __restrict__ sym, cplx<T>* __restrict__ out) {
  const long n3 = (long)n * n * n;
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n3; p += (long)gridDim.x * blockDim.x) {
    const int j1 = (int)(p % n), j2 = (int)((p / n) % n), j3 = (int)(p / ((long)n * n));
    cplx<T> acc = czero<T>();
    for (int s = 0; s < nsym; ++s) {
      const int* m = sym + 9 * s;
      const int i1 = (((m[0] * j1 + m[1] * j2 + m[2] * j3) % n) + n) % n;
      const int i2 = (((m[3] * j1 + m[4] * j2 + m[5] * j3) % n) + n) % n;
      const int i3 = (((m[6] * j1 + m[7] * j2 + m[8] * j3) % n) + n) % n;
      const long q = ((long)i3 * n + i2) * n + i1;
      cplx<T> v = czero<T>();
      for (int g = 0; g < ngroups; ++g) v = v + nprt[(long)g * n3 + q];
      acc = acc + v * scale;
    }
    out[p] = acc * (T(1) / (T)nsym);
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(64) k_hxc_z(cplx<T>* __restrict__ ng, const T* __restrict__ whart) {
  const int line = blockIdx.x * blockDim.x + threadIdx.x;   // (m2, m1)
  if (line >= N * N) return;
  const long plane = (long)N * N;
  cplx<T> l[N];
#pragma unroll
  for (int p = 0; p < N; ++p) l[p] = ng[p * plane + line];
  fft_line<T, N, -1>(l);
#pragma unroll
  for (int p = 0; p < N; ++p) l[p] = l[p] * whart[p * plane + line];
  fft_line<T, N, +1>(l);
#pragma unroll
  for (int p = 0; p < N; ++p) ng[p * plane + line] = l[p];
}

template <typename T, int N>
__global__ void __launch_bounds__(64) k_hxc_inv(const cplx<T>* __restrict__ ng, const cplx<T>* __restrict__ nr,
                                                const T* __restrict__ fxc, cplx<T>* __restrict__ vpr) {
  __shared__ cplx<T> P[N][N + 1];
  const int iz = blockIdx.x;
  const long plane = (long)N * N;
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) P[i / N][i % N] = ng[iz * plane + i];
  __syncthreads();
  if (threadIdx.x < N) {  // axis 2 inverse, column m1
    const int m1 = threadIdx.x;
    cplx<T> l[N];
#pragma unroll
    for (int p = 0; p < N; ++p) l[p] = P[p][m1];
    fft_line<T, N, +1>(l);
#pragma unroll
    for (int p = 0; p < N; ++p) P[p][m1] = l[p];
  }
  __syncthreads();
  if (threadIdx.x < N) {  // axis 1 inverse, row j2
    const int j2 = threadIdx.x;
    cplx<T> l[N];
#pragma unroll
    for (int p = 0; p < N; ++p) l[p] = P[j2][p];
    fft_line<T, N, +1>(l);
    const long base = iz * plane + (long)j2 * N;
#pragma unroll
    for (int p = 0; p < N; ++p) vpr[base + p] = l[p] + nr[base + p] * fxc[base + p];
  }
}

// ---------------------------------------------------------------------------------------
// The response potential where the orbitals are transformed on a work grid of W < n points a
// side (the chain's work_side): n' is on the W grid, which holds all its components, the Hartree
// term stays there, and f_xc n' is formed on the declared n grid.  Both directions between the
// grids are real n x W matrices per axis (rt [n][W], resample_table): a 24 x 32 matrix is a few
// dozen FMAs per point, in one pass where a pair of zero-padded FFTs would take two, and the axis-3
// product up, f_xc, and down again stay in one CTA.  Three launches, as on the declared grid alone.
//   k_hxcw_fwd  per plane s3: groups summed; slice 0: 2D FFT (Hartree); the other kHxcSlices:
//               n' interpolated to n x n points of the plane, columns j1 split over the slices
//               -> t1[s3][j2][j1]
//   k_hxcw_mid  Hartree lines (axis-3 FFT, kernel, inverse) and, per (j2, j1) column of t1, axis 3
//               up, times f_xc, axis 3 down, in place
//   k_hxcw_inv  per plane s3 and slice of s1: inverse 2D FFT of the Hartree part, t1 limited to
//               W x W points, their sum v'(s3) to vpr.  (Every slice repeats the plane's FFT: its
//               2 W lines are one warp's work beside the other warps' matrix product.)
constexpr int kHxcSlices = 4;
constexpr int kHxcCols = 8;      // t1 columns per CTA of k_hxcw_mid
static inline __host__ __device__ int hxcw_jslice(int n) { return (n + kHxcSlices - 1) / kHxcSlices; }
static inline __host__ __device__ int hxcw_sslice(int w) { return (w + kHxcSlices - 1) / kHxcSlices; }
template <typename T> size_t hxcw_fwd_smem(int w, int n) {
  return sizeof(cplx<T>) * ((size_t)w * (w + 1) + (size_t)w * hxcw_jslice(n)) + sizeof(T) * (size_t)n * w;
}
template <typename T> size_t hxcw_mid_smem(int w, int n) {
  return sizeof(cplx<T>) * (size_t)kHxcCols * (w + n) + sizeof(T) * (size_t)n * w;
}
template <typename T> size_t hxcw_inv_smem(int w, int n) {
  return sizeof(cplx<T>) * ((size_t)w * (w + 1) + (size_t)n * (n + 1) + (size_t)(n + w) * hxcw_sslice(w)) +
         sizeof(T) * (size_t)n * w;
}
static inline int hxcw_mid_blocks(int w, int n) { return (w * w + 31) / 32 + (n * n + kHxcCols - 1) / kHxcCols; }

template <typename T, int W>
__global__ void __launch_bounds__(256) k_hxcw_fwd(const cplx<T>* __restrict__ nprt, int ngroups, T scale, int n,
                                                 const T* __restrict__ rt, cplx<T>* __restrict__ ng,
                                                 cplx<T>* __restrict__ t1) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T>* P = reinterpret_cast<cplx<T>*>(smem_raw);        // [W][W + 1]
  const int js = hxcw_jslice(n);
  cplx<T>* Q = P + W * (W + 1);                              // [W][js]
  T* R = reinterpret_cast<T*>(Q + W * js);                   // [n][W]
  const int iz = blockIdx.x, sl = (int)blockIdx.y - 1;
  const long plane = (long)W * W;
  for (int i = threadIdx.x; i < W * W; i += blockDim.x) {
    const cplx<T>* src = nprt + iz * plane + i;
    cplx<T> acc = czero<T>();
#pragma unroll 8
    for (int gi = 0; gi < ngroups; ++gi) acc = acc + src[(long)gi * W * plane];
    P[(i / W) * (W + 1) + i % W] = acc * scale;
  }
  if (sl >= 0)
    for (int i = threadIdx.x; i < n * W; i += blockDim.x) R[i] = rt[i];
  __syncthreads();
  if (sl < 0) {
    if (threadIdx.x < W) {  // axis 1, row s2
      cplx<T>* row = P + threadIdx.x * (W + 1);
      cplx<T> l[W];
#pragma unroll
      for (int p = 0; p < W; ++p) l[p] = row[p];
      fft_line<T, W, -1>(l);
#pragma unroll
      for (int p = 0; p < W; ++p) row[p] = l[p];
    }
    __syncthreads();
    if (threadIdx.x < W) {  // axis 2, column m1
      const int m1 = threadIdx.x;
      cplx<T> l[W];
#pragma unroll
      for (int p = 0; p < W; ++p) l[p] = P[p * (W + 1) + m1];
      fft_line<T, W, -1>(l);
#pragma unroll
      for (int p = 0; p < W; ++p) ng[iz * plane + p * W + m1] = l[p];
    }
    return;
  }
  const int j0 = sl * js, nj = min(js, n - j0);
  for (int i = threadIdx.x; i < W * nj; i += blockDim.x) {   // axis 1
    const int s2 = i / nj, jl = i - s2 * nj;
    const T* r = R + (j0 + jl) * W;
    const cplx<T>* row = P + s2 * (W + 1);
    cplx<T> acc = czero<T>();
#pragma unroll
    for (int s = 0; s < W; ++s) acc = acc + row[s] * r[s];
    Q[s2 * js + jl] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * nj; i += blockDim.x) {   // axis 2
    const int j2 = i / nj, jl = i - j2 * nj;
    const T* r = R + j2 * W;
    cplx<T> acc = czero<T>();
#pragma unroll
    for (int s = 0; s < W; ++s) acc = acc + Q[s * js + jl] * r[s];
    t1[((long)iz * n + j2) * n + j0 + jl] = acc;
  }
}

template <typename T, int W>
__global__ void __launch_bounds__(128) k_hxcw_mid(cplx<T>* __restrict__ ng, const T* __restrict__ whart, int n,
                                                 const T* __restrict__ rt, const T* __restrict__ fxc,
                                                 cplx<T>* __restrict__ t1) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NH = (W * W + 31) / 32;   // CTAs of the Hartree lines
  const long plane = (long)W * W;
  if (blockIdx.x < NH) {
    const int line = blockIdx.x * 32 + threadIdx.x;   // (m2, m1)
    if (threadIdx.x >= 32 || line >= W * W) return;
    cplx<T> l[W];
#pragma unroll
    for (int p = 0; p < W; ++p) l[p] = ng[p * plane + line];
    fft_line<T, W, -1>(l);
#pragma unroll
    for (int p = 0; p < W; ++p) l[p] = l[p] * whart[p * plane + line];
    fft_line<T, W, +1>(l);
#pragma unroll
    for (int p = 0; p < W; ++p) ng[p * plane + line] = l[p];
    return;
  }
  cplx<T>* X = reinterpret_cast<cplx<T>*>(smem_raw);   // [W][kHxcCols]
  cplx<T>* Y = X + W * kHxcCols;                        // [n][kHxcCols]
  T* R = reinterpret_cast<T*>(Y + n * kHxcCols);        // [n][W]
  const int c0 = (blockIdx.x - NH) * kHxcCols, nn = n * n;
  const int cl = threadIdx.x % kHxcCols, ln = threadIdx.x / kHxcCols, nl = blockDim.x / kHxcCols;
  const bool on = c0 + cl < nn;
  for (int i = threadIdx.x; i < n * W; i += blockDim.x) R[i] = rt[i];
  for (int s = ln; s < W; s += nl) X[s * kHxcCols + cl] = on ? t1[(long)s * nn + c0 + cl] : czero<T>();
  __syncthreads();
  for (int j = ln; j < n; j += nl) {
    const T* r = R + j * W;
    cplx<T> acc = czero<T>();
#pragma unroll
    for (int s = 0; s < W; ++s) acc = acc + X[s * kHxcCols + cl] * r[s];
    Y[j * kHxcCols + cl] = acc * (on ? fxc[(long)j * nn + c0 + cl] : T(0));
  }
  __syncthreads();
  const T sc = T(W) / T(n);
  for (int s = ln; s < W; s += nl) {
    cplx<T> acc = czero<T>();
    for (int j = 0; j < n; ++j) acc = acc + Y[j * kHxcCols + cl] * R[j * W + s];
    if (on) t1[(long)s * nn + c0 + cl] = acc * sc;
  }
}

template <typename T, int W>
__global__ void __launch_bounds__(256) k_hxcw_inv(const cplx<T>* __restrict__ ng, int n, const T* __restrict__ rt,
                                                 const cplx<T>* __restrict__ t1, cplx<T>* __restrict__ vpr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ss = hxcw_sslice(W), s0 = blockIdx.y * ss, ns = min(ss, W - s0);
  cplx<T>* F = reinterpret_cast<cplx<T>*>(smem_raw);       // [W][W + 1] the Hartree part
  cplx<T>* X = F + W * (W + 1);                             // [n][n + 1] f_xc n'
  cplx<T>* Q = X + n * (n + 1);                             // [n][ss]
  cplx<T>* O = Q + n * ss;                                  // [W][ss]
  T* R = reinterpret_cast<T*>(O + W * ss);                  // [n][W]
  const int iz = blockIdx.x;
  const long plane = (long)W * W;
  for (int i = threadIdx.x; i < W * W; i += blockDim.x) F[(i / W) * (W + 1) + i % W] = ng[iz * plane + i];
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) X[(i / n) * (n + 1) + i % n] = t1[(long)iz * n * n + i];
  for (int i = threadIdx.x; i < n * W; i += blockDim.x) R[i] = rt[i];
  __syncthreads();
  constexpr int NF = (W + 31) / 32 * 32;   // threads of the FFT lines, the rest: the matrix product
  const T sc = T(W) / T(n);
  if (threadIdx.x < NF) {
    if (threadIdx.x < W) {  // axis 2 inverse, column m1
      const int m1 = threadIdx.x;
      cplx<T> l[W];
#pragma unroll
      for (int p = 0; p < W; ++p) l[p] = F[p * (W + 1) + m1];
      fft_line<T, W, +1>(l);
#pragma unroll
      for (int p = 0; p < W; ++p) F[p * (W + 1) + m1] = l[p];
    }
  } else {
    for (int i = threadIdx.x - NF; i < n * ns; i += blockDim.x - NF) {   // axis 1
      const int j2 = i / ns, sl = i - j2 * ns;
      cplx<T> acc = czero<T>();
      for (int j = 0; j < n; ++j) acc = acc + X[j2 * (n + 1) + j] * R[j * W + s0 + sl];
      Q[j2 * ss + sl] = acc * sc;
    }
  }
  __syncthreads();
  if (threadIdx.x < NF) {
    if (threadIdx.x < W) {  // axis 1 inverse, row s2
      cplx<T>* row = F + threadIdx.x * (W + 1);
      cplx<T> l[W];
#pragma unroll
      for (int p = 0; p < W; ++p) l[p] = row[p];
      fft_line<T, W, +1>(l);
#pragma unroll
      for (int p = 0; p < W; ++p) row[p] = l[p];
    }
  } else {
    for (int i = threadIdx.x - NF; i < W * ns; i += blockDim.x - NF) {   // axis 2
      const int s2 = i / ns, sl = i - s2 * ns;
      cplx<T> acc = czero<T>();
      for (int j = 0; j < n; ++j) acc = acc + Q[j * ss + sl] * R[j * W + s2];
      O[s2 * ss + sl] = acc * sc;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < W * ns; i += blockDim.x) {
    const int s2 = i / ns, sl = i - s2 * ns;
    vpr[iz * plane + s2 * W + s0 + sl] = F[s2 * (W + 1) + s0 + sl] + O[s2 * ss + sl];
  }
}

// ---------------------------------------------------------------------------------------
// Reductions.  Every sum below runs in a fixed order (per-thread strided partial sums, lanes,
// then warps), so results are bitwise reproducible.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Warp sums of NV values per lane at once (NV a power of two <= 32): at every step a lane keeps
// half of its values and gives its partner the other half, so 32 values take 31 exchanges
// instead of 5 each.  Returns the total of value number lane / (32 / NV).
template <typename T, int NV>
__device__ __forceinline__ T warp_sums(T (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = NV / 2; n > 0; n /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const T give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  T t = v[0];
#pragma unroll
  for (; o > 0; o /= 2) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// f(NV) with the block of bands (or of rows of a dot tile) that a thread takes per plane wave: four,
// and one or two for groups of as many, which a block of four would make four or two times the
// arithmetic.  FP64, 8 k-points of 4820 plane waves, groups of one band, us per step: blocks of four 481,
// so 291, the pair-by-pair form before 420.
template <int N> struct IntC { static constexpr int v = N; };
template <typename F>
__device__ __forceinline__ void band_blocks(int nv, F&& f) {
  if (nv == 1) f(IntC<1>{});
  else if (nv == 2) f(IntC<2>{});
  else f(IntC<4>{});
}

// Dot blocks of the per-k kernels, in tiles of 4 x NJ pairs whose sums a thread keeps in registers
// (4 + NJ loads per 4 NJ complex products); warp sums in T by halving exchange (warp_sums), warps
// summed with DSum.  `red`: kRedPairs complex T per warp; the tiles fill it before the block
// synchronises.  Bound by latency and by the reductions, not by the products: at 570 plane waves
// a thread of 256 holds 2 of them per tile, 128 FMAs beside the 31 exchanges (160 with a warp
// reduction per value; in FP64, where an add takes 16 cycles of the SM's pipe, the reductions
// were most of the block).
constexpr int kRedPairs = 128;
__host__ __device__ constexpr size_t red_elems(int threads) { return (size_t)(threads / 32) * 2 * kRedPairs; }

template <typename T, int NI, int NJ>
__device__ __forceinline__ void dots_tile(const cplx<T>* __restrict__ A, long lda, const cplx<T>* B, long ldb, int npw,
                                          int ni, int nj, T* red) {
  T acc[2 * NI * NJ];   // [i][j][re, im]
#pragma unroll
  for (int q = 0; q < 2 * NI * NJ; ++q) acc[q] = T(0);
  const cplx<T>*pa[NI], *pb[NJ];   // rows past the block's edge repeat its last one
#pragma unroll
  for (int i = 0; i < NI; ++i) pa[i] = A + (long)min(i, ni - 1) * lda;
#pragma unroll
  for (int j = 0; j < NJ; ++j) pb[j] = B + (long)min(j, nj - 1) * ldb;
  for (int g = threadIdx.x; g < npw; g += blockDim.x) {
    cplx<T> x[NI], y[NJ];
#pragma unroll
    for (int i = 0; i < NI; ++i) x[i] = pa[i][g];
#pragma unroll
    for (int j = 0; j < NJ; ++j) y[j] = pb[j][g];
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        acc[(i * NJ + j) * 2] += x[i].x * y[j].x + x[i].y * y[j].y;
        acc[(i * NJ + j) * 2 + 1] += x[i].x * y[j].y - x[i].y * y[j].x;
      }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp * 32 >= npw) return;   // a warp without plane waves
  constexpr int NV = 2 * NI * NJ;
  const T t = warp_sums<T, NV>(acc);
  if (lane % (32 / NV) == 0) red[(long)warp * 2 * kRedPairs + lane / (32 / NV)] = t;
}

// Two dot blocks at once (n1 = 0: one): out[i*nj + j] = mult[i] sum_{g < npw} conj(A0_i[g]) B0_j[g]
// for i < n0 (mult null: 1), then conj(A1_i) B1_j for i < n1 in the n1 rows after them; every row
// stride ld.  Called by the whole block; ends synchronised.
template <typename T, int NJ>
__device__ __forceinline__ void block_dots_nj(const cplx<T>* A0, const cplx<T>* B0, int n0, const double* mult,
                                              const cplx<T>* A1, const cplx<T>* B1, int n1, long ld, int npw, int nj,
                                              cplx<double>* out, T* red) {
  constexpr int TP = 4 * NJ, TB = kRedPairs / TP;   // pairs per tile, tiles per batch
  const int tj = (nj + NJ - 1) / NJ, t0n = ((n0 + 3) / 4) * tj, nt = t0n + ((n1 + 3) / 4) * tj;
  const int nw = min((int)blockDim.x, npw + 31) >> 5;   // warps with plane waves
  for (int b0 = 0; b0 < nt; b0 += TB) {
    const int n = min(TB, nt - b0);
    for (int q = 0; q < n; ++q) {
      const bool first = b0 + q < t0n;
      const int t = first ? b0 + q : b0 + q - t0n, i0 = t / tj * 4, j0 = t % tj * NJ;
      auto tile = [&](auto nc) {
        dots_tile<T, decltype(nc)::v, NJ>((first ? A0 : A1) + i0 * ld, ld, (first ? B0 : B1) + j0 * ld, ld, npw,
                                          (first ? n0 : n1) - i0, nj - j0, red + q * 2 * TP);
      };
      // (FP64: the pipe bounds the block, so that no row is done for nothing)
      if constexpr (sizeof(T) == 8) band_blocks((first ? n0 : n1) - i0, tile);
      else tile(IntC<4>{});
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * n * TP; e += blockDim.x) {   // a component of a pair
      const int p = e >> 1, q = b0 + p / TP;
      const bool first = q < t0n;
      const int t = first ? q : q - t0n, i = t / tj * 4 + (p % TP) / NJ, j = t % tj * NJ + p % NJ;
      if (i < (first ? n0 : n1) && j < nj) {
        DSum<T> sum;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) sum.add(red[w * 2 * kRedPairs + e]);
        const double a = sum.value();
        reinterpret_cast<double*>(out + ((first ? 0 : n0) + i) * nj + j)[e & 1] = first && mult ? a * mult[i] : a;
      }
    }
    __syncthreads();
  }
}

template <typename T>
__device__ __forceinline__ void block_dots2(const cplx<T>* A0, const cplx<T>* B0, int n0, const double* mult,
                                            const cplx<T>* A1, const cplx<T>* B1, int n1, long ld, int npw, int nj,
                                            cplx<double>* out, T* red) {
  if (nj == 1) block_dots_nj<T, 1>(A0, B0, n0, mult, A1, B1, n1, ld, npw, nj, out, red);
  else if (nj == 2) block_dots_nj<T, 2>(A0, B0, n0, mult, A1, B1, n1, ld, npw, nj, out, red);
  else block_dots_nj<T, 4>(A0, B0, n0, mult, A1, B1, n1, ld, npw, nj, out, red);
}
template <typename T>
__device__ __forceinline__ void block_dots(const cplx<T>* A, const cplx<T>* B, long ld, int npw, int ni, int nj,
                                           cplx<double>* out, T* red) {
  block_dots2<T>(A, B, ni, nullptr, A, B, 0, ld, npw, nj, out, red);
}

// The sums over the block of every thread's (re, im), lanes in T, warps with DSum, to thread 0 as
// out[0].  `red`: two T per warp.  Called by the whole block; ends synchronised.
template <typename T>
__device__ __forceinline__ void block_sum2(T re, T im, cplx<double>* out, T* red) {
  T v[2] = {re, im};
  const int lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  const T t = warp_sums<T, 2>(v);
  if (lane % 16 == 0) red[(threadIdx.x >> 5) * 2 + lane / 16] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    DSum<T> a, b;
    for (int w = 0; w < nw; ++w) a.add(red[2 * w]), b.add(red[2 * w + 1]);
    out[0] = mk(a.value(), b.value());
  }
  __syncthreads();
}

// acc[v] += sign sum_r M[r][g] C[r*ldc + v], v < nv <= NV, over nr rows of M (row stride ldm; C in
// shared memory): every value of M is loaded once for NV bands.
template <typename T, int SIGN, int NV>
__device__ __forceinline__ void rows_times(cplx<T> (&acc)[NV], const cplx<T>* __restrict__ M, long ldm, int nr,
                                           const cplx<T>* C, int ldc, int nv) {
#pragma unroll 4
  for (int r = 0; r < nr; ++r) {
    const cplx<T> m = M[r * ldm];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const cplx<T> c = C[r * ldc + min(v, nv - 1)];
      if (SIGN > 0) {
        acc[v].x += m.x * c.x - m.y * c.y;
        acc[v].y += m.x * c.y + m.y * c.x;
      } else {
        acc[v].x -= m.x * c.x - m.y * c.y;
        acc[v].y -= m.x * c.y + m.y * c.x;
      }
    }
  }
}

// x[v][g] -= sum_w U[w][g] S[w][v] for nv orbitals x of one k against its nbnd occupied
// states U (S = U^H x, nbnd x nv).  The coefficients are rounded to T once: conversions from
// double run on the slow FP64 pipe.
// nv <= NB nbnd: NB blocks of bands (v_hat and w_hat of the non-Hermitian update: 2).
template <typename T, int NB = 1>
__device__ __forceinline__ void subtract_projection(cplx<T>* x, const cplx<T>* __restrict__ uk, const cplx<double>* S, int nbnd,
                                                    int nv, int npw_pad) {
  __shared__ cplx<T> St[NB * 32 * 32];
  for (int i = threadIdx.x; i < nbnd * nv; i += blockDim.x) St[i] = mk((T)S[i].x, (T)S[i].y);
  __syncthreads();
  band_blocks(nv, [&](auto nc) {
    constexpr int NV = decltype(nc)::v;
    const int nb = (nv + NV - 1) / NV;
    for (int i = threadIdx.x; i < nb * npw_pad; i += blockDim.x) {
      const int v0 = i / npw_pad * NV, gi = i % npw_pad, n = min(NV, nv - v0);
      cplx<T> acc[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = v < n ? x[(long)(v0 + v) * npw_pad + gi] : czero<T>();
      rows_times<T, -1>(acc, uk + gi, npw_pad, nbnd, St + v0, nv, n);
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (v < n) x[(long)(v0 + v) * npw_pad + gi] = acc[v];
    }
  });
  __syncthreads();
}

// Metals (Sec. 2.6; smeared occupations f).  With c_mv = max(1 - f_m/f_v, 0) the weight of the
// projector on empty states P_{c,v} for the states m of k+Q and band v of k, the library
// iterates on z = Q^-1 (sqrt(f_v) x), Q = P_{c,v}^{1/2} (weight sqrt(c_mv) on the states of
// k+Q kept, 1 off them): there the operator D + Q W Q is symmetric (W: the Hartree-XC response
// of the density of Q z with the weights sqrt(f_v) folded into u_k), so the recursions need no
// metric, and the components along the kept states are not scaled down by sqrt(c) (in FP32 a
// scaled-down component would carry rounding blown up by 1/sqrt(c) into the scalar products).
// The image Q z feeds the FFT pipeline; the per-k projections restore Q^-1.  With Delta_mv =
// eps_{m,k+Q} - eps_{vk}, four [nks][nbnd (m)][nbnd (v)] tables in double:
//   sp   = 1 - sqrt(c) (1 where c = 0)  coefficient of S = U^H t in the operator's projection
//   da   = [c > 0] (1 - c) Delta        coefficient of Z = U^H z there (D's component along m)
//   keep = [c == 0]                     the projection P'_v of the Lanczos vectors
//   qh   = [c > 0] (1 - sqrt(c))        the image: Q z = z - U (qh Z)
// All null: an insulator.
struct MetalDev {
  const double* sp;
  const double* da;
  const double* keep;
  const double* qh;
};

static __device__ __forceinline__ long metal_idx(int k, int m, int v, int nbnd) {
  return ((long)k * nbnd + m) * nbnd + v;
}

// The sum of one double per thread over the block, in a fixed order (threads' values by warp,
// then the warps in order); every thread gets it.  Ends synchronised.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double wsum[32];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += wsum[w];
  __syncthreads();
  return t;
}

// x <- P_c x for every orbital of k (in place); with coef ([nks][nbnd][nbnd], m-major), the
// component along u_m of band v is removed with weight coef[k][m][v] instead of 1.  The bands
// of k are independent: grid (nks, nvec, nsplit) with nsplit dividing nbnd, each CTA taking
// nbnd/nsplit of them.  block 128.
template <typename T>
__global__ void __launch_bounds__(128) k_project(int nks, int nbnd, int npw_pad, const int* __restrict__ npw,
                                                 const cplx<T>* __restrict__ ukq, cplx<T>* __restrict__ x,
                                                 const double* __restrict__ coef) {
  __shared__ cplx<double> cf[32 * 32];
  __shared__ T red[red_elems(128)];
  const int k = blockIdx.x, vec = blockIdx.y;
  const int nv = nbnd / gridDim.z, v0 = blockIdx.z * nv;
  const long base = (((long)vec * nks + k) * nbnd + v0) * npw_pad;
  const cplx<T>* uk = ukq + (long)k * nbnd * npw_pad;
  block_dots<T>(uk, x + base, npw_pad, npw[k], nbnd, nv, cf, red);
  if (coef) {
    for (int i = threadIdx.x; i < nbnd * nv; i += blockDim.x) {
      const int m = i / nv;
      const double c = coef[((long)k * nbnd + m) * nbnd + v0 + i - m * nv];
      cf[i] = mk(cf[i].x * c, cf[i].y * c);
    }
    __syncthreads();
  }
  subtract_projection<T>(x + base, uk, cf, nbnd, nv, npw_pad);
}

// A metal's image of a batch vector z for the FFT pipeline: img = Q z = z - U (qh Z) and
// zp = [c > 0] Z, Z = U^H z (double), per (vector, k).  grid (nks, nvec), block 256.
template <typename T>
__global__ void __launch_bounds__(256) k_metal_image(int nks, int nbnd, int npw_pad, const int* __restrict__ npw,
                                                     const cplx<T>* __restrict__ ukq, const cplx<T>* __restrict__ z,
                                                     cplx<T>* __restrict__ img, cplx<double>* __restrict__ zp,
                                                     MetalDev md) {
  __shared__ cplx<double> cf[32 * 32];
  __shared__ T red[red_elems(256)];
  const int k = blockIdx.x, vec = blockIdx.y;
  const long base = ((long)vec * nks + k) * nbnd * npw_pad;
  const cplx<T>* uk = ukq + (long)k * nbnd * npw_pad;
  block_dots<T>(uk, z + base, npw_pad, npw[k], nbnd, nbnd, cf, red);
  for (int i = threadIdx.x; i < nbnd * nbnd; i += blockDim.x) {
    const long ci = (long)k * nbnd * nbnd + i;
    const cplx<double> v = cf[i];
    const double kept = md.keep[ci] == 0.0 ? 1.0 : 0.0, q = md.qh[ci];
    zp[(long)vec * nks * nbnd * nbnd + ci] = mk(v.x * kept, v.y * kept);
    cf[i] = mk(v.x * q, v.y * q);
  }
  for (int i = threadIdx.x; i < nbnd * npw_pad; i += blockDim.x) img[base + i] = z[base + i];
  __syncthreads();
  subtract_projection<T>(img + base, uk, cf, nbnd, nbnd, npw_pad);
}

// ---------------------------------------------------------------------------------------
// Device-side Lanczos bookkeeping.
struct Coef {
  double* beta;            // [cap]
  cplx<double>* gamma;     // [cap]
  cplx<double>* zpart;     // [cap][nks]  per-k partials of z_j
  int* err;                // [2] code, first failing step
};

__device__ __forceinline__ void flag_error(int* err, int code, int step) {
  if (atomicCAS(err, 0, code) == 0) err[1] = step;
}

// Start of pseudo-Hermitian step j: the device step counter is advanced to j (so that a captured
// step can be replayed), and beta_j from the n partials of Re(r_j^H X_j) in a fixed order;
// scal = {beta_j, 1/beta_j} for the update kernels.  One block.  (Every CTA of the update
// reduced the partials and divided by itself before: on the KB workload 512 CTAs x 256 threads of
// FP64 adds and divisions, 2 FP64 lanes per SM and cycle.)
static __global__ void __launch_bounds__(256) k_ph_beta(int* __restrict__ jdev, const double* __restrict__ part, int n,
                                                       int nks, Coef co, double tol, double* __restrict__ scal) {
  __shared__ double wsum[8];
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 256) s += part[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    const int j = *jdev + 1;
    double t = 0.0, b = 1.0;
    for (int w = 0; w < 8; ++w) t += wsum[w];
    const double b2 = t / nks;
    if (!(b2 > tol)) flag_error(co.err, b2 <= 0.0 ? DEV_NOTPD : DEV_BREAKDOWN, j);
    else b = sqrt(b2);
    co.beta[j - 1] = b;
    co.gamma[j - 1] = mk(b, 0.0);
    scal[0] = b;
    scal[1] = 1.0 / b;
    *jdev = j;
  }
}

// Pseudo-Hermitian step j (device step counter) for one band group of one k-point (P_c, the norm
// and z act band by band, so groups of bpc bands are independent): with beta_j from k_ph_beta,
// the group's z_j partial, r_{j+1} = P_c(X_j/beta_j - beta_j v_{j-1}) formed in shared memory and
// written to R (a metal: keep = MetalDev::keep, the projection P'_v), v_j = r_j/beta_j.  The
// sphere columns of r_{j+1} are then inverse-FFT'd along axis 3 by k_zinv.  grid (nks, ngrp),
// block proj_threads.  smem: r [bpc][npw_pad], S [nbnd*bpc] (double complex), reduction scratch.
template <typename T>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1) k_ph_update(const int* __restrict__ jdev, SphereDev s, int nbnd, int bpc,
                                                   const double* __restrict__ scal, cplx<T>* __restrict__ R,
                                                   const cplx<T>* __restrict__ X, cplx<T>* __restrict__ Vp,
                                                   const cplx<T>* __restrict__ y, const cplx<T>* __restrict__ ukq,
                                                   Coef co, const double* __restrict__ keep) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int j = *jdev, r_upper = (j % 2 == 0) ? 1 : 0;   // step index from the device counter
  const int npw_pad = s.npw_pad, nks = s.nks;
  const int k = blockIdx.x, grp = blockIdx.y, ngrp = gridDim.y;
  cplx<T>* rs = reinterpret_cast<cplx<T>*>(smem_raw);
  cplx<double>* cf = reinterpret_cast<cplx<double>*>(rs + bpc * npw_pad);
  T* red = reinterpret_cast<T*>(cf + nbnd * bpc);
  const long base = ((long)k * nbnd + grp * bpc) * npw_pad;
  const int np = s.npw[k];
  const long zi = (long)(j - 1) * nks * ngrp + (long)k * ngrp + grp;
  const T ib = (T)scal[1], bb = (T)scal[0];
  T zr = T(0), zim = T(0);   // z_j partial = (y, r_j) over the group's bands (r_j upper; beta_j: k_reduce_z)
#pragma unroll 4
  for (int i = threadIdx.x; i < bpc * npw_pad; i += blockDim.x) {
    const cplx<T> r = R[base + i], x = X[base + i], v = Vp[base + i];
    if (r_upper) {
      const cplx<T> yv = y[base + i];
      zr += yv.x * r.x + yv.y * r.y;
      zim += yv.x * r.y - yv.y * r.x;
    }
    rs[i] = x * ib - v * bb;
    Vp[base + i] = r * ib;
  }
  if (r_upper) block_sum2<T>(zr, zim, cf, red);
  else __syncthreads();
  if (threadIdx.x == 0) co.zpart[zi] = r_upper ? cf[0] : mk(0.0, 0.0);
  const cplx<T>* uk = ukq + (long)k * nbnd * npw_pad;
  block_dots<T>(uk, rs, npw_pad, np, nbnd, bpc, cf, red);
  if (keep) {  // a metal: only the states with c_mv = 0 are removed
    for (int i = threadIdx.x; i < nbnd * bpc; i += blockDim.x) {
      const int m = i / bpc;
      const double c = keep[metal_idx(k, m, grp * bpc + i - m * bpc, nbnd)];
      cf[i] = mk(cf[i].x * c, cf[i].y * c);
    }
    __syncthreads();
  }
  subtract_projection<T>(rs, uk, cf, nbnd, bpc, npw_pad);
  for (int i = threadIdx.x; i < bpc * npw_pad; i += blockDim.x) R[base + i] = rs[i];
}

// A metal's projection coefficients of the operator for one band group of k (kept out of line:
// the insulators' kernel keeps its registers): cf <- sp S - da Z (Z = U^H z of the input, from
// k_metal_image), so that the output's component along a kept u_m is sqrt(c) S + (1 - c)
// Delta Z; returns the term sum qh Re(conj(Z) <u_m|X>) that turns the partial Re(Q z, X) the
// kernel forms into Re(z, X) (to every thread).
static __device__ __noinline__ double metal_operator_coefs(const MetalDev md, int k, int v0, int nbnd, int bpc,
                                                    const cplx<double>* zp, cplx<double>* cf) {
  double corr = 0.0;
  for (int i = threadIdx.x; i < nbnd * bpc; i += blockDim.x) {
    const int m = i / bpc;
    const long ci = metal_idx(k, m, v0 + i - m * bpc, nbnd);
    const cplx<double> sv = cf[i], zv = zp[ci];
    const double p = md.sp[ci], d = md.da[ci];
    const cplx<double> c = mk(p * sv.x - d * zv.x, p * sv.y - d * zv.y);
    corr += md.qh[ci] * (zv.x * (sv.x - c.x) + zv.y * (sv.y - c.y));   // Re conj(Z) <u_m|X>
    cf[i] = c;
  }
  return block_sum(corr);
}

// Columns -> sphere: forward FFT of the columns along axis 3, gather (1/N^3) and the kinetic term,
// t = (1/2|k+Q+G|^2 - eps_vk) x + gathered, written to xout.  One thread per column line;
// grid (nks, nvec, lines), block kLines.  PR as for k_zinv.
constexpr int kLines = 128;
template <typename T, int N, int PR = 0>
__global__ void __launch_bounds__(kLines) k_zfwd(SphereDev s, int nbnd, const cplx<T>* __restrict__ cbuf, int cb_ncol,
                                                 const cplx<T>* __restrict__ xin, const T* __restrict__ kin,
                                                 const double* __restrict__ eps, cplx<T>* __restrict__ xout) {
  const int k = blockIdx.x, vec = blockIdx.y, nks = s.nks, npw_pad = s.npw_pad;
  const int nc = s.ncol[k];
  const int it = blockIdx.z * kLines + threadIdx.x;
  if (it >= nbnd * nc) return;
  const int v = it / nc, c = it - v * nc;
  const long o = ((long)vec * nks + k) * nbnd + v;
  const int4 cl = s.col[k * s.ncol_max + c];
  if (!LL_INB(c < cb_ncol)) return;
  const cplx<T>* src = cbuf + o * (long)N * cb_ncol + c;
  cplx<T> a[N];
#pragma unroll
  for (int p = 0; p < N; ++p) a[p] = src[(long)p * cb_ncol];
  const T ev = (T)eps[k * nbnd + v];
  const int st = s.colstart[k * s.ncol_max + c];
  const cplx<T>* x = xin + o * npw_pad + st;
  const T* kn = kin + (long)k * npw_pad + st;
  cplx<T>* t = xout + o * npw_pad + st;
  line_transform<T, N, -1>(a);
  const T scale = T(1) / T(N * N * N);
#pragma unroll
  for (int p = 0; p < N; ++p)
    if (line_kept<N, PR>(p)) {
      const int i = PR > 0 ? line_m<N, PR>(p, cl.z) - cl.z : wrapn<N>(p - cl.z);
      if ((unsigned)i < (unsigned)cl.w && LL_INB(st >= 0 && st + i < npw_pad)) t[i] = x[i] * (kn[i] - ev) + a[p] * scale;
    }
}

// Threads of the per-k projection kernels: 512 beyond three rounds of 256 (a band's 1632 plane waves
// of the eight-atom cell are then four long rounds of loads in flight; it has 1.7 CTAs per SM), else
// 256 (four CTAs per SM: the KB workload's 512 k-points of 570 plane waves are one wave).  In FP64
// on the KB workload, us per launch at 128 | 256: k_op_proj 411 | 429, k_ph_update 176 | 170.
static inline int proj_threads(int npw_pad) { return npw_pad > 768 ? 512 : 256; }

// Last stage of the operator, for one group of bpc bands of one k-point (the KB and P_c terms act
// band by band): from t (k_zfwd's output, in xout), + KB sum_p beta_p D_p <beta_p|x>, then P_c,
// the output X (in place) and the group's partial Re(x^H X) (a metal: x is the image Q z, zp
// holds Z = U^H z per vector; the output is the operator on z through the MetalDev tables, and the
// partial Re(z^H X)).
// P_c of the KB term goes through the overlaps ub = U^H B of the set-up, S = U^H t + ub c, so
// both dot blocks are formed on the same data and KB, P_c, the output and the norm partial
// are one pass over the plane waves, a block of bands of a plane wave per thread (band_blocks).
// grid (nks, nvec, ngrp), block proj_threads.  smem: coefficients, scratch.
// A kernel of its own: with the column transforms in front it needed 123 registers, two CTAs per
// SM and 1.7 waves on the KB workload's 512 k-points, and shared memory for x and t.  Measured
// (GB300, FP32, us per launch; the one kernel -> k_zfwd + this one): eight-atom cell (16 bands,
// 1632 plane waves) 128 -> 27 + 77, KB workload (4 bands, 570) 61 -> 19 + 40, two-atom 10 Ry cell
// (147) 15 -> 6 + 9.
template <typename T>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1) k_op_proj(SphereDev s, int nbnd, int bpc,
                                                   const cplx<T>* __restrict__ xin, const cplx<T>* __restrict__ ukq,
                                                   const cplx<T>* __restrict__ bkq, const double* __restrict__ dij,
                                                   const cplx<double>* __restrict__ ub, int nproj,
                                                   cplx<T>* xout, double* __restrict__ part, MetalDev md,
                                                   const cplx<double>* __restrict__ zp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int npw_pad = s.npw_pad, nks = s.nks;
  const int k = blockIdx.x, vec = blockIdx.y, grp = blockIdx.z, ngrp = gridDim.z;
  const int v0 = grp * bpc;
  cplx<double>* cf = reinterpret_cast<cplx<double>*>(smem_raw);   // [nproj + nbnd][bpc]: c, then S
  cplx<T>* ct = reinterpret_cast<cplx<T>*>(cf + (nproj + nbnd) * bpc);      // the coefficients in T
  T* red = reinterpret_cast<T*>(ct + (nproj + nbnd) * bpc);
  const long base = (((long)vec * nks + k) * nbnd + v0) * npw_pad;          // first orbital of the group
  const int np = s.npw[k];
  const cplx<T>* bk = bkq + (long)k * nproj * npw_pad;
  const cplx<T>* uk = ukq + (long)k * nbnd * npw_pad;
  cplx<T>* ts = xout + base;   // a thread meets the same plane waves of t in both passes (L1)
  cplx<double>* sf = cf + nproj * bpc;
  block_dots2<T>(bk, xin + base, nproj, dij, uk, ts, nbnd, npw_pad, np, bpc, cf, red);   // D_p <beta_p|x_v>, U^H t
  if (nproj > 0) {
    const cplx<double>* ubk = ub + (long)k * nbnd * nproj;
    for (int i = threadIdx.x; i < nbnd * bpc; i += blockDim.x) {   // + U^H B c
      const int w = i / bpc, v = i - w * bpc;
      cplx<double> a = sf[i];
      for (int p = 0; p < nproj; ++p) a = a + cmul(ubk[w * nproj + p], cf[p * bpc + v]);
      sf[i] = a;
    }
    __syncthreads();
  }
  const double corr =
      md.sp ? metal_operator_coefs(md, k, v0, nbnd, bpc, zp + (long)vec * nks * nbnd * nbnd, sf) : 0.0;
  for (int i = threadIdx.x; i < (nproj + nbnd) * bpc; i += blockDim.x) ct[i] = mk((T)cf[i].x, (T)cf[i].y);
  __syncthreads();
  T nr = T(0);
  band_blocks(bpc, [&](auto nc) {
    constexpr int NV = decltype(nc)::v;
    const int nb = (bpc + NV - 1) / NV;
    for (int i = threadIdx.x; i < nb * npw_pad; i += blockDim.x) {
      const int b0 = i / npw_pad * NV, gi = i % npw_pad, n = min(NV, bpc - b0);
      cplx<T> acc[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = v < n ? ts[(b0 + v) * npw_pad + gi] : czero<T>();
      rows_times<T, +1>(acc, bk + gi, npw_pad, nproj, ct + b0, bpc, n);
      rows_times<T, -1>(acc, uk + gi, npw_pad, nbnd, ct + nproj * bpc + b0, bpc, n);
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (v < n) {
          const long o = base + (long)(b0 + v) * npw_pad + gi;
          const cplx<T> x = xin[o];
          (void)LL_INB(gi < np || (acc[v].x == T(0) && acc[v].y == T(0)));   // the padding is zero
          nr += x.x * acc[v].x + x.y * acc[v].y;
          xout[o] = acc[v];
        }
    }
  });
  block_sum2<T>(nr, T(0), cf, red);
  if (threadIdx.x == 0) part[((long)vec * nks + k) * ngrp + grp] = cf[0].x + corr;
}

// Non-Hermitian step j after the two operator applications XV = L v_j, XW = L^dag w_j, for
// one group of bpc bands of one k-point: v_hat = P_c(XV - gamma_j v_{j-1}), w_hat =
// P_c(XW - conj(beta_j) w_{j-1}) (stored in XV, XW), the group's partials of s = (w_hat,
// v_hat) and of z_j = (y, v_j) (a metal: keep = MetalDev::keep, the projection P'_v).
// grid (nks, ngrp), block proj_threads.
template <typename T>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1) k_nh_update(int j, int upper, int nks, int nbnd, int bpc, int npw_pad,
                                                   const int* __restrict__ npw, cplx<T>* __restrict__ XV,
                                                   cplx<T>* __restrict__ XW, const cplx<T>* __restrict__ Vp,
                                                   const cplx<T>* __restrict__ Wp, const cplx<T>* __restrict__ Vc,
                                                   const cplx<T>* __restrict__ y, const cplx<T>* __restrict__ ukq,
                                                   Coef co, cplx<double>* __restrict__ spart,
                                                   const double* __restrict__ keep) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<T>* vs = reinterpret_cast<cplx<T>*>(smem_raw);          // [bpc][npw_pad]
  cplx<T>* ws = vs + bpc * npw_pad;
  cplx<double>* cf = reinterpret_cast<cplx<double>*>(ws + bpc * npw_pad);   // [nbnd * 2 bpc]
  T* red = reinterpret_cast<T*>(cf + nbnd * 2 * bpc);
  const int k = blockIdx.x, grp = blockIdx.y, ngrp = gridDim.y;
  const long base = ((long)k * nbnd + grp * bpc) * npw_pad;
  const long zi = (long)(j - 1) * nks * ngrp + (long)k * ngrp + grp;
  const int np = npw[k];
  const double bj = co.beta[j - 1];
  const cplx<double> gj = co.gamma[j - 1];
  const cplx<T> g = mk((T)gj.x, (T)gj.y), bc = mk((T)bj, (T)0);
  T zr = T(0), zim = T(0);   // z_j partial = (y, v_j) over the group's bands
#pragma unroll 2
  for (int i = threadIdx.x; i < bpc * npw_pad; i += blockDim.x) {
    if (upper) {
      const cplx<T> yv = y[base + i], v = Vc[base + i];
      zr += yv.x * v.x + yv.y * v.y;
      zim += yv.x * v.y - yv.y * v.x;
    }
    vs[i] = XV[base + i] - cmul(g, Vp[base + i]);
    ws[i] = XW[base + i] - cmul(bc, Wp[base + i]);
  }
  if (upper) block_sum2<T>(zr, zim, cf, red);
  else __syncthreads();
  if (threadIdx.x == 0) co.zpart[zi] = upper ? cf[0] : mk(0.0, 0.0);
  const cplx<T>* uk = ukq + (long)k * nbnd * npw_pad;
  // v_hat and w_hat are 2 bpc consecutive rows: one dot block and one pass of P_c for both
  block_dots<T>(uk, vs, npw_pad, np, nbnd, 2 * bpc, cf, red);
  if (keep) {  // a metal: P'_v, only the states with c_mv = 0 removed
    for (int i = threadIdx.x; i < nbnd * 2 * bpc; i += blockDim.x) {
      const int m = i / (2 * bpc), v = (i - m * 2 * bpc) % bpc;
      const double c = keep[metal_idx(k, m, grp * bpc + v, nbnd)];
      cf[i] = mk(cf[i].x * c, cf[i].y * c);
    }
    __syncthreads();
  }
  subtract_projection<T, 2>(vs, uk, cf, nbnd, 2 * bpc, npw_pad);
  T sr = T(0), si = T(0);
  for (int i = threadIdx.x; i < bpc * npw_pad; i += blockDim.x) {
    const cplx<T> v = vs[i], w = ws[i];
    XV[base + i] = v;
    XW[base + i] = w;
    sr += w.x * v.x + w.y * v.y;
    si += w.x * v.y - w.y * v.x;
  }
  block_sum2<T>(sr, si, cf, red);
  if (threadIdx.x == 0) spart[(long)k * ngrp + grp] = cf[0];
}

// Non-Hermitian scalars at the end of step j from the n partials of s = (w_hat, v_hat) (fixed
// order): beta_{j+1} = sqrt|s|, gamma_{j+1} = s/beta_{j+1}; scal = {1/beta, Re, Im of
// 1/conj(gamma)}.  One block.
static __global__ void __launch_bounds__(256) k_nh_scalars(int j, int n, int nks, const cplx<double>* __restrict__ spart,
                                                           Coef co, double tol, double* __restrict__ scal) {
  __shared__ double wr[8], wi[8];
  double sr = 0.0, si = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 256) {
    sr += spart[i].x;
    si += spart[i].y;
  }
  sr = warp_sum(sr);
  si = warp_sum(si);
  if ((threadIdx.x & 31) == 0) { wr[threadIdx.x >> 5] = sr; wi[threadIdx.x >> 5] = si; }
  __syncthreads();
  if (threadIdx.x == 0) {
    sr = si = 0.0;
    for (int w = 0; w < 8; ++w) sr += wr[w], si += wi[w];
    sr /= nks;
    si /= nks;
    const double a = sqrt(sr * sr + si * si);
    double b = sqrt(a);
    cplx<double> gm = mk(sr / b, si / b);
    if (!(a > tol)) { flag_error(co.err, DEV_BREAKDOWN, j + 1); b = 1.0; gm = mk(1.0, 0.0); }
    co.beta[j] = b;
    co.gamma[j] = gm;
    const double gg = gm.x * gm.x + gm.y * gm.y;   // 1/conj(gamma) = gamma/|gamma|^2
    scal[0] = 1.0 / b;
    scal[1] = gm.x / gg;
    scal[2] = gm.y / gg;
  }
}

// Non-Hermitian normalisation in place, v_hat/beta and w_hat/conj(gamma) (one vector's n values
// after the other): they are v_{j+1}, w_{j+1}, and the chain's three pairs of vectors take turns
// (v_j stays where it is and is v_{j-1} of the next step).  Bound by memory: 4 n values moved
// (8 n when v_j was copied).
template <typename T>
__global__ void __launch_bounds__(256) k_nh_normalize(long n, cplx<T>* __restrict__ XV, cplx<T>* __restrict__ XW,
                                                      const double* __restrict__ scal) {
  const T ib = (T)scal[0];
  const cplx<T> igc = mk((T)scal[1], (T)scal[2]);
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    XV[i] = XV[i] * ib;
    XW[i] = cmul(XW[i], igc);
  }
}

// The device step counter of the pseudo-Hermitian recursion before a run of steps (k_ph_beta
// advances it).
static __global__ void k_step_set(int* jdev, int j) { *jdev = j; }

// z_j = (1/nks) sum zpart[j][0..nzp) for j in [j0, j0 + gridDim.x), divided by beta_j where given (the
// pseudo-Hermitian partials are (y, r_j), v_j = r_j/beta_j): nzp partials per step, one per (k, band
// group) or (k, chunk) on the split path, one block per step, fixed order.  (One thread per step
// took 68 us for the KB workload's 512 partials.)
static __global__ void __launch_bounds__(128) k_reduce_z(const cplx<double>* __restrict__ zpart, int nzp, int nks, int j0,
                                                        const double* __restrict__ beta, cplx<double>* __restrict__ z) {
  __shared__ double wr[4], wi[4];
  const int j = j0 + blockIdx.x;
  double zr = 0, zi = 0;
  for (int k = threadIdx.x; k < nzp; k += 128) { zr += zpart[(long)j * nzp + k].x; zi += zpart[(long)j * nzp + k].y; }
  zr = warp_sum(zr);
  zi = warp_sum(zi);
  if ((threadIdx.x & 31) == 0) { wr[threadIdx.x >> 5] = zr; wi[threadIdx.x >> 5] = zi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double d = beta ? beta[j] * nks : (double)nks;
    z[j] = mk((wr[0] + wr[1] + wr[2] + wr[3]) / d, (wi[0] + wi[1] + wi[2] + wi[3]) / d);
  }
}

// ---------------------------------------------------------------------------------------
// Set-up kernels.
// For each Miller of sphere(k+Q): its index in sphere(k) (both lexicographic), or -1.
static __global__ void k_intersection_map(int nks, const int* __restrict__ off_k, const int* __restrict__ npw_k,
                                   const int* __restrict__ mil_k, const int* __restrict__ off_q,
                                   const int* __restrict__ npw_q, const int* __restrict__ mil_q, int npw_pad,
                                   int* __restrict__ map) {
  const int k = blockIdx.x;
  const int* mk_ = mil_k + 3L * off_k[k];
  const int n = npw_k[k];
  for (int i = threadIdx.x; i < npw_pad; i += blockDim.x) {
    int res = -1;
    if (i < npw_q[k]) {
      const int* q = mil_q + 3L * (off_q[k] + i);
      int lo = 0, hi = n - 1;
      while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int* m = mk_ + 3 * mid;
        int c = (m[0] != q[0]) ? (m[0] < q[0] ? -1 : 1)
              : (m[1] != q[1]) ? (m[1] < q[1] ? -1 : 1)
              : (m[2] != q[2]) ? (m[2] < q[2] ? -1 : 1) : 0;
        if (c == 0) { res = mid; break; }
        if (c < 0) lo = mid + 1; else hi = mid - 1;
      }
    }
    map[(long)k * npw_pad + i] = res;
  }
}

// y_{vk}(G) = u_{vk}(G) where G is also in sphere(k), else 0 (projection follows).
// grid (nks, nbnd), block 128.
template <typename T>
__global__ void k_gather_y(int nks, int nbnd, int npw_pad_q, int npw_pad_k, const int* __restrict__ map,
                           const cplx<T>* __restrict__ uk, cplx<T>* __restrict__ y) {
  const int k = blockIdx.x, v = blockIdx.y;
  for (int g = threadIdx.x; g < npw_pad_q; g += blockDim.x) {
    const int m = map[(long)k * npw_pad_q + g];
    y[((long)k * nbnd + v) * npw_pad_q + g] =
        (m >= 0 && LL_INB(m < npw_pad_k)) ? uk[((long)k * nbnd + v) * npw_pad_k + m] : czero<T>();
  }
}

// ALDA kernel f_xc = d v_xc/dn of Slater exchange + Perdew-Zunger 1981 correlation, in
// double, from the ground-state density; 0 where n <= 1e-10.
__device__ __forceinline__ double pz81_fxc(double n) {
  if (!(n > 1e-10)) return 0.0;
  const double pi = 3.14159265358979323846;
  const double rs = cbrt(3.0 / (4.0 * pi * n));
  const double cx = 0.75 * cbrt(3.0 / pi);
  const double fx = -4.0 / 9.0 * cx * pow(n, -2.0 / 3.0);
  double d1, d2;
  if (rs >= 1.0) {
    const double g = -0.1423, b1 = 1.0529, b2 = 0.3334;
    const double s = sqrt(rs);
    const double den = 1.0 + b1 * s + b2 * rs;
    const double dden = b1 / (2.0 * s) + b2;
    const double d2den = -b1 / (4.0 * s * s * s);
    d1 = -g * dden / (den * den);
    d2 = -g * (d2den * den - 2.0 * dden * dden) / (den * den * den);
  } else {
    const double A = 0.0311, C = 0.0020, D = -0.0116;
    d1 = A / rs + C * (log(rs) + 1.0) + D;
    d2 = -A / (rs * rs) + C / rs;
  }
  const double dvc = 2.0 / 3.0 * d1 - rs / 3.0 * d2;
  return fx + dvc * (-rs / (3.0 * n));
}

// ---- set-up from device-resident inputs (ll_system_desc.where = LL_WHERE_DEVICE) --------

// The smallest index of a NaN or infinity among n values into *first, which the caller sets
// to all ones beforehand (left so when every value is finite).
static __global__ void k_first_nonfinite(const double* __restrict__ p, long n, unsigned long long* first) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    if (!isfinite(p[i])) atomicMin(first, (unsigned long long)i);
}

// Packed complex rows [k][row][npw[k]] (k blocks at nrow * off[k]) -> padded [k][row][npw_pad]
// in T, zero on the padding, each row times rscale[k][row] when given.  grid (nks, nrow),
// block 256.
template <typename T>
__global__ void k_pad_rows(const double* __restrict__ src, const int* __restrict__ off, const int* __restrict__ npw,
                           int nrow, int npw_pad, const double* __restrict__ rscale, cplx<T>* __restrict__ dst) {
  const int k = blockIdx.x, r = blockIdx.y, n = npw[k];
  const double* s = src + 2 * ((long)nrow * off[k] + (long)r * n);
  // u_k only: sqrt of the k-point weight times sqrt of the band's occupation (a metal)
  const double f = rscale ? rscale[(long)k * nrow + r] : 1.0;
  cplx<T>* d = dst + ((long)k * nrow + r) * npw_pad;
  for (int g = threadIdx.x; g < npw_pad; g += blockDim.x)
    d[g] = g < n ? mk((T)(f * s[2 * g]), (T)(f * s[2 * g + 1])) : czero<T>();
}

// The padded rows of one batch vector back in the packed layout, in double.  grid (nks, nrow), block 256.
template <typename T>
__global__ void k_unpad_rows(const cplx<T>* __restrict__ src, const int* __restrict__ off, const int* __restrict__ npw,
                             int nrow, int npw_pad, double* __restrict__ dst) {
  const int k = blockIdx.x, r = blockIdx.y, n = npw[k];
  const cplx<T>* s = src + ((long)k * nrow + r) * npw_pad;
  double* d = dst + 2 * ((long)nrow * off[k] + (long)r * n);
  for (int g = threadIdx.x; g < n; g += blockDim.x) {
    const cplx<T> v = s[g];
    d[2 * g] = (double)v.x;
    d[2 * g + 1] = (double)v.y;
  }
}

// A grid [j1][j2][j3] -> [j3][j2][j1] in T.
template <typename T>
__global__ void k_grid_in(int n, const double* __restrict__ src, T* __restrict__ dst) {
  const long n3 = (long)n * n * n;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += (long)gridDim.x * blockDim.x) {
    const long j1 = i % n, j2 = (i / n) % n, j3 = i / ((long)n * n);
    dst[i] = (T)src[(j1 * n + j2) * n + j3];
  }
}

// One axis of a grid band-limited and sampled on w of its n points: in [na][n][nb] ->
// out [na][w][nb] = (w/n) sum_j r[j][s] in[.][j][.] (r: the resampling table [n][w]).
static __global__ void k_resample_axis(long na, int n, long nb, int w, const double* __restrict__ r,
                                       const double* __restrict__ in, double* __restrict__ out) {
  const double sc = (double)w / (double)n;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < na * w * nb; i += (long)gridDim.x * blockDim.x) {
    const long b = i % nb, s = (i / nb) % w, a = i / (nb * w);
    double t = 0.0;
    for (int j = 0; j < n; ++j) t += r[(long)j * w + s] * in[(a * n + j) * nb + b];
    out[i] = t * sc;
  }
}

template <typename T>
__global__ void k_fxc(long n3, const double* __restrict__ rho, T* __restrict__ fxc, int on) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n3; i += (long)gridDim.x * blockDim.x)
    fxc[i] = on ? (T)pz81_fxc(rho[i]) : T(0);
}

template <typename T>
__global__ void k_scale(long n, const cplx<T>* __restrict__ a, double s, cplx<T>* __restrict__ out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    out[i] = a[i] * (T)s;
}

// part[k] = Re sum conj(a) b over the k block (for norms).
template <typename T>
__global__ void __launch_bounds__(128) k_dot_re(int nks, int nbnd, int npw_pad, const cplx<T>* __restrict__ a,
                                                const cplx<T>* __restrict__ b, double* __restrict__ part) {
  __shared__ double red[4];
  const int k = blockIdx.x;
  const long base = (long)k * nbnd * npw_pad;
  double acc = 0;
  for (int i = threadIdx.x; i < nbnd * npw_pad; i += blockDim.x) {
    const cplx<T> t = cjmul(a[base + i], b[base + i]);
    acc += (double)t.x;
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    part[k] = s;
  }
}

// ---------------------------------------------------------------------------------------
// Spectrum (Eqs. 32-33, 5): per frequency, with A = (w + i eta) I - T, chi_LL = z^T A^-1 e_1
// = u_1 where A^T u = z, eliminated from the bottom row up (the continued fraction):
//   d_M = w, r_M = z_M;  d_j = w - beta_{j+1} gamma_{j+1} / d_{j+1},
//   r_j = z_j + beta_{j+1} r_{j+1} / d_{j+1};  u_1 = r_1 / d_1.
// chi = pref b_1 u_1, eps^-1 = 1 + v_Q chi, eps = 1/eps^-1.
__device__ __forceinline__ cplx<double> cdiv(cplx<double> a, cplx<double> b) {
  const double d = b.x * b.x + b.y * b.y;
  return mk((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

// Continuation of the coefficients past the m computed ones (Sec. 2.5, Sec. 3.3): for an
// index i >= m, beta_i = b[i % 2] and gamma_i = g[i % 2] ('constant': b[0] = b[1]); z_i = 0.
struct ExtrapTail {
  double b[2];
  cplx<double> g[2];
};

// The tail constants: means over the positions max(1, m/2)..m-1, both parities together
// (kind 1, constant) or each parity apart (kind 2, bi-constant), fixed summation order.
// One block of 256 threads.
static __global__ void __launch_bounds__(256) k_extrap_tail(int m, int kind, const double* __restrict__ beta,
                                                            const cplx<double>* __restrict__ gamma,
                                                            ExtrapTail* __restrict__ tail) {
  __shared__ double red[8][6];
  const int h = m / 2 > 1 ? m / 2 : 1;
  double s[6] = {0, 0, 0, 0, 0, 0};   // per parity: beta, Re gamma, Im gamma
  for (int i = h + threadIdx.x; i < m; i += blockDim.x) {
    const int p = (kind == 2) ? (i & 1) : 0;
    s[3 * p] += beta[i];
    s[3 * p + 1] += gamma[i].x;
    s[3 * p + 2] += gamma[i].y;
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const double v = warp_sum(s[c]);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][c] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[6] = {0, 0, 0, 0, 0, 0};
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
      for (int c = 0; c < 6; ++c) t[c] += red[w][c];
    int n[2] = {0, 0};
    for (int i = h; i < m; ++i) ++n[(kind == 2) ? (i & 1) : 0];
    for (int p = 0; p < 2; ++p) {
      const int q = (kind == 2) ? p : 0;
      const double c = n[q] > 0 ? 1.0 / n[q] : 0.0;
      tail->b[p] = t[3 * q] * c;
      tail->g[p] = mk(t[3 * q + 1] * c, t[3 * q + 2] * c);
    }
  }
}

// 2^-e with e the largest exponent among the arguments (1 where they vanish or are not finite):
// multiplying by it is exact.
__device__ __forceinline__ double pow2_scale(double a, double b, double c, double d) {
  const int e = max(max(__double2hiint(a) & 0x7ff00000, __double2hiint(b) & 0x7ff00000),
                    max(__double2hiint(c) & 0x7ff00000, __double2hiint(d) & 0x7ff00000));
  return (e == 0 || e >= 0x7fe00000) ? 1.0 : __hiloint2double(0x7fe00000 - e, 0);
}

// Double-double values h + l, |l| <= ulp(h)/2 (Dekker 1971; Knuth's two-sum), and their complex
// products, for the matrix power below.
struct dd { double h, l; };
__device__ __forceinline__ dd dd_norm(double h, double l) {   // |h| >= |l|
  const double s = __dadd_rn(h, l);
  return {s, __dadd_rn(l, -__dadd_rn(s, -h))};
}
__device__ __forceinline__ dd dd_prod(double a, double b) {
  const double p = __dmul_rn(a, b);
  return {p, __fma_rn(a, b, -p)};
}
__device__ __forceinline__ dd operator+(dd a, dd b) {
  const double s = __dadd_rn(a.h, b.h), t = __dadd_rn(s, -a.h);
  const double e = __dadd_rn(__dadd_rn(a.h, -__dadd_rn(s, -t)), __dadd_rn(b.h, -t));
  return dd_norm(s, __dadd_rn(e, __dadd_rn(a.l, b.l)));
}
__device__ __forceinline__ dd operator-(dd a) { return {-a.h, -a.l}; }
__device__ __forceinline__ dd operator-(dd a, dd b) { return a + -b; }
__device__ __forceinline__ dd operator*(dd a, dd b) {
  const dd p = dd_prod(a.h, b.h);
  return dd_norm(p.h, __fma_rn(a.h, b.l, __fma_rn(a.l, b.h, p.l)));
}
__device__ __forceinline__ cplx<dd> operator*(cplx<dd> a, cplx<dd> b) { return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ cplx<dd> dd_sqr(cplx<dd> a) {
  const dd t = a.x * a.y;
  return mk(a.x * a.x - a.y * a.y, dd{2.0 * t.h, 2.0 * t.l});
}
__device__ __forceinline__ cplx<double> dd_hi(cplx<dd> a) { return mk(a.x.h, a.y.h); }
__device__ __forceinline__ cplx<dd> dd_scale(cplx<dd> a, double s) {   // s a power of two
  return mk(dd{a.x.h * s, a.x.l * s}, dd{a.y.h * s, a.y.l * s});
}

// The elimination without its divisions: with d_j = P_j / P_{j+1} and r_j = R_j / P_{j+1},
//   P_j = w P_{j+1} - beta_{j+1} gamma_{j+1} P_{j+2},   R_j = z_j P_{j+1} + beta_{j+1} R_{j+1},
// u_1 = R_1 / P_1; P, P_{j+1} and R are scaled together by an exact power of two every fourth
// row.  m_total > m continues the chain with `tail` (T grows to m_total x m_total; z stays m
// long): there R = 0 and the rows repeat with period two, so the whole tail is the
// floor((m_total - m)/2)-th power of one 2 x 2 matrix, formed by repeated squaring.  A squaring
// doubles the relative error of its argument, so the k-th power would carry k roundings where
// the rows carry about sqrt(k): the squarings run in double-double, the power is applied in double.
// Bound by the FP64 pipe (one warp instruction per 16 cycles and SM): 14 FP64 instructions per row
// against about 70 with two complex divisions; one warp per CTA puts 4001 frequencies on 126 SMs
// where 128-thread CTAs used 32.  1000 coefficients continued to 20000 at 4001 frequencies, us per
// call: divisions 68900, this form 740 with every squaring in double, 850 with double-double.  Errors
// against extended precision, divisions / double squarings / this form: 8.6e-15 / 2.1e-15 / 1e-15
// there; 60 coefficients continued to 400 2.0e-14 / 3.0e-14 / 2.1e-15.  Block 32.
static __global__ void __launch_bounds__(32) k_spectrum(int m, int m_total, const ExtrapTail* __restrict__ tail,
                                                        const double* __restrict__ beta,
                                                        const cplx<double>* __restrict__ gamma,
                                                        const cplx<double>* __restrict__ z, int nw,
                                                        const double* __restrict__ w_ha, double eta, double pref,
                                                        double vq, cplx<double>* __restrict__ chi,
                                                        cplx<double>* __restrict__ epsi, cplx<double>* __restrict__ eps) {
  __shared__ cplx<double> sbg[32], sz[32];
  __shared__ double sb[32];
  const int lane = threadIdx.x, i = blockIdx.x * 32 + lane;
  const cplx<double> w = mk(w_ha[min(i, nw - 1)], eta);
  cplx<double> P = w, P1 = mk(1.0, 0.0);
  const int nt = (tail && m_total > m) ? m_total - m : 0;
  if (nt > 0) {
    const int pa = m & 1, pb = pa ^ 1;   // row c takes the constants of parity c % 2; the rows c = m, m + 2, ...: pa
    const cplx<double> ca = tail->g[pa] * tail->b[pa], cb = tail->g[pb] * tail->b[pb];
    if (nt & 1) {
      const cplx<double> t = cmul(w, P) - cmul(ca, P1);
      P1 = P;
      P = t;
    }
    // one period: [[w, -ca], [1, 0]] [[w, -cb], [1, 0]]
    const cplx<dd> wd = mk(dd{w.x, 0.0}, dd{w.y, 0.0}), cad = mk(dd_prod(tail->g[pa].x, tail->b[pa]), dd_prod(tail->g[pa].y, tail->b[pa])),
                   cbd = mk(dd_prod(-tail->g[pb].x, tail->b[pb]), dd_prod(-tail->g[pb].y, tail->b[pb]));
    cplx<dd> a = dd_sqr(wd) - cad, b = cbd * wd, c = wd, d = cbd;
    for (int h = nt >> 1; h; h >>= 1) {
      if (h & 1) {
        const cplx<double> t = cmul(dd_hi(a), P) + cmul(dd_hi(b), P1), u = cmul(dd_hi(c), P) + cmul(dd_hi(d), P1);
        const double s = pow2_scale(t.x, t.y, u.x, u.y);
        P = t * s;
        P1 = u * s;
      }
      if (h == 1) break;
      const cplx<dd> bc = b * c, tr = a + d;
      const cplx<dd> na = dd_sqr(a) + bc, nd = dd_sqr(d) + bc, nb = b * tr, nc = c * tr;
      const double s = fmin(pow2_scale(na.x.h, na.y.h, nb.x.h, nb.y.h), pow2_scale(nc.x.h, nc.y.h, nd.x.h, nd.y.h));
      a = dd_scale(na, s);
      b = dd_scale(nb, s);
      c = dd_scale(nc, s);
      d = dd_scale(nd, s);
    }
  }
  cplx<double> R = cmul(z[m - 1], P1);
  for (int j0 = m - 2; j0 >= 0; j0 -= 32) {   // rows j0, j0 - 1, ...
    __syncwarp();
    if (j0 - lane >= 0) {
      const int j = j0 - lane;
      const double b = beta[j + 1];
      sb[lane] = b;
      sbg[lane] = gamma[j + 1] * b;
      sz[lane] = z[j];
    }
    __syncwarp();
    const int n = min(32, j0 + 1);
    auto row = [&](int q) {
      const cplx<double> zj = sz[q], g = sbg[q];
      const double b = sb[q];
      R = mk(zj.x * P.x - zj.y * P.y + b * R.x, zj.x * P.y + zj.y * P.x + b * R.y);
      const cplx<double> t = mk(w.x * P.x - w.y * P.y - (g.x * P1.x - g.y * P1.y),
                                w.x * P.y + w.y * P.x - (g.x * P1.y + g.y * P1.x));
      P1 = P;
      P = t;
    };
    auto rescale = [&]() {
      const double s = pow2_scale(P.x, P.y, P1.x, P1.y);
      P = P * s;
      P1 = P1 * s;
      R = R * s;
    };
    int q = 0;
    for (; q + 4 <= n; q += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) row(q + u);
      rescale();
    }
    for (; q < n; ++q) row(q);
    rescale();
  }
  if (i >= nw) return;
  const cplx<double> u1 = cdiv(R, P);
  const cplx<double> c = u1 * (pref * beta[0]);
  chi[i] = c;
  const cplx<double> ei = mk(1.0 + vq * c.x, vq * c.y);
  epsi[i] = ei;
  eps[i] = cdiv(mk(1.0, 0.0), ei);
}

}  // namespace ll
