// The per-plane pass of k_xy (kernels.cuh) for spheres whose Miller indices lie within
// |m| <= PR < W/2 on every axis (PR = W/2 - 1: -W/2 too; signed indices are then unique on the grid),
// pipelined with
// bulk copies.  grid (W planes, groups); a CTA takes SL orbitals per batch, one per line slot,
// so every thread (P = 1) or lane pair (P = 2) has exactly one axis-1 row and one axis-2 line of
// the batch:
//   rows     item (b, r) = orbital b of the batch, sphere row r: axis-1 inverse transform of the
//            row's columns in Cs into Ys[b][r][j1]
//   lines    (slot, j1): axis-2 inverse transform of Ys[slot][.][j1], V(r) x(r) (density:
//            conj(u) x added to the thread's own column), axis-2 forward transform back to Ys;
//            pass 2: v'(r) u(r) and the forward transform only
//   rows     axis-1 forward transform, back into Cs (pass 2: added to the columns there)
// Data movement is bulk copies by one warp, off the threads' instruction stream: the plane's
// column-buffer row of every orbital (one contiguous run) two batches ahead into one of two Cs
// buffers and back from it, and in the modes that read the orbital grids u(r) the plane of every
// orbital, one batch ahead, while the rows of this batch and the next are transformed.
//
// FP64 chains run the same pass with fixed-point lines (plane64.cuh).
//
// What bounds it and why this shape (KB workload, FP32, W = 24, 2048 orbitals; the line FFTs are
// 28 us of FMA issue, u(r) 34 us of HBM): the pass it replaces (128 threads, columns staged by
// hand) took 94 / 135 / 87 us (pass 1 / density / pass 2): half its issue slots were index
// arithmetic (m mod W per point), 24-point lines left its warps partly filled, and its u(r) loads
// waited on HBM inside the line loop.  With signed indices every point's offset is a compile-time
// constant and its test one compare, W SL P threads fill their warps for W = 16, 24, 32, 48, and
// the bulk copies are in flight two phases ahead: 63 / 91 / 55 us.  Eight-atom cell (W = 32):
// 115 / 176 / 108 -> 68 / 129 / 62 us; sixteen-atom cell (W = 48): 1654 / 1969 / 1080 -> 868 /
// 1024 / 664 us.
#pragma once
#include "kernels.cuh"
#include "tc.cuh"

namespace ll {

// ---- bulk copies (contiguous, 16-byte aligned addresses and sizes) ----------------------
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the sources of this thread's stores may be overwritten
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// Every wait on a copy is bounded (XYArgs::polls).  A thread whose wait has run out waits for no
// other; once one of warp 0's has, no further copy is asked for (a barrier's next phase is armed only
// when its last one is known to be complete), so the others' waits run out as well and the CTA
// reaches its end.  There one thread records the error and waits, again with a limit, for the copies
// still in flight: cols, us: batches whose columns and u(r) have been asked for.
__device__ __forceinline__ void plane_gave_up(uint64_t* full, uint64_t* ufull, int cols, int us, int* err) {
  flag_error(err, DEV_TIMEOUT, 1);
  for (int b = cols > 2 ? cols - 2 : 0; b < cols; ++b) mbar_wait(&full[b & 1], (b >> 1) & 1);
  if (us > 0) mbar_wait(ufull, (us - 1) & 1);
}

// ---- launch shape ------------------------------------------------------------------------
// P lanes per line and SL line slots for a side, type and mode.  A lane holds W/P points; two
// lanes where one would not keep a line in registers beside its temporaries (W >= 36 in FP32,
// W >= 24 in FP64) or beside the density's column (W = 32).
template <typename T, int W, int MODE> struct PlaneCfg {
  static constexpr bool f64 = sizeof(T) == 8;
  static constexpr int P = (W >= 36 || (W >= 24 && f64) || (W >= 32 && MODE == XY_PASS1_DENS)) ? 2 : 1;
  static constexpr int SL = W == 48 ? (f64 ? 1 : 2) : W == 36 ? 2 : W == 32 ? (P == 2 ? 2 : 4) : W == 24 ? (f64 ? 4 : 8) : 8;
  static constexpr int H = W / P, TH = SL * W * P;
  static constexpr bool acc_reg = MODE == XY_PASS1_DENS && !f64;   // density column in registers (FP64: in shared memory)
  // CTAs per SM that the registers allow, a scheduler's quarter of them (512 per thread of a warp) shared by whole warps
  static constexpr int regs = (f64 ? 4 * H + 96 : 2 * H + (acc_reg ? 2 * H : 0) + 52) + 7;
  static constexpr int warps = (TH + 31) / 32;
  static constexpr int ctas = f64 ? 4 * (512 / (regs / 8 * 8)) / warps : 65536 / (warps * 32 * (regs / 8 * 8));
  static constexpr int min_ctas = ctas < 1 ? 1 : ctas;
};

// Dynamic shared memory: Cs [2][SL][cb_ncol], Us [SL][W][W] (modes with u), Ys [SL][nrow][W + 1],
// density planes [SL][W][W] (not in registers) or one [W][W] (the slots' sum), v' or V [W][W].
template <typename T, int W, int MODE>
size_t plane_smem(int cb_ncol, int nrow) {
  using C = PlaneCfg<T, W, MODE>;
  size_t n = 2 * (size_t)C::SL * cb_ncol + (size_t)C::SL * nrow * (W + 1);
  if (MODE != XY_PASS1) n += (size_t)C::SL * W * W;
  if (MODE == XY_PASS2) n += (size_t)W * W;
  if (MODE == XY_PASS1_DENS) n += (size_t)(C::acc_reg ? 1 : C::SL) * W * W;
  return n * sizeof(cplx<T>) + (MODE == XY_PASS2 ? 0 : (size_t)W * W * sizeof(T));
}

template <typename T, int W, int MODE, int PR>
__global__ void __launch_bounds__(PlaneCfg<T, W, MODE>::TH, PlaneCfg<T, W, MODE>::min_ctas)
    k_plane(XYArgs a, cplx<T>* __restrict__ cbuf, const T* __restrict__ vloc, const cplx<T>* __restrict__ vpr,
            const cplx<T>* __restrict__ ur, cplx<T>* __restrict__ nprt, int* __restrict__ err) {
  using C = PlaneCfg<T, W, MODE>;
  constexpr int P = C::P, SL = C::SL, H = C::H, TH = C::TH;
  constexpr int NP = W + 1, WW = W * W;
  constexpr bool HAS_U = MODE != XY_PASS1;
  // kept points of a lane's half line (P = 2: p = 2 i + h), i <= LO or i >= H - HI
  constexpr int LO = P == 1 ? PR : PR / 2, HI = P == 1 ? line_hi(W, PR) : (PR + 1) / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[2], ufull;
  __shared__ int s_asked[2];   // batches whose columns, u(r) have been asked for
  const SphereDev& s = a.s;
  const int iz = blockIdx.x, g = blockIdx.y, cb = a.cb_ncol;
  cplx<T>* Cs = reinterpret_cast<cplx<T>*>(smem_raw);
  cplx<T>* Us = Cs + 2 * SL * cb;
  cplx<T>* Ys = Us + (HAS_U ? SL * WW : 0);
  cplx<T>* Pb = Ys + SL * s.nrow_max * NP;
  cplx<T>* Pl = Pb + (MODE == XY_PASS1_DENS ? WW : 0);
  T* Pv = reinterpret_cast<T*>(Pl);
  const int t = threadIdx.x;
  if (t == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    mbar_init(&ufull, 1);
    s_asked[0] = s_asked[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (MODE == XY_PASS2) {
    for (int i = t; i < WW; i += TH) Pl[i] = vpr[(long)iz * WW + i];
  } else {
    for (int i = t; i < WW; i += TH) Pv[i] = vloc[(long)iz * WW + i];
  }
  __syncthreads();

  const int o_begin = a.o_off + g * a.per_group;
  const int o_end = a.o_off + min(a.norb, g * a.per_group + a.per_group);
  const int nbat = o_end > o_begin ? (o_end - o_begin + SL - 1) / SL : 0;
  const uint32_t cbytes = (uint32_t)(cb * sizeof(cplx<T>));
  auto dens_orb = [&](int o) { return MODE == XY_PASS2 || a.f_pervec.div(o) == a.dens_vec; };
  auto row_of = [&](int o) { return cbuf + (long)o * W * cb + (long)iz * cb; };
  // warp 0: the columns of batch `it` into its buffer; u(r) of batch `it`
  auto load_cols = [&](int it) {
    const int nb = min(SL, o_end - o_begin - it * SL);
    if (t == 0) {
      s_asked[0] = it + 1;
      mbar_expect(&full[it & 1], nb * cbytes);
    }
    __syncwarp();
    if (t < nb) bulk_load(Cs + ((it & 1) * SL + t) * cb, row_of(o_begin + it * SL + t), cbytes, &full[it & 1]);
  };
  auto load_u = [&](int it) {
    const int o = o_begin + it * SL + t;
    const bool on = t < SL && o < o_end && dens_orb(o);
    const uint32_t n = __popc(__ballot_sync(0xffffffffu, on));
    if (t == 0) {
      s_asked[1] = it + 1;
      mbar_expect(&ufull, n * (uint32_t)(WW * sizeof(cplx<T>)));
    }
    __syncwarp();
    if (on)
      bulk_load(Us + t * WW, ur + ((long)a.f_pervec.mod(o) * W + iz) * WW, (uint32_t)(WW * sizeof(cplx<T>)), &ufull);
  };
  if (t < 32 && nbat > 0) {
    load_cols(0);
    if (HAS_U) load_u(0);
    if (nbat > 1) load_cols(1);
  }
  // this thread's row (b, r) and line (slot, j1) of every batch; P = 2: h = lane of the pair
  const int pr = t / P, h = t % P;
  const unsigned pmask = 3u << (t & 30);
  const int rb = a.f_nrow.div(pr), rr = pr - rb * s.nrow_max;
  const int ls = pr / W, j1 = pr - ls * W;
  int4 rw = make_int4(0, 0, 0, 0);   // row: (m2, first column, m1 of it, columns); none: 0 columns
  bool row_on = false;
  int nr = 0, m2min = 0;             // the line's orbital: rows, first m2
  auto tables = [&](int ob) {
    const int orow = ob + rb, ol = ob + ls;
    row_on = false;
    if (rb < SL && orow < o_end) {
      const int k = a.f_nks.mod(a.f_nbnd.div(orow));
      row_on = rr < s.nrow[k];
      rw = s.row[k * s.nrow_max + rr];
    }
    nr = 0;
    if (ol < o_end) {
      const int k = a.f_nks.mod(a.f_nbnd.div(ol));
      nr = s.nrow[k];
      m2min = s.row[k * s.nrow_max].x;
    }
  };
  if (nbat > 0) tables(o_begin);
  cplx<T> acc[MODE == XY_PASS1_DENS ? H : 1];
#pragma unroll
  for (int i = 0; i < (MODE == XY_PASS1_DENS ? H : 1); ++i) acc[i] = czero<T>();
  // signed index of point i of this lane, in a run of indices that starts at lo: m(i) = (p <= PR ? p : p - W)
  // at h = 0, + h; the middle point of a whole line is -W/2 or W/2 (line_m)
  auto m_of = [&](int i, int lo) {
    if (PR == W / 2 - 1 && i == H / 2 && (P == 1 || h == 0)) return lo > -W / 2 ? W / 2 : -W / 2;
    return P == 1 ? (i <= LO ? i : i - W) : (i <= LO ? 2 * i : 2 * i - W);
  };
  auto kept = [](int i) constexpr { return i <= LO || i >= H - HI; };
  bool bad = false;

  for (int it = 0; it < nbat; ++it) {
    const int ob = o_begin + it * SL;
    cplx<T>* cs = Cs + (it & 1) * SL * cb + (row_on ? rb * cb + rw.y - rw.z : 0);
    cplx<T>* ysr = Ys + (row_on ? pr * NP : 0);
    if (MODE != XY_PASS2) {
      if (!bad) bad = !mbar_wait(&full[it & 1], (it >> 1) & 1, a.polls);
      if (row_on) {
        cplx<T> l[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
          l[i] = czero<T>();
          if (kept(i)) {
            const int m = m_of(i, rw.z) + h, j = m - rw.z;
            if ((unsigned)j < (unsigned)rw.w && LL_INB(rw.y >= 0 && rw.y + j < cb)) l[i] = cs[m];
          }
        }
        line_inv<T, W, P, LO, HI>(l, h, pmask);
#pragma unroll
        for (int i = 0; i < H; ++i) ysr[H * h + i] = l[i];
      }
      __syncthreads();
    }
    const bool line_on = ob + ls < o_end;
    const int lnr = nr, lm2 = m2min;
    const int4 rwc = rw;
    const bool rowc = row_on;
    if (it + 1 < nbat) tables(ob + SL);
    if (HAS_U && !bad) bad = !mbar_wait(&ufull, it & 1, a.polls);
    if (line_on) {
      cplx<T> l[H];
      cplx<T>* ysl = Ys + (ls * s.nrow_max - lm2) * NP + j1;
      const cplx<T>* u = Us + ls * WW + H * h * W + j1;
      if (MODE == XY_PASS2) {
#pragma unroll
        for (int i = 0; i < H; ++i) l[i] = cmul_rn(Pl[(H * h + i) * W + j1], u[i * W]);
      } else {
#pragma unroll
        for (int i = 0; i < H; ++i) {
          l[i] = czero<T>();
          if (kept(i)) {
            const int m = m_of(i, lm2) + h;
            if ((unsigned)(m - lm2) < (unsigned)lnr && LL_INB(m - lm2 < s.nrow_max)) l[i] = ysl[m * NP];
          }
        }
        line_inv<T, W, P, LO, HI>(l, h, pmask);
        if (MODE == XY_PASS1_DENS && dens_orb(ob + ls)) {
#pragma unroll
          for (int i = 0; i < H; ++i) {
            const cplx<T> x = u[i * W];
            acc[i].x = fma_rn(x.y, l[i].y, fma_rn(x.x, l[i].x, acc[i].x));
            acc[i].y = fma_rn(-x.y, l[i].x, fma_rn(x.x, l[i].y, acc[i].y));
          }
        }
#pragma unroll
        for (int i = 0; i < H; ++i) l[i] = l[i] * Pv[(H * h + i) * W + j1];
      }
      line_fwd<T, W, P>(l, h, pmask);
#pragma unroll
      for (int i = 0; i < H; ++i)
        if (kept(i)) {
          const int m = m_of(i, lm2) + h;
          if ((unsigned)(m - lm2) < (unsigned)lnr && LL_INB(m - lm2 < s.nrow_max)) ysl[m * NP] = l[i];
        }
    }
    __syncthreads();
    if (HAS_U && t < 32 && it + 1 < nbat && !__any_sync(0xffffffffu, bad)) load_u(it + 1);
    if (MODE == XY_PASS2 && !bad) bad = !mbar_wait(&full[it & 1], (it >> 1) & 1, a.polls);
    if (rowc) {
      cplx<T> l[H];
#pragma unroll
      for (int i = 0; i < H; ++i) l[i] = ysr[H * h + i];
      line_fwd<T, W, P>(l, h, pmask);
#pragma unroll
      for (int i = 0; i < H; ++i)
        if (kept(i)) {
          const int m = m_of(i, rwc.z) + h, j = m - rwc.z;
          if ((unsigned)j < (unsigned)rwc.w && LL_INB(rwc.y >= 0 && rwc.y + j < cb)) {
            if (MODE == XY_PASS2) cs[m] = cs[m] + l[i];
            else cs[m] = l[i];
          }
        }
    }
    fence_async_smem();
    __syncthreads();
    if (t < 32) {
      const int nb = min(SL, o_end - ob);
      if (t < nb) {
        bulk_store(row_of(ob + t), Cs + ((it & 1) * SL + t) * cb, cbytes);
        bulk_commit();
      }
      if (it + 2 < nbat && !__any_sync(0xffffffffu, bad)) {   // the same buffer's next batch, once the store has read it
        if (t < nb) bulk_wait_read();
        __syncwarp();
        load_cols(it + 2);
      }
    }
  }
  if (__syncthreads_or(bad) && t == 0) plane_gave_up(full, &ufull, s_asked[0], s_asked[1], err);
  if (MODE == XY_PASS1_DENS) {   // the slots summed in order
    __syncthreads();
    for (int q = 0; q < SL; ++q) {
      if (ls == q) {
#pragma unroll
        for (int i = 0; i < H; ++i) {
          cplx<T>* p = Pb + (H * h + i) * W + j1;
          *p = q == 0 ? acc[i] : *p + acc[i];
        }
      }
      __syncthreads();
    }
    for (int i = t; i < WW; i += TH) nprt[((long)g * W + iz) * WW + i] = Pb[i];
  }
  if (t < SL) bulk_wait();   // the stores leave shared memory before the CTA does
}

}  // namespace ll
