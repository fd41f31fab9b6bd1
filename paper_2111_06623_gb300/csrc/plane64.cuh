// The plane pass of the FP64 path: k_plane's work (plane.cuh) with the lines in 64-bit block fixed
// point (fixed.cuh).  Same grid, batches, bulk copies and shared tables; what differs:
//
//   exponents  a row has one exponent after its inverse transform (s_er), an axis-2 line one after
//              its forward transform (s_el); the next transform's inputs are shifted to the
//              largest of their line.  V and v' are limbs of one exponent per plane.  The density
//              is accumulated in doubles, and doubles are what the column buffer and u(r) hold.
//   phases     rows inverse, lines, rows forward run through ONE inverse and one forward transform
//              in the code (a loop over the phases, not unrolled): written out, the four integer
//              transforms do not fit the instruction caches and the warps wait for instructions.
//   lanes      two per line from W = 24 on: half the registers and half the code per transform.
//
// What bounds it: instruction issue at three warps per scheduler (fixed latencies, the barriers of a
// batch).  KB workload, one GB300, us per launch (pass 1 / density / pass 2): FP64 arithmetic on
// one lane per line 2206 / 2478 / 1423, bound by the FP64 pipe; fixed point written out phase by
// phase on one lane per line 867 / 2196 / 1142 (half the issue slots lost to instruction
// fetch, six warps per SM in the modes with u(r)); shared transforms, two lanes per line 956 / 1166 /
// 640; the pair's butterflies halved between the lanes (below) 757 / 936 / 565; one product per twiddled
// input, every line shifted up again after its transform 748 / 944 / 592.  Two CTAs per SM:
// the 96 registers that a third would leave spill 580 bytes per thread.
#pragma once
#include "plane.cuh"

namespace ll {

// A line of 2H points on a lane pair (h: the lane).  In grid order lane h holds the points
// Q h + (0 .. Q-1) and those H further on (Q = H/2), so that each lane computes Q of the H twiddled
// butterflies and exchanges Q values with its partner (fft_pair_dit's lanes hold a half each: lane
// 1 multiplies all H values while lane 0 waits, and all H are exchanged).  In sphere order lane h
// holds the points 2 i + h.  The twiddle of butterfly Q h + k is W^k, turned by +-i at h = 1.
template <int SIGN>
__device__ __forceinline__ cplx<fx64> fx_turn(cplx<fx64> a, int h) {   // h: times SIGN i
  if (SIGN > 0) return mk(h ? -a.y : a.x, h ? a.x : a.y);
  return mk(h ? a.y : a.x, h ? -a.x : a.y);
}
template <int SIGN> __device__ __forceinline__ FxTw fx_turn(FxTw w, int h) {
  const FxTw r = turn_tw<SIGN>(w);
  return FxTw{h ? r.xh : w.xh, h ? r.xl : w.xl, h ? r.yh : w.yh, h ? r.yl : w.yl, h ? r.nh : w.nh, h ? r.nl : w.nl};
}
__device__ __forceinline__ cplx<fx64> fx_sel(int h, cplx<fx64> a, cplx<fx64> b) {   // h ? a : b
  return mk(h ? a.x : b.x, h ? a.y : b.y);
}
template <int W, int P, int LO, int HI>
__device__ __forceinline__ void fx_line_inv(cplx<fx64> (&l)[W / P], int h, unsigned mask) {
  if constexpr (P == 1) {
    fft_line_in<fx64, W, +1, LO, HI>(l);
  } else {
    constexpr int H = W / 2, Q = H / 2;
    static_assert(H % 2 == 0, "half lines of an even length");
    fft_line_in<fx64, H, +1, LO, HI>(l);   // Y_h
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const cplx<fx64> r = shfl_pair(fx_sel(h, l[k], l[k + Q]), mask);
      const cplx<fx64> y0 = fx_sel(h, r, l[k]), y1 = fx_sel(h, l[k + Q], r);
      const cplx<fx64> p = k == 0 ? fx_turn<+1>(y1, h) : cmul_rn(y1, fx_turn<+1>(twiddle<fx64, W, +1>(k), h));
      l[k] = cadd(y0, p);
      l[k + Q] = csub(y0, p);
    }
  }
}
template <int W, int P>
__device__ __forceinline__ void fx_line_fwd(cplx<fx64> (&l)[W / P], int h, unsigned mask) {
  if constexpr (P == 1) {
    fft_line<fx64, W, -1>(l);
  } else {
    constexpr int H = W / 2, Q = H / 2;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const cplx<fx64> a = cadd(l[k], l[k + Q]), b = csub(l[k], l[k + Q]);
      const cplx<fx64> d = k == 0 ? fx_turn<-1>(b, h) : cmul_rn(b, fx_turn<-1>(twiddle<fx64, W, -1>(k), h));
      const cplx<fx64> r = shfl_pair(fx_sel(h, a, d), mask);
      l[k] = fx_sel(h, r, a);
      l[k + Q] = fx_sel(h, d, r);
    }
    fft_line<fx64, H, -1>(l);              // even (h = 0) or odd (h = 1) outputs
  }
}

template <int W, int MODE, int PR>
__global__ void __launch_bounds__(PlaneCfg<double, W, MODE>::TH, PlaneCfg<double, W, MODE>::min_ctas)
    k_plane64(XYArgs a, cplx<double>* __restrict__ cbuf, const double* __restrict__ vloc,
              const cplx<double>* __restrict__ vpr, const cplx<double>* __restrict__ ur, cplx<double>* __restrict__ nprt,
              int* __restrict__ err) {
  using T = double;
  using C = PlaneCfg<double, W, MODE>;
  constexpr int P = C::P, SL = C::SL, H = C::H, TH = C::TH;
  constexpr int NP = W + 1, WW = W * W;
  constexpr bool HAS_U = MODE != XY_PASS1;
  // kept points of a lane's half line (P = 2: p = 2 i + h), i <= LO or i >= H - HI
  constexpr int LO = P == 1 ? PR : PR / 2, HI = P == 1 ? line_hi(W, PR) : (PR + 1) / 2;
  // headroom of a transform's inputs (of the whole line, so that results do not depend on PR)
  constexpr int G = fx_growth(W);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[2], ufull;
  __shared__ int s_asked[2];   // batches whose columns, u(r) have been asked for
  __shared__ int s_er[SL * W], s_el[SL * W], s_ev;   // exponents of the rows and lines; largest of V or v'
  const SphereDev& s = a.s;
  const int iz = blockIdx.x, g = blockIdx.y, cb = a.cb_ncol;
  cplx<T>* Cs = reinterpret_cast<cplx<T>*>(smem_raw);
  cplx<T>* Us = Cs + 2 * SL * cb;
  cplx<fx64>* Ys = reinterpret_cast<cplx<fx64>*>(Us + (HAS_U ? SL * WW : 0));
  cplx<T>* Pb = reinterpret_cast<cplx<T>*>(Ys + SL * s.nrow_max * NP);
  int2* Pv = reinterpret_cast<int2*>(Pb + (MODE == XY_PASS1_DENS ? SL * WW : 0));   // limbs of V, or of v' (re, im)
  const int t = threadIdx.x;
  if (t == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    mbar_init(&ufull, 1);
    s_asked[0] = s_asked[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    s_ev = 0;
  }
  __syncthreads();
  int ev = 0;
  {
    constexpr int n = MODE == XY_PASS2 ? 2 * WW : WW;
    const T* src = MODE == XY_PASS2 ? reinterpret_cast<const T*>(vpr + (long)iz * WW) : vloc + (long)iz * WW;
    for (int i = t; i < n; i += TH) ev = max(ev, fx_hiword(fx_raw(src[i])) & 0x7fffffff);
    atomicMax(&s_ev, ev);
    __syncthreads();
    ev = max(s_ev >> 20, 1);
    for (int i = t; i < n; i += TH) {
      int2 w;
      fx_coef(fx_raw(src[i]), ev, w.x, w.y);
      Pv[i] = w;
    }
    ev = fx_coef_exp(ev);
  }
  if (MODE == XY_PASS1_DENS)
    for (int i = t; i < SL * WW; i += TH) Pb[i] = czero<T>();
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
  // signed index of point i of this lane, in a run of indices that starts at lo: m(i) = (p <= PR ? p : p - W)
  // at h = 0, + h; the middle point of a whole line is -W/2 or W/2 (line_m)
  auto m_of = [&](int i, int lo) {
    if (PR == W / 2 - 1 && i == H / 2 && (P == 1 || h == 0)) return lo > -W / 2 ? W / 2 : -W / 2;
    return P == 1 ? (i <= LO ? i : i - W) : (i <= LO ? 2 * i : 2 * i - W);
  };
  auto kept = [](int i) constexpr { return i <= LO || i >= H - HI; };
  // the next batch's row: (m2, first column, m1 of it, columns); line: the orbital's rows and first m2
  int4 rw_n = make_int4(0, 0, 0, 0);
  bool row_n = false;
  int lnr_n = 0, lm2_n = 0;
  auto tables = [&](int ob) {
    row_n = false;
    lnr_n = 0;
    if (rb < SL && ob + rb < o_end) {
      const int k = a.f_nks.mod(a.f_nbnd.div(ob + rb));
      row_n = rr < s.nrow[k];
      rw_n = s.row[k * s.nrow_max + rr];
    }
    if (ob + ls < o_end) {
      const int k = a.f_nks.mod(a.f_nbnd.div(ob + ls));
      lnr_n = s.nrow[k];
      lm2_n = s.row[k * s.nrow_max].x;
    }
  };
  if (nbat > 0) tables(o_begin);
  // grid point i of this lane: hb + pos(i)
  auto pos = [](int i) constexpr { return P == 1 || i < H / 2 ? i : i + H / 2; };
  const int hb = P == 1 ? 0 : H / 2 * h;
  bool bad = false;

  for (int it = 0; it < nbat; ++it) {
    const int ob = o_begin + it * SL;
    const int4 rw = rw_n;
    const bool row_on = row_n, line_on = ob + ls < o_end;
    const int lnr = lnr_n, lm2 = lm2_n;
    if (it + 1 < nbat) tables(ob + SL);
    cplx<T>* cs = Cs + (it & 1) * SL * cb + (row_on ? rb * cb + rw.y - rw.z : 0);
    cplx<fx64>* ysr = Ys + (row_on ? pr * NP : 0);
    cplx<fx64>* ysl = Ys + (ls * s.nrow_max - lm2) * NP + j1;
    const int* er = s_er + ls * s.nrow_max;
    // phase 0: rows inverse; 1: lines; 2: rows forward (pass 2 has no inverse transforms)
#pragma unroll 1
    for (int ph = MODE == XY_PASS2 ? 1 : 0; ph < 3; ++ph) {
      if (HAS_U && ph == 1 && !bad) bad = !mbar_wait(&ufull, it & 1, a.polls);
      if (ph == (MODE == XY_PASS2 ? 2 : 0) && !bad) bad = !mbar_wait(&full[it & 1], (it >> 1) & 1, a.polls);
      cplx<fx64> l[H];
      int e = 0;
      if (ph == 1 ? line_on : row_on) {
        if (ph == 0) {
#pragma unroll
          for (int i = 0; i < H; ++i) {
            l[i] = czero<fx64>();
            if (kept(i)) {
              const int m = m_of(i, rw.z) + h, j = m - rw.z;
              if ((unsigned)j < (unsigned)rw.w && LL_INB(rw.y >= 0 && rw.y + j < cb)) l[i] = fx_raw(cs[m]);
            }
          }
          e = fx_line_exp<P>(l, pmask);
          fx_line_from<8 - G>(l, e);
          e = fx_exp(e, 8 - G);
        } else if (ph == 1 && MODE != XY_PASS2) {   // the rows brought to one exponent
          e = -(1 << 30);
          for (int r = 0; r < lnr; ++r) e = max(e, er[r]);
#pragma unroll
          for (int i = 0; i < H; ++i) {
            l[i] = czero<fx64>();
            if (kept(i)) {
              const int m = m_of(i, lm2) + h;
              if ((unsigned)(m - lm2) < (unsigned)lnr && LL_INB(m - lm2 < s.nrow_max))
                l[i] = fx_down(ysl[m * NP], min(e - er[m - lm2] + G, 63));
            }
          }
          e += G;
        } else if (ph == 1) {                       // v'(r) u(r)
          const cplx<T>* u = Us + ls * WW + hb * W + j1;
#pragma unroll
          for (int i = 0; i < H; ++i) l[i] = fx_raw(u[pos(i) * W]);
          e = fx_line_exp<P>(l, pmask);
          fx_line_from<8>(l, e);
          e = fx_exp(e, 8) + ev;
          const int4* pl = reinterpret_cast<const int4*>(Pv) + hb * W + j1;
#pragma unroll
          for (int i = 0; i < H; ++i) {
            const int4 w = pl[pos(i) * W];
            l[i] = cmul_rn(l[i], FxTw{w.x, w.y, w.z, w.w, -w.z, -w.w});
          }
        } else {                                    // the lines brought to one exponent
          const int* el = s_el + rb * W + hb;
          e = -(1 << 30);
#pragma unroll
          for (int i = 0; i < H; ++i) e = max(e, el[pos(i)]);
          if (P == 2) e = max(e, __shfl_xor_sync(pmask, e, 1));
#pragma unroll
          for (int i = 0; i < H; ++i) l[i] = fx_down(ysr[hb + pos(i)], min(e - el[pos(i)] + G, 63));
          e += G;
        }
        if (MODE != XY_PASS2 && ph < 2) fx_line_inv<W, P, LO, HI>(l, h, pmask);
        if (ph == 1 && MODE != XY_PASS2) {
          if (MODE == XY_PASS1_DENS && dens_orb(ob + ls)) {
            cplx<T>* pb = Pb + ls * WW + hb * W + j1;
            const cplx<T>* u = Us + ls * WW + hb * W + j1;
#pragma unroll
            for (int i = 0; i < H; ++i) {
              const cplx<T> x = u[pos(i) * W], r = fx_value(l[i], e);
              cplx<T> q = pb[pos(i) * W];
              q.x = fma_rn(x.y, r.y, fma_rn(x.x, r.x, q.x));
              q.y = fma_rn(-x.y, r.x, fma_rn(x.x, r.y, q.y));
              pb[pos(i) * W] = q;
            }
          }
          const int2* pv = Pv + hb * W + j1;
#pragma unroll
          for (int i = 0; i < H; ++i) {
            const int2 w = pv[pos(i) * W];
            l[i] = mk(fx_mul(l[i].x, w.x, w.y), fx_mul(l[i].y, w.x, w.y));
          }
          e += ev;
        }
        if (ph < 2) {   // back up to the full range; a line: with the forward transform's headroom
          const int c = fx_top<P>(l, pmask);
          e -= c;
          if (ph == 0) {
            fx_up<0>(l, c);
          } else {
            fx_up<G>(l, c);
            e += G;
          }
          if (ph == 0 && h == 0) s_er[pr] = e;
        }
        if (ph > 0) fx_line_fwd<W, P>(l, h, pmask);
        if (ph == 1) {   // the rows' transform reads the line at its own headroom: up again first
          const int c = fx_top<P>(l, pmask);
          fx_up<0>(l, c);
          if (h == 0) s_el[pr] = e - c;
        }
        if (ph == 0) {
#pragma unroll
          for (int i = 0; i < H; ++i) ysr[hb + pos(i)] = l[i];
        } else if (ph == 1) {
#pragma unroll
          for (int i = 0; i < H; ++i)
            if (kept(i)) {
              const int m = m_of(i, lm2) + h;
              if ((unsigned)(m - lm2) < (unsigned)lnr && LL_INB(m - lm2 < s.nrow_max)) ysl[m * NP] = l[i];
            }
        } else {
#pragma unroll
          for (int i = 0; i < H; ++i)
            if (kept(i)) {
              const int m = m_of(i, rw.z) + h, j = m - rw.z;
              if ((unsigned)j < (unsigned)rw.w && LL_INB(rw.y >= 0 && rw.y + j < cb)) {
                const cplx<T> r = fx_value(l[i], e);
                if (MODE == XY_PASS2) cs[m] = cs[m] + r;
                else cs[m] = r;
              }
            }
        }
      }
      if (ph == 2) fence_async_smem();
      __syncthreads();
      if (HAS_U && ph == 1 && t < 32 && it + 1 < nbat && !__any_sync(0xffffffffu, bad)) load_u(it + 1);
    }
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
    for (int i = t; i < WW; i += TH) {
      cplx<T> v = Pb[i];
      for (int q = 1; q < SL; ++q) v = v + Pb[q * WW + i];
      nprt[((long)g * W + iz) * WW + i] = v;
    }
  }
  if (t < SL) bulk_wait();   // the stores leave shared memory before the CTA does
}

// The plane pass of a type.
template <typename T, int W, int MODE, int PR> constexpr auto plane_kernel() {
  if constexpr (sizeof(T) == 8) return &k_plane64<W, MODE, PR>;
  else return &k_plane<T, W, MODE, PR>;
}

}  // namespace ll
