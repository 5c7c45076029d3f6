// qt_me_small.cuh -- master-equation solver (paper section 3.1,
// Eq. (master_equation)) for small systems: one CTA, or one thread-block
// cluster, integrates one density matrix that stays in shared memory.
//
// What bounds it: GB300 has two FP64 multiply-adds per cycle and SM, so a
// warp's FP64 instruction takes 16 cycles of its SM, and a small system on
// one SM is bound by the number of FP64 instructions (and by the latency of
// its barriers in FP32).  The solver therefore does as little arithmetic as
// the generator allows:
//   * the diagonal of the generator, D_ij = -i (h_ii - conj h_jj) +
//     sum_n c_n,ii conj(c_n,jj) over the diagonal collapse operators, is one
//     coefficient per entry, formed once;
//   * the other terms are a list per entry, each a source and a coefficient;
//     the terms of operators that are all real (ladder operators, spin flips)
//     take two multiply-adds instead of four;
//   * for a Hermitian state only the upper triangle is evaluated (herm);
//   * the Dormand-Prince step is evaluated in powers of the generator (DPP,
//     qt_device.cuh): no stage combinations;
//   * the step-size control runs on one warp, which hands the next step to
//     the others through shared memory; divisions and the fifth root are
//     Newton iterations.
// The vectors that the generator is applied to are full matrices in shared
// memory, in two alternating buffers (every CTA of a cluster holds a copy and
// writes its entries to all of them); rho, L rho, and the sums of the new
// state and of the error are private to the thread that owns the entry, in
// shared memory when they fit (KS), else in the caller's workspace.  One
// barrier per right-hand side.
//
// One solve (before: the general solver of qt_me_impl.cuh on one CTA): the
// Jaynes-Cummings model, dim 20, 3722 right-hand sides in FP64 33.3 -> 7.2 ms,
// 2486 mixed ones 8.0 -> 2.1 ms; the 304 x 151 correlation (304 CTAs) 189 ->
// 57 ms in FP64, 33.9 -> 10.5 ms mixed; an XXZ chain of 6 spins 588 -> 35 ms
// in FP64 (8 CTAs).  Bound: FP64 pipe (one warp issues an FP64 instruction
// every 65 cycles), mixed: latency of one right-hand side on one CTA.
#pragma once

#include <cooperative_groups.h>

#include "qt_device.cuh"
#include "qt_internal.h"

namespace qt {

namespace {

// Coefficients of a term: real (or, for the terms of a real H_eff, imaginary),
// or complex.  The mixed solver keeps each as an FP32 value and its FP32
// remainder, formed from the FP64 product, so that the generator carries no
// systematic FP32 rounding and the jump terms and the anticommutator in H_eff
// use the same collapse operators.
template <typename T> struct SCoef;
template <> struct SCoef<double> {
  using R = double;
  using C = double2;
  __device__ __forceinline__ static R real(double x) { return x; }
  __device__ __forceinline__ static C make(double re, double im) { return make_double2(re, im); }
};
template <> struct SCoef<float> {
  using R = float2;  // value, remainder
  using C = float4;  // value re, im, remainder re, im
  __device__ __forceinline__ static R real(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
  }
  __device__ __forceinline__ static C make(double re, double im) {
    const float2 x = real(re), y = real(im);
    return make_float4(x.x, y.x, x.y, y.y);
  }
};

// out += c x (the mixed form adds the product with the remainder to lo).
__device__ __forceinline__ void smac(double c, double2 x, double2 &out, double2 &) {
  out = vfma(c, x, out);
}
__device__ __forceinline__ void smac(float2 c, float2 x, float2 &out, float2 &lo) {
  out = vfma(c.x, x, out);
  lo = vfma(c.y, x, lo);
}
__device__ __forceinline__ void smac(double2 c, double2 x, double2 &out, double2 &) {
  cmac(out, c, x);
}
__device__ __forceinline__ void smac(float4 c, float2 x, float2 &out, float2 &lo) {
  const float2 ix = make_float2(-x.y, x.x);
  out = vfma(c.x, x, out);
  out = vfma(c.y, ix, out);
  lo = vfma(c.z, x, lo);
  lo = vfma(c.w, ix, lo);
}

constexpr int kSmallMaxRanks = 8;
// Dynamic shared memory of one CTA: the 227 KB that a CTA may have, less 1 KB
// for the static variables of the kernels that call the solver; the limit of
// every launch, whatever its size (see kSmemPerCta).
constexpr size_t kSmallSmemMax = kSmemPerCta - 1024;

// What warp 0 of each CTA hands to the others after each step attempt.
struct SmallCtl {
  double h;      // length of the next attempt
  double c[8];   // FP64: c_k h^k
  double e[8];   // FP64: e_k h^k
  int accepted;  // the last attempt was accepted (its state is in y1)
  int out;       // output index to write from y1, or -1
  int done;
  int skip;      // the next output time is not ahead: write it without a step
};

// Shared-memory layout, the same on host and device.
constexpr int kSmallArrays = 4;  // entry arrays private to a thread

struct SmallSmem {
  size_t y, k, dt, ij, ho, hc, co, cc, red, red2, ctl, total;
};

__host__ __device__ inline int small_entries(int d, bool herm) {
  return herm ? d * (d + 1) / 2 : d * d;
}

// Entries that one CTA of a team stores: its threads take them in rounds.
__host__ __device__ inline int small_local(int nent, int ranks, int threads) {
  return (nent + ranks * threads - 1) / (ranks * threads) * threads;
}

// in_smem: the entry arrays and the terms in shared memory, else only the
// matrices (the rest in the workspace).
__host__ __device__ inline SmallSmem small_smem(int precision, int d, int nent, SmallInfo f,
                                                int ranks, int threads, bool in_smem) {
  const size_t nloc = in_smem ? (size_t)small_local(nent, ranks, threads) : 0;
  const size_t ev = precision == QT_MIXED ? 8 : 16, ld = (size_t)(d | 1);
  SmallSmem s;
  size_t p = 0;
  auto take = [&p](size_t b) {
    const size_t at = p;
    p = (p + b + 15) / 16 * 16;
    return at;
  };
  s.y = take(2 * d * ld * ev);
  s.k = take(kSmallArrays * nloc * ev);
  s.dt = take(nloc * 16);
  s.hc = take(2 * f.nl * nloc * (f.hreal ? 8 : 16));
  s.cc = take(f.kc * nloc * (f.creal ? 8 : 16));
  s.ij = take(nloc * 4);
  s.ho = take(2 * f.nl * nloc * 4);
  s.co = take(f.kc * nloc * 4);
  s.red = take((size_t)threads * 2 * 8);
  s.red2 = take((size_t)kSmallMaxRanks * 2 * 8);
  s.ctl = take(sizeof(SmallCtl));
  s.total = p;
  return s;
}

// Bytes of the workspace of one CTA when the entry arrays and the terms do not
// fit in shared memory, laid out from its start in the order of SmallSmem::k
// .. co (without the matrices).
__host__ __device__ inline size_t small_ws_bytes(int precision, int d, int nent, SmallInfo f,
                                                 int ranks, int threads) {
  return small_smem(precision, d, nent, f, ranks, threads, true).red -
         small_smem(precision, d, nent, f, ranks, threads, true).k;
}

// Systems that the solver takes: time-independent, in units in which the powers
// of the generator are in the FP64 range, with at most kSmallTerms
// terms per entry (operators with wider rows go to the general solver, which
// forms their products row by row).
constexpr int kSmallTerms = 64;
__host__ __device__ inline bool small_takes(SmallInfo f) {
  return f.in_range && 2 * f.nl + f.kc <= kSmallTerms;
}
inline bool small_fits(const MeArgs &a) {
  return a.n_td == 0 && a.ops.d <= kMeSmallDim && small_takes(a.small);
}

// CTAs of a solve on its own.  A cluster divides the FP64 work but adds about
// 0.5 us of cluster barrier per right-hand side: up to one round of one CTA's
// threads (256 entries) one CTA is faster, above that four, then eight.
// Measured per solve in ms on 1 / 4 / 8 CTAs, FP64 (mixed): 210 entries 7.3 /
// 8.1 / 9.2 (2.2 / 3.4 / 3.7), 820 entries 2.5 / 1.24 / 1.29 (0.94 / 0.86 /
// 0.93), 1830 entries 2.4 / 0.75 / 0.69 (0.83 / 0.49 / 0.51), 2080 entries
// with 12 more terms 123 / 46 / 35 (24.8 / 10.8 / 8.8).
inline int small_ranks(int nent) { return nent <= 256 ? 1 : nent <= 1024 ? 4 : 8; }

// One solve by a CTA (CL = false) or by all CTAs of a cluster (CL = true).
// KS: the entry arrays and the terms in shared memory, else at work
// (small_ws_bytes per CTA).
template <typename T, bool CL, bool KS>
struct SmallSolver {
  using V = typename CT<T>::V;
  using C = typename SCoef<T>::C;
  using R = typename SCoef<T>::R;
  const MeArgs &a;
  const bool herm;
  const int d, ld, nent, rank, nranks, nthr, e0, nloc;
  const int kh, kc;        // terms of H_eff and of the collapse operators per entry
  const bool hreal, creal;
  V *y0, *y1, *kb;  // the two matrices; the entry arrays
  C *dt;            // the diagonal of the generator
  unsigned char *hco, *cco;  // coefficients [term][entry], R or C
  int *ij, *hof, *cof;       // row and column of an entry; sources [term][entry]
  double *red, *red2;
  SmallCtl *ctl;

  __device__ SmallSolver(const MeArgs &a_, bool herm_, unsigned char *sm, unsigned char *work,
                         int rank_, int nranks_)
      : a(a_), herm(herm_), d(a_.ops.d), ld(a_.ops.d | 1), nent(small_entries(a_.ops.d, herm_)),
        rank(rank_), nranks(nranks_), nthr((int)blockDim.x * nranks_),
        // the entries of a warp are consecutive, the warps alternate over the CTAs
        e0(((int)(threadIdx.x >> 5) * nranks_ + rank_) * 32 + (int)(threadIdx.x & 31)),
        nloc(small_local(nent, nranks_, (int)blockDim.x)), kh(2 * a_.small.nl), kc(a_.small.kc),
        hreal(a_.small.hreal != 0), creal(a_.small.creal != 0) {
    const int prec = sizeof(T) == 4 ? QT_MIXED : QT_FP64;
    const SmallSmem L = small_smem(prec, d, nent, a_.small, nranks_, (int)blockDim.x, KS);
    const SmallSmem W = small_smem(prec, d, nent, a_.small, nranks_, (int)blockDim.x, true);
    unsigned char *base = KS ? sm + W.k : work;
    y0 = reinterpret_cast<V *>(sm + L.y);
    y1 = y0 + d * ld;
    kb = reinterpret_cast<V *>(base);
    dt = reinterpret_cast<C *>(base + (W.dt - W.k));
    hco = base + (W.hc - W.k);
    cco = base + (W.cc - W.k);
    ij = reinterpret_cast<int *>(base + (W.ij - W.k));
    hof = reinterpret_cast<int *>(base + (W.ho - W.k));
    cof = reinterpret_cast<int *>(base + (W.co - W.k));
    red = reinterpret_cast<double *>(sm + L.red);
    red2 = reinterpret_cast<double *>(sm + L.red2);
    ctl = reinterpret_cast<SmallCtl *>(sm + L.ctl);
  }

  __device__ __forceinline__ void sync() const {
    if constexpr (CL) cooperative_groups::this_cluster().sync();
    else __syncthreads();
  }

  // fn(l, i, j) for the entries of this thread, l their place in its arrays.
  template <typename F> __device__ __forceinline__ void each(F &&fn) const {
    for (int e = e0, l = threadIdx.x; e < nent; e += nthr, l += blockDim.x)
      fn(l, ij[l] & 0xffff, ij[l] >> 16);
  }

  // Entry (i, j) of the matrix buf in every CTA's copy, with its mirror
  // for a Hermitian state.
  __device__ __forceinline__ void put(V *buf, int i, int j, V v) const {
    if (herm && i == j) v.y = (T)0;
    V w = v;
    w.y = -v.y;
    if constexpr (CL) {
      for (int r = 0; r < nranks; ++r) {
        V *b = cooperative_groups::this_cluster().map_shared_rank(buf, r);
        b[i * ld + j] = v;
        if (herm && i != j) b[j * ld + i] = w;
      }
    } else {
      buf[i * ld + j] = v;
      if (herm && i != j) buf[j * ld + i] = w;
    }
  }

  // Totals of nv (1 or 2) values per thread over the team, in v on the lanes
  // of warp 0 of every CTA (in a fixed order, the same in every CTA).
  __device__ void reduce(double *v, int nv) const {
    for (int q = 0; q < nv; ++q) red[q * blockDim.x + threadIdx.x] = v[q];
    // the threads of warps without entries add nothing
    const int nact = min((int)blockDim.x, ((nent + 31) / 32 + nranks - 1) / nranks * 32);
    __syncthreads();
    if (threadIdx.x < 32) {
      for (int q = 0; q < nv; ++q) {
        double x = 0.0;
        for (int s = threadIdx.x; s < nact; s += 32) x += red[q * blockDim.x + s];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        v[q] = x;
        if constexpr (CL)
          if ((int)threadIdx.x < nranks)
            cooperative_groups::this_cluster().map_shared_rank(red2, (int)threadIdx.x)[rank * 2 + q] = x;
      }
    }
    if constexpr (CL) {
      sync();
      if (threadIdx.x < 32)
        for (int q = 0; q < nv; ++q) {
          double x = 0.0;
          for (int r = 0; r < nranks; ++r) x += red2[r * 2 + q];
          v[q] = x;
        }
    }
  }

  // The generator by entry: the diagonal D and the terms, from the ELL rows of
  // the operators.  Rows shorter than the widest are padded with zero terms
  // on the entry itself.
  __device__ void build() {
    const int w0 = a.ops.w[0];
    const int64_t off0 = a.ops.off[0];
    const int *col = a.ops.col;
    const double2 *val = a.ops.val64;
    for (int e = e0, l = threadIdx.x; e < nent; e += nthr, l += blockDim.x) {
      int i = 0, j = e;  // entry e, row by row; columns i..d-1 when herm
      if (herm) {
        while (j >= d - i) j -= d - i++;
        j += i;
      } else {
        i = e / d;
        j = e - i * d;
      }
      ij[l] = i | (j << 16);
      double2 D = make_double2(0.0, 0.0);
      int k = 0;
      auto term = [&](int off, double re, double im) {  // an H_eff term with coefficient -i (re, im)
        hof[k * nloc + l] = off;
        if (hreal) reinterpret_cast<R *>(hco)[k * nloc + l] = SCoef<T>::real(-re);
        else reinterpret_cast<C *>(hco)[k * nloc + l] = SCoef<T>::make(im, -re);
        ++k;
      };
      for (int s = 0; s < w0; ++s) {  // -i H_eff y
        const int64_t p = off0 + (int64_t)s * d + i;
        const double2 v = val[p];
        if (col[p] != i) term(col[p] * ld + j, v.x, v.y);
        else { D.x += v.y; D.y -= v.x; }
      }
      while (k < kh / 2) term(i * ld + j, 0.0, 0.0);
      for (int s = 0; s < w0; ++s) {  // +i y H_eff^dag
        const int64_t p = off0 + (int64_t)s * d + j;
        const double2 v = val[p];
        if (col[p] != j) term(i * ld + col[p], -v.x, v.y);
        else { D.x += v.y; D.y += v.x; }
      }
      while (k < kh) term(i * ld + j, 0.0, 0.0);
      reinterpret_cast<double2 *>(dt)[l] = D;  // FP64 until the collapse terms are in
    }
    int k = 0;
    for (int c = 1; c <= a.n_c; ++c) {
      const int w = a.ops.w[c];
      const int64_t off = a.ops.off[c];
      int diag = 1;
      for (int r = threadIdx.x; r < d; r += blockDim.x)
        for (int s = 0; s < w; ++s) {
          const double2 v = val[off + (int64_t)s * d + r];
          if (col[off + (int64_t)s * d + r] != r && (v.x != 0.0 || v.y != 0.0)) diag = 0;
        }
      diag = __syncthreads_and(diag);
      each([&](int l, int i, int j) {
        int q = k;
        for (int s = 0; s < w; ++s)
          for (int t = 0; t < w; ++t) {
            const int64_t pi = off + (int64_t)s * d + i, pj = off + (int64_t)t * d + j;
            const double2 u = val[pi], v = val[pj];  // u conj(v)
            const double re = u.x * v.x + u.y * v.y, im = u.y * v.x - u.x * v.y;
            if (diag) {
              double2 &D = reinterpret_cast<double2 *>(dt)[l];
              D.x += re;
              D.y += im;
              continue;
            }
            cof[q * nloc + l] = col[pi] * ld + col[pj];
            if (creal) reinterpret_cast<R *>(cco)[q * nloc + l] = SCoef<T>::real(re);
            else reinterpret_cast<C *>(cco)[q * nloc + l] = SCoef<T>::make(re, im);
            ++q;
          }
      });
      if (!diag) k += w * w;
    }
    each([&](int l, int, int) {
      const double2 D = reinterpret_cast<double2 *>(dt)[l];
      dt[l] = SCoef<T>::make(D.x, D.y);
    });
  }

  // n terms of entry l added to (o, ol): coefficients c, sources from; rot:
  // the coefficients are imaginary.
  template <typename K, bool ROT>
  __device__ __forceinline__ void terms(const unsigned char *c, const int *from, int n,
                                        const V *__restrict__ y, int l, V &o, V &ol) const {
    const K *ck = reinterpret_cast<const K *>(c);
    for (int q = 0; q < n; ++q, l += nloc) {
      V g = y[from[l]];
      if (ROT) {
        const T x = g.x;
        g.x = -g.y;
        g.y = x;
      }
      smac(ck[l], g, o, ol);
    }
  }

  // Entry (i, j), the l-th of this thread, of the right-hand side at y.
  __device__ __forceinline__ V f(const V *__restrict__ y, int l, int i, int j) const {
    V o = cmake<V>(0.0, 0.0), ol = o;
    smac(dt[l], y[i * ld + j], o, ol);
    if (hreal) terms<R, true>(hco, hof, kh, y, l, o, ol);
    else terms<C, false>(hco, hof, kh, y, l, o, ol);
    if (creal) terms<R, false>(cco, cof, kc, y, l, o, ol);
    else terms<C, false>(cco, cof, kc, y, l, o, ol);
    if constexpr (sizeof(T) == 4) o = vadd(o, ol);
    return o;
  }

  // Expectation values Tr(O rho) and the optional state at output m, from
  // the matrix y (one warp of the team per observable).
  __device__ void output(int m, const V *y) const {
    if (a.states)
      for (int x = (int)threadIdx.x + rank * (int)blockDim.x; x < d * d; x += nthr) {
        const V r = y[x / d * ld + x % d];
        a.states[(int64_t)m * d * d + x] = make_double2((double)r.x, (double)r.y);
      }
    const int lane = threadIdx.x & 31;
    const V *val = sizeof(T) == 8 ? reinterpret_cast<const V *>(a.ops.val64)
                                  : reinterpret_cast<const V *>(a.ops.val32);
    for (int q = ((int)threadIdx.x >> 5) * nranks + rank; q < a.n_e; q += nthr >> 5) {
      const int op = 1 + a.n_c + q, w = a.ops.w[op];
      const int64_t off = a.ops.off[op];
      double re = 0.0, im = 0.0;
      for (int i = lane; i < d; i += 32)
        for (int s = 0; s < w; ++s) {
          const int64_t p = off + (int64_t)s * d + i;
          const V o = val[p];
          const V r = y[__ldg(a.ops.col + p) * ld + i];  // O[i,c] rho[c,i]
          re += (double)o.x * r.x - (double)o.y * r.y;
          im += (double)o.x * r.y + (double)o.y * r.x;
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (lane == 0) a.expect[(int64_t)m * a.n_e + q] = make_double2(re, im);
    }
  }

  __device__ void solve() {
    build();
    // rho, L rho, the sum of the step (added to rho once, so that rho is
    // rounded once per step), the sum of the error (which then receives L of
    // the new state)
    V *rho = kb, *v1 = kb + nloc, *sum = kb + 2 * nloc, *err = kb + 3 * nloc;
    double v[2];
    const bool lead = threadIdx.x < 32;  // this CTA's control warp

    // ---- initial state: rho0 = |psi><psi| / <psi|psi> or the given matrix
    double scale = 1.0;
    if (a.state_is_ket) {
      double s = 0.0;  // every warp forms the norm itself
      for (int i = threadIdx.x & 31; i < d; i += 32)
        s += a.state0[i].x * a.state0[i].x + a.state0[i].y * a.state0[i].y;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (!(s > 0.0)) {
        if (threadIdx.x == 0 && rank == 0) set_status(a.status, QT_ENORM);
        return;
      }
      scale = 1.0 / s;
    }
    if constexpr (CL) sync();  // every CTA of the cluster has started
    each([&](int, int i, int j) {
      double2 r;
      if (a.state_is_ket) {
        const double2 p = a.state0[i], q = a.state0[j];  // p conj(q)
        r = make_double2((p.x * q.x + p.y * q.y) * scale, (p.y * q.x - p.x * q.y) * scale);
      } else {
        r = a.state0[i * d + j];
      }
      put(y1, i, j, cmake<V>(r.x, r.y));
    });
    sync();
    unsigned long long n_acc = 0, n_rej = 0, n_rhs = 1;
    each([&](int l, int i, int j) { err[l] = f(y1, l, i, j); });

    // ---- starting step (Hairer-Norsett-Wanner), by FP64 sums
    double t = a.tlist[0], hprop = a.h0;
    if (a.n_t > 1 && !(hprop > 0.0)) {
      v[0] = v[1] = 0.0;
      each([&](int l, int i, int j) {
        const V r = y1[i * ld + j], g = err[l];
        const double sx = a.atol + a.rtol * fabs((double)r.x);
        const double sy = a.atol + a.rtol * fabs((double)r.y);
        const double wt = herm && i != j ? 2.0 : 1.0;
        v[0] += wt * (((double)r.x / sx) * ((double)r.x / sx) + ((double)r.y / sy) * ((double)r.y / sy));
        v[1] += wt * (((double)g.x / sx) * ((double)g.x / sx) + ((double)g.y / sy) * ((double)g.y / sy));
      });
      reduce(v, 2);
      const double nr = 2.0 * (double)d * (double)d;
      double h0 = 0.0, d1 = 0.0;
      if (lead) {
        const double d0 = sqrt(v[0] / nr);
        d1 = sqrt(v[1] / nr);
        h0 = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
        if (threadIdx.x == 0) ctl->h = h0;
      }
      __syncthreads();
      h0 = ctl->h;
      each([&](int l, int i, int j) {
        const V r = y1[i * ld + j], g = err[l];
        put(y0, i, j, cmake<V>((double)r.x + h0 * (double)g.x, (double)r.y + h0 * (double)g.y));
      });
      sync();
      ++n_rhs;
      v[0] = 0.0;
      each([&](int l, int i, int j) {
        const V r = y1[i * ld + j], g = err[l], g1 = f(y0, l, i, j);
        const double sx = a.atol + a.rtol * fabs((double)r.x);
        const double sy = a.atol + a.rtol * fabs((double)r.y);
        const double ex = ((double)g1.x - (double)g.x) / sx;
        const double ey = ((double)g1.y - (double)g.y) / sy;
        v[0] += (herm && i != j ? 2.0 : 1.0) * (ex * ex + ey * ey);
      });
      reduce(v, 1);
      if (lead) {
        const double d2 = sqrt(v[0] / nr) / h0;
        const double dm = fmax(d1, d2);
        const double h1 = (dm <= 1e-15) ? fmax(1e-6, h0 * 1e-3) : pow(0.01 / dm, 0.2);
        hprop = fmin(100.0 * h0, h1);
      }
    }
    // ---- the control warp's state: next output m at tk, attempts towards it
    int m = 1, status = QT_OK;
    int64_t attempts = 0;
    bool after_reject = false, clipped = false;
    double tk = a.n_t > 1 ? a.tlist[1] : t, h = 0.0;
    const double inv_n = 1.0 / (2.0 * (double)d * (double)d);
    // length of the next attempt, or an error status
    auto next = [&]() {
      if (attempts++ >= a.max_steps) { status = QT_ESTEP; return; }
      const double rest = tk - t;  // positive
      clipped = !pos_less(hprop, rest);
      h = clipped ? rest : hprop;
      if (!clipped && pos_less(h, 16.0 * 2.220446049250313e-16 * max_abs(t, tk))) status = QT_ESTEP;
    };
    auto hand_over = [&](bool accepted, int out) {
      const int last = a.n_t - 1;
      const bool done = status != QT_OK || (out >= 0 && out == last);
      const bool skip = !done && !(t < tk);
      if (!done && !skip) next();
      if (sizeof(T) == 8 && threadIdx.x >= 1 && threadIdx.x <= 7) {  // coefficients of v_k
        double p = h;
        for (int q = 1; q < (int)threadIdx.x; ++q) p *= h;
        ctl->c[threadIdx.x] = dpp_c(threadIdx.x) * p;
        // L ynew takes one power of h
        ctl->e[threadIdx.x] = dpp_e(threadIdx.x) * (threadIdx.x == 7 ? h : p);
      }
      if (threadIdx.x == 0) {
        ctl->h = h;
        ctl->accepted = accepted;
        ctl->out = out;
        ctl->done = done || status != QT_OK;
        ctl->skip = skip;
      }
    };
    if (lead) hand_over(true, 0);
    __syncthreads();

    for (;;) {
      const bool accepted = ctl->accepted != 0;
      const int out = ctl->out, done = ctl->done, skip = ctl->skip;
      const T ht = (T)ctl->h;
      if (out >= 0) output(out, y1);
      if (done) break;
      if (skip) {
        __syncthreads();
        if (lead) {
          const int om = m;
          if (++m < a.n_t) tk = a.tlist[m];
          hand_over(true, om);
        }
        __syncthreads();
        continue;
      }
      if (accepted) {  // first same as last
        V *sw = v1;
        v1 = err;
        err = sw;
      }
      // FP64: v_k with the coefficients c_k h^k, e_k h^k; mixed: h^k v_k (an
      // FP32 power of a large generator would overflow) with c_k, e_k
      auto ck = [&](int q) { return sizeof(T) == 8 ? (T)ctl->c[q] : (T)dpp_c(q); };
      auto ek = [&](int q) { return sizeof(T) == 8 ? (T)ctl->e[q] : (T)dpp_e(q); };
      // v_1; the accepted state becomes rho
      {
        const T c = ck(1), ce = ek(1);
        each([&](int l, int i, int j) {
          const V r = accepted ? y1[i * ld + j] : rho[l];
          if (accepted) rho[l] = r;
          V g = v1[l];
          if constexpr (sizeof(T) == 4) g = vmul(ht, g);
          sum[l] = vmul(c, g);
          err[l] = vmul(ce, g);
          put(y0, i, j, g);
        });
      }
      sync();
      // v_2 .. v_6, the last fused with the new state (into y1)
#pragma unroll 1
      for (int q = 2; q <= 6; ++q) {
        const V *in = (q & 1) ? y1 : y0;
        V *nxt = (q & 1) ? y0 : y1;
        const T c = ck(q), ce = ek(q);
        each([&](int l, int i, int j) {
          V g = f(in, l, i, j);
          if constexpr (sizeof(T) == 4) g = vmul(ht, g);
          const V s = vfma(c, g, sum[l]);
          sum[l] = s;
          err[l] = vfma(ce, g, err[l]);
          put(nxt, i, j, q == 6 ? vadd(rho[l], s) : g);
        });
        sync();
      }
      // L ynew fused with the error norm
      {
        const T at = (T)a.atol, rt = (T)a.rtol;
        const T ce = sizeof(T) == 8 ? (T)ctl->e[7] : (T)DPP::e7 * ht;
        T acc = (T)0;
        each([&](int l, int i, int j) {
          const V g = f(y1, l, i, j);
          const V er = vfma(ce, g, err[l]);
          err[l] = g;
          const V r = rho[l], yn = y1[i * ld + j];
          const T qx = ratio(er.x, tfma(rt, max_abs(r.x, yn.x), at));
          const T qy = ratio(er.y, tfma(rt, max_abs(r.y, yn.y), at));
          const T q2 = tfma(qx, qx, qy * qy);
          acc += herm && i != j ? (T)2 * q2 : q2;
        });
        v[0] = (double)acc;
      }
      reduce(v, 1);
      if (lead) {
        n_rhs += 6;
        // err^2; err <= 1 exactly when err^2 <= 1
        const double x = v[0] * inv_n;
        bool ok = false;
        int outm = -1;
        if (!isfinite(x)) {
          status = QT_ENUMERIC;
        } else {
          ok = x <= 1.0;
          hprop = dp_control_sq<T>(h, x, ok, after_reject, clipped, hprop);
          after_reject = !ok;
          if (ok) {
            ++n_acc;
            t = clipped ? tk : t + h;
            if (!(t < tk)) {
              outm = m;
              attempts = 0;
              if (++m < a.n_t) tk = a.tlist[m];
            }
          } else {
            ++n_rej;
          }
        }
        hand_over(ok, outm);
      }
      __syncthreads();
    }
    if (threadIdx.x == 0 && rank == 0) {
      if (status != QT_OK) set_status(a.status, status);
      atomicAdd(a.counters + 0, n_acc);
      atomicAdd(a.counters + 1, n_rej);
      atomicAdd(a.counters + 2, n_rhs);
    }
    if constexpr (CL) sync();  // no CTA leaves while its copy may be written
  }
};

}  // namespace

}  // namespace qt
