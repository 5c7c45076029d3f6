// qt_adjoint.cu -- gradients of a master-equation loss by the discrete
// adjoint (an extension beyond the paper's solvers; the forward problem is
// Eq. (master_equation) of section 3.1).
//
// The generator of segment s is
//   F_s(rho) = -i [H0 + Omega_s Hd, rho]
//              + sum_k gamma_k (A_k rho A_k^dag - 1/2 {A_k^dag A_k, rho}),
// Omega_s constant on each segment of length t_seg, and the loss
//   L = Re Tr(P1 rho(T)) + Re q(T),   dq/dt = Tr(P2 rho),
// q carried by the same Runge-Kutta stages as rho.  The forward pass is the
// adaptive Dormand-Prince solve of the library's controller with the segment
// ends as output times; it records every accepted step length (the frozen
// grid) and rho at the segment ends.  F_s is linear and constant on a segment,
// so a step is evaluated in powers of it (DPP, qt_device.cuh): with
// v_k = F v_(k-1), v_0 = rho,
//   rho <- sum_k c_k h^k v_k,   q <- q + sum_k c_(k+1) h^(k+1) Tr(P2 v_k)
// (the stage sums of the tableau multiplied out; c_0 = 1, k = 0..6 and 0..5).
// The backward pass walks the segments in reverse: it recomputes the
// segment's states and their v_k from its checkpoint, then for each step
// (last first) applies the adjoint of the step,
//   a_6 = c_6 h^6 lambda,
//   a_(k-1) = c_(k-1) h^(k-1) lambda + c_k h^k P2 + F^dag(a_k),   k = 6..1,
//   lambda <- a_0,                                      lambda(T) = P1,
//   dL/dOmega_s += sum_k <i [Hd, a_k], v_(k-1)>,
//   dL/dgamma_j += sum_k <A_j^dag a_k A_j - 1/2 {A_j^dag A_j, a_k}, v_(k-1)>,
// with F^dag(X) = i [H, X] + sum_k gamma_k (A_k^dag X A_k - 1/2 {A_k^dag A_k, X})
// and <X, Y> = Re Tr(X^dag Y).  This is the exact derivative of the discrete
// map, so it agrees with finite differences taken on the same grid; the
// parameter derivatives take their products from F^dag(a_k) and cost only the
// inner products with v_(k-1).
//
// One CTA integrates one parameter vector; everything is FP64, and the FP64
// pipe bounds it (two multiply-adds per cycle and SM).  So the diagonal of
// the generator is one coefficient per entry, off-diagonal products with real
// operators take two multiply-adds, and when the initial state is Hermitian
// (lambda always is) only the upper triangle is evaluated.  The two matrices
// that the generator reads from and writes to alternate in shared memory; the
// arrays private to an entry (the states and their v_k, lambda, sums) are in
// the workspace.
// Transmon x cavity, dim 60, 256 drive vectors of 16 segments, forward and
// backward: 571 -> 63 ms (before: every product complex and from the full
// matrix, the stage sums of the tableau, 97 generator products and parameter
// products per backward step, the FP64 pipe 90 % busy).
#include <type_traits>

#include "qt_device.cuh"
#include "qt_internal.h"

namespace qt {

namespace {

constexpr int kAdjBlock = 512;

__device__ __forceinline__ double2 cj(double2 v) { return make_double2(v.x, -v.y); }
__device__ __forceinline__ double nan_value() { return __longlong_as_double(0x7ff8000000000000ll); }

struct AdjCtl {
  double h;
  // the weights of F v_(k-1) and Tr(P2 v_(k-1)), c_k h^k, those of the error, e_k h^k
  // (e_7: h alone), and those of lambda in a_k, c_k h^k; for a step that is
  // dpp_scaled c_k h, e_k h and c_k
  double c[8], e[8], l[8];
  int accepted, done, status;
};

// Shared memory: two matrices, the reduction scratch, the gamma sums.
struct AdjSmem {
  size_t y, red, gk, ctl, total;
};
__host__ __device__ inline AdjSmem adj_smem(int d, int nk) {
  AdjSmem s;
  size_t p = 0;
  s.y = p;
  p += 2 * (size_t)d * (d | 1) * 16;
  s.red = p;
  p += (size_t)kAdjBlock * 2 * 8;
  s.gk = p;
  p += (size_t)kAdjBlock * nk * 8;
  s.ctl = p;
  p += (sizeof(AdjCtl) + 15) / 16 * 16;
  s.total = p;
  return s;
}

struct Adj {
  const AdjArgs &a;
  const int d, ld, nent, nk;
  const bool herm;
  double2 *y0, *y1;
  double *red, *gk;
  AdjCtl *ctl;
  double2 *ws;        // this CTA's workspace: arrays of nent entries
  const double *gam;  // [nk]

  __device__ Adj(const AdjArgs &a_, unsigned char *sm)
      : a(a_), d(a_.ops.d), ld(a_.ops.d | 1),
        nent(a_.herm ? a_.ops.d * (a_.ops.d + 1) / 2 : a_.ops.d * a_.ops.d), nk(a_.nk),
        herm(a_.herm != 0), gam(a_.gamma + (int64_t)blockIdx.x * a_.nk) {
    const AdjSmem L = adj_smem(d, nk);
    y0 = reinterpret_cast<double2 *>(sm + L.y);
    y1 = y0 + d * ld;
    red = reinterpret_cast<double *>(sm + L.red);
    gk = reinterpret_cast<double *>(sm + L.gk);
    ctl = reinterpret_cast<AdjCtl *>(sm + L.ctl);
    ws = a.work + (int64_t)blockIdx.x * a.slots * ((int64_t)d * d);
  }
  __device__ __forceinline__ double2 *array(int q) const { return ws + (int64_t)q * nent; }

  // fn(e, i, j) for the entries of this thread: row by row, columns i..d-1
  // when herm.
  template <typename F> __device__ __forceinline__ void each(F &&fn) const {
    int i = 0, j = (int)threadIdx.x;
    for (int e = threadIdx.x; e < nent; e += kAdjBlock, j += kAdjBlock) {
      while (j >= d) {  // j counts from the row's first stored column
        j -= herm ? d - i - 1 : d;
        ++i;
      }
      fn(e, i, j);
    }
  }
  __device__ __forceinline__ void put(double2 *m, int i, int j, double2 v) const {
    if (herm && i == j) v.y = 0.0;
    m[i * ld + j] = v;
    if (herm && i != j) m[j * ld + i] = cj(v);
  }
  __device__ __forceinline__ double weight(int i, int j) const { return herm && i != j ? 2.0 : 1.0; }

  // Totals over the CTA of nv (1 or 2) values per thread, on the lanes of warp 0.
  __device__ void reduce(double *v, int nv) const {
    for (int q = 0; q < nv; ++q) red[q * kAdjBlock + threadIdx.x] = v[q];
    __syncthreads();
    if (threadIdx.x < 32)
      for (int q = 0; q < nv; ++q) {
        double x = 0.0;
        for (int s = threadIdx.x; s < kAdjBlock; s += 32) x += red[q * kAdjBlock + s];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        v[q] = x;
      }
  }

  // (Op M)_ij and (M Op^dag)_ij over the stored (off-diagonal) entries,
  // l += ..., r += ...
  template <bool REAL>
  __device__ __forceinline__ void lr(const AdjOp &o, const double2 *__restrict__ M, int i, int j,
                                     double2 &l, double2 &r) const {
    for (int s = 0; s < o.w; ++s) {
      const int pi = o.off + s * d + i, pj = o.off + s * d + j;
      const double2 vi = __ldg(a.ops.val64 + pi), vj = __ldg(a.ops.val64 + pj);
      const double2 g = M[__ldg(a.ops.col + pi) * ld + j], h = M[i * ld + __ldg(a.ops.col + pj)];
      if (REAL) {
        l = vfma(vi.x, g, l);
        r = vfma(vj.x, h, r);
      } else {
        cmac(l, vi, g);
        cmac(r, cj(vj), h);
      }
    }
  }
  __device__ __forceinline__ void lr(const AdjOp &o, const double2 *M, int i, int j, double2 &l,
                                     double2 &r) const {
    if (o.real) lr<true>(o, M, i, j, l, r);
    else lr<false>(o, M, i, j, l, r);
  }
  // [Op, M]_ij over the off-diagonal entries
  __device__ __forceinline__ double2 commutator(const AdjOp &o, const double2 *M, int i, int j) const {
    double2 l = make_double2(0.0, 0.0), r = l;
    lr(o, M, i, j, l, r);
    return make_double2(l.x - r.x, l.y - r.y);
  }
  // (A M A^dag)_ij from the rows i and j of A
  template <bool REAL>
  __device__ __forceinline__ double2 sand(const AdjOp &o, const double2 *__restrict__ M, int i,
                                          int j) const {
    double2 acc = make_double2(0.0, 0.0);
    for (int s = 0; s < o.w; ++s) {
      const int ps = o.off + s * d + i;
      const double2 u = __ldg(a.ops.val64 + ps);
      const double2 *row = M + __ldg(a.ops.col + ps) * ld;
      for (int t = 0; t < o.w; ++t) {
        const int pt = o.off + t * d + j;
        const double2 v = __ldg(a.ops.val64 + pt), m = row[__ldg(a.ops.col + pt)];
        if (REAL) acc = vfma(u.x * v.x, m, acc);
        else cmac(acc, make_double2(u.x * v.x + u.y * v.y, u.y * v.x - u.x * v.y), m);
      }
    }
    return acc;
  }
  // A_k M A_k^dag (or A_k^dag M A_k) - 1/2 {A_k^dag A_k, M}, its off-diagonal parts
  __device__ __forceinline__ double2 dissipator(int k, bool dagger, const double2 *M, int i, int j) const {
    const AdjOp &o = dagger ? a.op_ad[k] : a.op_a[k];
    double2 t = o.real ? sand<true>(o, M, i, j) : sand<false>(o, M, i, j);
    if (a.op_n[k].w > 0) {
      double2 l = make_double2(0.0, 0.0), r = l;
      lr(a.op_n[k], M, i, j, l, r);
      t = vfma(-0.5, vadd(l, r), t);
    }
    return t;
  }
  // The diagonal coefficient of dissipator k at (i, j).
  __device__ __forceinline__ double2 diag_k(int k, int i, int j) const {
    const double2 u = a.diag_a[k * d + i], v = a.diag_a[k * d + j];
    return make_double2(u.x * v.x + u.y * v.y - 0.5 * (a.diag_n[k * d + i] + a.diag_n[k * d + j]),
                        u.y * v.x - u.x * v.y);
  }
  // D_ij of the generator without the drive: -i (h0_i - h0_j) + sum_k gamma_k d_k.
  __device__ double2 diag(int i, int j) const {
    double2 D = make_double2(0.0, a.diag_h[j].x - a.diag_h[i].x);
    for (int k = 0; k < nk; ++k) D = vfma(gam[k], diag_k(k, i, j), D);
    return D;
  }

  // Entry (i, j) of F(M): D the diagonal, w the drive.
  __device__ __forceinline__ double2 gen(double2 D, double w, const double2 *M, int i, int j) const {
    double2 o = make_double2(0.0, 0.0);
    cmac(o, D, M[i * ld + j]);
    if (a.op_hd.w > 0) {
      const double2 z = commutator(a.op_hd, M, i, j);
      o.x = fma(w, z.y, o.x);  // -i w z
      o.y = fma(-w, z.x, o.y);
    }
    if (a.op_h0.w > 0) {
      const double2 z = commutator(a.op_h0, M, i, j);
      o.x += z.y;
      o.y -= z.x;
    }
    for (int k = 0; k < nk; ++k)
      if (a.op_a[k].w > 0 || a.op_n[k].w > 0) o = vfma(gam[k], dissipator(k, false, M, i, j), o);
    return o;
  }
  // D with the drive's diagonal, for segments with drive w
  __device__ __forceinline__ double2 drive(double2 D, double w, int i, int j) const {
    if (a.hd_diag) D.y = fma(w, a.diag_h[j].y - a.diag_h[i].y, D.y);
    return D;
  }

  // Re Tr(P M) over this thread's rows.
  __device__ double trace_rows(const AdjOp &o, const double2 *M) const {
    double x = 0.0;
    for (int r = threadIdx.x; r < d; r += kAdjBlock)
      for (int s = 0; s < o.w; ++s) {
        const int p = o.off + s * d + r;
        const double2 v = __ldg(a.ops.val64 + p), m = M[__ldg(a.ops.col + p) * ld + r];
        x = fma(v.x, m.x, x);
        x = fma(-v.y, m.y, x);
      }
    return x;
  }
  // Entry (i, j) of an operator.
  __device__ double2 dense(const AdjOp &o, int i, int j) const {
    double2 acc = make_double2(0.0, 0.0);
    for (int s = 0; s < o.w; ++s) {
      const int p = o.off + s * d + i;
      if (a.ops.col[p] == j) acc = vadd(acc, a.ops.val64[p]);
    }
    return acc;
  }
  // This thread's entries of m by h (a step that is dpp_scaled).
  __device__ void scale(double2 *m, double h) const {
    each([&](int, int i, int j) { put(m, i, j, vmul(h, m[i * ld + j])); });
  }
  // The last forward pass of this vector did not reach the final time: its
  // grid and checkpoints end before.
  __device__ bool failed() const {
    return a.nsteps[(int64_t)blockIdx.x * a.n_seg + a.n_seg - 1] == 0;
  }
  // The coefficients of a step of length h by lanes 0..7 of warp 0.
  __device__ __forceinline__ void powers(double h) const {
    if (threadIdx.x < 8) {
      const bool scaled = dpp_scaled(h);
      double p = 1.0;
      for (int q = 0; q < (int)threadIdx.x; ++q) p = scaled ? h : p * h;
      const double c = threadIdx.x == 0 ? 1.0 : dpp_c(threadIdx.x);
      ctl->c[threadIdx.x] = c * p;
      ctl->e[threadIdx.x] = dpp_e(threadIdx.x) * (threadIdx.x == 7 ? h : p);
      ctl->l[threadIdx.x] = scaled ? c : c * p;
    }
  }
};

// Forward solve of one parameter vector: adaptive (recording the grid and
// the segment checkpoints) or on the recorded grid (a.fixed, loss only).
// nsteps[s] stays 0 for a segment that was not completed (an error status), so
// a vector's grid is whole exactly when that of its last segment is not 0:
// Adj::failed() tells the passes on the recorded grid, which return NaN then
// (as does the loss of the failing pass itself).
__global__ void __launch_bounds__(kAdjBlock, 1) adjoint_forward_kernel(const __grid_constant__ AdjArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  Adj A(a, smem);
  const int b = blockIdx.x, d = A.d, ld = A.ld;
  const int64_t n = (int64_t)d * d;
  const double *om = a.omega + (int64_t)b * a.n_seg;
  int *nsteps = a.nsteps + (int64_t)b * a.n_seg;
  double *hgrid = a.hgrid + (int64_t)b * a.n_seg * a.maxs;
  double2 *ckpt = a.ckpt + (int64_t)b * (a.n_seg + 1) * n;
  double2 *rho = A.array(0), *v1 = A.array(1), *sum = A.array(2), *err = A.array(3),
          *Dst = A.array(4);
  double2 *y0 = A.y0, *y1 = A.y1;
  AdjCtl *ctl = A.ctl;
  const bool lead = threadIdx.x < 32;
  if (a.fixed && A.failed()) {
    if (threadIdx.x == 0) a.loss[b] = nan_value();
    return;
  }
  if (!a.fixed)
    for (int s = threadIdx.x; s < a.n_seg; s += kAdjBlock) nsteps[s] = 0;
  auto checkpoint = [&](int s) {
    for (int x = threadIdx.x; x < n; x += kAdjBlock) ckpt[(int64_t)s * n + x] = y1[x / d * ld + x % d];
  };
  A.each([&](int e, int i, int j) {
    A.put(y1, i, j, a.rho0[i * d + j]);
    Dst[e] = A.diag(i, j);
  });
  __syncthreads();
  if (!a.fixed) checkpoint(0);
  double q = 0.0;  // this thread's share of q
  double hprop = 0.0, v[2];
  bool after_reject = false;
  int status = QT_OK;
  unsigned long long n_acc = 0, n_rej = 0, n_rhs = 0;
  const double inv_n = 1.0 / (2.0 * (double)n);
  for (int s = 0; s < a.n_seg && status == QT_OK; ++s) {
    const double w = om[s];
    A.each([&](int e, int i, int j) { v1[e] = A.gen(A.drive(Dst[e], w, i, j), w, y1, i, j); });
    ++n_rhs;
    if (!a.fixed && s == 0) {
      // Hairer-Norsett-Wanner starting step
      v[0] = v[1] = 0.0;
      A.each([&](int e, int i, int j) {
        const double2 r = y1[i * ld + j], f = v1[e];
        const double sx = a.atol + a.rtol * fabs(r.x), sy = a.atol + a.rtol * fabs(r.y);
        const double wt = A.weight(i, j);
        v[0] += wt * ((r.x / sx) * (r.x / sx) + (r.y / sy) * (r.y / sy));
        v[1] += wt * ((f.x / sx) * (f.x / sx) + (f.y / sy) * (f.y / sy));
      });
      A.reduce(v, 2);
      double d1 = 0.0;
      if (lead) {
        const double d0 = sqrt(v[0] / (2.0 * n));
        d1 = sqrt(v[1] / (2.0 * n));
        if (threadIdx.x == 0) ctl->h = (d0 < 1e-5 || d1 < 1e-5) ? 1e-6 : 0.01 * d0 / d1;
      }
      __syncthreads();
      const double h0 = ctl->h;
      A.each([&](int e, int i, int j) { A.put(y0, i, j, vfma(h0, v1[e], y1[i * ld + j])); });
      __syncthreads();
      v[0] = 0.0;
      A.each([&](int e, int i, int j) {
        const double2 r = y1[i * ld + j], f = v1[e];
        const double2 g = A.gen(A.drive(Dst[e], w, i, j), w, y0, i, j);
        const double sx = a.atol + a.rtol * fabs(r.x), sy = a.atol + a.rtol * fabs(r.y);
        const double ex = (g.x - f.x) / sx, ey = (g.y - f.y) / sy;
        v[0] += A.weight(i, j) * (ex * ex + ey * ey);
      });
      ++n_rhs;
      A.reduce(v, 1);
      if (lead) {
        const double d2 = sqrt(v[0] / (2.0 * n)) / h0;
        const double dm = fmax(d1, d2);
        const double h1 = (dm <= 1e-15) ? fmax(1e-6, h0 * 1e-3) : pow(0.01 / dm, 0.2);
        hprop = fmin(100.0 * h0, h1);
      }
    }
    // the control warp's view of the segment
    double u = 0.0, h = 0.0;
    int ns = 0;
    int64_t attempts = 0;
    bool clipped = false;
    const int fixed_ns = a.fixed ? nsteps[s] : 0;
    auto next = [&]() {
      const bool more = a.fixed ? ns < fixed_ns : u < a.t_seg;
      if (more && attempts++ >= a.max_steps) status = QT_ESTEP;
      if (more && status == QT_OK) {
        if (a.fixed) {
          h = hgrid[ns];
        } else {
          const double rest = a.t_seg - u;
          clipped = !pos_less(hprop, rest);
          h = clipped ? rest : hprop;
        }
        A.powers(h);
      }
      if (threadIdx.x == 0) {
        ctl->h = h;
        ctl->done = !more;
        ctl->status = status;
      }
    };
    __syncthreads();
    if (lead) {
      next();
      if (threadIdx.x == 0) ctl->accepted = 1;
    }
    __syncthreads();
    bool first = true;
    for (;;) {
      const bool accepted = ctl->accepted != 0;
      status = ctl->status;
      if (ctl->done || status != QT_OK) break;
      if (accepted && !first) {  // err holds F of the new state
        double2 *sw = v1;
        v1 = err;
        err = sw;
      }
      // v_1; the accepted state becomes rho
      const double c1 = ctl->c[1], e1 = ctl->e[1], hs = ctl->h;
      if (first || accepted) {
        A.each([&](int e, int i, int j) { rho[e] = y1[i * ld + j]; });
      }
      first = false;
      double dq = 0.0;
      if (!accepted) {  // Tr(P2 rho) needs the state's matrix again
        A.each([&](int e, int i, int j) { A.put(y1, i, j, rho[e]); });
        __syncthreads();
      }
      auto powers = [&](auto scaled) {
        constexpr bool SC = decltype(scaled)::value;  // dpp_scaled
        if (threadIdx.x < d) dq = c1 * A.trace_rows(a.op_p2, y1);
        A.each([&](int e, int i, int j) {
          const double2 g = v1[e];
          sum[e] = vmul(c1, g);
          err[e] = vmul(e1, g);
          A.put(y0, i, j, g);
        });
        if constexpr (SC) A.scale(y0, hs);
        __syncthreads();
#pragma unroll 1
        for (int k = 2; k <= 6; ++k) {
          const double2 *in = (k & 1) ? y1 : y0;
          double2 *nxt = (k & 1) ? y0 : y1;
          const double c = ctl->c[k], ce = ctl->e[k];
          if (threadIdx.x < d) dq = fma(c, A.trace_rows(a.op_p2, in), dq);
          A.each([&](int e, int i, int j) {
            const double2 g = A.gen(A.drive(Dst[e], w, i, j), w, in, i, j);
            const double2 sk = vfma(c, g, sum[e]);
            sum[e] = sk;
            if (!a.fixed) err[e] = vfma(ce, g, err[e]);
            A.put(nxt, i, j, k == 6 ? vadd(rho[e], sk) : g);
          });
          if constexpr (SC)
            if (k < 6) A.scale(nxt, hs);
          __syncthreads();
        }
      };
      if (dpp_scaled(hs)) powers(std::true_type());
      else powers(std::false_type());
      // F of the new state, fused with the error norm
      {
        const double e7 = ctl->e[7];
        double acc = 0.0;
        A.each([&](int e, int i, int j) {
          const double2 g = A.gen(A.drive(Dst[e], w, i, j), w, y1, i, j);
          if (!a.fixed) {
            const double2 er = vfma(e7, g, err[e]);
            const double2 r = rho[e], yn = y1[i * ld + j];
            const double qx = ratio(er.x, fma(a.rtol, max_abs(r.x, yn.x), a.atol));
            const double qy = ratio(er.y, fma(a.rtol, max_abs(r.y, yn.y), a.atol));
            acc = fma(A.weight(i, j), fma(qx, qx, qy * qy), acc);
          }
          err[e] = g;
        });
        v[0] = acc;
      }
      n_rhs += a.fixed && ns == 0 ? 5 : 6;
      A.reduce(v, 1);
      if (lead) {
        bool ok = true;
        if (!a.fixed) {
          const double x = v[0] * inv_n;
          if (!finite_bits(x)) {
            status = QT_ENUMERIC;
            ok = false;
          } else {
            ok = !pos_less(1.0, x);
            hprop = dp_control_sq<double>(h, x, ok, after_reject, clipped, hprop);
            after_reject = !ok;
          }
        }
        if (ok) {
          if (!a.fixed) {
            if (ns >= a.maxs) status = QT_ESTEP;
            else if (threadIdx.x == 0) hgrid[(int64_t)s * a.maxs + ns] = h;
            u = clipped ? a.t_seg : u + h;
          }
          ++ns;
          ++n_acc;
        } else {
          ++n_rej;
        }
        next();
        if (threadIdx.x == 0) {
          ctl->accepted = ok;
          ctl->status = status;
        }
      }
      __syncthreads();
      if (ctl->accepted) q += dq;
    }
    if (a.fixed) hgrid += a.maxs;
    if (status != QT_OK) break;
    if (!a.fixed) {
      if (threadIdx.x == 0) nsteps[s] = ns;
      checkpoint(s + 1);
    }
    __syncthreads();
  }
  v[0] = A.trace_rows(a.op_p1, y1) + q;
  __syncthreads();
  A.reduce(v, 1);
  if (threadIdx.x == 0) {
    if (status != QT_OK) set_status(a.status, status);
    a.loss[b] = status == QT_OK ? v[0] : nan_value();
    atomicAdd(a.counters + 0, n_acc);
    atomicAdd(a.counters + 1, n_rej);
    atomicAdd(a.counters + 2, n_rhs);
  }
}

// Backward pass of one parameter vector on its recorded grid.
__global__ void __launch_bounds__(kAdjBlock, 1) adjoint_backward_kernel(const __grid_constant__ AdjArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  Adj A(a, smem);
  const int b = blockIdx.x, d = A.d, ld = A.ld, nk = A.nk;
  const int64_t n = (int64_t)d * d;
  const double *om = a.omega + (int64_t)b * a.n_seg;
  const int *nsteps = a.nsteps + (int64_t)b * a.n_seg;
  const double *hgrid = a.hgrid + (int64_t)b * a.n_seg * a.maxs;
  const double2 *ckpt = a.ckpt + (int64_t)b * (a.n_seg + 1) * n;
  double2 *y0 = A.y0, *y1 = A.y1;
  AdjCtl *ctl = A.ctl;
  double *gk = A.gk;
  const double scale = a.dloss ? a.dloss[b] : 1.0;
  if (A.failed()) {
    for (int s = threadIdx.x; s < a.n_seg; s += kAdjBlock) a.g_omega[(int64_t)b * a.n_seg + s] = nan_value();
    for (int k = threadIdx.x; k < nk; k += kAdjBlock) a.g_gamma[(int64_t)b * nk + k] = nan_value();
    return;
  }
  // workspace: lambda, D, P2, the sums of conj(a) v, a step sum, v_1..v_5 of
  // one recomputed step, the segment's states, then v_1..v_5 of its first
  // `kept` steps
  double2 *lam = A.array(0), *Dst = A.array(1), *P2 = A.array(2), *S = A.array(3),
          *sum = A.array(4), *one = A.array(5), *X = A.array(10), *V = A.array(11 + a.maxs);
  const int64_t room = a.slots * n / A.nent - (11 + a.maxs);
  const int kept = (int)(room / 5 < a.maxs ? room / 5 : a.maxs);
  const int nent = A.nent;
  // lambda(T) = P1
  A.each([&](int e, int i, int j) {
    lam[e] = A.dense(a.op_p1, i, j);
    P2[e] = A.dense(a.op_p2, i, j);
    Dst[e] = A.diag(i, j);
    S[e] = make_double2(0.0, 0.0);
  });
  for (int k = 0; k < nk; ++k) gk[k * kAdjBlock + threadIdx.x] = 0.0;
  // v_1..v_5 of the step of length h from the state x (already in y1 unless
  // load) into vk; with xn also the state after the step (its matrix in y1)
  auto powers_of = [&](double w, double h, const double2 *x, bool load, double2 *vk, double2 *xn) {
    if (load) {
      __syncthreads();
      A.each([&](int e, int i, int j) { A.put(y1, i, j, x[e]); });
      __syncthreads();
    }
    auto powers = [&](auto scaled) {
      constexpr bool SC = decltype(scaled)::value;  // dpp_scaled
#pragma unroll 1
      for (int k = 1; k <= (xn ? 6 : 5); ++k) {
        const double2 *in = (k & 1) ? y1 : y0;
        double2 *nxt = (k & 1) ? y0 : y1;
        const double c = ctl->c[k];
        A.each([&](int e, int i, int j) {
          const double2 g = A.gen(A.drive(Dst[e], w, i, j), w, in, i, j);
          if (xn) {
            const double2 sk = k == 1 ? vmul(c, g) : vfma(c, g, sum[e]);
            if (k < 6) {
              sum[e] = sk;
            } else {
              const double2 y = vadd(x[e], sk);
              xn[e] = y;
              A.put(y1, i, j, y);
            }
          }
          if (k < 6) {
            const double2 v = SC ? vmul(h, g) : g;
            vk[(int64_t)(k - 1) * nent + e] = v;
            if (k < 5 || xn) A.put(nxt, i, j, v);
          }
        });
        __syncthreads();
      }
    };
    if (dpp_scaled(h)) powers(std::true_type());
    else powers(std::false_type());
  };
  double v[2];
  for (int s = a.n_seg - 1; s >= 0; --s) {
    const double w = om[s];
    const int ns = nsteps[s];
    const double *hs = hgrid + (int64_t)s * a.maxs;
    __syncthreads();
    A.each([&](int e, int i, int j) {
      const double2 x = ckpt[(int64_t)s * n + i * d + j];
      X[e] = x;
      A.put(y1, i, j, x);
    });
    // the segment's states and their v_k
    for (int m = 0; m < ns; ++m) {
      if (threadIdx.x < 32) A.powers(hs[m]);
      __syncthreads();
      double2 *x = X + (int64_t)m * nent;
      powers_of(w, hs[m], x, false, m < kept ? V + (int64_t)m * 5 * nent : one,
                m + 1 < ns ? x + nent : nullptr);
    }
    double gom = 0.0;
    for (int m = ns - 1; m >= 0; --m) {
      const double h = hs[m];
      const double2 *x = X + (int64_t)m * nent;
      const double2 *vk = V + (int64_t)m * 5 * nent;
      __syncthreads();
      if (threadIdx.x < 32) A.powers(h);
      __syncthreads();
      if (m >= kept) {
        if (m + 1 < ns) powers_of(w, h, x, true, one, nullptr);
        vk = one;
      }
      {
        const double c6 = ctl->c[6];
        __syncthreads();
        A.each([&](int e, int i, int j) { A.put(y0, i, j, vmul(c6, lam[e])); });
        __syncthreads();
      }
      // a_k (of a scaled step: a_k / h^(k-1)) in y0 (k even) or y1 (k odd)
      auto adjoint = [&](auto scaled) {
        constexpr bool SC = decltype(scaled)::value;  // dpp_scaled
#pragma unroll 1
        for (int k = 6; k >= 1; --k) {
          const double2 *in = (k & 1) ? y1 : y0;
          double2 *nxt = (k & 1) ? y0 : y1;
          const double2 *vp = k == 1 ? x : vk + (int64_t)(k - 2) * nent;
          const double cl = ctl->l[k - 1], cp = ctl->c[k];
          A.each([&](int e, int i, int j) {
            const double wt = A.weight(i, j);
            const double2 av = in[i * ld + j], y = vp[e];
            double2 yw = make_double2(wt * y.x, wt * y.y);
            // the diagonal of F^dag, and conj(a) v for its parameter derivatives
            double2 o = make_double2(0.0, 0.0), sv = S[e];
            cmac(o, cj(A.drive(Dst[e], w, i, j)), av);
            sv.x = fma(av.x, yw.x, sv.x);
            sv.x = fma(av.y, yw.y, sv.x);
            if (a.dk_complex) {
              sv.y = fma(av.x, yw.y, sv.y);
              sv.y = fma(-av.y, yw.x, sv.y);
            }
            S[e] = sv;
            double2 z = make_double2(0.0, 0.0);
            if (a.op_hd.w > 0) {
              z = A.commutator(a.op_hd, in, i, j);
              o.x = fma(-w, z.y, o.x);  // +i w z
              o.y = fma(w, z.x, o.y);
            }
            if (a.hd_diag) z = vfma(a.diag_h[i].y - a.diag_h[j].y, av, z);
            gom = fma(-z.y, yw.x, gom);  // <i z, v>
            gom = fma(z.x, yw.y, gom);
            if (a.op_h0.w > 0) {
              const double2 c = A.commutator(a.op_h0, in, i, j);
              o.x -= c.y;
              o.y += c.x;
            }
            for (int q = 0; q < nk; ++q)
              if (a.op_a[q].w > 0 || a.op_n[q].w > 0) {
                const double2 t = A.dissipator(q, true, in, i, j);
                o = vfma(A.gam[q], t, o);
                double g = gk[q * kAdjBlock + threadIdx.x];
                g = fma(t.x, yw.x, g);
                gk[q * kAdjBlock + threadIdx.x] = fma(t.y, yw.y, g);
              }
            o = vfma(cl, lam[e], o);
            o = vfma(cp, P2[e], o);
            if (k == 1) lam[e] = o;
            else A.put(nxt, i, j, o);
          });
          if constexpr (SC)
            if (k > 1) A.scale(nxt, h);
          __syncthreads();
        }
      };
      if (dpp_scaled(h)) adjoint(std::true_type());
      else adjoint(std::false_type());
    }
    v[0] = gom;
    A.reduce(v, 1);
    if (threadIdx.x == 0) a.g_omega[(int64_t)b * a.n_seg + s] = scale * v[0];
  }
  for (int k = 0; k < nk; ++k) {
    // the diagonal part: sum of Re(d_k conj(a) v)
    double g = gk[k * kAdjBlock + threadIdx.x];
    A.each([&](int e, int i, int j) {
      const double2 D = A.diag_k(k, i, j), sv = S[e];
      g = fma(D.x, sv.x, g);
      g = fma(-D.y, sv.y, g);
    });
    v[0] = g;
    __syncthreads();
    A.reduce(v, 1);
    if (threadIdx.x == 0) a.g_gamma[(int64_t)b * nk + k] = scale * v[0];
  }
}

// The kernels' limit is that of the largest problem (dim 64, 8 decay rates),
// whatever this one takes: it belongs to the process, and one set for a
// smaller problem on another thread would refuse this thread's launch.
cudaError_t smem_for(const void *kern, const AdjArgs &a, size_t *bytes) {
  *bytes = adj_smem(a.ops.d, a.nk).total;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)adj_smem(64, 8).total);
}

}  // namespace

size_t adjoint_slots(int maxs) { return 28 + (size_t)maxs + 1; }

cudaError_t launch_adjoint_forward(const AdjArgs &a, cudaStream_t s) {
  size_t smem;
  cudaError_t e = smem_for((const void *)adjoint_forward_kernel, a, &smem);
  if (e != cudaSuccess) return e;
  adjoint_forward_kernel<<<a.batch, kAdjBlock, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_backward(const AdjArgs &a, cudaStream_t s) {
  size_t smem;
  cudaError_t e = smem_for((const void *)adjoint_backward_kernel, a, &smem);
  if (e != cudaSuccess) return e;
  adjoint_backward_kernel<<<a.batch, kAdjBlock, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace qt
