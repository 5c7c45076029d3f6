// qt_corr.cu -- two-time correlation functions <A(t + tau) B(t)> by the
// quantum regression theorem (the ODE form of the paper's correlation
// functions, section 5 function list): with rho(t_k) from one master-equation
// solve, X_k = B rho(t_k) is evolved over tau by the same Lindblad generator
// and C(t_k, tau_j) = Tr[A X_k(t_k + tau_j)].
//
// Small systems: one CTA per X_k (the solver of qt_me_small.cuh on all d*d
// entries; the general solver of qt_me_impl.cuh for the systems that it does
// not take), X_k and the shifted output times formed by the CTA itself.  With
// two CTAs per SM the dim-20 FP64 correlation keeps the FP64 pipe 80 % busy.
// Larger systems: corr_prepare_kernel forms one X_k and its times, and the
// cooperative solver of qt_me.cu evolves it.
//
// The same one-CTA-per-start-matrix scheme gives the propagator (the paper's
// propagator): every matrix unit evolved, its states scattered into the
// columns of U(t_k).
#include "qt_me_impl.cuh"
#include "qt_me_small.cuh"

namespace qt {

namespace {

// X = B rho_k (FP64; B is table operator b_op in ELL rows) and the output
// times t_k + tau_j of the k-th evolution, by threads tid, tid + stride, ...
__device__ __forceinline__ void corr_prepare(const OpTable &ops, const CorrArgs &c, int k,
                                             double2 *X, double *times, int64_t tid,
                                             int64_t stride) {
  const int d = ops.d;
  const int64_t n = (int64_t)d * d;
  const double2 *rho = c.rho_t + (int64_t)k * n;
  const int w = ops.w[c.b_op];
  const int64_t off = ops.off[c.b_op];
  for (int64_t idx = tid; idx < n; idx += stride) {
    const int i = (int)(idx / d), j = (int)(idx - (int64_t)i * d);
    double2 acc = make_double2(0.0, 0.0);
    for (int s = 0; s < w; ++s) {
      const int64_t p = off + (int64_t)s * d + i;
      cmac(acc, ops.val64[p], rho[(int64_t)__ldg(ops.col + p) * d + j]);
    }
    X[idx] = acc;
  }
  const double tk = c.tlist[k];
  for (int64_t j = tid; j < c.n_tau; j += stride) times[j] = __dadd_rn(tk, c.taulist[j]);
}

__global__ void corr_prepare_kernel(const __grid_constant__ OpTable ops,
                                    const __grid_constant__ CorrArgs c, int k, double2 *X,
                                    double *times) {
  corr_prepare(ops, c, k, X, times, (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
               (int64_t)gridDim.x * blockDim.x);
}

// How a CTA solves: the shared-memory solver of qt_me_small.cuh with the
// entry arrays in shared memory or in the workspace, or the general solver
// (time-dependent terms, wide operators).
enum class SmallMode { kShared, kWork, kGeneral };

template <typename T, SmallMode MODE>
__device__ void cta_solve(const MeArgs &m) {
  if constexpr (MODE == SmallMode::kGeneral) {
    using V = typename CT<T>::V;
    __shared__ double sh[kMePartialMax * (kMeBlock / 32) + kMePartialMax];
    __shared__ double tot[kMePartialMax];
    __shared__ double tdcoef[kTdMax];
    BlockTeam team;
    SparseRhs<T> rhs(m, sizeof(T) == 8 ? reinterpret_cast<const V *>(m.ops.val64)
                                       : reinterpret_cast<const V *>(m.ops.val32), tdcoef);
    me_solve<T>(m, team, rhs, sh, tot);
  } else {
    extern __shared__ double2 dyn_smem[];
    SmallSolver<T, false, MODE == SmallMode::kShared> s(
        m, false, reinterpret_cast<unsigned char *>(dyn_smem),
        reinterpret_cast<unsigned char *>(m.work), 0, 1);
    s.solve();
  }
}

// CTA b evolves X_k for k = b, b + grid, ...; its slab of a.work holds the
// solver workspace, X_k and the times.  a carries the tau evolution (n_t =
// n_tau, expect = the correlation array, all d*d entries of X_k).
// MODE: the solver of the CTA (SmallMode above).
template <typename T, SmallMode MODE>
__global__ void __launch_bounds__(kMeBlock) corr_block_kernel(const __grid_constant__ MeArgs a,
                                                              const __grid_constant__ CorrArgs c) {
  __shared__ MeArgs m;
  char *slab = reinterpret_cast<char *>(a.work) + (size_t)blockIdx.x * c.ws_stride;
  double2 *X = reinterpret_cast<double2 *>(slab + c.x_off);
  double *times = reinterpret_cast<double *>(slab + c.times_off);
  for (int k = blockIdx.x; k < c.n_t; k += gridDim.x) {
    corr_prepare(a.ops, c, k, X, times, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) {
      m = a;
      m.state0 = X;
      m.tlist = times;
      m.expect = a.expect + (int64_t)k * a.n_t * a.n_e;
      m.work = slab;
    }
    __syncthreads();
    cta_solve<T, MODE>(m);
    __syncthreads();  // m, X and times are rewritten for the next k
  }
}

// The propagator: CTA b evolves the matrix units E_k (k = a d + b') for
// k = b, b + grid, ... from tlist[0] by the solver of MODE and scatters each
// output state rho_k(t_m) into column k of U(t_m): U[m][ij][k].
template <typename T, SmallMode MODE>
__global__ void __launch_bounds__(kMeBlock) prop_block_kernel(const __grid_constant__ MeArgs a,
                                                              const __grid_constant__ PropArgs p) {
  __shared__ MeArgs m;
  const int64_t n = (int64_t)a.ops.d * a.ops.d;
  char *slab = reinterpret_cast<char *>(a.work) + (size_t)blockIdx.x * p.ws_stride;
  double2 *X = reinterpret_cast<double2 *>(slab + p.x_off);
  double2 *st = reinterpret_cast<double2 *>(slab + p.st_off);
  for (int64_t k = blockIdx.x; k < n; k += gridDim.x) {
    for (int64_t idx = threadIdx.x; idx < n; idx += blockDim.x)
      X[idx] = make_double2(idx == k ? 1.0 : 0.0, 0.0);
    if (threadIdx.x == 0) {
      m = a;
      m.state0 = X;
      m.states = st;
      m.work = slab;
    }
    __syncthreads();
    cta_solve<T, MODE>(m);
    __syncthreads();
    for (int t = 0; t < a.n_t; ++t)
      for (int64_t idx = threadIdx.x; idx < n; idx += blockDim.x)
        p.U[((int64_t)t * n + idx) * n + k] = st[(int64_t)t * n + idx];
    __syncthreads();  // m, X and st are rewritten for the next k
  }
}

// The mode and the dynamic shared memory of a system (general matrices: all
// d*d entries).
SmallMode small_mode(const MeArgs &a, int precision, size_t *smem) {
  *smem = 0;
  if (!small_fits(a)) return SmallMode::kGeneral;
  const int d = a.ops.d, nent = small_entries(d, false);
  *smem = small_smem(precision, d, nent, a.small, 1, kMeBlock, true).total;
  if (*smem <= kSmallSmemMax) return SmallMode::kShared;
  *smem = small_smem(precision, d, nent, a.small, 1, kMeBlock, false).total;
  return SmallMode::kWork;
}

static_assert(sizeof(MeArgs) <= 1024, "static shared memory beside kSmallSmemMax");

// The limit of every instance with dynamic shared memory (one value for all
// sizes: see kSmallSmemMax).
template <typename K>
cudaError_t set_smem_limit(K kern, size_t smem) {
  if (smem == 0) return cudaSuccess;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmallSmemMax);
}

// Resident CTAs of a kernel with smem bytes of dynamic shared memory, at most
// units (negative on error).
template <typename K>
int block_grid(K kern, size_t smem, int64_t units) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (set_smem_limit(kern, smem) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMeBlock, smem) != cudaSuccess)
    return -1;
  if (per_sm < 1) return -1;
  const int64_t cap = (int64_t)sms * per_sm;
  return (int)(units < cap ? units : cap);
}

// fn(kernel) for the instance of the given precision and mode.
template <typename F>
auto with_corr_kernel(int precision, SmallMode m, F &&fn) {
  if (precision == QT_MIXED)
    return m == SmallMode::kShared  ? fn(corr_block_kernel<float, SmallMode::kShared>)
           : m == SmallMode::kWork  ? fn(corr_block_kernel<float, SmallMode::kWork>)
                                    : fn(corr_block_kernel<float, SmallMode::kGeneral>);
  return m == SmallMode::kShared ? fn(corr_block_kernel<double, SmallMode::kShared>)
         : m == SmallMode::kWork ? fn(corr_block_kernel<double, SmallMode::kWork>)
                                 : fn(corr_block_kernel<double, SmallMode::kGeneral>);
}
template <typename F>
auto with_prop_kernel(int precision, SmallMode m, F &&fn) {
  if (precision == QT_MIXED)
    return m == SmallMode::kShared  ? fn(prop_block_kernel<float, SmallMode::kShared>)
           : m == SmallMode::kWork  ? fn(prop_block_kernel<float, SmallMode::kWork>)
                                    : fn(prop_block_kernel<float, SmallMode::kGeneral>);
  return m == SmallMode::kShared ? fn(prop_block_kernel<double, SmallMode::kShared>)
         : m == SmallMode::kWork ? fn(prop_block_kernel<double, SmallMode::kWork>)
                                 : fn(prop_block_kernel<double, SmallMode::kGeneral>);
}

}  // namespace

int corr_block_grid(const MeArgs &a, int n_t, int precision) {
  size_t smem;
  const SmallMode m = small_mode(a, precision, &smem);
  return with_corr_kernel(precision, m, [&](auto *k) { return block_grid(k, smem, n_t); });
}

cudaError_t launch_corr_block(const MeArgs &a, const CorrArgs &c, int grid, int precision,
                              cudaStream_t s) {
  size_t smem;
  const SmallMode m = small_mode(a, precision, &smem);
  return with_corr_kernel(precision, m, [&](auto *k) {
    const cudaError_t e = set_smem_limit(k, smem);
    if (e != cudaSuccess) return e;
    k<<<grid, kMeBlock, smem, s>>>(a, c);
    return cudaGetLastError();
  });
}

int prop_block_grid(const MeArgs &a, int64_t units, int precision) {
  size_t smem;
  const SmallMode m = small_mode(a, precision, &smem);
  return with_prop_kernel(precision, m, [&](auto *k) { return block_grid(k, smem, units); });
}

cudaError_t launch_prop_block(const MeArgs &a, const PropArgs &p, int grid, int precision,
                              cudaStream_t s) {
  size_t smem;
  const SmallMode m = small_mode(a, precision, &smem);
  return with_prop_kernel(precision, m, [&](auto *k) {
    const cudaError_t e = set_smem_limit(k, smem);
    if (e != cudaSuccess) return e;
    k<<<grid, kMeBlock, smem, s>>>(a, p);
    return cudaGetLastError();
  });
}

cudaError_t launch_corr_prepare(const OpTable &ops, const CorrArgs &c, int k, double2 *X,
                                double *times, cudaStream_t s) {
  const int64_t n = (int64_t)ops.d * ops.d;
  const int64_t blocks = (n + 255) / 256;
  corr_prepare_kernel<<<(unsigned)(blocks < 2048 ? blocks : 2048), 256, 0, s>>>(ops, c, k, X,
                                                                              times);
  return cudaGetLastError();
}

}  // namespace qt
