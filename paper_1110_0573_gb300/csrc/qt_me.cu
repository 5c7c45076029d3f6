// qt_me.cu -- the master-equation solver as one cooperative launch over the
// whole grid: the Hermitian-state solver of qt_me_herm.cuh with the sparse
// product on the CUDA cores, or the general solver of qt_me_impl.cuh (no
// symmetry assumed) for non-Hermitian initial matrices and on request.
#include "qt_me_herm.cuh"
#include "qt_me_small.cuh"

namespace qt {

namespace {

template <typename T>
__global__ void __launch_bounds__(kMeBlock) me_kernel(const __grid_constant__ MeArgs a) {
  using V = typename CT<T>::V;
  extern __shared__ double2 dyn_smem[];  // tiles of the Hermitian combine phase
  __shared__ double sh[kMePartialMax * (kMeBlock / 32) + kMePartialMax];
  __shared__ double tot[kMePartialMax];
  __shared__ double tdcoef[kTdMax];
  GridTeam team(a.partial);
  const V *val = sizeof(T) == 8 ? reinterpret_cast<const V *>(a.ops.val64)
                                : reinterpret_cast<const V *>(a.ops.val32);
  bool herm = a.herm == 1;
  if (a.herm == 2) {
    const double2 *m = a.rhs_in ? a.rhs_in : a.state0;
    herm = (!a.rhs_in && a.state_is_ket) || herm_check(m, a.ops.d, team, sh, tot);
  }
  if (herm) {
    SpmmY<T> prod(a, val, tdcoef);
    V *tiles = reinterpret_cast<V *>(dyn_smem);
    if (a.rhs_in)
      me_rhs_once_herm<T>(a, team, prod, val, tiles);
    else
      me_solve_herm<T>(a, team, prod, val, tiles, sh, tot);
  } else {
    SparseRhs<T> rhs(a, val, tdcoef);
    if (a.rhs_in)
      me_rhs_once<T>(a, team, rhs, sh, tot);
    else
      me_solve<T>(a, team, rhs, sh, tot);
  }
}

// Small systems: the whole solve on one CTA (CL = false) or one cluster.
template <typename T, bool CL, bool KS>
__global__ void __launch_bounds__(kMeBlock, 1) me_small_kernel(const __grid_constant__ MeArgs a) {
  extern __shared__ double2 dyn_smem[];
  int rank = 0, nranks = 1;
  if constexpr (CL) {
    rank = (int)cg::this_cluster().block_rank();
    nranks = (int)cg::this_cluster().num_blocks();
  }
  unsigned char *work = nullptr;
  if constexpr (!KS)
    work = reinterpret_cast<unsigned char *>(a.work) +
           rank * small_ws_bytes(sizeof(T) == 4 ? QT_MIXED : QT_FP64, a.ops.d,
                                 small_entries(a.ops.d, a.small_herm != 0), a.small, nranks,
                                 (int)blockDim.x);
  SmallSolver<T, CL, KS> s(a, a.small_herm != 0, reinterpret_cast<unsigned char *>(dyn_smem), work,
                           rank, nranks);
  s.solve();
}

// Small systems with time-dependent terms, with operators too wide for the
// shared-memory copy, and single right-hand sides: the general solver on one
// CTA (team barriers are __syncthreads, no grid-wide synchronisation).
template <typename T>
__global__ void __launch_bounds__(kMeBlock) me_block_kernel(const __grid_constant__ MeArgs a) {
  using V = typename CT<T>::V;
  __shared__ double sh[kMePartialMax * (kMeBlock / 32) + kMePartialMax];
  __shared__ double tot[kMePartialMax];
  __shared__ double tdcoef[kTdMax];
  BlockTeam team;
  const V *val = sizeof(T) == 8 ? reinterpret_cast<const V *>(a.ops.val64)
                                : reinterpret_cast<const V *>(a.ops.val32);
  SparseRhs<T> rhs(a, val, tdcoef);
  if (a.rhs_in)
    me_rhs_once<T>(a, team, rhs, sh, tot);
  else
    me_solve<T>(a, team, rhs, sh, tot);
}

template <typename T>
size_t dyn_bytes(int n_cslots, int n_cterms) {
  return herm_smem_bytes<typename CT<T>::V>(n_cslots, n_cterms);
}

// The limit of me_kernel: the Hermitian solver with the most collapse operators
// that it stages (one value for all launches: see kSmemPerCta).
template <typename T>
cudaError_t set_me_limit() {
  return cudaFuncSetAttribute(me_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)dyn_bytes<T>(kCSlotsMax, kCTermsMax));
}

template <typename T>
int grid_for(int d, bool herm, int n_cslots, int n_cterms) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  const size_t dyn = herm ? dyn_bytes<T>(n_cslots, n_cterms) : 0;
  if (set_me_limit<T>() != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, me_kernel<T>, kMeBlock, dyn) !=
      cudaSuccess)
    return -1;
  if (per_sm < 1) return -1;
  const int64_t n = (int64_t)d * d;
  const int64_t nt = (d + kHT - 1) / kHT;
  int64_t want = herm ? nt * (nt + 1) / 2 : (n + kMeBlock - 1) / kMeBlock;
  int64_t cap = (int64_t)sms * per_sm;
  return (int)(want < cap ? want : cap);
}

}  // namespace

int me_grid(int d, int precision) {
  return precision == QT_MIXED ? grid_for<float>(d, false, 0, 0) : grid_for<double>(d, false, 0, 0);
}

int me_herm_grid(int d, int precision, int n_cslots, int n_cterms) {
  return precision == QT_MIXED ? grid_for<float>(d, true, n_cslots, n_cterms)
                               : grid_for<double>(d, true, n_cslots, n_cterms);
}

size_t me_workspace_bytes(int d, int precision, int grid) {
  const size_t elem = precision == QT_MIXED ? sizeof(float2) : sizeof(double2);
  return 11 * (size_t)d * d * elem + (size_t)grid * kMePartialMax * sizeof(double) + 256;
}

// Workspace of the small solver for a system it takes (0: it does not).
size_t small_workspace_bytes(const MeArgs &a, int precision, bool herm, bool cluster) {
  if (!small_fits(a)) return 0;
  const int d = a.ops.d, nent = small_entries(d, herm), ranks = cluster ? small_ranks(nent) : 1;
  return ranks * small_ws_bytes(precision, d, nent, a.small, ranks, kMeBlock);
}

namespace {

template <typename T, bool CL, bool KS>
cudaError_t launch_small_inst(const MeArgs &a, size_t smem, int ranks, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(me_small_kernel<T, CL, KS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmallSmemMax);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ranks);
  cfg.blockDim = dim3(kMeBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ranks;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = CL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, me_small_kernel<T, CL, KS>, a);
}

template <typename T>
cudaError_t launch_small(const MeArgs &a, cudaStream_t s) {
  const int prec = sizeof(T) == 4 ? QT_MIXED : QT_FP64;
  const int d = a.ops.d, nent = small_entries(d, a.small_herm != 0);
  const int ranks = small_ranks(nent);
  for (int ks = 1; ks >= 0; --ks) {
    const size_t smem = small_smem(prec, d, nent, a.small, ranks, kMeBlock, ks != 0).total;
    if (smem > kSmallSmemMax) continue;
    if (ranks > 1)
      return ks ? launch_small_inst<T, true, true>(a, smem, ranks, s)
                : launch_small_inst<T, true, false>(a, smem, ranks, s);
    return ks ? launch_small_inst<T, false, true>(a, smem, ranks, s)
              : launch_small_inst<T, false, false>(a, smem, ranks, s);
  }
  return cudaErrorInvalidValue;  // the matrices of kMeSmallDim always fit
}

}  // namespace

template <typename T>
cudaError_t launch_me_t(const MeArgs &a, cudaStream_t s) {
  if (a.single_cta) {
    if (!a.rhs_in && small_fits(a)) return launch_small<T>(a, s);
    me_block_kernel<T><<<1, kMeBlock, 0, s>>>(a);
    return cudaGetLastError();
  }
  const size_t dyn = a.herm ? dyn_bytes<T>(a.n_cslots, a.n_cterms) : 0;
  const cudaError_t e = set_me_limit<T>();
  if (e != cudaSuccess) return e;
  void *args[] = {const_cast<MeArgs *>(&a)};
  return cudaLaunchCooperativeKernel((const void *)me_kernel<T>, dim3(a.grid), dim3(kMeBlock),
                                     args, dyn, s);
}

cudaError_t launch_me(const MeArgs &a, int precision, cudaStream_t s) {
  return precision == QT_MIXED ? launch_me_t<float>(a, s) : launch_me_t<double>(a, s);
}

}  // namespace qt
