// k_adjoint.inl - launchers of the adjoint kernels of one storage form.  Included
// by k_storage.inl inside its anonymous namespace (S = the storage element type),
// kept apart from the forward launchers.

// Adjoint arithmetic type: FP64 for the FP64 form, else FP32.
using L = std::conditional<std::is_same<S, double>::value, double, float>::type;

// Blocks of an adjoint step (one dL/domega partial each).
long long adjoint_blocks(const Grid& g) {
  return std::is_same<S, double>::value ? (g.ncell + 31) / 32 : cell_blocks(g);
}

// The adjoint kernel for this grid: 32-bit element indices (FP32 adjoint) when
// Q ncell fits them.
using AdjointFn = void (*)(const S*, const L*, const double*, L*, double*, Grid, double);
template <int M, bool kFirst>
AdjointFn adjoint_kernel(const Grid& g) {
  if ((unsigned long long)Model<M>::Q * (unsigned long long)g.ncell <= 0xFFFFFFFFull)
    return k_adjoint<M, S, L, kFirst, true>;
  return k_adjoint<M, S, L, kFirst, false>;
}

// FP64 form: warps per 32 cells, by the blocks of 32 cells an SM gets, as step64_warps.  All
// measured (us an adjoint step with 1 / 2 / 4 warps, 152 SMs):
//   D3Q95, blocks an SM 1: 61.9 / 41.2 / 35.0, 2: 66.8 / 51.1 / 53.7, 3: 65.2 / 54.6 / 60.3,
//   5: 88.7 / 85.5 / 103, 6: 100 / 97 / 125, 7: 106 / 127 / 145, 8: 122 / 128 / 167,
//   9: 186 / 156 / 184, 14: 247 / 220 / 283, 27: 453 / 429 / 532, 432: 6852 / 6542 / 8282
//   D2Q33, 64 blocks: 25.6 / 16.5 / 14.0, 112: 26.6 / 17.2 / 15.4, 128: 25.8 / 17.3 / 18.3, an SM
//   2: 25.6 / 20.7 / 25.2, 3: 28.6 / 25.0 / 32.7, 4: 30.3 / 31.9 / 42.1, 5: 38.7 / 41.4 / 53.2,
//   14: 96 / 100 / 140, 432: 2475 / 2967 / 4258.
template <int M>
int adjoint64_warps(long long ncell, int sms) {
  const long long all = (ncell + 31) / 32, blocks = (all + sms - 1) / sms;
  if (M == 0) return 4 * all <= 3 * sms ? 4 : blocks <= 3 ? 2 : 1;
  return blocks == 1 ? 4 : blocks == 7 || blocks == 8 ? 1 : 2;
}

template <int M>
cudaError_t adjoint64_m(const void* state_n, const void* nu_next, const double* dldrho,
                        void* nu_out, double* omega_acc, const Grid& g, double omega,
                        cudaStream_t st) {
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  const int w = adjoint64_warps<M>(g.ncell, sms);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((g.ncell + 31) / 32));
  cfg.blockDim = dim3(32 * w);
  cfg.dynamicSmemBytes = dldrho ? 0 : Model<M>::Q * 32 * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto kern = k_adjoint64<M, false, 1>;
  if (dldrho) kern = w == 1 ? k_adjoint64<M, true, 1> : w == 2 ? k_adjoint64<M, true, 2> : k_adjoint64<M, true, 4>;
  else kern = w == 1 ? k_adjoint64<M, false, 1> : w == 2 ? k_adjoint64<M, false, 2> : k_adjoint64<M, false, 4>;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<const double*>(state_n),
                            static_cast<const double*>(nu_next), dldrho,
                            static_cast<double*>(nu_out), omega_acc, g, omega);
}

template <int M>
cudaError_t adjoint_m(const void* state_n, const void* nu_next, const double* dldrho, void* nu_out,
                      double* omega_acc, const Grid& g, double omega, cudaStream_t st) {
  if constexpr (std::is_same<S, double>::value) {
    return adjoint64_m<M>(state_n, nu_next, dldrho, nu_out, omega_acc, g, omega, st);
  } else {
  const int bx = cell_block_x(g.nx);
  const dim3 grid((unsigned)((g.nx + bx - 1) / bx), (unsigned)g.ny, (unsigned)g.nz);
  constexpr int smem = adj_smem_bytes<M, L>();
  const AdjointFn kern = dldrho ? adjoint_kernel<M, true>(g) : adjoint_kernel<M, false>(g);
  {
    // Dynamic shared memory above the 48 KB default needs the opt-in, once per device.
    static std::mutex mu;
    static int done_dev[16] = {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done_dev[dev & 15] != dev) {
      const AdjointFn all[4] = {k_adjoint<M, S, L, true, false>, k_adjoint<M, S, L, false, false>,
                                k_adjoint<M, S, L, true, true>, k_adjoint<M, S, L, false, true>};
      for (int k = 0; k < 4 && e == cudaSuccess; ++k)
        e = cudaFuncSetAttribute(all[k], cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
      done_dev[dev & 15] = dev;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(bx);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (dldrho)
    return cudaLaunchKernelEx(&cfg, kern, static_cast<const S*>(state_n),
                              static_cast<const L*>(nullptr), dldrho, static_cast<L*>(nu_out),
                              omega_acc, g, omega);
  return cudaLaunchKernelEx(&cfg, kern, static_cast<const S*>(state_n),
                            static_cast<const L*>(nu_next), static_cast<const double*>(nullptr),
                            static_cast<L*>(nu_out), omega_acc, g, omega);
  }
}

template <int M>
cudaError_t grad_init_m(const void* nu0, const double* fields, double* d_rho, double* d_U,
                        double* d_T, const Grid& g, cudaStream_t st) {
  // blocks of one warp where the FP64 pipe bounds the kernel (see k_stream_collide64)
  const int bs = std::is_same<L, double>::value ? 32 : 128;
  k_grad_init<M, L><<<(unsigned)((g.ncell + bs - 1) / bs), bs, 0, st>>>(static_cast<const L*>(nu0), fields, d_rho, d_U, d_T, g);
  return cudaGetLastError();
}

cudaError_t adjoint_step(int m, const void* state_n, const void* nu_next, const double* dldrho,
                         void* nu_out, double* omega_acc, const Grid& g, double omega,
                         cudaStream_t st) {
  return m == 0 ? adjoint_m<0>(state_n, nu_next, dldrho, nu_out, omega_acc, g, omega, st)
                : adjoint_m<1>(state_n, nu_next, dldrho, nu_out, omega_acc, g, omega, st);
}
cudaError_t grad_init(int m, const void* nu0, const double* fields, double* d_rho, double* d_U,
                      double* d_T, const Grid& g, cudaStream_t st) {
  return m == 0 ? grad_init_m<0>(nu0, fields, d_rho, d_U, d_T, g, st)
                : grad_init_m<1>(nu0, fields, d_rho, d_U, d_T, g, st);
}
