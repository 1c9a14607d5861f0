// Diagnostic kernels and host launchers of the batched stiff-chemistry integrator
// (sm_103a); the device code shared with chem_kernels_w.cu is in chem_device.cuh.
// This translation unit instantiates the integration kernel with the RODAS4 stepper.

#include "chem_device.cuh"

namespace chem {

size_t smem_bytes(int Kmax, int Imax, int prec, bool m0_global, bool x_tab) {
  return make_layout(Kmax, Imax, prec, m0_global, x_tab).total;
}

int64_t matrix_slot_entries(int Kmax) { return (int64_t)slot_entries(Kmax); }

// W-method instantiations (chem_kernels_w.cu)
cudaError_t launch_integrate_w(const IntegrateArgs& a, int block, int prec, int grid, cudaStream_t st);

struct DiagArgs {
  DevMech m;
  int64_t n;
  const double *T, *p, *Y;
  double* out;
  double dt, rtol, atol;
  int what;    // 0 rhs, 1 jacobian, 2 h0
  int jac_fd;  // FP64 form: forward-difference Jacobian for what = 1
  int q;       // starting-step exponent 1/q (the method's embedded order + 1)
};

template <int NW, int PREC>
__global__ void __launch_bounds__(NW * 32) k_diag(const __grid_constant__ DiagArgs a) {
  using A = typename Policy<PREC>::ASM;
  const Layout L = make_layout(a.m.K, a.m.I, PREC, false, true);
  Cta<NW> c;
  c.bind(L);

  constexpr int NT = NW * 32;
  const int K = a.m.K, n = K + 1, ld = odd_ld(n);
#pragma unroll 1
  for (int64_t cell = blockIdx.x; cell < a.n; cell += gridDim.x) {
    if (c.tid == 0) c.y()[0] = a.T[cell];
#pragma unroll 1
    for (int k = c.tid; k < K; k += NT) c.y()[1 + k] = a.Y[(size_t)cell * K + k];
    const double p = a.p[cell];
    c.set_cell(a.m, p);
    c.set_matrix(K, nullptr);
    __syncthreads();
    if (a.what == 0) {
      eval_rhs<NW, false, Policy<PREC>::IR>(a.m, c, c.y(), p, c.f0());
#pragma unroll 1
      for (int i = c.tid; i < n; i += NT) a.out[(size_t)cell * n + i] = c.f0()[i];
    } else if (a.what == 1) {
      if (PREC == PREC_FP64 && a.jac_fd) {
        eval_rhs<NW, false, false>(a.m, c, c.y(), p, c.f0());
        fd_matrix<NW, true>(a.m, c, p, c.y(), c.f0(), 0.0);
      } else {
        const Scal s = eval_rhs<NW, true, Policy<PREC>::IR>(a.m, c, c.y(), p, c.f0());
        build_matrix<NW, PREC, true>(a.m, c, s, c.f0(), 0.0);
      }
      // (the mixed forms hold it by columns)
      const A* J = reinterpret_cast<const A*>(Policy<PREC>::IR ? c.M0 : c.M());
      const int si = Policy<PREC>::IR ? 1 : ld, sj = Policy<PREC>::IR ? ld : 1;
#pragma unroll 1
      for (int i = c.warp; i < n; i += NW)
#pragma unroll 1
        for (int j = c.lane; j < n; j += 32) a.out[(size_t)cell * n * n + i * n + j] = to_double(J[i * si + j * sj]);
    } else {
      eval_rhs<NW, false, Policy<PREC>::IR>(a.m, c, c.y(), p, c.f0());
      const double h = starting_step<NW, Policy<PREC>::IR>(a.m, c, p, a.dt, a.rtol, a.atol, a.q);
      if (c.tid == 0) a.out[cell] = h;
    }
    __syncthreads();
  }
}

// The rate kernels' elementary functions, elementwise (diagnostic): op 0 exp, 1 log,
// 2 1/x; 3 and 4 the hi and lo parts of the float-float split (widened exactly).
__global__ void k_math(int op, const double* x, double* y, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (op >= 3) {
      const ff2 s = ff_split(x[i]);
      y[i] = f32_to_f64(op == 3 ? s.hi : s.lo);
    } else {
      y[i] = op == 0 ? xexp(x[i]) : op == 1 ? xlog(x[i]) : xrcp(x[i]);
    }
  }
}

struct LuArgs {
  int64_t n_mat;
  int dim;
  const double *A, *b;
  double* x;
  int* info;
  int ir;
};

// Batched solves: a CTA takes a matrix from its load to the solution, bound by the chain of
// its n dependent pivots, so what counts is how many matrices an SM holds and that nothing
// else adds to the chain. A warp that waited for one row's loads at a time took 28 memory
// latencies for n = 55; with eight loads in flight per thread a matrix takes three. The
// layout leaves out the species arrays and registers are limited to five CTAs of 128 threads
// (four before) or sixteen of 64 (n <= 32, which needs half of them); beyond n = 64 the
// inverse stays in the registers of 256 threads instead of the shared memory of 128.
// Mixed form: 8,192 of n = 55 712 -> 501 us, 65,536 of n = 16 1398 -> 490 us, 592 of
// n = 101 3434 -> 311 us; FP64 form: 3,970 of n = 55 1619 -> 1535 us, 296 of n = 128 1737 ->
// 1133 us, 100 of n = 55 158 -> 123 us. (Of these 3 % at most are what the test of the
// pivots' range and the rounding of the entries cost.)
template <int NW, int PREC>
__global__ void __launch_bounds__(NW * 32, NW == 2 ? 16 : NW == 4 ? 5 : 2) k_lu_solve(const __grid_constant__ LuArgs a) {
  using P = Policy<PREC>;
  using R = typename P::LU;
  const Layout L = make_layout(a.dim - 1, 1, PREC, false, false, 0);
  Cta<NW> c;
  c.bind(L);
  constexpr int NT = NW * 32, B = 8;  // B loads in flight per thread
  const int n = a.dim, nn = n * n, ld = odd_ld(n);
  const unsigned rn = 0xffffffffu / (unsigned)n + 1u;  // e / n = umulhi(e, rn) for e < 2^16 (n = 1: 0)
  R* M = reinterpret_cast<R*>(c.M());
#pragma unroll 1
  for (int64_t s = blockIdx.x; s < a.n_mat; s += gridDim.x) {
    const double* As = a.A + (size_t)s * nn;
#pragma unroll 1
    for (int e0 = c.tid; e0 < nn; e0 += B * NT) {
      double v[B];
#pragma unroll
      for (int u = 0; u < B; ++u) v[u] = e0 + u * NT < nn ? As[e0 + u * NT] : 0.0;
#pragma unroll
      for (int u = 0; u < B; ++u) {
        const int e = e0 + u * NT, i = (int)__umulhi((unsigned)e, rn), j = e - i * n;
        if (e >= nn) break;
        if constexpr (P::IR) reinterpret_cast<typename P::ASM*>(c.M0)[j * ld + i] = from_double<typename P::ASM>(v[u]);
        else M[i * ld + j] = v[u];
      }
    }
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) c.fv()[i] = a.b[(size_t)s * n + i];
    __syncthreads();
    const int info = factor<NW, PREC, NW == 2 ? 32 : 128>(c, n);
    if (info == 0) solve<NW, PREC>(c, n, c.fv(), c.u(), a.ir);
#pragma unroll 1
    for (int i = c.tid; i < n; i += NT) a.x[(size_t)s * n + i] = info == 0 ? c.u()[i] : NAN;
    if (c.tid == 0 && a.info) a.info[s] = info;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
template <int NW, int PREC>
static cudaError_t launch_integrate_t(const IntegrateArgs& a, int grid, cudaStream_t st) {
  return launch_integrate_m<NW, PREC, METHOD_RODAS4>(a, grid, st);
}

cudaError_t launch_integrate(const IntegrateArgs& a, int block, int prec, int grid, cudaStream_t st) {
  if (a.tab.s == 4) return launch_integrate_w(a, block, prec, grid, st);
#define LI(P)                                                                       \
  do {                                                                              \
    if (block == 64) return launch_integrate_t<2, P>(a, grid, st);                  \
    if (block == 256) return launch_integrate_t<8, P>(a, grid, st);                 \
    return launch_integrate_t<4, P>(a, grid, st);                                   \
  } while (0)
  if (prec == PREC_FP64) LI(PREC_FP64);
  if (prec == PREC_MIXED) LI(PREC_MIXED);
  LI(PREC_FP32ASM);
#undef LI
}

cudaError_t occupancy_integrate(int block, int prec, int K, int I, int* ctas_per_sm, bool m0_global) {
  const size_t smem = smem_bytes(K, I, prec, m0_global);
  cudaError_t e;
#define OCC(NW, P)                                                                                    \
  do {                                                                                                \
    e = prep(k_integrate<NW, P, METHOD_RODAS4>, smem);                                                \
    if (e != cudaSuccess) return e;                                                                   \
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k_integrate<NW, P, METHOD_RODAS4>, \
                                                         NW * 32, smem);                              \
  } while (0)
#define OCCP(P)                  \
  do {                           \
    if (block == 64) OCC(2, P);  \
    if (block == 256) OCC(8, P); \
    OCC(4, P);                   \
  } while (0)
  if (prec == PREC_FP64) OCCP(PREC_FP64);
  if (prec == PREC_MIXED) OCCP(PREC_MIXED);
  OCCP(PREC_FP32ASM);
#undef OCCP
#undef OCC
}

template <int PREC, class ArgT, class KernelT>
static cudaError_t launch_simple(KernelT k, const ArgT& a, size_t smem, int grid, cudaStream_t st, int block = 128) {
  cudaError_t e = prep(k, smem);
  if (e != cudaSuccess) return e;
  k<<<grid, block, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_diag(const DevMech& m, int64_t n, const double* T, const double* p, const double* Y,
                        double* out, double dt, double rtol, double atol, int what, int prec,
                        cudaStream_t st, int jac_fd, int q) {
  DiagArgs a;
  a.jac_fd = jac_fd;
  a.q = q;
  a.m = m;
  a.n = n;
  a.T = T;
  a.p = p;
  a.Y = Y;
  a.out = out;
  a.dt = dt;
  a.rtol = rtol;
  a.atol = atol;
  a.what = what;
  const size_t smem = smem_bytes(m.K, m.I, prec);
  const int grid = (int)(n < 65535 ? n : 65535);
  if (prec == PREC_FP64) return launch_simple<PREC_FP64>(k_diag<4, PREC_FP64>, a, smem, grid, st);
  if (prec == PREC_MIXED) return launch_simple<PREC_MIXED>(k_diag<4, PREC_MIXED>, a, smem, grid, st);
  return launch_simple<PREC_FP32ASM>(k_diag<4, PREC_FP32ASM>, a, smem, grid, st);
}

cudaError_t launch_math(int op, const double* x, double* y, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  k_math<<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(op, x, y, n);
  return cudaGetLastError();
}

// Threads per matrix: the register inverse takes 64 threads up to n = 32, 128 up to 64 and
// 256 up to 128. The FP64 LU is quicker with more threads while the SMs are not full.
// (FP64, us with 64 / 128 / 256 threads: 100 matrices of n = 32 86 / 62 / 55, 11,722 of them
// 1335 / 1385 / 1502; 100 of n = 55 236 / 152 / 123, 3,970 of them 1516 / 1535 / 1609; 296 of
// n = 128 - / 1682 / 1129. Mixed: 100 of n = 55 35 / 28 / 30, 3,970 of them 283 / 277 / 440.)
// At 86 us a matrix and 0.114 us a matrix for the full GPU, 64 threads reach that rate with
// some 750 matrices in flight, five per SM.
static int lu_block(int64_t n_mat, int dim, int prec) {
  const int block = dim <= 32 ? 64 : dim <= 64 ? 128 : 256;
  int dev = 0, sms = 0;
  if (prec != PREC_FP64 || block == 256 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return block;
  return n_mat <= 4 * (int64_t)sms ? 2 * block : block;
}

cudaError_t launch_lu_solve(int64_t n_mat, int dim, const double* A, const double* b, double* x,
                            int* info, int prec, int ir, cudaStream_t st) {
  LuArgs a;
  a.n_mat = n_mat;
  a.dim = dim;
  a.A = A;
  a.b = b;
  a.x = x;
  a.info = info;
  a.ir = ir;
  const size_t smem = make_layout(dim - 1, 1, prec, false, false, 0).total;
  const int grid = (int)(n_mat < 65535 ? n_mat : 65535);
  const int block = lu_block(n_mat, dim, prec);
#define LU(P)                                                                               \
  do {                                                                                      \
    if (block == 64) return launch_simple<P>(k_lu_solve<2, P>, a, smem, grid, st, block);   \
    if (block == 256) return launch_simple<P>(k_lu_solve<8, P>, a, smem, grid, st, block);  \
    return launch_simple<P>(k_lu_solve<4, P>, a, smem, grid, st, block);                    \
  } while (0)
  if (prec == PREC_FP64) LU(PREC_FP64);
  if (prec == PREC_MIXED) LU(PREC_MIXED);
  LU(PREC_FP32ASM);
#undef LU
}

}  // namespace chem
