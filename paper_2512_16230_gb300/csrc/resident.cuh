// Many steps of a small 2D grid in one launch: the populations stay in the shared memory of one
// thread-block cluster.
//
// A step of a small grid is all latency: a chained launch costs 1.6 to 1.9 us on GB300 whatever the grid
// (rD2Q17 64x48: 1.7 us a step), of which the collision is a fraction. Here the rows of the grid are dealt
// to the CTAs of one cluster (up to 16, one per SM), a step gathers its sources (Eq. (2-2b)) from the
// shared memory of the CTAs that own them (distributed shared memory), collides with the code of
// k_step and writes the other of two buffers; the step ends with a cluster barrier (0.21-0.24 us), and
// global memory is touched at the ends of the call only. A population is contiguous over the CTA's cells, as in
// global memory: consecutive threads read consecutive cells, and a source is at its row's address + its column + the
// velocity times the population's bytes, which the grid fixes at run time. (With a cell's populations contiguous the
// remote loads of a warp split into 32 pieces: rD2Q21 64x48 3.1 us a step against 1.1.)
#pragma once

namespace lbm {

constexpr int kResidentThreads = 512;   // at most, one CTA per SM
constexpr int kResidentSmem = 160 * 1024;  // above what the largest grid taken asks for
constexpr int kResidentCtas = 16;       // CTAs of the cluster, at most (above 8 the size is opt-in)

struct ResidentParams {
  int nsteps;
  int rows;  // grid rows per CTA
};

namespace cluster {
__device__ __forceinline__ uint32_t rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address in the cluster's shared memory of `addr` (shared memory of this CTA) in CTA `r`.
__device__ __forceinline__ uint32_t map(uint32_t addr, uint32_t r) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(r));
  return a;
}
__device__ __forceinline__ void sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <class ST>
__device__ __forceinline__ float load(uint32_t addr) {
  if constexpr (std::is_same<ST, float>::value) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
  } else {
    uint16_t v;
    asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    if constexpr (std::is_same<ST, __half>::value) return __half2float(__ushort_as_half(v));
    else return __uint_as_float(uint32_t(v) << 16);
  }
}
}  // namespace cluster

// Bytes of shared memory of a CTA that owns `rows` rows.
template <class L, class ST>
inline size_t resident_smem(const lbm_model* m, int64_t rows) {
  const size_t cells = size_t(rows * m->n[0]);
  const size_t head = (size_t(m->n[1]) * 4 + 15) / 16 * 16;
  return head + (2 * cells * L::Q * sizeof(ST) + 15) / 16 * 16 + (m->eq == LBM_NCDE ? cells * 4 : 0);
}

template <class L, class ST, int EQ, bool KEEP>
__global__ void __launch_bounds__(kResidentThreads, 1)
    k_steps_resident(const StepParams<float> p, const ResidentParams rp, ST* cur, ST* other, float* phi) {
  constexpr int Q = L::Q, RM = L::RMAX;
  constexpr uint32_t CELL = sizeof(ST);
  constexpr bool DEV = is_deviation_storage<ST>();
  extern __shared__ __align__(16) uint8_t res_smem[];
  chain_release();
  const int nx = p.n[0], ny = p.n[1];
  const uint32_t me = cluster::rank();
  const int y0 = int(me) * rp.rows, own = max(0, min(rp.rows, ny - y0)) * nx, cells = rp.rows * nx;
  uint32_t* row_addr = reinterpret_cast<uint32_t*>(res_smem);  // of every grid row, first buffer
  ST* f0 = reinterpret_cast<ST*>(res_smem + (ny * 4 + 15) / 16 * 16);
  float* s_phi = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(f0) + (2 * cells * Q * int(CELL) + 15) / 16 * 16);
  const uint32_t f0_s = static_cast<uint32_t>(__cvta_generic_to_shared(f0));
  const uint32_t pop_bytes = uint32_t(cells) * CELL, buf_bytes = pop_bytes * Q;
  for (int y = threadIdx.x; y < ny; y += blockDim.x) {
    const int r = y / rp.rows;
    row_addr[y] = cluster::map(f0_s, uint32_t(r)) + uint32_t((y - r * rp.rows) * nx) * CELL;
  }
  chain_wait();
  const size_t N = size_t(p.ncells);
  const size_t g0 = size_t(y0) * nx;
  static_for<Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    for (int c = threadIdx.x; c < own; c += blockDim.x) f0[I * cells + c] = cur[size_t(I) * N + g0 + c];
  });
  if constexpr (EQ == LBM_NCDE) {
    for (int c = threadIdx.x; c < own; c += blockDim.x) s_phi[c] = phi[g0 + c];
  }
  cluster::sync();
  for (int s = 0; s < rp.nsteps; ++s) {
    const uint32_t src = (s & 1) ? buf_bytes : 0u;
    ST* out = f0 + ((s & 1) ? 0 : size_t(cells) * Q);
    for (int c = threadIdx.x; c < own; c += blockDim.x) {
      const int ly = int(__umulhi(unsigned(c), p.div_m[0]) >> p.div_s[0]);
      const int x = c - ly * nx, y = y0 + ly;
      uint32_t ra[2 * RM + 1], xa[2 * RM + 1];
#pragma unroll
      for (int k = -RM; k <= RM; ++k) {
        ra[k + RM] = row_addr[Neigh<L>::wrap1(y - k, k, ny)] + src;
        xa[k + RM] = uint32_t(Neigh<L>::wrap1(x - k, k, nx)) * CELL;
      }
      float f[Q];
      static_for<Q>([&](auto i) {
        constexpr int I = decltype(i)::value;
        constexpr Vel v = L::e(I);
        f[I] = cluster::load<ST>(ra[RM + v.y] + xa[RM + v.x] + I * pop_bytes);
      });
      float F[3];
      const bool forced = body_force(p.force_a, p.force_b, p.force_tab, p.invc, x, y, 0, F);
      float phi_prev = 0.f, phi_now = 0.f;
      if constexpr (EQ == LBM_NCDE) phi_prev = s_phi[c];
      float gr[3];
      const float* grad = nullptr;
      if constexpr (EQ == LBM_NCDE) grad = cell_field_gradient<L>(p, p.n, p.grad_in, int(g0) + c, x, y, 0, gr);
      collide<L, float, EQ, DEV, KEEP>(f, p, p, forced, F, phi_prev, phi_now, grad);
      if constexpr (EQ == LBM_NCDE) s_phi[c] = phi_now;
      static_for<Q>([&](auto i) {
        constexpr int I = decltype(i)::value;
        if constexpr (DEV) out[I * cells + c] = RawCodec<ST>::enc(f[I]);
        else out[I * cells + c] = f[I];
      });
    }
    cluster::sync();
  }
  // both buffers go back to where a launch per step would have left them: an even number of steps ends in `cur`
  const ST* f1 = f0 + size_t(cells) * Q;
  static_for<Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    for (int c = threadIdx.x; c < own; c += blockDim.x) {
      const size_t g = size_t(I) * N + g0 + c;
      cur[g] = f0[I * cells + c];
      other[g] = f1[I * cells + c];
    }
  });
  if constexpr (EQ == LBM_NCDE) {
    for (int c = threadIdx.x; c < own; c += blockDim.x) phi[g0 + c] = s_phi[c];
  }
}

// Whether a call of nsteps steps runs resident, and the cluster's size. Single-speed NSE models with the
// density-gradient term of M2G (a field of the neighbours' last step in global memory) do not.
template <class L, class ST>
bool resident_plan(const lbm_model* m, int64_t nsteps, int* ctas) {
  if (L::D != 2 || m->m2g_aniso || m->gather != LBM_GATHER_AUTO) return false;
  int n = kResidentCtas;
  while (n > 1 && n > m->n[1]) n /= 2;
  const int64_t rows = (m->n[1] + n - 1) / n, cells = rows * m->n[0], pops = cells * L::Q;
  // Per CTA, a cell a thread at most and the populations up to which a step is the faster one. us a step, resident /
  // chained: rD2Q17 32x32 0.74 / 1.60, 64x48 0.98 / 1.71, 80x60 1.27 / 1.76; rD2Q25 64x48 1.30 / 1.91, 80x60 (8000
  // populations) 1.66 / 1.91, 100x76 2.07 / 2.01; with a second cell for some threads rD2Q13 630x16 2.33 / 1.76,
  // rD2Q9 630x16 1.83 / 1.71.
  if (cells > kResidentThreads || pops > 8192) return false;
  // Loading and storing the grid costs a call 4 to 9 us, so that a short one is faster step by step. Steps from which
  // one launch is faster, measured (on NSE and NCDE, FP32 and FP16): 576 populations 4.2 .. 5.5, 1600 5.0 .. 9.3,
  // 3264 8.0 .. 8.7, 5440 11 .. 14, 6500 19 .. 24, 8000 9 .. 32.
  if (nsteps < 4 + pops / 512) return false;
  *ctas = n;
  return resident_smem<L, ST>(m, rows) <= size_t(kResidentSmem);
}

template <class L, class ST, int EQ, bool KEEP>
cudaError_t launch_resident(const lbm_model* m, const StepParams<float>& p, int nsteps, int ctas, float* phi) {
  ResidentParams rp;
  rp.nsteps = nsteps;
  rp.rows = int((m->n[1] + ctas - 1) / ctas);
  const size_t smem = resident_smem<L, ST>(m, rp.rows);
  auto kernel = k_steps_resident<L, ST, EQ, KEEP>;
  // (one limit for every grid: a thread that launches another grid must not lower it in between)
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem);
  if (err == cudaSuccess && ctas > 8)
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (err != cudaSuccess) return err;
  const int cells = int(rp.rows * m->n[0]);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(ctas));
  cfg.blockDim = dim3(unsigned(std::min(kResidentThreads, (cells + 31) / 32 * 32)));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = m->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(ctas);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, p, rp, static_cast<ST*>(m->f[m->cur]), static_cast<ST*>(m->f[m->cur ^ 1]), phi);
}

}  // namespace lbm
