// Kernels around the time step, one instantiation per lattice: population I/O in FP64, the macroscopic
// fields (Eq. (2-4-2) / (2-4-1)) and the FP64 conservation sums. The velocity loops are unrolled, so
// the Q loads of a cell are independent and in flight together. (A first form read the velocities
// from a table with a run-time index, one load after another. rD3Q53 256x256x192 fields FP32 950 -> 497
// us (452 us at the copy bandwidth), FP16 1000 -> 452 us; 128x128x96 FP32 populations in FP64 190 ->
// 173 us (147), into the model 170 -> 152 us (147), conservation sums 111 -> 68 us (49).)
#pragma once

namespace lbm {

// Exact widening FP32 -> FP64 in integer arithmetic: the conversion instruction runs on the FP64 pipe,
// which on GB300 takes 2 values per clock and SM and would alone cost more time than the memory traffic
// of a population read-out. Zeros, subnormals, infinities and NaN take the instruction.
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = __float_as_uint(v), e = b & 0x7F800000u;
  if (e == 0u || e == 0x7F800000u) return double(v);
  const uint32_t hi = (b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20));
  return __hiloint2double(int(hi), int(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

// f-bar_i(x) = A_i(x - e_i): the pre-collision populations from the stored array.
template <class L, class CT, class ST>
__global__ void __launch_bounds__(kBlock) k_gather(const StepParams<CT> p, const ST* __restrict__ A,
                                                   double* __restrict__ out) {
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  const size_t N = size_t(p.ncells);
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    out[size_t(I) * N + cell] =
        widen(Codec<ST>::template dec<CT>(A[size_t(I) * N + nb.template src<I>()], p.wref[I]));
  });
}

// A_i(x - e_i) = f-bar_i(x)
template <class L, class CT, class ST>
__global__ void __launch_bounds__(kBlock) k_scatter(const StepParams<CT> p, const double* __restrict__ in,
                                                    ST* __restrict__ A) {
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  const size_t N = size_t(p.ncells);
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    A[size_t(I) * N + nb.template src<I>()] =
        Codec<ST>::template enc<CT>(CT(in[size_t(I) * N + cell]), p.wref[I]);
  });
}

// sum_i f_i and sum_i e_i f_i
template <class L, class V>
__device__ __forceinline__ void moments01(const V (&f)[L::Q], V& m0, V (&m1)[3]) {
  m0 = f[0];
  m1[0] = m1[1] = m1[2] = V(0);
  static_for<num_pairs<L>()>([&](auto q) {
    constexpr int ip = pair_plus<L>(decltype(q)::value), im = opposite<L>(ip);
    constexpr Vel e = L::e(ip);
    m0 = m0 + (f[ip] + f[im]);
    const V d = f[ip] - f[im];
    if constexpr (e.x != 0) m1[0] = axpy_c<e.x>(d, m1[0]);
    if constexpr (e.y != 0) m1[1] = axpy_c<e.y>(d, m1[1]);
    if constexpr (e.z != 0) m1[2] = axpy_c<e.z>(d, m1[2]);
  });
}

// Eq. (2-4-2): rho = sum f, u = (sum c f + F/2) / rho; Eq. (2-4-1): phi = sum f (+ S_G / 2 for
// the CDE variant), computed in the model's compute dtype from the gathered f-bar.
template <class L, class CT, class ST>
__global__ void __launch_bounds__(kBlock) k_fields(const StepParams<CT> p, const double3 c, int nse,
                                                   const ST* __restrict__ A, double* __restrict__ rho_out,
                                                   double* __restrict__ u_out) {
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  const size_t N = size_t(p.ncells);
  CT f[L::Q], rho, m1[3];
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    f[I] = Codec<ST>::template dec<CT>(A[size_t(I) * N + nb.template src<I>()], p.wref[I]);
  });
  moments01<L>(f, rho, m1);
  if (!nse) {
    if (p.ncde_variant == LBM_NCDE_CDE) {
      static_for<L::D>([&](auto a) {
        constexpr int X = decltype(a)::value;
        rho = fmaf_t(CT(0.5) * p.cde_coef[X], m1[X], rho);
      });
    }
    rho_out[cell] = widen(rho);
    return;
  }
  rho_out[cell] = widen(rho);
  if (u_out == nullptr) return;
  CT F[3] = {CT(0), CT(0), CT(0)};
  body_force(p.force_a, p.force_b, p.force_tab, p.invc, nb.x, nb.y, nb.z, F);
  static_for<L::D>([&](auto a) {
    constexpr int X = decltype(a)::value;
    const CT ca = CT(X == 0 ? c.x : (X == 1 ? c.y : c.z));
    u_out[size_t(X) * N + cell] = widen(ca * (fmaf_t(CT(0.5), F[X], m1[X]) / rho));
  });
}

// NCDE: phi_prev(x) = sum_i f-bar_i(x); for the NSE (S = 0) the same sum is the density
template <class L, class CT, class ST>
__global__ void __launch_bounds__(kBlock) k_phi(const StepParams<CT> p, const ST* __restrict__ A,
                                                CT* __restrict__ phi) {
  const int cell = blockIdx.x * kBlock + threadIdx.x;
  if (cell >= p.ncells) return;
  const Neigh<L> nb(cell, p);
  const size_t N = size_t(p.ncells);
  CT s = CT(0);
  static_for<L::Q>([&](auto i) {
    constexpr int I = decltype(i)::value;
    s += Codec<ST>::template dec<CT>(A[size_t(I) * N + nb.template src<I>()], p.wref[I]);
  });
  phi[cell] = s;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Conservation sums, pass 1: each thread sums whole cells (per-cell sums in the compute dtype,
// cross-cell accumulation in FP64) over a fixed grid-stride; each block reduces in a fixed
// order and writes its four partial sums. Streaming is a permutation, so the stored array has
// the same totals as f-bar and needs no gather.
template <class L, class CT, class ST>
__global__ void __launch_bounds__(256, 4) k_sums_partial(const StepParams<CT> p, const double3 c,
                                                      const ST* __restrict__ A, double* __restrict__ partials) {
  // (a block without cells leaves the FP64 pipe alone, which takes two operations per clock and SM: on 64x48 rD2Q17 the
  // reduction of all blocks was 5 of 16.4 us)
  if (int64_t(blockIdx.x) * blockDim.x >= p.ncells) {
    if (threadIdx.x < 4) partials[size_t(blockIdx.x) * 4 + threadIdx.x] = 0.0;
    return;
  }
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const size_t N = size_t(p.ncells);
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t cell = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; cell < p.ncells; cell += stride) {
    CT f[L::Q], m0, m1[3];
    static_for<L::Q>([&](auto i) {
      constexpr int I = decltype(i)::value;
      f[I] = Codec<ST>::template dec<CT>(A[size_t(I) * N + cell], p.wref[I]);
    });
    moments01<L>(f, m0, m1);
    acc[0] += double(m0);
    for (int a = 0; a < L::D; ++a) acc[1 + a] += double(m1[a]);
  }
  __shared__ double red[4][256 / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int q = 0; q < 4; ++q) {
    const double v = warp_sum(acc[q]);
    if (lane == 0) red[q][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int w = 0; w < int(blockDim.x / 32); ++w) s += red[threadIdx.x][w];
    const double scale = threadIdx.x == 0 ? 1.0 : (threadIdx.x == 1 ? c.x : (threadIdx.x == 2 ? c.y : c.z));
    partials[size_t(blockIdx.x) * 4 + threadIdx.x] = scale * s;
  }
}

// Pass 2: one warp per quantity sums the block partials in a fixed order.
static __global__ void k_sums_final(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s = 0.0;
  for (int b = lane; b < nblocks; b += 32) s += partials[size_t(b) * 4 + q];
  s = warp_sum(s);
  if (lane == 0) out[q] = s;
}

template <class F>
lbm_status dispatch_store(const lbm_model* m, F&& f) {
  switch (m->store) {
    case LBM_F64: return f(double(), double());
    case LBM_F32: return f(float(), float());
    case LBM_BF16_DEV: return f(__nv_bfloat16(), float());
    case LBM_F16_DEV: return f(__half(), float());
  }
  return set_error(LBM_ERR_ARG, "unknown storage dtype");
}

template <int KIND>
lbm_status Launch<KIND>::io(lbm_model* m, const IoCall& io) {
  using L = Lat<KIND>;
  return dispatch_store(m, [&](auto st, auto ct) -> lbm_status {
    using ST = decltype(st);
    using CT = decltype(ct);
    StepParams<CT> p;
    make_step_params(m, &p);
    const int grid = (m->ncells + kBlock - 1) / kBlock;
    ST* A = static_cast<ST*>(m->f[m->cur]);
    const double* c = m->lat->c;
    const double3 cc = make_double3(c[0], c[1], L::D == 3 ? c[2] : 0.0);
    int launches = 1;
    switch (io.what) {
      case IoCall::kGather: k_gather<L, CT, ST><<<grid, kBlock, 0, m->stream>>>(p, A, io.out); break;
      case IoCall::kScatter: k_scatter<L, CT, ST><<<grid, kBlock, 0, m->stream>>>(p, io.in, A); break;
      case IoCall::kFields:
        k_fields<L, CT, ST><<<grid, kBlock, 0, m->stream>>>(p, cc, m->eq == LBM_NSE ? 1 : 0, A, io.out, io.out2);
        break;
      case IoCall::kPhi: k_phi<L, CT, ST><<<grid, kBlock, 0, m->stream>>>(p, A, static_cast<CT*>(io.field)); break;
      case IoCall::kSums:
        k_sums_partial<L, CT, ST><<<kRedBlocks, 256, 0, m->stream>>>(p, cc, A, io.out2);
        k_sums_final<<<1, 128, 0, m->stream>>>(io.out2, kRedBlocks, io.out);
        launches = 2;
        break;
    }
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_error(err, io.name);
    m->launches += launches;
    return LBM_OK;
  });
}

}  // namespace lbm
