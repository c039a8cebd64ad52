// Block products with eight interleaved right-hand sides (the block product
// of the multi-right-hand-side solve): every operator of the solver acts on
// the interleaved vectors as M (x) I_8, so one pass over M's stored blocks
// serves all eight columns.
#include "spmv_kernels.cuh"

namespace scr {

// A lane holds CV = 16 bytes of columns and all BR scalar rows: the L = 8 / CV
// lanes of a block load its values together and its BC source rows with one
// 16-byte load each, S such lane sets share a block row.  Per block a lane
// issues 1 + BR BC + BC loads for BR BC CV multiply-adds (3x3, FP32: 13 for
// 36), against 28 for 24 in the scalar-row kernel with eight columns, whose
// source loads bound it (0.27 of HBM on the bifurcation); FP64 is bound by the
// FP64 pipe, whose lanes the S-way sums and the epilogue now fill (the scalar
// rows are dealt to the S sets).
template <int BR, int BC, int S, typename VT, typename XT, Epi E>
__global__ void __launch_bounds__(256) k_spmm(int nbr, const int* __restrict__ rp, const int* __restrict__ col,
                                              const VT* __restrict__ val, const XT* x, Epilogue<XT, E> epi, int pf,
                                              const int* __restrict__ lrow, int nl, int lthr) {
  constexpr int K = kSpmmCols, CV = 16 / (int)sizeof(XT), L = K / CV, G = S * L;
  pdl_allow_next();
  if ((int)blockIdx.x < nl) {
    long_row_cta<BR, BC, K>(__ldg(lrow + blockIdx.x), rp, col, val, x, epi);
    return;
  }
  const long long cta = (long long)blockIdx.x - nl;
  const long long i = (cta * blockDim.x + threadIdx.x) / G;
  const int lane = threadIdx.x % G, set = lane / L, c0 = (lane % L) * CV;
  int s = 0, k = 0;
  if (i < nbr) s = __ldg(rp + i), k = __ldg(rp + i + 1) - s;
  const bool active = i < nbr && k <= lthr;  // the others still join the shuffles
  if (!active) k = 0;
  pdl_wait_prev();
  if (pf > 0 && threadIdx.x == 0) {
    const long long i0 = (cta + pf) * (256 / G), i1 = i0 + 256 / G < nbr ? i0 + 256 / G : nbr;
    if (i0 < nbr) l2_prefetch_blocks<BR * BC>(col, val, __ldg(rp + i0), __ldg(rp + i1));
  }
  const VT* v = val + (long long)s * BR * BC;
  XT acc[BR][CV];
#pragma unroll
  for (int r = 0; r < BR; ++r)
#pragma unroll
    for (int e = 0; e < CV; ++e) acc[r][e] = (XT)0;
#pragma unroll 2
  for (int t = set; t < k; t += S) {
    const XT* xb = x + (long long)__ldg(col + s + t) * BC * K + c0;
    XT xv[BC][CV];
#pragma unroll
    for (int c = 0; c < BC; ++c) load16(xb + c * K, xv[c]);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int c = 0; c < BC; ++c) {
        const XT a = (XT)__ldg(v + (long long)r * k * BC + t * BC + c);
#pragma unroll
        for (int e = 0; e < CV; ++e) acc[r][e] = fma(a, xv[c][e], acc[r][e]);
      }
  }
#pragma unroll
  for (int off = L; off < G; off <<= 1)
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int e = 0; e < CV; ++e) acc[r][e] += __shfl_xor_sync(0xffffffffu, acc[r][e], off, G);
  if (active) {
#pragma unroll
    for (int r = 0; r < BR; ++r) {
      if (r % S != set) continue;
      const long long o = i * BR + r;
      typename Epilogue<XT, E>::Operands op[CV];
#pragma unroll
      for (int e = 0; e < CV; ++e) op[e] = epi.load(o * K + c0 + e, o);
#pragma unroll
      for (int e = 0; e < CV; ++e) epi.store(o * K + c0 + e, acc[r][e], op[e]);
    }
  }
}

template <int BR, int BC, typename VT, typename XT, Epi E>
static void launch_spmm(int G, const DBsr<VT>& M, const XT* x, XT* y, const EpiArgs& e, cudaStream_t s) {
  const Epilogue<XT, E> epi = make_epilogue<XT, E>(x, y, e);
  constexpr int L = kSpmmCols * (int)sizeof(XT) / 16;
  auto go = [&](auto* kern, int S) {
    launch_rows(M, kern, ceil_div((long long)M.nbr * S * L, 256), s, M.nbr, (const int*)M.rp, (const int*)M.col,
                (const VT*)M.val, x, epi, g_l2_prefetch);
  };
  if (G <= 1) go(k_spmm<BR, BC, 1, VT, XT, E>, 1);
  else if (G <= 2) go(k_spmm<BR, BC, 2, VT, XT, E>, 2);
  else if (G <= 4) go(k_spmm<BR, BC, 4, VT, XT, E>, 4);
  else go(k_spmm<BR, BC, 8, VT, XT, E>, 8);
  SCR_LAUNCH();
}

template <int BR, int BC, typename VT, typename XT>
static void launch_spmm_e(int G, const DBsr<VT>& M, const XT* x, XT* y, const EpiArgs& e, cudaStream_t s) {
  switch (e.kind) {
    case Epi::Set: launch_spmm<BR, BC, VT, XT, Epi::Set>(G, M, x, y, e, s); break;
    case Epi::Axpby: launch_spmm<BR, BC, VT, XT, Epi::Axpby>(G, M, x, y, e, s); break;
    case Epi::Resid: launch_spmm<BR, BC, VT, XT, Epi::Resid>(G, M, x, y, e, s); break;
    case Epi::Jacobi: launch_spmm<BR, BC, VT, XT, Epi::Jacobi>(G, M, x, y, e, s); break;
    case Epi::ScaledSub: launch_spmm<BR, BC, VT, XT, Epi::ScaledSub>(G, M, x, y, e, s); break;
    case Epi::ChebFirst:
    case Epi::ChebStep:
    case Epi::ChebZero:
      if constexpr (BR == BC) {
        if (e.kind == Epi::ChebFirst) launch_spmm<BR, BC, VT, XT, Epi::ChebFirst>(G, M, x, y, e, s);
        else if (e.kind == Epi::ChebZero) launch_spmm<BR, BC, VT, XT, Epi::ChebZero>(G, M, x, y, e, s);
        else launch_spmm<BR, BC, VT, XT, Epi::ChebStep>(G, M, x, y, e, s);
      } else {
        throw CudaError{cudaErrorInvalidValue, "Chebyshev epilogue on a non-square block shape"};
      }
      break;
  }
}

template <typename VT, typename XT>
void spmm_launch(int G, const DBsr<VT>& M, const XT* x, XT* y, const EpiArgs& e, cudaStream_t s) {
  const int br = M.br, bc = M.bc;
  // 16-byte source loads: every interleaved vector starts at a multiple of eight entries
  if (reinterpret_cast<uintptr_t>(x) % 16) throw CudaError{cudaErrorInvalidValue, "spmm: source vector not aligned"};
  if (br == 3 && bc == 3) launch_spmm_e<3, 3, VT, XT>(G, M, x, y, e, s);
  else if (br == 3 && bc == 1) launch_spmm_e<3, 1, VT, XT>(G, M, x, y, e, s);
  else if (br == 1 && bc == 3) launch_spmm_e<1, 3, VT, XT>(G, M, x, y, e, s);
  else if (br == 1 && bc == 1) launch_spmm_e<1, 1, VT, XT>(G, M, x, y, e, s);
  else throw CudaError{cudaErrorInvalidValue, "spmm: unsupported block shape"};
}
template void spmm_launch<double, double>(int, const DBsr<double>&, const double*, double*, const EpiArgs&,
                                          cudaStream_t);
template void spmm_launch<float, float>(int, const DBsr<float>&, const float*, float*, const EpiArgs&,
                                        cudaStream_t);
template void spmm_launch<__nv_bfloat16, float>(int, const DBsr<__nv_bfloat16>&, const float*, float*,
                                                const EpiArgs&, cudaStream_t);

}  // namespace scr
