// Fused epilogues of the block products: what a product kernel does with
// the row sum acc of M x for scalar output row o (flat index gi = o * nrhs
// + h for right-hand side h).  Shared by the product kernels.
#pragma once
#include "kernels.h"

namespace scr {

template <typename XT, Epi E>
struct Epilogue {
  XT* y;
  const XT* z;
  const XT* xs;
  const XT* dinv;
  const XT* xin;  // the product's source vector (ChebStep: the direction)
  XT* r;
  XT* dout;
  XT* xsol;
  XT alpha, beta;
  // what the epilogue reads at (gi, o).  A product kernel loads it before its
  // sums are done, so that these reads are in flight with the product's own
  // instead of starting after the last multiply-add (gi is read and written
  // by its owner only, so the early read sees what a late one would)
  struct Operands {
    XT p, q, t, d;
  };
  __device__ __forceinline__ Operands load(long long gi, long long o) const {
    Operands v{(XT)0, (XT)0, (XT)0, (XT)0};
    if constexpr (E == Epi::Axpby) {
      if (z) v.p = z[gi];
    } else if constexpr (E == Epi::Resid) {
      v.p = z[gi];
    } else if constexpr (E == Epi::Jacobi || E == Epi::ChebFirst) {
      v.p = z[gi], v.q = xs[gi], v.d = dinv[o];
    } else if constexpr (E == Epi::ScaledSub) {
      v.p = z[gi], v.d = dinv[o];
    } else if constexpr (E == Epi::ChebStep) {
      v.p = r[gi], v.q = xin[gi], v.t = xsol[gi], v.d = dinv[o];
    } else if constexpr (E == Epi::ChebZero) {
      v.d = dinv[o];
    }
    return v;
  }
  template <typename AT>
  __device__ __forceinline__ void store(long long gi, AT acc, const Operands& v) const {
    if constexpr (E == Epi::Set) {
      y[gi] = (XT)acc;
    } else if constexpr (E == Epi::Axpby) {
      XT w = alpha * (XT)acc;
      if (z) w += beta * v.p;
      y[gi] = w;
    } else if constexpr (E == Epi::Resid) {
      y[gi] = v.p - (XT)acc;
    } else if constexpr (E == Epi::Jacobi) {
      y[gi] = v.q + (v.p - (XT)acc) * v.d;
    } else if constexpr (E == Epi::ScaledSub) {
      y[gi] = v.p - (XT)acc * v.d;
    } else if constexpr (E == Epi::ChebFirst) {
      const XT ri = (v.p - (XT)acc) * v.d;
      const XT di = alpha * ri;
      r[gi] = ri;
      dout[gi] = di;
      y[gi] = v.q + di;
    } else if constexpr (E == Epi::ChebZero) {
      const XT ri = (XT)acc * v.d;
      const XT di = ri * alpha;
      y[gi] = (XT)acc;
      r[gi] = ri;
      dout[gi] = di;
      xsol[gi] = di;
    } else {
      const XT ri = v.p - (XT)acc * v.d;
      const XT di = alpha * v.q + beta * ri;
      r[gi] = ri;
      dout[gi] = di;
      xsol[gi] = v.t + di;
    }
  }
  template <typename AT>
  __device__ __forceinline__ void operator()(long long gi, long long o, AT acc) const {
    store(gi, acc, load(gi, o));
  }
};

template <typename XT, Epi E>
Epilogue<XT, E> make_epilogue(const XT* x, XT* y, const EpiArgs& e) {
  Epilogue<XT, E> epi;
  epi.y = y;
  epi.z = static_cast<const XT*>(e.z);
  epi.xs = static_cast<const XT*>(e.xs);
  epi.dinv = static_cast<const XT*>(e.dinv);
  epi.xin = x;
  epi.r = static_cast<XT*>(e.r);
  epi.dout = static_cast<XT*>(e.dout);
  epi.xsol = static_cast<XT*>(e.xsol);
  epi.alpha = (XT)e.alpha;
  epi.beta = (XT)e.beta;
  return epi;
}

}  // namespace scr
