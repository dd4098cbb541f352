// The Wilson Dslash hopping term with its spin structure: the operator whose
// port to GPUs the paper names as its next step (Sec. 6, Summary and Outlook),
// beyond the site-local expression engine.
//
//   out(x) = sum_mu [ (1 - gamma_mu) U_mu(x) psi(x+mu)
//                   + (1 + gamma_mu) U_mu(x-mu)^dagger psi(x-mu) ]
//
// psi and out are spinor fields, stored as colour-vector fields with four
// objects per site (object s = spin component s), U the four links of every
// site.  Euclidean gamma matrices in the chiral basis,
//   gamma_mu = [[0, s_mu], [s_mu^dagger, 0]] in 2x2 spin blocks,
//   s_x = [[0, i], [i, 0]], s_y = [[0, -1], [1, 0]], s_z = [[i, 0], [0, -i]],
//   s_t = 1, so gamma_5 = diag(1, 1, -1, -1).
// (1 + sg gamma_mu) has rank 2: with psi = (u; l) in upper and lower spin
// pairs, (1 + sg gamma_mu) psi = (h; sg s_mu^dagger h) with the half spinor
// h = u + sg s_mu l.  The colour matrix acts on each spin component, so each
// of the 8 terms multiplies only the two components of h by the link (2
// matrix-vector products instead of 4) and rebuilds the lower pair from the
// product.  Every s_mu has one entry per row, a phase in {1, i, -1, -i}, so
// the projection and the rebuild are sums with swapped and negated parts.
//
// Algorithmic traffic per site (FP64, every input read once): the 4 links
// (576 B), the spinor (192 B) and the output (192 B), 960 B; 1320 flops
// (per term: 12 for the projection, 2 x 66 for the products, 24 to
// accumulate; the first term's accumulation is a copy).
#include <cuda_runtime.h>

#include <type_traits>

#include "dev_stencil.cuh"
#include "internal.h"

namespace su3s {

// Multiplication by a phase P = i^ph, ph uniform across the warp, without
// branches: P (xr + i xi) = (sr a, si b) with (a, b) = (xr, xi) or (xi, xr)
// (odd ph), sr = -1 for ph = 1, 2 and si = -1 for ph = 2, 3.  Negation is exact
// in every arithmetic, so the result is the phase times the value exactly.
struct Phase {
  bool swap, neg_re, neg_im;
  __device__ __forceinline__ explicit Phase(int ph)
      : swap((ph & 1) != 0), neg_re(ph == 1 || ph == 2), neg_im(ph >= 2) {}
};

template <class M>
__device__ __forceinline__ typename M::A neg_acc(const typename M::A& a) {
  if constexpr (std::is_same<typename M::A, FAcc>::value) return FAcc{-a.hh, -a.cr, a.e};
  else return -a;
}

// h = u + P l for one spin component pair (colour vectors of reals).
template <class M>
__device__ __forceinline__ void half_spinor(typename M::R* h, const typename M::R* u,
                                            const typename M::R* l, Phase P) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const typename M::R a = P.swap ? l[2 * c + 1] : l[2 * c];
    const typename M::R b = P.swap ? l[2 * c] : l[2 * c + 1];
    typename M::A re, im;
    M::template add<true, 1>(re, u[2 * c]);
    M::template add<true, 1>(im, u[2 * c + 1]);
    M::template add<false, 1>(re, P.neg_re ? M::neg(a) : a);
    M::template add<false, 1>(im, P.neg_im ? M::neg(b) : b);
    h[2 * c] = M::finish(re);
    h[2 * c + 1] = M::finish(im);
  }
}

// out += P chi for a colour vector of accumulators.
template <class M>
__device__ __forceinline__ void add_rebuilt(typename M::A* out, const typename M::A* chi, Phase P) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const typename M::A a = P.swap ? chi[2 * c + 1] : chi[2 * c];
    const typename M::A b = P.swap ? chi[2 * c] : chi[2 * c + 1];
    M::template combine<1>(out[2 * c], P.neg_re ? neg_acc<M>(a) : a);
    M::template combine<1>(out[2 * c + 1], P.neg_im ? neg_acc<M>(b) : b);
  }
}

template <class M>
__device__ __noinline__ void dslash_site_f64(const FieldDesc& dst, const FieldDesc& U,
                                             const FieldDesc& psi, const LatGeo& g, int64_t s);

// The eight terms at site s, then the store (or, for a site whose inputs are
// outside the FP64-accurate arithmetics' range, native FP64 instead).  The
// terms run in a rolled loop: unrolled, the eight bodies (~10,000 instructions
// per site in the pair arithmetic) overflowed the instruction cache and
// instruction fetch was the leading stall.  Direction and sense are uniform
// across the warp, so the phase and column choices are uniform branches; the
// backward link's adjoint is taken in its load.
template <class M>
__device__ __forceinline__ void dslash_site(const FieldDesc& dst, const FieldDesc& U,
                                            const FieldDesc& psi, const LatGeo& g, int64_t s) {
  typename M::A out[4][6];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int r = 0; r < 6; ++r) out[k][r] = M::zero();
  uint32_t gm = 0;
#pragma unroll 1
  for (int t = 0; t < 8; ++t) {
    const int mu = t >> 1;
    const bool bwd = (t & 1) != 0;          // sense: SG = +1 backward, -1 forward
    const int64_t n = shift_site_rt(g, s, mu, bwd ? -1 : 1);
    // s_mu: row k has its entry in column k ^ sw with phase code ph_k
    const bool sw = mu < 2;
    const int ph0 = mu == 0 ? 1 : mu == 1 ? 2 : mu == 2 ? 1 : 0;
    const int ph1 = mu == 0 ? 1 : mu == 1 ? 0 : mu == 2 ? 3 : 0;
    const int sg = bwd ? 0 : 2;             // phase code of SG
    typename M::R h[2][6];
    {
      typename M::R sp[4][6];
#pragma unroll
      for (int k = 0; k < 4; ++k) load_nc<M, 6>(psi, n, k, sp[k], gm);
      if (sw) {
        half_spinor<M>(h[0], sp[0], sp[3], Phase((ph0 + sg) & 3));
        half_spinor<M>(h[1], sp[1], sp[2], Phase((ph1 + sg) & 3));
      } else {
        half_spinor<M>(h[0], sp[0], sp[2], Phase((ph0 + sg) & 3));
        half_spinor<M>(h[1], sp[1], sp[3], Phase((ph1 + sg) & 3));
      }
    }
    if constexpr (M::kScaled) {
      // fixed point: the half spinor's components share one exponent
      typename M::A a[12];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int r = 0; r < 6; ++r) a[6 * k + r] = M::to_acc(h[k][r]);
      M::template finish_obj<12>(&h[0][0], a);
    }
    typename M::R u[18];
    load_link<M>(U, bwd ? n : s, mu, bwd, u, gm);
    // upper spin k += U h_k; lower spin (k ^ sw) += SG conj(P_k) U h_k
    const Phase q0((((4 - ph0) & 3) + sg) & 3), q1((((4 - ph1) & 3) + sg) & 3), one(0);
    {
      typename M::A chi[6];
      mv_acc<M, true, 1, false>(chi, u, h[0]);
      add_rebuilt<M>(out[0], chi, one);
      if (sw) add_rebuilt<M>(out[3], chi, q0);
      else add_rebuilt<M>(out[2], chi, q0);
    }
    {
      typename M::A chi[6];
      mv_acc<M, true, 1, false>(chi, u, h[1]);
      add_rebuilt<M>(out[1], chi, one);
      if (sw) add_rebuilt<M>(out[2], chi, q1);
      else add_rebuilt<M>(out[3], chi, q1);
    }
  }
  if constexpr (M::kGuard) {
    if (gm >= guard_hi(2)) {
      dslash_site_f64<MathF64>(dst, U, psi, g, s);
      return;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const typename M::A(*o)[6] = reinterpret_cast<const typename M::A(*)[6]>(out[k]);
    store_obj<KV, P_F64, M, 1, 6>(dst, s, k, o);
  }
}

template <class M>
__device__ __noinline__ void dslash_site_f64(const FieldDesc& dst, const FieldDesc& U,
                                             const FieldDesc& psi, const LatGeo& g, int64_t s) {
  dslash_site<M>(dst, U, psi, g, s);
}

// ------------------------------------------------ staged (asynchronous) loads
// Each thread stages the operands of its next term (the neighbour spinor's 12
// complex components and the link's 9) in its own slots of shared memory with
// asynchronous copies (cp.async) while it computes the current term, so the
// loads' latency is hidden behind a term's arithmetic without holding the
// next operands in registers.  Slots are [element][thread], 16 bytes each.
constexpr int kDslashElems = 21;
constexpr int kDslashThreads = 128;

// Issue the copies of term t (direction t >> 1, backward if t is odd) of site s.
__device__ __forceinline__ void stage_term(uint4* slot, int nt, const FieldDesc& U,
                                           const FieldDesc& psi, const LatGeo& g, int64_t s, int t) {
  const int mu = t >> 1;
  const bool bwd = (t & 1) != 0;
  const int64_t n = shift_site_rt(g, s, mu, bwd ? -1 : 1);
  const uint4* pp = reinterpret_cast<const uint4*>(psi.ptr);
  const uint4* pu = reinterpret_cast<const uint4*>(U.ptr);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t b = elem_base(psi, n, k);
#pragma unroll
    for (int c = 0; c < 3; ++c) cp_async16(slot + (3 * k + c) * nt, pp + b + c * psi.s_c);
  }
  const int64_t bu = elem_base(U, bwd ? n : s, mu);
#pragma unroll
  for (int e = 0; e < 9; ++e) cp_async16(slot + (12 + e) * nt, pu + bu + e * U.s_c);
  cp_async_commit();
}

template <class M, int W>
__device__ __forceinline__ void read_staged(const uint4* slot, int nt, int first, typename M::R* out,
                                            uint32_t& gm) {
#pragma unroll
  for (int c = 0; c < W / 2; ++c) {
    const uint4 v = slot[(first + c) * nt];
    if constexpr (M::kGuard) gm = guard_max(gm, v.y, v.w);
    split_complex<M>(v, out[2 * c], out[2 * c + 1]);
  }
  M::template normalize_obj<W>(out);
}

// The link of the term from its slots, its adjoint for the backward term
// (element (i, j) read from (j, i), imaginary part negated).
template <class M>
__device__ __forceinline__ void read_staged_link(const uint4* slot, int nt, bool dag,
                                                 typename M::R* out, uint32_t& gm) {
  if (dag) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const uint4 v = slot[(12 + 3 * j + i) * nt];
        if constexpr (M::kGuard) gm = guard_max(gm, v.y, v.w);
        split_complex<M>(make_uint4(v.x, v.y, v.z, v.w ^ 0x80000000u), out[2 * (3 * i + j)],
                         out[2 * (3 * i + j) + 1]);
      }
    M::template normalize_obj<18>(out);
  } else {
    read_staged<M, 18>(slot, nt, 12, out, gm);
  }
}

// The Wilson term at the thread's sites s, s + stride, ...: each term's
// operands were staged during the previous term (the first site's first term
// before the loop), and the next term's copies are issued as soon as this
// term's slots have been read into registers.
template <class M>
__device__ __forceinline__ void dslash_staged(const FieldDesc& dst, const FieldDesc& U,
                                              const FieldDesc& psi, const LatGeo& g, int64_t s,
                                              int64_t stride, uint4* slot, int nt) {
  if (s < g.V) stage_term(slot, nt, U, psi, g, s, 0);
  while (s < g.V) {
    typename M::A out[4][6];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int r = 0; r < 6; ++r) out[k][r] = M::zero();
    uint32_t gm = 0;
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
      const int mu = t >> 1;
      const bool bwd = (t & 1) != 0;
      const bool sw = mu < 2;
      const int ph0 = mu == 0 ? 1 : mu == 1 ? 2 : mu == 2 ? 1 : 0;
      const int ph1 = mu == 0 ? 1 : mu == 1 ? 0 : mu == 2 ? 3 : 0;
      const int sg = bwd ? 0 : 2;
      cp_async_wait_all();
      typename M::R h[2][6];
      {
        typename M::R sp[4][6];
#pragma unroll
        for (int k = 0; k < 4; ++k) read_staged<M, 6>(slot, nt, 3 * k, sp[k], gm);
        if (sw) {
          half_spinor<M>(h[0], sp[0], sp[3], Phase((ph0 + sg) & 3));
          half_spinor<M>(h[1], sp[1], sp[2], Phase((ph1 + sg) & 3));
        } else {
          half_spinor<M>(h[0], sp[0], sp[2], Phase((ph0 + sg) & 3));
          half_spinor<M>(h[1], sp[1], sp[3], Phase((ph1 + sg) & 3));
        }
      }
      if constexpr (M::kScaled) {
        typename M::A a[12];
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int r = 0; r < 6; ++r) a[6 * k + r] = M::to_acc(h[k][r]);
        M::template finish_obj<12>(&h[0][0], a);
      }
      typename M::R u[18];
      read_staged_link<M>(slot, nt, bwd, u, gm);
      // this term's slots are in registers: stage the next term
      if (t < 7) stage_term(slot, nt, U, psi, g, s, t + 1);
      else if (s + stride < g.V) stage_term(slot, nt, U, psi, g, s + stride, 0);
      const Phase q0((((4 - ph0) & 3) + sg) & 3), q1((((4 - ph1) & 3) + sg) & 3), one(0);
      {
        typename M::A chi[6];
        mv_acc<M, true, 1, false>(chi, u, h[0]);
        add_rebuilt<M>(out[0], chi, one);
        if (sw) add_rebuilt<M>(out[3], chi, q0);
        else add_rebuilt<M>(out[2], chi, q0);
      }
      {
        typename M::A chi[6];
        mv_acc<M, true, 1, false>(chi, u, h[1]);
        add_rebuilt<M>(out[1], chi, one);
        if (sw) add_rebuilt<M>(out[2], chi, q1);
        else add_rebuilt<M>(out[3], chi, q1);
      }
    }
    if (M::kGuard && gm >= guard_hi(2)) {
      dslash_site_f64<MathF64>(dst, U, psi, g, s);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const typename M::A(*o)[6] = reinterpret_cast<const typename M::A(*)[6]>(out[k]);
        store_obj<KV, P_F64, M, 1, 6>(dst, s, k, o);
      }
    }
    s += stride;
  }
  cp_async_wait_all();
}

// Native FP64 and fixed point: one thread per site, each with 21 staging slots.
template <class M>
__global__ void __launch_bounds__(kDslashThreads) k_dslash(FieldDesc dst, FieldDesc U, FieldDesc psi, LatGeo g) {
  extern __shared__ __align__(16) uint4 d_slots[];
  dslash_staged<M>(dst, U, psi, g, (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                   (int64_t)gridDim.x * blockDim.x, d_slots + threadIdx.x, (int)blockDim.x);
}

// ------------------------------------- pair arithmetic: both spins of h per lane pair
// The pair arithmetic has a kernel of its own, bound by instruction issue and
// the FMA pipe (62% busy, issue 62%), not by memory.  It packs every FP32
// operation over the two components k = 0, 1 of the half spinor (the two lanes
// of f32x2): both are multiplied by the same link element, so the link's reals
// are duplicated and nothing else is swapped or negated (packing (re, im) of
// one output instead needs swapped copies of h and signed copies of the link).
//   - Phases ride along as +-1 factors of packed FMAs.  Directions go in the
//     order x, y, t, z; s_mu has the entries i f_k (x, z) or f_k (y, t), so
//     h_k = u_k + f_k (i) l, where the factor i only exchanges the addresses of
//     l's real and imaginary parts, and the lower accumulators hold the lower
//     spins (times i for x, z) in the lane order of the direction's columns;
//     they are turned where that changes, three times per site.
//   - The projections are formed in FP64 (one DFMA per real on a pipe that is
//     idle otherwise): only the 12 reals of h are split into pairs, not the 24
//     of the spinor, and h enters rounded to nearest.
//   - Operands come one colour at a time (two spins of u, two of l, three link
//     elements).  The next colour is read and split, work of the ALU pipe,
//     between the products of the current one, work of the FMA pipe; each
//     colour's slots are refilled for the next term as soon as they are read.
// Measured at 32^3 x 64 (pair arithmetic, default launch): 1,031 us before (one
// (re, im) pair per lane pair, 242 registers, 10,870 instructions per site),
// 884 us with the spins packed, 787 with the colours pipelined (8,580
// instructions), 755 with four waves of blocks, 740 with walked addresses, 728
// with the six terms of a colour side by side (dp_fma_shared).
// Not kept: tiles of sites in 2, 3 or 4 dimensions per block with and without
// L1 (863-880 against 873 us), 128 registers (815), the first term opening the
// accumulators (761 against 755).

// a += f * b lane-wise (MathDF::combine with a sign per lane: f = +-1, so every
// product is exact)
__device__ __forceinline__ void dp_combine_sign(dpa& a, const dpa& b, float2 f) {
  const float2 s = f2_fma(b.S, f, a.S);
  const float2 nbp = f2_sub(a.S, s);
  const float2 ap = f2_add(s, nbp);
  const float2 db = f2_fma(b.S, f, nbp);
  const float2 da = f2_sub(a.S, ap);
  float2 t = f2_add(da, db);
  t = f2_fma(b.lo, f, t);
  a.S = s;
  a.lo = f2_add(a.lo, t);
}

__device__ __forceinline__ void dp_swap_lanes(dpa& a) {
  a.S = make_float2(a.S.y, a.S.x);
  a.lo = make_float2(a.lo.y, a.lo.x);
}

// One real of the half spinors k = 0, 1 into pairs, the leading part rounded to
// nearest (the split truncates), which halves the trailing part the products
// round with.  The range guard takes h's words instead of the spinor's: NaN and
// infinities reach h, and large components that cancel leave an h that FP64
// holds and the pairs can represent.
__device__ __forceinline__ dp dslash_half(double x0, double x1, uint32_t& gm) {
  const uint32_t h0 = (uint32_t)__double2hiint(x0), h1 = (uint32_t)__double2hiint(x1);
  gm = guard_max(gm, h0, h1);
  const dp a = dp_split((uint32_t)__double2loint(x0), h0, (uint32_t)__double2loint(x1), h1);
  const float2 h = f2_add(a.h, a.l);
  return dp{h, f2_sub(a.l, f2_sub(h, a.h))};
}

// Direction of position t >> 1 in the order x, y, t, z.
__device__ __forceinline__ int dir_at(int t) {
  const int p = t >> 1;
  return p < 2 ? p : 5 - p;
}

// Where one term's operands lie: the neighbour spinor's and the link's first
// elements.
struct TermSrc {
  const uint4* psi;
  const uint4* U;
};
__device__ __forceinline__ TermSrc term_src(const FieldDesc& U, const FieldDesc& psi, const LatGeo& g,
                                            const Coords& c, int32_t s, int t) {
  const int mu = dir_at(t);
  const bool bwd = (t & 1) != 0;
  const int32_t n = neighbour(g, c, s, mu, bwd);
  return TermSrc{reinterpret_cast<const uint4*>(psi.ptr) + elem_base(psi, n, 0),
                 reinterpret_cast<const uint4*>(U.ptr) + elem_base(U, bwd ? n : s, mu)};
}

// Stage colour j of a term: the four spin components and the link's column j
// (backward: row j).  Slots: [colour][4 spins, 3 link elements][thread].
__device__ __forceinline__ void stage_colour(uint4* slot, const TermSrc& src, const FieldDesc& U,
                                             const FieldDesc& psi, bool bwd, int j) {
  const uint4* p = src.psi + j * psi.s_c;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    cp_async16(slot + (7 * j + k) * kDslashThreads, p);
    p += psi.s_mu;
  }
  const int64_t step = bwd ? U.s_c : 3 * U.s_c;
  p = src.U + (bwd ? 3 * j : j) * U.s_c;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cp_async16(slot + (7 * j + 4 + i) * kDslashThreads, p);
    p += step;
  }
  cp_async_commit();
}

// One colour's operands in pairs: h_k of that colour (lanes k = 0, 1) and the
// link's three elements (lanes re, im).
struct ColourOps {
  dp hr, hm;
  df2 u[3];
};

// How a term reads its operands (uniform across the grid).
struct TermForm {
  int l0, l1;           // byte offsets of the spin components added to u_0 and u_1
  int flip;             // 8: real and imaginary parts of l exchanged (factor i)
  uint32_t r0, r1, i0, i1;  // high words of the +-1.0 factors
  uint32_t neg;         // sign flip of the link's imaginary parts (adjoint)
};
__device__ __forceinline__ TermForm term_form(int t) {
  const int mu = dir_at(t);
  const bool bwd = (t & 1) != 0;
  const bool im = (mu & 1) == 0, sw = mu < 2;
  const bool p0 = (mu != 1) == bwd, p1 = (mu != 2) == bwd;  // f_k = +1
  TermForm f;
  f.l0 = (sw ? 3 : 2) * kDslashThreads * 16;
  f.l1 = (sw ? 2 : 3) * kDslashThreads * 16;
  f.flip = im ? 8 : 0;
  f.i0 = p0 ? 0x3FF00000u : 0xBFF00000u;
  f.i1 = p1 ? 0x3FF00000u : 0xBFF00000u;
  f.r0 = p0 != im ? 0x3FF00000u : 0xBFF00000u;
  f.r1 = p1 != im ? 0x3FF00000u : 0xBFF00000u;
  f.neg = bwd ? 0x80000000u : 0u;
  return f;
}

// h_k = u_k + f_k (i) l of colour j: with the factor i the real part takes
// -im(l) and the imaginary part re(l).
__device__ __forceinline__ void read_half(ColourOps& o, const uint4* slot, const TermForm& f, int j,
                                          uint32_t& gm) {
  const unsigned char* base = reinterpret_cast<const unsigned char*>(slot + 7 * j * kDslashThreads);
  const double2 u0 = *reinterpret_cast<const double2*>(base);
  const double2 u1 = *reinterpret_cast<const double2*>(base + kDslashThreads * 16);
  const double a0 = *reinterpret_cast<const double*>(base + f.l0 + f.flip);
  const double b0 = *reinterpret_cast<const double*>(base + f.l0 + (8 - f.flip));
  const double a1 = *reinterpret_cast<const double*>(base + f.l1 + f.flip);
  const double b1 = *reinterpret_cast<const double*>(base + f.l1 + (8 - f.flip));
  o.hr = dslash_half(fma(a0, __hiloint2double((int)f.r0, 0), u0.x),
                     fma(a1, __hiloint2double((int)f.r1, 0), u1.x), gm);
  o.hm = dslash_half(fma(b0, __hiloint2double((int)f.i0, 0), u0.y),
                     fma(b1, __hiloint2double((int)f.i1, 0), u1.y), gm);
}
__device__ __forceinline__ void read_link_elem(ColourOps& o, const uint4* slot, const TermForm& f, int j,
                                               int i, uint32_t& gm) {
  const uint4 v = slot[(7 * j + 4 + i) * kDslashThreads];
  gm = guard_max(gm, v.y, v.w);
  o.u[i] = df2_split(v.x, v.y, v.z, v.w ^ f.neg);
}

__global__ void __launch_bounds__(kDslashThreads, 3)
    k_dslash_df(const __grid_constant__ FieldDesc dst, const __grid_constant__ FieldDesc U,
                const __grid_constant__ FieldDesc psi, const __grid_constant__ LatGeo g) {
  extern __shared__ __align__(16) uint4 d_slots[];
  uint4* slot = d_slots + threadIdx.x;
  const int32_t V = (int32_t)g.V;
  const int64_t stride = (int64_t)gridDim.x * kDslashThreads;
  int64_t s = (int64_t)blockIdx.x * kDslashThreads + threadIdx.x;
  if (s >= V) return;
  Coords co = site_coords(g, s);
  uint32_t gm = 0, gm_next = 0;
  ColourOps cur;
  {
    const TermSrc src = term_src(U, psi, g, co, (int32_t)s, 0);
#pragma unroll
    for (int j = 0; j < 3; ++j) stage_colour(slot, src, U, psi, false, j);
    cp_async_wait<2>();
    const TermForm f = term_form(0);
    read_half(cur, slot, f, 0, gm_next);
#pragma unroll
    for (int i = 0; i < 3; ++i) read_link_elem(cur, slot, f, 0, i, gm_next);
  }
  for (;;) {
    const int64_t sn = s + stride;
    dpa up[6], low[6];   // [2 colour + re/im]
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      up[r] = dpa{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
      low[r] = up[r];
    }
    gm = 0;
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
      // this term's first colour was read during the term before (at t = 0 the
      // previous site's last): its range guard counts from here
      gm = max(gm, gm_next);
      gm_next = 0;
      // where the next term's operands come from (past the last site: this
      // site again, read and not used)
      if (t == 7 && sn < V) co = site_coords(g, sn);
      const int tn = (t + 1) & 7;
      const bool bwd_n = (tn & 1) != 0;
      const TermSrc src = term_src(U, psi, g, co, (int32_t)(t == 7 && sn < V ? sn : s), tn);
      const TermForm fc = term_form(t), fn = term_form(tn);
      dpa re[3], im[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        // colour j is in registers: refill its slots with the next term's, and
        // read colour j + 1 (after the last, the next term's first)
        ColourOps nxt;
        stage_colour(slot, src, U, psi, bwd_n, j);
        cp_async_wait<2>();
        const int jn = j < 2 ? j + 1 : 0;
        const TermForm& fr = j < 2 ? fc : fn;
        uint32_t& gr = j < 2 ? gm : gm_next;
        read_half(nxt, slot, fr, jn, gr);
        dp er[3], em[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const df2& e = cur.u[i];
          er[i] = dp{make_float2(e.h.x, e.h.x), make_float2(e.l.x, e.l.x)};
          em[i] = dp{make_float2(e.h.y, e.h.y), make_float2(e.l.y, e.l.y)};
        }
        dpa* const a0[6] = {&re[0], &re[1], &re[2], &im[0], &im[1], &im[2]};
        const dp* const y0[6] = {&er[0], &er[1], &er[2], &em[0], &em[1], &em[2]};
        const dp* const y1[6] = {&em[0], &em[1], &em[2], &er[0], &er[1], &er[2]};
        if (j == 0) dp_fma_shared<6, true, 0u>(a0, cur.hr, y0);
        else dp_fma_shared<6, false, 0u>(a0, cur.hr, y0);
        read_link_elem(nxt, slot, fr, jn, 0, gr);
        read_link_elem(nxt, slot, fr, jn, 1, gr);
        dp_fma_shared<6, false, 7u>(a0, cur.hm, y1);
        read_link_elem(nxt, slot, fr, jn, 2, gr);
        cur = nxt;
      }
      const float2 f = make_float2(__uint_as_float((fc.i0 & 0x80000000u) | 0x3F800000u),
                                   __uint_as_float((fc.i1 & 0x80000000u) | 0x3F800000u));
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        df2_combine<1>(up[2 * i], re[i]);
        df2_combine<1>(up[2 * i + 1], im[i]);
        dp_combine_sign(low[2 * i], re[i], f);
        dp_combine_sign(low[2 * i + 1], im[i], f);
      }
      // lower accumulators: x holds i * lower in lanes (3, 2); y lower in lanes
      // (3, 2); t lower in lanes (2, 3); z i * lower in lanes (2, 3)
      if (t == 3) {
#pragma unroll
        for (int r = 0; r < 6; ++r) dp_swap_lanes(low[r]);
      } else if (t == 1 || t == 5) {
        // x -> y: lower = -i (i lower); t -> z: i lower
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const dpa a = low[2 * c], b = low[2 * c + 1];
          const dpa na{f2_neg(a.S), f2_neg(a.lo)}, nb{f2_neg(b.S), f2_neg(b.lo)};
          low[2 * c] = t == 1 ? b : nb;
          low[2 * c + 1] = t == 1 ? na : a;
        }
      }
    }
    if (gm >= guard_hi(2)) {
      dslash_site_f64<MathF64>(dst, U, psi, g, s);
    } else {
      const int64_t b = elem_base(dst, s, 0);
      char* p = reinterpret_cast<char*>(dst.ptr);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int64_t e = b + c * dst.s_c;
        pair_store_c(p, e, e + dst.s_mu, true, up[2 * c], up[2 * c + 1]);
        // lower = -i (i lower)
        const dpa n{f2_neg(low[2 * c].S), f2_neg(low[2 * c].lo)};
        pair_store_c(p, e + 2 * dst.s_mu, e + 3 * dst.s_mu, true, low[2 * c + 1], n);
      }
    }
    if (sn >= V) break;
    s = sn;
  }
  cp_async_wait_all();
}

// `waves` waves of blocks, the threads' sites strided by the grid.
static cudaError_t dslash_grid(const void* kernel, size_t smem, int64_t V, int waves, dim3* grid) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 1;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kDslashThreads, smem);
  if (e != cudaSuccess) return e;
  const int64_t nb = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count() * waves;
  const int64_t need = (V + kDslashThreads - 1) / kDslashThreads;
  *grid = dim3((unsigned)(nb < need ? nb : need));
  return cudaSuccess;
}

static cudaError_t launch_dslash_df(const su3s_field* dest, const su3s_field* U, const su3s_field* psi,
                                    cudaStream_t st) {
  const LatGeo g = lat_geo(psi);
  const size_t smem = (size_t)kDslashElems * 16 * kDslashThreads;
  dim3 grid;
  // four waves: blocks do not all take the same time, and what one finishes
  // early the next ones use (one wave 787 us, two 769, four 755, one site per
  // thread 766 at 32^3 x 64)
  const cudaError_t e = dslash_grid((const void*)k_dslash_df, smem, g.V, 4, &grid);
  if (e != cudaSuccess) return e;
  k_dslash_df<<<grid, kDslashThreads, smem, st>>>(dest->desc, U->desc, psi->desc, g);
  return cudaGetLastError();
}

template <class M>
static cudaError_t launch_dslash(const su3s_field* dest, const su3s_field* U, const su3s_field* psi,
                                 cudaStream_t st) {
  const LatGeo g = lat_geo(psi);
  const size_t smem = (size_t)kDslashElems * 16 * kDslashThreads;
  dim3 grid;
  // 32 waves: each wave of a grid-stride loop lets its blocks drift apart, new
  // blocks start in the order of the sites, so that the neighbours of those in
  // flight stay in the L2 cache.  Fixed point: one wave 2,094 us, four 2,086,
  // eight 2,064, 32 1,985, one site per thread 2,044 at 32^3 x 64; at 16^3 x 32
  // one wave 156, 32 waves 145.  FP64 at 32^3 x 64: one wave 4,037, 32 waves 4,002.
  const cudaError_t e = dslash_grid((const void*)k_dslash<M>, smem, g.V, 32, &grid);
  if (e != cudaSuccess) return e;
  k_dslash<M><<<grid, kDslashThreads, smem, st>>>(dest->desc, U->desc, psi->desc, g);
  return cudaGetLastError();
}

}  // namespace su3s

using namespace su3s;

SU3S_EXPORT int su3s_dslash(su3s_field* dest, const su3s_field* U, const su3s_field* psi, int math,
                            void* stream) {
  if (!dest || !U || !psi) return fail(SU3S_EINVAL, "null argument");
  if (U->kind != SU3S_MATRIX || U->nmu != 4)
    return fail(SU3S_ETYPE, "the links must be a matrix field with 4 links per site");
  if (psi->kind != SU3S_VECTOR || psi->nmu != 4 || dest->kind != SU3S_VECTOR || dest->nmu != 4)
    return fail(SU3S_ETYPE, "spinor fields are colour-vector fields with 4 spin components per site");
  if (U->prec != SU3S_F64 || psi->prec != SU3S_F64 || dest->prec != SU3S_F64)
    return fail(SU3S_EUNSUPPORTED, "the Wilson hopping term needs FP64 storage");
  for (int d = 0; d < 4; ++d)
    if (U->L[d] != psi->L[d] || dest->L[d] != psi->L[d])
      return fail(SU3S_ESHAPE, "fields live on different lattices");
  if (overlap(dest, psi) || overlap(dest, U)) return fail(SU3S_EINVAL, "destination overlaps an input");
  if (!valid_math(math)) return fail(SU3S_EINVAL, "bad arithmetic %d", math);
  const int m = resolve_math(SU3S_F64, math);
  cudaStream_t st = (cudaStream_t)stream;
  if (psi->V == 0) return SU3S_OK;
  cudaError_t ce = m == MATH_F64  ? launch_dslash<MathF64>(dest, U, psi, st)
                   : m == MATH_FX ? launch_dslash<MathFX>(dest, U, psi, st)
                                  : launch_dslash_df(dest, U, psi, st);
  if (ce != cudaSuccess) return cuda_fail(ce, "Wilson hopping-term kernel launch");
  return SU3S_OK;
}
