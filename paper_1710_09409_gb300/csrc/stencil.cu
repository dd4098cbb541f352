// Nearest-neighbour operations: the Cshift and the colour part of the Dslash
// hopping term, which the paper names as the next step beyond its site-local
// expression engine (Sec. 6, Summary and Outlook: porting Grid's Dslash
// operator, whose Cshift operations lie outside the expression templates).
//
//   su3s_cshift  dst(x) = src(x + shift e_dim), periodic in every direction:
//                a gather of whole site objects in their storage format.
//   su3s_hop     out(x) = sum_mu U_mu(x) v(x+mu) + U_mu(x-mu)^dagger v(x-mu)
//                for a colour-vector or colour-matrix field v and the four
//                links U of every site, FP64 storage, in the arithmetic of
//                the site-local kernels.
//
// Sites are s = x + Lx (y + Ly (z + Lz t)); one thread per site.  Neighbour
// objects are read through the read-only data cache: every object is read
// by up to eight neighbouring sites, so L1 and L2 supply most of the reuse.
#include <cuda_runtime.h>

#include "dev_stencil.cuh"
#include "internal.h"

namespace su3s {

// ------------------------------------------------------------- Cshift
// One thread per (site, object element); EB bytes per stored element.
template <int EB>
struct Raw;
template <>
struct Raw<16> {
  using T = uint4;
};
template <>
struct Raw<8> {
  using T = uint2;
};
template <>
struct Raw<4> {
  using T = uint32_t;
};

// One thread per site of one element (blockIdx.y = link * ncomp + component);
// consecutive threads take consecutive sites, so reads and writes coalesce
// except where the shift wraps around.
// The shifted direction is passed as its stride and extent (no per-thread
// indexing of the geometry).
template <int EB>
__global__ void __launch_bounds__(256) k_cshift(FieldDesc dst, FieldDesc src, int64_t V,
                                                uint32_t stride, uint32_t extent, int ncomp,
                                                int shift) {
  using T = typename Raw<EB>::T;
  const int q = blockIdx.y;
  const int mu = q / ncomp, c = q - mu * ncomp;
  const int64_t qo_d = (int64_t)mu * dst.s_mu + (int64_t)c * dst.s_c;
  const int64_t qo_s = (int64_t)mu * src.s_mu + (int64_t)c * src.s_c;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < V;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int32_t co = (int32_t)(((uint32_t)s / stride) % extent);
    int32_t c2 = co + shift;   // shift in [0, extent)
    c2 = c2 >= (int32_t)extent ? c2 - (int32_t)extent : c2;
    const int64_t n = s + (int64_t)(c2 - co) * stride;
    const T v = __ldg(reinterpret_cast<const T*>(src.ptr) + elem_base(src, n, 0) + qo_s);
    reinterpret_cast<T*>(dst.ptr)[elem_base(dst, s, 0) + qo_d] = v;
  }
}

// ---------------------------------------------------------- hopping term
// The hopping term at site s in the arithmetic M.  Every term's operands are
// range-checked (see dev_math.cuh); a site out of range is computed again in
// native FP64 before its store (the destination overlaps no input).
template <int KIND>
__device__ __noinline__ void hop_site_f64(const FieldDesc& dst, const FieldDesc& U,
                                          const FieldDesc& v, const LatGeo& g, int64_t s);

template <class M, int KIND>
__device__ __forceinline__ void hop_site(const FieldDesc& dst, const FieldDesc& U, const FieldDesc& v,
                                         const LatGeo& g, int64_t s) {
  constexpr int W = KIND == KM ? 18 : 6;
  typename M::A acc[W];
  uint32_t gm = 0;
  if constexpr (KIND == KM) {
#pragma unroll
    for (int r = 0; r < W; ++r) acc[r] = M::zero();
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
      // t = 2 mu: forward U_mu(x) v(x + mu); t = 2 mu + 1: backward
      // U_mu(x - mu)^dagger v(x - mu)
      const int mu = t >> 1;
      const bool bwd = (t & 1) != 0;
      const int64_t n = shift_site_rt(g, s, mu, bwd ? -1 : 1);
      typename M::R u[18], x[W];
      load_link<M>(U, bwd ? n : s, mu, bwd, u, gm);
      load_nc<M, W>(v, n, 0, x, gm);
      mm_combine<M, 1, false, false>(acc, u, x);
    }
  } else {
    {
      typename M::R u[18], x[W];
      load_nc<M, 18>(U, s, 0, u, gm);
      load_nc<M, W>(v, shift_site_rt(g, s, 0, 1), 0, x, gm);
      mv_acc<M, true, 1, false>(acc, u, x);
    }
#pragma unroll 1
    for (int t = 1; t < 8; ++t) {
      const int mu = t >> 1;
      typename M::R u[18], x[W];
      if ((t & 1) == 0) {
        load_nc<M, 18>(U, s, mu, u, gm);
        load_nc<M, W>(v, shift_site_rt(g, s, mu, 1), 0, x, gm);
        mv_combine<M, 1, false>(acc, u, x);
      } else {
        const int64_t bw = shift_site_rt(g, s, mu, -1);
        load_nc<M, 18>(U, bw, mu, u, gm);
        load_nc<M, W>(v, bw, 0, x, gm);
        mv_combine<M, 1, true>(acc, u, x);
      }
    }
  }
  if constexpr (M::kGuard) {
    if (gm >= guard_hi(2)) {
      hop_site_f64<KIND>(dst, U, v, g, s);
      return;
    }
  }
  typename M::A out[1][W];
#pragma unroll
  for (int r = 0; r < W; ++r) out[0][r] = acc[r];
  store_obj<KIND, P_F64, M, 1, W>(dst, s, 0, out);
}

template <int KIND>
__device__ __noinline__ void hop_site_f64(const FieldDesc& dst, const FieldDesc& U,
                                          const FieldDesc& v, const LatGeo& g, int64_t s) {
  hop_site<MathF64, KIND>(dst, U, v, g, s);
}

// One thread per site; up to 32 waves of blocks (launch_hop), which start in the
// order of the sites, so that the sites in flight (and the backward links and
// neighbours they share) stay together in the L2 cache; the loop over the 8
// terms is rolled.  Colour matrices: the terms run through a single
// product routine (the backward link's adjoint is taken in its load), which
// keeps the matrix-product code small enough for the instruction cache (+29%
// at 48^4 over separate forward and backward routines).  Colour vectors (native
// FP64 and fixed point): the matrix-vector code is small, and separate forward
// and backward routines, with the first term opening the accumulators, are
// faster (+13%).
template <class M, int KIND>
__global__ void __launch_bounds__(128) k_hop(FieldDesc dst, FieldDesc U, FieldDesc v, LatGeo g) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < g.V;
       s += (int64_t)gridDim.x * blockDim.x)
    hop_site<M, KIND>(dst, U, v, g, s);
}

// ------------------------------- pair arithmetic on vectors: both senses per lane pair
// The pair arithmetic's kernel for colour vectors takes the forward and the
// backward term of a direction together, one in each lane of the packed FP32
// operations: lane 0 U_mu(x) v(x+mu), lane 1 U_mu(x-mu)^dagger v(x-mu), the
// adjoint a transposed address and a sign folded into the split.  The two
// products share nothing but their shape, so no operand is duplicated, swapped
// or negated; each product is accumulated on its own and added to its lane's
// sum over the directions, and the two lanes' sums are added at the end.  The
// operands come one colour at a time through slots in shared memory
// (asynchronous copies): the next colour is read and split, work of the ALU
// pipe, between the products of the current one, work of the FMA pipe, and its
// slots are refilled for the next direction as soon as they are read.
// Bound by issue with the ALU and FMA pipes 53% and 56% busy (4,190 instructions
// per site, 4,510 before).  Measured at 47x45x46x49: 1,069 -> 815 us (672 B per
// site: 2,998 -> 3,932 GB/s); three blocks of 144 registers per SM 824.  The
// order of the sites (one wave, four, contiguous runs of 1 to 16 tiles per
// block) moves the DRAM reads between 3.6 and 4.3 GB and the time by 4% only.
constexpr int kHopThreads = 128;
constexpr int kHopSlots = 8;   // per colour: v forward, v backward, 3 + 3 link elements

struct HopSrc {
  const uint4 *vf, *vb, *uf, *ub;   // first elements of direction mu's operands
};
__device__ __forceinline__ HopSrc hop_src(const FieldDesc& U, const FieldDesc& v, const LatGeo& g,
                                          const Coords& c, int32_t s, int mu) {
  const int32_t nf = neighbour(g, c, s, mu, false), nb = neighbour(g, c, s, mu, true);
  const uint4* pv = reinterpret_cast<const uint4*>(v.ptr);
  const uint4* pu = reinterpret_cast<const uint4*>(U.ptr);
  return HopSrc{pv + elem_base(v, nf, 0), pv + elem_base(v, nb, 0), pu + elem_base(U, s, mu),
                pu + elem_base(U, nb, mu)};
}

// Stage colour j of a direction: v_j of both neighbours, column j of the
// forward link, row j of the backward one.
__device__ __forceinline__ void hop_stage(uint4* slot, const HopSrc& src, const FieldDesc& U,
                                          const FieldDesc& v, int j) {
  uint4* d = slot + kHopSlots * j * kHopThreads;
  cp_async16(d, src.vf + j * v.s_c);
  cp_async16(d + kHopThreads, src.vb + j * v.s_c);
  const uint4* pf = src.uf + j * U.s_c;
  const uint4* pb = src.ub + 3 * j * U.s_c;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cp_async16(d + (2 + i) * kHopThreads, pf);
    cp_async16(d + (5 + i) * kHopThreads, pb);
    pf += 3 * U.s_c;
    pb += U.s_c;
  }
  cp_async_commit();
}

// One colour's operands in pairs, lanes (forward, backward).
struct HopOps {
  dp vr, vm, ur[3], um[3];
};
__device__ __forceinline__ void hop_read_v(HopOps& o, const uint4* slot, int j, uint32_t& gm) {
  const uint4 f = slot[kHopSlots * j * kHopThreads], b = slot[(kHopSlots * j + 1) * kHopThreads];
  gm = guard_max(guard_max(gm, f.y, f.w), b.y, b.w);
  o.vr = dp_split(f.x, f.y, b.x, b.y);
  o.vm = dp_split(f.z, f.w, b.z, b.w);
}
__device__ __forceinline__ void hop_read_u(HopOps& o, const uint4* slot, int j, int i, uint32_t& gm) {
  const uint4 f = slot[(kHopSlots * j + 2 + i) * kHopThreads];
  const uint4 b = slot[(kHopSlots * j + 5 + i) * kHopThreads];
  gm = guard_max(guard_max(gm, f.y, f.w), b.y, b.w);
  o.ur[i] = dp_split(f.x, f.y, b.x, b.y);
  o.um[i] = dp_split(f.z, f.w, b.z, b.w ^ 0x80000000u);
}

__global__ void __launch_bounds__(kHopThreads, 4)
    k_hop_df(const __grid_constant__ FieldDesc dst, const __grid_constant__ FieldDesc U,
             const __grid_constant__ FieldDesc v, const __grid_constant__ LatGeo g) {
  extern __shared__ __align__(16) uint4 h_slots[];
  uint4* slot = h_slots + threadIdx.x;
  const int32_t V = (int32_t)g.V;
  const int64_t stride = (int64_t)gridDim.x * kHopThreads;
  int64_t s = (int64_t)blockIdx.x * kHopThreads + threadIdx.x;
  if (s >= V) return;
  Coords co = site_coords(g, s);
  uint32_t gm = 0, gm_next = 0;
  HopOps cur;
  {
    const HopSrc src = hop_src(U, v, g, co, (int32_t)s, 0);
#pragma unroll
    for (int j = 0; j < 3; ++j) hop_stage(slot, src, U, v, j);
    cp_async_wait<2>();
    hop_read_v(cur, slot, 0, gm_next);
#pragma unroll
    for (int i = 0; i < 3; ++i) hop_read_u(cur, slot, 0, i, gm_next);
  }
  for (;;) {
    const int64_t sn = s + stride;
    dpa acc[6];   // [2 colour + re/im], lanes: forward, backward
#pragma unroll
    for (int r = 0; r < 6; ++r) acc[r] = dpa{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
    gm = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      // this direction's first colour was read during the one before (at mu = 0
      // the previous site's last): its range guard counts from here
      gm = max(gm, gm_next);
      gm_next = 0;
      // where the next direction's operands come from (past the last site:
      // this site again, read and not used)
      if (mu == 3 && sn < V) co = site_coords(g, sn);
      const HopSrc src = hop_src(U, v, g, co, (int32_t)(mu == 3 && sn < V ? sn : s), (mu + 1) & 3);
      dpa re[3], im[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        HopOps nxt;
        hop_stage(slot, src, U, v, j);
        cp_async_wait<2>();
        const int jn = j < 2 ? j + 1 : 0;
        uint32_t& gr = j < 2 ? gm : gm_next;
        hop_read_v(nxt, slot, jn, gr);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          if (j == 0) dp_cterm<true, 1, false, false>(re[i], im[i], cur.ur[i], cur.um[i], cur.vr, cur.vm);
          else dp_cterm<false, 1, false, false>(re[i], im[i], cur.ur[i], cur.um[i], cur.vr, cur.vm);
          hop_read_u(nxt, slot, jn, i, gr);
        }
        cur = nxt;
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        df2_combine<1>(acc[2 * i], re[i]);
        df2_combine<1>(acc[2 * i + 1], im[i]);
      }
    }
    if (gm >= guard_hi(2)) {
      hop_site_f64<KV>(dst, U, v, g, s);
    } else {
      DAcc out[1][6];
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        out[0][r] = DAcc{acc[r].S.x, acc[r].lo.x};
        MathDF::combine<1>(out[0][r], DAcc{acc[r].S.y, acc[r].lo.y});
      }
      store_obj<KV, P_F64, MathDF, 1, 6>(dst, s, 0, out);
    }
    if (sn >= V) break;
    s = sn;
  }
  cp_async_wait_all();
}

template <class K>
static dim3 grid_for(K kernel, int threads, int64_t work) {
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
  int64_t nb = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count() * 4;
  const int64_t need = (work + threads - 1) / threads;
  if (nb > need) nb = need;
  return dim3((unsigned)(nb < 1 ? 1 : nb));
}

template <class M, int KIND>
static cudaError_t launch_hop(const su3s_field* dest, const su3s_field* U, const su3s_field* v,
                              cudaStream_t st) {
  const LatGeo g = lat_geo(v);
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hop<M, KIND>, 128, 0);
  // 32 waves: the blocks of one wave drift apart over a long grid-stride loop.
  // 32^3 x 64, one wave, four, 32: pair arithmetic on matrices 1,086, 998, 955 us;
  // fixed point on vectors 604, 548, 536, on matrices 1,361, 1,358, 1,345; FP64
  // 1,212, 1,177, 1,175 and 3,700, 3,602, 3,579.  Fixed-point matrices below eight
  // waves keep one; there the two come out alike.  One wave against 32 at 20 sizes:
  // within 1% at nine, one faster at eight (14^3 x 28 51.5 / 52.9 us, 16^3 x 32 94.4 /
  // 96.5, 20^3 x 30 164.6 / 169.9, 20^3 x 40 212 / 219 and others, 1.5 to 3%), 32 at
  // three (18^3 x 30 130 / 123, 18^3 x 36 155 / 146, 24^4 229 / 227): how full the
  // last round of blocks is decides, not the number of waves.
  const int64_t wave = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count();
  const int64_t need = (g.V + 127) / 128;
  const int64_t nb = M::kScaled && KIND == KM && need < 8 * wave ? wave : 32 * wave;
  const dim3 grid((unsigned)(nb < need ? nb : need));
  k_hop<M, KIND><<<grid, 128, 0, st>>>(dest->desc, U->desc, v->desc, g);
  return cudaGetLastError();
}

static cudaError_t launch_hop_df(const su3s_field* dest, const su3s_field* U, const su3s_field* v,
                                 cudaStream_t st) {
  const LatGeo g = lat_geo(v);
  const size_t smem = (size_t)3 * kHopSlots * 16 * kHopThreads;
  cudaError_t e = cudaFuncSetAttribute(k_hop_df, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 1;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hop_df, kHopThreads, smem);
  if (e != cudaSuccess) return e;
  // four waves of blocks, as the Wilson term
  const int64_t nb = (int64_t)(per_sm > 0 ? per_sm : 1) * sm_count() * 4;
  const int64_t need = (g.V + kHopThreads - 1) / kHopThreads;
  k_hop_df<<<(unsigned)(nb < need ? nb : need), kHopThreads, smem, st>>>(dest->desc, U->desc, v->desc, g);
  return cudaGetLastError();
}

}  // namespace su3s

using namespace su3s;

SU3S_EXPORT int su3s_cshift(su3s_field* dest, const su3s_field* src, int dim, int shift,
                            void* stream) {
  if (!dest || !src) return fail(SU3S_EINVAL, "null argument");
  if (dim < 0 || dim > 3) return fail(SU3S_EINVAL, "direction %d is not 0..3", dim);
  int rc = check_same_shape(dest, src, true);
  if (rc) return rc;
  if (dest->kind != src->kind) return fail(SU3S_ETYPE, "fields of different kinds");
  if (overlap(dest, src)) return fail(SU3S_EINVAL, "destination overlaps the source");
  const int L = src->L[dim];
  const int sh = ((shift % L) + L) % L;   // into [0, L)
  const LatGeo g = lat_geo(src);
  const int nelem = src->nmu * src->ncomp;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t ce = cudaSuccess;
  if (g.V == 0) return SU3S_OK;
  const auto grid = [&](dim3 gx) { return dim3(gx.x, (unsigned)nelem, 1); };
  switch (src->elem_bytes) {
    case 16:
      k_cshift<16><<<grid(grid_for(k_cshift<16>, 256, g.V)), 256, 0, st>>>(dest->desc, src->desc, g.V,
                                                                           (uint32_t)g.stride[dim], (uint32_t)g.L[dim], src->ncomp, sh);
      break;
    case 8:
      k_cshift<8><<<grid(grid_for(k_cshift<8>, 256, g.V)), 256, 0, st>>>(dest->desc, src->desc, g.V,
                                                                         (uint32_t)g.stride[dim], (uint32_t)g.L[dim], src->ncomp, sh);
      break;
    default:
      k_cshift<4><<<grid(grid_for(k_cshift<4>, 256, g.V)), 256, 0, st>>>(dest->desc, src->desc, g.V,
                                                                         (uint32_t)g.stride[dim], (uint32_t)g.L[dim], src->ncomp, sh);
      break;
  }
  ce = cudaGetLastError();
  if (ce != cudaSuccess) return cuda_fail(ce, "cshift kernel launch");
  return SU3S_OK;
}

SU3S_EXPORT int su3s_hop(su3s_field* dest, const su3s_field* U, const su3s_field* v, int math,
                         void* stream) {
  if (!dest || !U || !v) return fail(SU3S_EINVAL, "null argument");
  if (U->kind != SU3S_MATRIX || U->nmu != 4)
    return fail(SU3S_ETYPE, "the links must be a matrix field with 4 links per site");
  if (v->kind == SU3S_REAL || v->nmu != 1)
    return fail(SU3S_ETYPE, "the operand must be a matrix or vector field with one object per site");
  if (dest->kind != v->kind || dest->nmu != 1)
    return fail(SU3S_ETYPE, "the destination must have the operand's kind");
  if (U->prec != SU3S_F64 || v->prec != SU3S_F64 || dest->prec != SU3S_F64)
    return fail(SU3S_EUNSUPPORTED, "the hopping term needs FP64 storage");
  for (int d = 0; d < 4; ++d)
    if (U->L[d] != v->L[d] || dest->L[d] != v->L[d])
      return fail(SU3S_ESHAPE, "fields live on different lattices");
  if (overlap(dest, v) || overlap(dest, U)) return fail(SU3S_EINVAL, "destination overlaps an input");
  if (!valid_math(math)) return fail(SU3S_EINVAL, "bad arithmetic %d", math);
  const int m = resolve_math(SU3S_F64, math);
  cudaStream_t st = (cudaStream_t)stream;
  if (v->V == 0) return SU3S_OK;
  cudaError_t ce;
  const bool mat = v->kind == SU3S_MATRIX;
  if (m == MATH_F64) ce = mat ? launch_hop<MathF64, KM>(dest, U, v, st) : launch_hop<MathF64, KV>(dest, U, v, st);
  else if (m == MATH_FX) ce = mat ? launch_hop<MathFX, KM>(dest, U, v, st) : launch_hop<MathFX, KV>(dest, U, v, st);
  else ce = mat ? launch_hop<MathDFScalar, KM>(dest, U, v, st) : launch_hop_df(dest, U, v, st);
  if (ce != cudaSuccess) return cuda_fail(ce, "hopping-term kernel launch");
  return SU3S_OK;
}
