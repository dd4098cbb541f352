// Uniform per-site interpreter for expression trees outside the compiled
// catalogue (FP64 storage).  The tree is flattened on the host into a short
// register program; every thread runs the same program on its own site, so
// control flow is uniform across the grid (no divergence), and the whole tree
// is still evaluated in one read/write pass (Sec. 3, Listing 1).  The register
// file lives in shared memory, laid out [register][real][thread] so that
// consecutive threads touch consecutive words; an instruction copies its
// operands into fixed-size arrays (their widths are known per operation), so
// the arithmetic runs on registers, and writes its result back.  The host
// sizes the shared memory to the registers the program uses: leaves are
// loaded at their first use and every register is freed after the last operation
// that reads it (interp_prog.h).
#include <string.h>

#include <mutex>
#include <vector>

#include "dev_kernels.cuh"
#include "internal.h"
#include "interp_prog.h"

namespace su3s {

// The register file: real r of register g of this thread, in a slot of SLOT
// bytes.  The native FP64 path of the range guard runs on the register file of
// another arithmetic: a double in the thread's own slots, moved as two words
// where the slot is not aligned to it.
template <class M, int SLOT = (int)sizeof(typename M::R)>
struct IRegs {
  using R = typename M::R;
  unsigned char* base;
  int nt, tid;
  __device__ __forceinline__ unsigned char* slot(int g, int r) const {
    return base + (size_t)((g * 18 + r) * nt + tid) * SLOT;
  }
  __device__ __forceinline__ R ld(int g, int r) const {
    if constexpr (SLOT % alignof(R) == 0) {
      return *reinterpret_cast<const R*>(slot(g, r));
    } else {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(slot(g, r));
      return u2d(w[0], w[1]);
    }
  }
  __device__ __forceinline__ void st(int g, int r, const R& v) const {
    if constexpr (SLOT % alignof(R) == 0) {
      *reinterpret_cast<R*>(slot(g, r)) = v;
    } else {
      uint32_t* w = reinterpret_cast<uint32_t*>(slot(g, r));
      w[0] = (uint32_t)__double2loint(v);
      w[1] = (uint32_t)__double2hiint(v);
    }
  }
  template <int W>
  __device__ __forceinline__ void get(int g, R* v) const {
#pragma unroll
    for (int r = 0; r < W; ++r) v[r] = ld(g, r);
  }
  template <int W>
  __device__ __forceinline__ void put(int g, const R* v) const {
#pragma unroll
    for (int r = 0; r < W; ++r) st(g, r, v[r]);
  }
};

// Object of W reals of field f (FP64 storage) at site s, link mu; g is the
// site's range guard (largest input high word, see dev_math.cuh).
template <class M, int W>
__device__ __forceinline__ void i_load(const FieldDesc& f, int64_t s, int mu, typename M::R* r,
                                       uint32_t& g) {
  const int64_t b = elem_base(f, s, mu);
  if constexpr (W == 1) {
    const uint2 v = ld8((const char*)f.ptr + b * 8);
    if constexpr (M::kGuard) g = guard_max(g, v.y, v.y);
    r[0] = M::from_bits(v.x, v.y);
  } else {
#pragma unroll
    for (int c = 0; c < W / 2; ++c) {
      const uint4 v = ld16((const char*)f.ptr + (b + c * f.s_c) * 16);
      if constexpr (M::kGuard) g = guard_max(g, v.y, v.w);
      split_complex<M>(v, r[2 * c], r[2 * c + 1]);
    }
  }
  M::template normalize_obj<W>(r);
}

// A matrix register, or (FOLD and dag) its adjoint.
template <class M, bool FOLD, class Regs>
__device__ __forceinline__ void i_get_mat(const Regs& R, int g, bool dag, typename M::R* v) {
  R.template get<18>(g, v);
  if (FOLD && dag) {
    typename M::R t[18];
    adjoint<M>(t, v);
#pragma unroll
    for (int r = 0; r < 18; ++r) v[r] = t[r];
  }
}

template <class M, int W, class Regs>
__device__ __forceinline__ void i_add(const Regs& R, const IIns& in, int sg) {
  typename M::R x[W], y[W], d[W];
  typename M::A acc[W];
  R.template get<W>(in.a, x);
  R.template get<W>(in.b, y);
#pragma unroll
  for (int r = 0; r < W; ++r) {
    M::template add<true, 1>(acc[r], x[r]);
    if (sg > 0) M::template add<false, 1>(acc[r], y[r]);
    else M::template add<false, -1>(acc[r], y[r]);
  }
  finish<M, W>(d, acc);
  R.template put<W>(in.dst, d);
}

template <class M, int W, class Regs>
__device__ __forceinline__ void i_scale(const Regs& R, const IIns& in, const KParams& p) {
  typename M::R x[W], d[W];
  typename M::A acc[W];
  R.template get<W>(in.a, x);
  const typename M::R sc = M::scalar(p.sc[in.arg], p.sch[in.arg], p.scl[in.arg]);
#pragma unroll
  for (int r = 0; r < W; ++r) M::template fma<true, 1>(acc[r], sc, x[r]);
  finish<M, W>(d, acc);
  R.template put<W>(in.dst, d);
}

template <class M, int W, class Regs>
__device__ __forceinline__ void i_store(const FieldDesc& dst, int64_t s, int mu, const Regs& R,
                                        int g) {
  typename M::R z[W];
  R.template get<W>(g, z);
  const int64_t b = elem_base(dst, s, mu);
  if constexpr (W == 1) {
    StoreReal::template store_acc<M>(dst.ptr, b, M::to_acc(z[0]));
  } else {
#pragma unroll
    for (int c = 0; c < W / 2; ++c) {
      typename M::A re[1] = {M::to_acc(z[2 * c])}, im[1] = {M::to_acc(z[2 * c + 1])};
      Store<P_F64>::template store_acc<M>(dst.ptr, b + c * dst.s_c, re, im);
    }
  }
}

// Run the program on site s into the register file R (g: range guard).
// FOLD: products may read their operands' adjoints (the pair kernel's programs).
template <class M, bool FOLD, class Regs>
__device__ __forceinline__ void i_run(const KParams& p, const IProg& prog, const Regs& R,
                                      int64_t s, int mu, uint32_t& g) {
  using Rv = typename M::R;
  using Av = typename M::A;
  for (int pc = 0; pc < prog.n; ++pc) {
    const IIns in = prog.ins[pc];
    switch (in.op) {
      case I_LOAD: {
        Rv v[18];
        if (in.w == 18) {
          i_load<M, 18>(p.leaf[in.arg], s, mu, v, g);
          R.template put<18>(in.dst, v);
        } else if (in.w == 6) {
          i_load<M, 6>(p.leaf[in.arg], s, mu, v, g);
          R.template put<6>(in.dst, v);
        } else {
          i_load<M, 1>(p.leaf[in.arg], s, mu, v, g);
          R.template put<1>(in.dst, v);
        }
        break;
      }
      case I_MMUL: {
        Rv x[18], y[18], d[18];
        Av acc[18];
        i_get_mat<M, FOLD>(R, in.a, (in.adj & 1) != 0, x);
        i_get_mat<M, FOLD>(R, in.b, (in.adj & 2) != 0, y);
        mm_acc<M, true, 1, false, false>(acc, x, y);
        finish<M, 18>(d, acc);
        R.template put<18>(in.dst, d);
        break;
      }
      case I_MVMUL: {
        Rv x[18], y[6], d[6];
        Av acc[6];
        i_get_mat<M, FOLD>(R, in.a, (in.adj & 1) != 0, x);
        R.template get<6>(in.b, y);
        mv_acc<M, true, 1, false>(acc, x, y);
        finish<M, 6>(d, acc);
        R.template put<6>(in.dst, d);
        break;
      }
      case I_RMUL: {
        Rv x[1], y[1], d[1];
        Av acc[1];
        R.template get<1>(in.a, x);
        R.template get<1>(in.b, y);
        M::template fma<true, 1>(acc[0], x[0], y[0]);
        finish<M, 1>(d, acc);
        R.template put<1>(in.dst, d);
        break;
      }
      case I_ADD:
      case I_SUB: {
        const int sg = in.op == I_ADD ? 1 : -1;
        if (in.w == 18) i_add<M, 18>(R, in, sg);
        else if (in.w == 6) i_add<M, 6>(R, in, sg);
        else i_add<M, 1>(R, in, sg);
        break;
      }
      case I_SCALE: {
        if (in.w == 18) i_scale<M, 18>(R, in, p);
        else if (in.w == 6) i_scale<M, 6>(R, in, p);
        else i_scale<M, 1>(R, in, p);
        break;
      }
      default: {  // I_ADJ
        Rv x[18], t[18];
        R.template get<18>(in.a, x);
        adjoint<M>(t, x);
        R.template put<18>(in.dst, t);
        break;
      }
    }
  }
}

template <class M, class Regs>
__device__ __forceinline__ void i_store_root(const KParams& p, const IProg& prog, const Regs& R,
                                             int64_t s, int mu) {
  if (prog.root_kind == KR) i_store<M, 1>(p.dst, s, mu, R, prog.root);
  else if (prog.root_kind == KV) i_store<M, 6>(p.dst, s, mu, R, prog.root);
  else i_store<M, 18>(p.dst, s, mu, R, prog.root);
}

// The range guard's path: the program again in native FP64 on this thread's
// slots of the register file (a double is no wider than any arithmetic's
// real, so it fits its slot), then the store.  Out of line, off the hot loop.
template <int SLOT, bool FOLD>
__device__ __noinline__ void i_site_f64(const KParams& p, const IProg& prog, unsigned char* base, int nt,
                                        int tid, int64_t s, int mu) {
  const IRegs<MathF64, SLOT> R{base, nt, tid};
  uint32_t g = 0;
  i_run<MathF64, FOLD>(p, prog, R, s, mu, g);
  i_store_root<MathF64>(p, prog, R, s, mu);
}

template <class M>
__global__ void __launch_bounds__(128) k_interp(const __grid_constant__ KParams p,
                                                const __grid_constant__ IProg prog) {
  using Rv = typename M::R;
  extern __shared__ __align__(16) unsigned char i_smem[];
  const IRegs<M> R{i_smem, (int)blockDim.x, (int)threadIdx.x};
  const int mu = blockIdx.y;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < p.nvec; s += stride) {
    uint32_t g = p.gscal;
    i_run<M, false>(p, prog, R, s, mu, g);
    if (M::kGuard && g >= p.ghi)
      i_site_f64<(int)sizeof(Rv), false>(p, prog, i_smem, (int)blockDim.x, (int)threadIdx.x, s, mu);
    else i_store_root<M>(p, prog, R, s, mu);
  }
}

// ------------------------------------------- pair arithmetic: two sites per thread
// The pair arithmetic's interpreter packs every FP32 operation over two sites,
// s and s + blockDim.x of a run of 2 blockDim.x sites: half the instructions,
// program steps and operand fetches per site, and no operand is copied,
// swapped or signed (as in dev_pairs.cuh).  A register's real is 16 bytes per
// thread ([register][real][thread]: leading parts of both sites, trailing
// parts), one shared-memory access.  Each lane performs MathDF's operations in
// MathDF's order: the values are those of the one-site interpreter.
// The next load's object is fetched while the steps before it run.  Bound by
// latency at 8 warps per SM (the register file: 864 bytes per thread and three
// registers): 2,420 instructions per 32 sites (3,490), issue 35%.
// Measured against one site per thread (both with results in place): a (b + c) -
// d at 24^4 63.7 / 65.2 us, 28^4 113 / 121, 40^4 440 / 476 (506 before);
// adj(a) b + c at 40^4 348 / 406.  Programs of four registers run 6 warps and
// are slower here (a (b c - d) at 40^4 592 / 561), programs of three products
// and more too (a b c d at 32^4 228 / 223: their rolled rows keep fewer
// accumulations in flight), and small lattices, a thread's chain being longer.
struct PRegs {
  float4* base;
  int nt, tid;
  __device__ __forceinline__ dp get(int g, int r) const {
    const float4 v = base[(g * 18 + r) * nt + tid];
    return dp{make_float2(v.x, v.y), make_float2(v.z, v.w)};
  }
  __device__ __forceinline__ void put(int g, int r, const dp& v) const {
    base[(g * 18 + r) * nt + tid] = make_float4(v.h.x, v.h.y, v.l.x, v.l.y);
  }
  // element e (of 9) of a matrix register, or of its adjoint
  __device__ __forceinline__ void get_c(int g, int i, int j, bool dag, dp& re, dp& im) const {
    const int e = dag ? 3 * j + i : 3 * i + j;
    re = get(g, 2 * e);
    im = get(g, 2 * e + 1);
    const float sg = dag ? -1.0f : 1.0f;   // exact
    im.h = f2_mul_packed(im.h, make_float2(sg, sg));
    im.l = f2_mul_packed(im.l, make_float2(sg, sg));
  }
};

// accumulator -> operand (MathDF::finish)
__device__ __forceinline__ dp dp_norm(const dpa& a) {
  const float2 h = f2_add(a.S, a.lo);
  return dp{h, f2_sub(a.lo, f2_sub(h, a.S))};
}

// a + b or a - b of two operands, finished (MathDF::add twice, then finish)
template <bool NEG>
__device__ __forceinline__ dp dp_sum(const dp& a, const dp& b) {
  dpa z{a.h, a.l};
  df2_combine<NEG ? -1 : 1>(z, dpa{b.h, b.l});
  return dp_norm(z);
}

// The raw object of the next load, fetched while the steps before it run: the
// complex elements of both sites (a real field: its two values in v0[0]).
struct PNext {
  uint4 v0[9], v1[9];
  __device__ __forceinline__ void fetch(const KParams& p, const IProg& prog, int i, int64_t s0, int64_t s1,
                                        int mu) {
    const FieldDesc& f = p.leaf[prog.load_leaf[i]];
    const int w = prog.load_w[i];
    const int64_t b0 = elem_base(f, s0, mu), b1 = elem_base(f, s1, mu);
    if (w == 1) {
      const uint2 a = ld8((const char*)f.ptr + b0 * 8), b = ld8((const char*)f.ptr + b1 * 8);
      v0[0] = make_uint4(a.x, a.y, b.x, b.y);
      return;
    }
    const char* p0 = (const char*)f.ptr + b0 * 16;
    const char* p1 = (const char*)f.ptr + b1 * 16;
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      if (c == 3 && w == 6) break;
      v0[c] = ld16(p0 + c * f.s_c * 16);
      v1[c] = ld16(p1 + c * f.s_c * 16);
    }
  }
  template <int NC>
  __device__ __forceinline__ void put(const PRegs& R, int g, uint32_t& gm) const {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      gm = guard_max(guard_max(gm, v0[c].y, v0[c].w), v1[c].y, v1[c].w);
      R.put(g, 2 * c, dp_split(v0[c].x, v0[c].y, v1[c].x, v1[c].y));
      R.put(g, 2 * c + 1, dp_split(v0[c].z, v0[c].w, v1[c].z, v1[c].w));
    }
  }
};

// Reals r0 .. r0 + N - 1 of a sum (sg: +-1 of the second operand) and of a scaled
// operand: all operands first, so that their reads overlap.
template <int N>
__device__ __forceinline__ void p_add(const PRegs& R, const IIns& in, int r0, float2 sg) {
  dp a[N], b[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    a[q] = R.get(in.a, r0 + q);
    b[q] = R.get(in.b, r0 + q);
  }
#pragma unroll
  for (int q = 0; q < N; ++q)
    R.put(in.dst, r0 + q, dp_sum<false>(a[q], dp{f2_mul_packed(b[q].h, sg), f2_mul_packed(b[q].l, sg)}));
}
template <int N>
__device__ __forceinline__ void p_scale(const PRegs& R, const IIns& in, int r0, const dp& sc) {
  dp x[N];
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = R.get(in.a, r0 + q);
#pragma unroll
  for (int q = 0; q < N; ++q) {
    dpa a;
    dp_first<false>(a, sc, x[q]);
    R.put(in.dst, r0 + q, dp_norm(a));
  }
}

// The program on sites s0, s1; n0, n1: the sites after them (they are this
// thread's next ones, or these again), whose first load is fetched ahead.
__device__ __forceinline__ void p_run(const KParams& p, const IProg& prog, const PRegs& R, PNext& next,
                                      int64_t s0, int64_t s1, int64_t n0, int64_t n1, int mu, uint32_t& gm) {
  int loaded = 0;
  for (int pc = 0; pc < prog.n; ++pc) {
    const IIns in = prog.ins[pc];
    switch (in.op) {
      case I_LOAD: {
        if (in.w == 18) {
          next.put<9>(R, in.dst, gm);
        } else if (in.w == 6) {
          next.put<3>(R, in.dst, gm);
        } else {
          const uint4 v = next.v0[0];
          gm = guard_max(gm, v.y, v.w);
          R.put(in.dst, 0, dp_split(v.x, v.y, v.z, v.w));
        }
        if (++loaded < prog.nloads) next.fetch(p, prog, loaded, s0, s1, mu);
        else next.fetch(p, prog, 0, n0, n1, mu);
        break;
      }
      case I_MMUL: {
        // op(y) held, op(x) and the result one row at a time
        const bool dx = (in.adj & 1) != 0, dy = (in.adj & 2) != 0;
        dp y[18];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
          for (int k = 0; k < 3; ++k) R.get_c(in.b, j, k, dy, y[6 * j + 2 * k], y[6 * j + 2 * k + 1]);
        dp x[6];
#pragma unroll
        for (int j = 0; j < 3; ++j) R.get_c(in.a, 0, j, dx, x[2 * j], x[2 * j + 1]);
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {
          dpa re[3], im[3];
          dpa* const a[6] = {&re[0], &re[1], &re[2], &im[0], &im[1], &im[2]};
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const dp xr = x[2 * j], xm = x[2 * j + 1];
            if (i < 2) R.get_c(in.a, i + 1, j, dx, x[2 * j], x[2 * j + 1]);   // the next row's
            const dp* const yj = y + 6 * j;
            const dp* const y0[6] = {yj, yj + 2, yj + 4, yj + 1, yj + 3, yj + 5};
            const dp* const y1[6] = {yj + 1, yj + 3, yj + 5, yj, yj + 2, yj + 4};
            if (j == 0) dp_fma_shared<6, true, 0u>(a, xr, y0);
            else dp_fma_shared<6, false, 0u>(a, xr, y0);
            dp_fma_shared<6, false, 7u>(a, xm, y1);
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            R.put(in.dst, 6 * i + 2 * k, dp_norm(re[k]));
            R.put(in.dst, 6 * i + 2 * k + 1, dp_norm(im[k]));
          }
        }
        break;
      }
      case I_MVMUL: {
        const bool dx = (in.adj & 1) != 0;
        dp y[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) y[r] = R.get(in.b, r);
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {
          dpa re, im;
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            dp xr, xm;
            R.get_c(in.a, i, j, dx, xr, xm);
            if (j == 0) dp_cterm<true, 1, false, false>(re, im, xr, xm, y[2 * j], y[2 * j + 1]);
            else dp_cterm<false, 1, false, false>(re, im, xr, xm, y[2 * j], y[2 * j + 1]);
          }
          R.put(in.dst, 2 * i, dp_norm(re));
          R.put(in.dst, 2 * i + 1, dp_norm(im));
        }
        break;
      }
      case I_RMUL: {
        dpa a;
        dp_first<false>(a, R.get(in.a, 0), R.get(in.b, 0));
        R.put(in.dst, 0, dp_norm(a));
        break;
      }
      case I_ADD:
      case I_SUB: {
        const float sg = in.op == I_ADD ? 1.0f : -1.0f;   // exact
        const float2 s2 = make_float2(sg, sg);
        if (in.w == 1) {
          p_add<1>(R, in, 0, s2);
        } else {
#pragma unroll 1
          for (int r0 = 0; r0 < in.w; r0 += 6) p_add<6>(R, in, r0, s2);
        }
        break;
      }
      case I_SCALE: {
        const dp sc{make_float2(p.sch[in.arg], p.sch[in.arg]), make_float2(p.scl[in.arg], p.scl[in.arg])};
        if (in.w == 1) {
          p_scale<1>(R, in, 0, sc);
        } else {
#pragma unroll 1
          for (int r0 = 0; r0 < in.w; r0 += 6) p_scale<6>(R, in, r0, sc);
        }
        break;
      }
      default: {  // I_ADJ
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            dp re, im;
            R.get_c(in.a, i, j, true, re, im);
            R.put(in.dst, 2 * (3 * i + j), re);
            R.put(in.dst, 2 * (3 * i + j) + 1, im);
          }
        break;
      }
    }
  }
}

__device__ __forceinline__ void p_store_root(const KParams& p, const IProg& prog, const PRegs& R,
                                             int64_t s0, int64_t s1, bool has1, int mu) {
  char* base = (char*)p.dst.ptr;
  const int64_t e0 = elem_base(p.dst, s0, mu), e1 = elem_base(p.dst, s1, mu);
  if (prog.root_kind == KR) {
    const dp v = R.get(prog.root, 0);
    double d0, d1;
    df2_to_double(dpa{v.h, v.l}, d0, d1);
    st8(base + e0 * 8, make_uint2((uint32_t)__double2loint(d0), (uint32_t)__double2hiint(d0)));
    if (has1) st8(base + e1 * 8, make_uint2((uint32_t)__double2loint(d1), (uint32_t)__double2hiint(d1)));
    return;
  }
  const int nc = prog.root_kind == KV ? 3 : 9;
#pragma unroll 1
  for (int c0 = 0; c0 < nc; c0 += 3) {
    dp z[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) z[q] = R.get(prog.root, 2 * c0 + q);
#pragma unroll
    for (int q = 0; q < 3; ++q)
      pair_store_c(base, e0 + (c0 + q) * p.dst.s_c, e1 + (c0 + q) * p.dst.s_c, has1,
                   dpa{z[2 * q].h, z[2 * q].l}, dpa{z[2 * q + 1].h, z[2 * q + 1].l});
  }
}

__global__ void __launch_bounds__(128) k_interp_pair(const __grid_constant__ KParams p,
                                                     const __grid_constant__ IProg prog) {
  extern __shared__ __align__(16) unsigned char i_smem[];
  const int nt = (int)blockDim.x, tid = (int)threadIdx.x;
  const PRegs R{reinterpret_cast<float4*>(i_smem), nt, tid};
  const int mu = blockIdx.y;
  const int64_t step = (int64_t)gridDim.x * 2 * nt;
  int64_t s0 = (int64_t)blockIdx.x * 2 * nt + tid;
  if (s0 >= p.nvec) return;
  PNext next;
  next.fetch(p, prog, 0, s0, s0 + nt < p.nvec ? s0 + nt : s0, mu);
  for (; s0 < p.nvec; s0 += step) {
    const bool has1 = s0 + nt < p.nvec;
    const int64_t s1 = has1 ? s0 + nt : s0;
    const int64_t n0 = s0 + step < p.nvec ? s0 + step : s0, n1 = n0 + nt < p.nvec ? n0 + nt : n0;
    uint32_t gm = p.gscal;
    p_run(p, prog, R, next, s0, s1, n0, n1, mu, gm);
    if (gm >= p.ghi) {
      // native FP64, one site after the other
      i_site_f64<16, true>(p, prog, i_smem, nt, tid, s0, mu);
      if (has1) i_site_f64<16, true>(p, prog, i_smem, nt, tid, s1, mu);
    } else {
      p_store_root(p, prog, R, s0, s1, has1, mu);
    }
  }
}

// ------------------------------------------------------------------ host
namespace {
template <class M>
cudaError_t launch_interp(const KParams& p, const IProg& prog, cudaStream_t st) {
  static_assert(!M::kGuard || sizeof(typename M::R) >= sizeof(double),
                "the range guard reruns the program in FP64 on the same register file");
  // shared memory: nregs registers of 18 reals per thread; 128 threads per
  // block while that fits in 200 KB, fewer for long programs
  const size_t per_thread = (size_t)prog.nregs * 18 * sizeof(typename M::R);
  int threads = 128;
  while (threads > 32 && per_thread * threads > (200u << 10)) threads /= 2;
  const size_t smem = per_thread * threads;
  const void* k = (const void*)&k_interp<M>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 1;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int64_t blocks = (int64_t)per_sm * sm_count();               // one wave, grid-stride
  const int64_t need = (p.nvec + threads - 1) / threads;
  if (blocks > need) blocks = need;
  if (blocks < 1) blocks = 1;
  k_interp<M><<<dim3((unsigned)blocks, (unsigned)p.nmu), threads, smem, st>>>(p, prog);
  return cudaGetLastError();
}

// Two sites per thread: 288 bytes per register and thread.  The block size with
// the most warps per SM (the register file in shared memory sets it), larger
// blocks first.
cudaError_t launch_interp_pair(const KParams& p, const IProg& prog, cudaStream_t st) {
  struct Shape {
    int threads, per_sm;
  };
  static std::mutex mu;
  static Shape shapes[kPairRegs + 1];   // by registers used, looked up once each
  const size_t per_thread = (size_t)prog.nregs * 18 * sizeof(float4);
  Shape sh;
  {
    std::lock_guard<std::mutex> lk(mu);
    Shape& c = shapes[prog.nregs];
    if (c.threads == 0) {
      cudaError_t e = cudaFuncSetAttribute(k_interp_pair, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           smem_optin());
      Shape best{0, 0};
      for (int t = 128; t >= 32 && e == cudaSuccess; t -= 32) {
        if (per_thread * t > (size_t)smem_optin()) continue;
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_interp_pair, t, per_thread * t);
        if (n * t > best.per_sm * best.threads) best = Shape{t, n};
      }
      if (e != cudaSuccess) return e;
      if (best.threads == 0) return cudaErrorInvalidConfiguration;
      c = best;
    }
    sh = c;
  }
  const int threads = sh.threads, per_sm = sh.per_sm;
  int64_t blocks = (int64_t)per_sm * sm_count();               // one wave, grid-stride
  const int64_t need = (p.nvec + 2 * threads - 1) / (2 * threads);
  if (blocks > need) blocks = need;
  if (blocks < 1) blocks = 1;
  k_interp_pair<<<dim3((unsigned)blocks, (unsigned)p.nmu), threads, per_thread * threads, st>>>(p, prog);
  return cudaGetLastError();
}
}  // namespace

// Degree of a runtime tree (most factors in one term), as Degree<> of the
// compiled trees: it sets the range guard's bound.
static int degree(const su3s_expr* e) {
  switch (e->op) {
    case 0: return 1;
    case 1: return degree(e->a) + degree(e->b);
    case 4: return degree(e->a) + 1;
    case 5: return degree(e->a);
    default: {
      const int a = degree(e->a), b = degree(e->b);
      return a > b ? a : b;
    }
  }
}

int interp_eval(const su3s_expr* e, const Canon& c, su3s_field* dest, int math, cudaStream_t st) {
  // Two sites per thread from kPairSites on, for programs of at most two products
  // whose registers let 8 warps per SM run; else one site per thread.
  const bool large = math == MATH_DF && (int64_t)dest->Vpad * dest->nmu >= kPairSites;
  IProg prog;
  bool pairs;
  if (interp_program(e, c, large, &prog, &pairs))
    return fail(SU3S_EUNSUPPORTED, "expression too large for the interpreter (%d registers, %d steps)",
                kIRegs, kIMax);
  KParams p;
  build_params(c, dest, 1, &p);
  p.ghi = guard_hi(degree(e));
  cudaError_t ce = math == MATH_F64  ? launch_interp<MathF64>(p, prog, st)
                   : math == MATH_FX ? launch_interp<MathFX>(p, prog, st)
                                     : pairs ? launch_interp_pair(p, prog, st)
                                               : launch_interp<MathDFScalar>(p, prog, st);
  if (ce != cudaSuccess) return cuda_fail(ce, "interpreter kernel launch");
  return SU3S_OK;
}

}  // namespace su3s
