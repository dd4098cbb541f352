// Whole-field reduction (the loss sum_x Re tr(X^dagger Y)) and projection of
// matrix fields back to SU(3).
#include <math.h>

#include "dev_convert.cuh"
#include "dev_kernels.cuh"
#include "internal.h"

namespace su3s {

constexpr int kRedThreads = 256;

// Fixed-order block reduction of per-thread sums; the total in thread 0.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[kRedThreads / 32];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = sh[0];
#pragma unroll
  for (int w = 1; w < kRedThreads / 32; ++w) t += sh[w];
  return t;
}

// Sum over the real sites of link blockIdx.y and the NC complex components of
// x*y (FP64 storage; NC = 0: one real), one number per block.
// HBM-bound: all 2 NC loads of a site are issued before its products, and links
// are a grid dimension, so that no site index is divided by the volume.  Two
// blocks per SM cover HBM's latency; each further block costs small fields its
// start (vectors of 4 links on 16^3 x 32: 9.9 us, 10.8 with three, 12.2 with
// four; two or four vectors per thread at a time 11.2, 11.8).
// Both kernels, before and now: 48^4 matrices 327 -> 213 us (7.2 TB/s), 48^4
// vectors of 4 links 435 -> 284, 16^3 x 32 12.1 -> 9.9, 4^4 6.3 -> 4.3.
template <int NC>
__global__ void __launch_bounds__(kRedThreads, 2)
    k_redot_partial(FieldDesc x, FieldDesc y, int64_t V, double* __restrict__ partial) {
  // the final sum's block may take its place; it waits for this grid's results
  cudaTriggerProgrammaticLaunchCompletion();
  const int mu = blockIdx.y;
  const int64_t stride = (int64_t)gridDim.x * kRedThreads;
  double acc0 = 0.0, acc1 = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * kRedThreads + threadIdx.x; s < V; s += stride) {
    const int64_t bx = fbase(x, s, mu), by = fbase(y, s, mu);
    if constexpr (NC == 0) {
      acc0 = fma(reinterpret_cast<const double*>(x.ptr)[bx], reinterpret_cast<const double*>(y.ptr)[by], acc0);
    } else {
      double2 a[NC], b[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        a[c] = reinterpret_cast<const double2*>(x.ptr)[bx + c * x.s_c];
        b[c] = reinterpret_cast<const double2*>(y.ptr)[by + c * y.s_c];
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        acc0 = fma(a[c].x, b[c].x, acc0);
        acc1 = fma(a[c].y, b[c].y, acc1);
      }
    }
  }
  const double t = block_sum(acc0 + acc1);
  if (threadIdx.x == 0) partial[blockIdx.x + blockIdx.y * gridDim.x] = t;
}

__global__ void __launch_bounds__(kRedThreads)
    k_redot_final(const double* partial, int n, double* __restrict__ out) {
  cudaGridDependencySynchronize();
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += kRedThreads) acc += partial[i];
  const double t = block_sum(acc);
  if (threadIdx.x == 0) *out = t;
}

// One wave of blocks over all links, no more than there are sites for.
static dim3 redot_grid(const su3s_field* x) {
  int64_t nb = (2 * (int64_t)sm_count() + x->nmu - 1) / x->nmu;
  const int64_t need = (x->V + kRedThreads - 1) / kRedThreads;
  if (nb > need) nb = need;
  return dim3((unsigned)(nb < 1 ? 1 : nb), (unsigned)x->nmu);
}

cudaError_t launch_redot(const su3s_field* x, const su3s_field* y, double* out, double* partial,
                         dim3 grid, cudaStream_t st) {
  switch (x->kind) {
    case SU3S_MATRIX: k_redot_partial<9><<<grid, kRedThreads, 0, st>>>(x->desc, y->desc, x->V, partial); break;
    case SU3S_VECTOR: k_redot_partial<3><<<grid, kRedThreads, 0, st>>>(x->desc, y->desc, x->V, partial); break;
    default: k_redot_partial<0><<<grid, kRedThreads, 0, st>>>(x->desc, y->desc, x->V, partial);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // The final sum's block is resident when the partial sums end: 4^4 matrices
  // 6.9 -> 4.8 us with the shorter block sum.
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(kRedThreads);
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_redot_final, (const double*)partial, (int)(grid.x * grid.y), out);
}

int check_redot(const su3s_field* x, const su3s_field* y, const double* out) {
  if (!x || !y || !out) return fail(SU3S_EINVAL, "null argument");
  if (x->kind != y->kind) return fail(SU3S_ETYPE, "fields of different kinds");
  if (x->prec != SU3S_F64 || y->prec != SU3S_F64)
    return fail(SU3S_EUNSUPPORTED, "reduction needs FP64 storage");
  return check_same_shape(x, y, true);
}

// ------------------------------------------------------------ reunitarise
// The 9 elements of a stored matrix, and back.
template <int PREC>
__device__ __forceinline__ void reunit_load(const FieldDesc& f, int64_t b, double* r) {
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const double2 v = get_complex<PREC>(f.ptr, b + c * f.s_c);
    r[2 * c] = v.x;
    r[2 * c + 1] = v.y;
  }
}
template <int PREC>
__device__ __forceinline__ void reunit_store(const FieldDesc& f, int64_t b, const double* r) {
#pragma unroll
  for (int c = 0; c < 9; ++c) put_complex<PREC>(f.ptr, b + c * f.s_c, r[2 * c], r[2 * c + 1]);
}

// Projection of one matrix (rows r[0..5], r[6..11], r[12..17]) by the
// definition: Gram-Schmidt over rows, two sweeps, then division by the
// principal cube root of the determinant's phase.  Out of line and from the
// field itself: it serves the matrices whose norms leave the range in which
// reunit_fast is the same projection (see there).
template <int PREC>
__device__ __noinline__ void reunit_sweeps(const FieldDesc& src, const FieldDesc& dst, int64_t bs,
                                           int64_t bd) {
  double r[18];
  reunit_load<PREC>(src, bs, r);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int rep = 0; rep < 2; ++rep)
#pragma unroll
      for (int p = 0; p < i; ++p) {
        double cr = 0.0, ci = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const double pr = r[6 * p + 2 * j], pi = r[6 * p + 2 * j + 1];
          const double xr = r[6 * i + 2 * j], xi = r[6 * i + 2 * j + 1];
          cr += pr * xr + pi * xi;
          ci += pr * xi - pi * xr;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const double pr = r[6 * p + 2 * j], pi = r[6 * p + 2 * j + 1];
          r[6 * i + 2 * j] -= cr * pr - ci * pi;
          r[6 * i + 2 * j + 1] -= cr * pi + ci * pr;
        }
      }
    double nn = 0.0;
#pragma unroll
    for (int j = 0; j < 6; ++j) nn += r[6 * i + j] * r[6 * i + j];
    const double inv = rsqrt(nn);
#pragma unroll
    for (int j = 0; j < 6; ++j) r[6 * i + j] *= inv;
  }
  double dr = 0.0, di = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int a = (j + 1) % 3, b = (j + 2) % 3;
    const double xr = r[6 + 2 * a] * r[12 + 2 * b] - r[6 + 2 * a + 1] * r[12 + 2 * b + 1] -
                      (r[6 + 2 * b] * r[12 + 2 * a] - r[6 + 2 * b + 1] * r[12 + 2 * a + 1]);
    const double xi = r[6 + 2 * a] * r[12 + 2 * b + 1] + r[6 + 2 * a + 1] * r[12 + 2 * b] -
                      (r[6 + 2 * b] * r[12 + 2 * a + 1] + r[6 + 2 * b + 1] * r[12 + 2 * a]);
    dr += r[2 * j] * xr - r[2 * j + 1] * xi;
    di += r[2 * j] * xi + r[2 * j + 1] * xr;
  }
  const double phi = atan2(di, dr);
  double sn, cs;
  sincos(-phi / 3.0, &sn, &cs);
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const double re = r[2 * c], im = r[2 * c + 1];
    r[2 * c] = cs * re - sn * im;
    r[2 * c + 1] = cs * im + sn * re;
  }
  reunit_store<PREC>(dst, bd, r);
}

// a = b times c, complex
__device__ __forceinline__ void zmul(double& ar, double& ai, double br, double bi, double cr,
                                     double ci) {
  const double re = fma(br, cr, -(bi * ci));
  ai = fma(br, ci, bi * cr);
  ar = re;
}

// The part of row b along row a (not normalised; rn = 1/|a|^2) taken out of b:
// one Gram-Schmidt sweep.  Returns that part's squared norm.
__device__ __forceinline__ double project_out(const double* a, double rn, double* b) {
  double cr = 0.0, ci = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    cr = fma(a[2 * j], b[2 * j], fma(a[2 * j + 1], b[2 * j + 1], cr));
    ci = fma(a[2 * j], b[2 * j + 1], fma(-a[2 * j + 1], b[2 * j], ci));
  }
  const double part = fma(cr, cr, ci * ci) * rn;
  cr *= rn;
  ci *= rn;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    b[2 * j] = fma(-cr, a[2 * j], fma(ci, a[2 * j + 1], b[2 * j]));
    b[2 * j + 1] = fma(-cr, a[2 * j + 1], fma(-ci, a[2 * j], b[2 * j + 1]));
  }
  return part;
}
__device__ __forceinline__ double row_norm2(const double* a) {
  double n = 0.0;
#pragma unroll
  for (int j = 0; j < 6; ++j) n = fma(a[j], a[j], n);
  return n;
}

// 1/sqrt(n) as y (1 + g): y the hardware's approximation cut to its leading word
// (21 bits, so that y^2 is exact), e = 1 - n y^2, and g the series of
// (1 - e)^(-1/2) - 1, exact to e^3 < 2^-56.  Kept in two parts, the factor enters
// what it scales with one rounding.  1/n = y^2 / (1 - e).
struct Rsqrt {
  double y, g, w, e;   // w = y^2
  __device__ __forceinline__ explicit Rsqrt(double n) {
    double a;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(a) : "d"(n));
    y = __hiloint2double(__double2hiint(a), 0);
    w = y * y;
    e = fma(-n, w, 1.0);
    g = e * fma(e, 0.375, 0.5);
  }
  __device__ __forceinline__ double near() const { return fma(0.5 * y, e, y); }   // to e^2
  __device__ __forceinline__ double inverse() const { return fma(w, fma(e, e, e), w); }
  // (t + h) / sqrt(n), q = t + h rounded
  __device__ __forceinline__ double scale(double t, double h, double q) const {
    return fma(t, y, y * fma(q, g, h));
  }
};

// The same projection with fewer FP64 operations: the FP64 pipe bounds the
// kernel (91% busy; 2.59 M FP64 matrices: 1,989 us by the definition's sweeps with
// FP64 atan2 and sincos, which stay for the cases below, 948 here).
// Row 1 takes a second sweep only where the first took out a sixteenth or more
// of what it left (in norm squared): else one sweep leaves no more of row 0 than
// its own rounding, as two do.  Of row 2 only a phase is free: orthonormal to
// rows 0 and 1 it is e^{i alpha} w, w = conj(r0 x r1), so Gram-Schmidt's two
// sweeps and normalisation come down to the direction of d = <w, row 2>, and
// e^{i alpha} = d/|d| is also the determinant.  Dividing by its principal cube
// root leaves rows 0, 1 times q and w times conj(q)^2, q = e^{-i alpha/3}.  q is
// formed in FP32 (atan2f, sincosf: the branch of the cube root is that of the
// signs of d), rounded to multiples of 2^-22 (its square is then exact in FP64)
// and refined by one step on q^3 d/|d| = 1: with q^3 d/|d| = 1 + z, |z| < 1e-6,
// q (1 - z/3 + 2/9 z^2) is exact to z^3 < 1e-18.  d/|d| is brought back to the
// unit circle, and q and the norms' reciprocal roots kept in two parts until they
// are one factor of a row, as what such a factor rounds by is an error of the whole
// row.  rms error against extended precision and, in brackets, the definition's in
// FP64: projected matrices 3.40e-17 (3.45e-17), rounded to FP32 4.08e-17
// (4.31e-17), with noise of 1e-6 to 1e-1 4.22 to 4.28e-17 (4.48 to 4.52e-17),
// Gaussian 5.88e-17 (6.56e-17).  With rounded reciprocal roots noisy matrices had
// 4.69e-17, in the same time (951 us).
// Returns false where a norm is NaN, zero, or so large or small that it could
// overflow or underflow here and not in the definition.
__device__ __forceinline__ bool reunit_fast(double* r) {
  double* a = r;  // rows 0 and 1, not normalised until the end
  double* b = r + 6;
  const double n0 = row_norm2(a);
  const Rsqrt s0(n0);
  const double rn0 = s0.inverse();
  const double part = project_out(a, rn0, b);
  double n1 = row_norm2(b);
  if (part > n1 * 0.0625) {
    project_out(a, rn0, b);
    n1 = row_norm2(b);
  }
  const Rsqrt s1(n1);
  // x = a x b; d = sum_j x_j row2_j
  double x[6], dr = 0.0, di = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int k = (j + 1) % 3, l = (j + 2) % 3;
    x[2 * j] = fma(a[2 * k], b[2 * l], fma(-a[2 * k + 1], b[2 * l + 1],
               fma(-a[2 * l], b[2 * k], a[2 * l + 1] * b[2 * k + 1])));
    x[2 * j + 1] = fma(a[2 * k], b[2 * l + 1], fma(a[2 * k + 1], b[2 * l],
                   fma(-a[2 * l], b[2 * k + 1], -(a[2 * l + 1] * b[2 * k]))));
    dr = fma(x[2 * j], r[12 + 2 * j], fma(-x[2 * j + 1], r[12 + 2 * j + 1], dr));
    di = fma(x[2 * j], r[12 + 2 * j + 1], fma(x[2 * j + 1], r[12 + 2 * j], di));
  }
  const double nd = fma(dr, dr, di * di);
  const double invd = Rsqrt(nd).near();   // |d|'s rest goes with the step to the unit circle
  if (!(n0 > 0x1p-200 && n0 < 0x1p200 && n1 > 0x1p-200 && n1 < 0x1p200 && nd > 0x1p-800 &&
        nd < 0x1p800))
    return false;
  double er = dr * invd, ei = di * invd;
  const double ue = -0.5 * fma(er, er, fma(ei, ei, -1.0));
  er = fma(er, ue, er);
  ei = fma(ei, ue, ei);
  float qs, qc;
  sincosf(atan2f(__double2float_rn(ei), __double2float_rn(er)) * (-1.0f / 3.0f), &qs, &qc);
  const double tr = (double)__fsub_rn(__fadd_rn(qc, 3.0f), 3.0f);
  const double ti = (double)__fsub_rn(__fadd_rn(qs, 3.0f), 3.0f);
  double sr = fma(tr, tr, -(ti * ti)), si = (tr + tr) * ti, zr, zi;
  zmul(zr, zi, sr, si, tr, ti);
  sr = fma(zr, er, fma(-zi, ei, -1.0));
  si = fma(zr, ei, zi * er);
  // 1 - z/3 + 2/9 z^2 = 1 + z (2/9 z - 1/3)
  zmul(zr, zi, sr, si, fma(sr, 2.0 / 9.0, -1.0 / 3.0), si * (2.0 / 9.0));
  const double hr = fma(tr, zr, -(ti * zi)), hi = fma(tr, zi, ti * zr);  // q = t + h
  const double qr = tr + hr, qi = ti + hi;
  // rows 0, 1: q over the norms, times the rows; row 2: e^{i alpha} q conj(x) /
  // |x|, the conjugate of x times conj(e^{i alpha} q) over its norm
  const Rsqrt s2(row_norm2(x));
  const double yg = s2.y * s2.g;
  double pr = fma(er, qr, -(ei * qi)), pi = -fma(er, qi, ei * qr);
  pr = fma(pr, s2.y, pr * yg);
  pi = fma(pi, s2.y, pi * yg);
  const double q0r = s0.scale(tr, hr, qr), q0i = s0.scale(ti, hi, qi);
  const double q1r = s1.scale(tr, hr, qr), q1i = s1.scale(ti, hi, qi);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    zmul(r[2 * j], r[2 * j + 1], a[2 * j], a[2 * j + 1], q0r, q0i);
    zmul(r[6 + 2 * j], r[6 + 2 * j + 1], b[2 * j], b[2 * j + 1], q1r, q1i);
    zmul(r[12 + 2 * j], r[12 + 2 * j + 1], x[2 * j], x[2 * j + 1], pr, pi);
    r[12 + 2 * j + 1] = -r[12 + 2 * j + 1];
  }
  return true;
}

template <int PREC>
__global__ void __launch_bounds__(256) k_reunit(FieldDesc src, FieldDesc dst, int64_t V, int nmu) {
  const int64_t n = V * nmu;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
    const int mu = (int)(q / V);
    const int64_t s = q - (int64_t)mu * V;
    const int64_t bs = fbase(src, s, mu), bd = fbase(dst, s, mu);
    double r[18];
    reunit_load<PREC>(src, bs, r);
    if (reunit_fast(r)) reunit_store<PREC>(dst, bd, r);
    else reunit_sweeps<PREC>(src, dst, bs, bd);
  }
}

template <int PREC>
static cudaError_t reunit_t(const su3s_field* src, su3s_field* dst, cudaStream_t st) {
  const int64_t n = src->V * src->nmu;
  int64_t nb = (n + 255) / 256;
  if (nb > (int64_t)sm_count() * 16) nb = (int64_t)sm_count() * 16;
  if (nb < 1) nb = 1;
  k_reunit<PREC><<<(unsigned)nb, 256, 0, st>>>(src->desc, dst->desc, src->V, src->nmu);
  return cudaGetLastError();
}

}  // namespace su3s

using namespace su3s;

SU3S_EXPORT int su3s_field_redot(const su3s_field* x, const su3s_field* y, double* dev_out,
                                 void* stream) {
  int rc = check_redot(x, y, dev_out);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const dim3 grid = redot_grid(x);
  void* partial = nullptr;
  cudaError_t e = scratch_alloc(&partial, (size_t)grid.x * grid.y * sizeof(double), st);
  if (e != cudaSuccess) return fail(SU3S_ENOMEM, "reduction scratch: %s", cudaGetErrorString(e));
  e = launch_redot(x, y, dev_out, (double*)partial, grid, st);
  cudaError_t e2 = scratch_free(partial, st);
  if (e != cudaSuccess) return cuda_fail(e, "reduction kernels");
  if (e2 != cudaSuccess) return cuda_fail(e2, "reduction scratch release");
  return SU3S_OK;
}

SU3S_EXPORT int su3s_reunitarize(su3s_field* dst, const su3s_field* src, void* stream) {
  if (!dst || !src) return fail(SU3S_EINVAL, "null argument");
  if (src->kind != SU3S_MATRIX || dst->kind != SU3S_MATRIX)
    return fail(SU3S_ETYPE, "projection to SU(3) needs matrix fields");
  int rc = check_same_shape(src, dst, true);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  switch (src->prec) {
    case SU3S_F64: e = reunit_t<P_F64>(src, dst, st); break;
    case SU3S_F32: e = reunit_t<P_F32>(src, dst, st); break;
    case SU3S_BF16: e = reunit_t<P_BF16>(src, dst, st); break;
    case SU3S_F16: e = reunit_t<P_F16>(src, dst, st); break;
    default: return fail(SU3S_EUNSUPPORTED, "two-row storage is special unitary by construction");
  }
  if (e != cudaSuccess) return cuda_fail(e, "projection kernel");
  return SU3S_OK;
}
