// Conversion between the canonical AoS FP64 array and a field's device layout
// and storage precision (the scalar/vector data layouts of Sec. 4-5: the
// canonical array is the naive AoS order, the field is the coalesced one).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dev_convert.cuh"
#include "dev_kernels.cuh"
#include "internal.h"

namespace su3s {

// Both directions are transposes: a site's elements are contiguous in the host
// order, an element's sites in the field.  A block takes a tile of consecutive
// sites through shared memory ([site][element], the element stride odd, so
// that neither side has bank conflicts): one side of the copy walks the host
// array's run of the tile, the other whole 32-site rows of an element, and both
// are full 128-byte lines.  HBM-bound.  Measured, FP64 links of 23x25x24x47
// (747 MB of canonical array and field): pack 379 -> 127 us, unpack 231 -> 119 us
// against one element per thread in host order (16-byte pieces of the field at a
// time, four 64-bit divisions each).

// One host element and its stored form.  H: the host array's element, moved as
// two doubles when the array is not aligned to it.
template <int PREC>
struct CanonElem {  // canonical complex <-> stored complex
  using H = double2;
  __device__ static __forceinline__ H load(const void* p, int64_t i, bool aligned) {
    if (aligned) return reinterpret_cast<const double2*>(p)[i];
    const double* q = reinterpret_cast<const double*>(p) + 2 * i;
    return make_double2(q[0], q[1]);
  }
  __device__ static __forceinline__ void store(void* p, int64_t i, H v, bool aligned) {
    if (aligned) {
      reinterpret_cast<double2*>(p)[i] = v;
    } else {
      double* q = reinterpret_cast<double*>(p) + 2 * i;
      q[0] = v.x;
      q[1] = v.y;
    }
  }
  __device__ static __forceinline__ void put(void* f, int64_t e, H v) { put_complex<PREC>(f, e, v.x, v.y); }
  __device__ static __forceinline__ H get(const void* f, int64_t e) { return get_complex<PREC>(f, e); }
};
template <typename T>
struct RawElem {  // stored bytes unchanged (and real fields: one double)
  using H = T;
  __device__ static __forceinline__ H load(const void* p, int64_t i, bool) {
    return reinterpret_cast<const T*>(p)[i];
  }
  __device__ static __forceinline__ void store(void* p, int64_t i, H v, bool) {
    reinterpret_cast<T*>(p)[i] = v;
  }
  __device__ static __forceinline__ void put(void* f, int64_t e, H v) { reinterpret_cast<T*>(f)[e] = v; }
  __device__ static __forceinline__ H get(const void* f, int64_t e) {
    return reinterpret_cast<const T*>(f)[e];
  }
};

constexpr int kTileThreads = 128;

// Sites of a block's tile: 32 k, with about as many elements as a tile of 32
// sites of 4 matrices (1,152, nine loads per thread in flight).
struct TileGeo {
  int64_t V, Vpad;
  int nmu, nc_host, nc_field;  // elements per site object in the host array and in the field
  int sites;                   // multiple of 32
  int E, P;                    // host elements per site, and the padded (odd) stride
  uint32_t magic;              // i / E = umulhi(i, magic) for i < sites * E
  bool aligned;                // host array aligned to its element
};

// Host order -> field; pad sites are zeroed.  Host elements past nc_field
// (row 2 of a two-row matrix) are skipped.
template <class El>
__global__ void __launch_bounds__(kTileThreads)
    k_put_tile(FieldDesc d, const void* __restrict__ host, TileGeo g) {
  using H = typename El::H;
  extern __shared__ __align__(16) unsigned char t_smem[];
  H* sm = reinterpret_cast<H*>(t_smem);
  const int64_t s0 = (int64_t)blockIdx.x * g.sites;
  const int64_t left = g.V - s0;
  const int n = (int)(left < 0 ? 0 : left < g.sites ? left : g.sites) * g.E;
  const int64_t base = s0 * g.E;
  for (int i0 = threadIdx.x; i0 < n; i0 += 4 * kTileThreads) {
    H v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u * kTileThreads < n) v[u] = El::load(host, base + i0 + u * kTileThreads, g.aligned);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * kTileThreads;
      const int s = g.E > 1 ? (int)__umulhi((uint32_t)i, g.magic) : i;
      if (i < n) sm[s * g.P + (i - s * g.E)] = v[u];
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, k = g.sites / 32;
  for (int w = threadIdx.x / 32; w < g.nmu * g.nc_field * k; w += kTileThreads / 32) {
    const int r = w / k, mu = r / g.nc_field, c = r - mu * g.nc_field;
    const int sl = (w - r * k) * 32 + lane;
    const int64_t s = s0 + sl;
    if (s < g.Vpad)
      El::put(d.ptr, fbase(d, s, mu) + c * d.s_c,
              s < g.V ? sm[sl * g.P + mu * g.nc_host + c] : H{});
  }
}

// Field -> host order.  C12: one matrix per thread, row 2 rebuilt in FP64.
template <class El, bool C12>
__global__ void __launch_bounds__(kTileThreads)
    k_get_tile(FieldDesc d, void* __restrict__ host, TileGeo g) {
  using H = typename El::H;
  extern __shared__ __align__(16) unsigned char t_smem[];
  H* sm = reinterpret_cast<H*>(t_smem);
  const int64_t s0 = (int64_t)blockIdx.x * g.sites;
  const int64_t left = g.V - s0;
  const int ns = (int)(left < g.sites ? left : g.sites);
  const int lane = threadIdx.x & 31, k = g.sites / 32;
  constexpr int NW = kTileThreads / 32;
  if constexpr (C12) {
    for (int w = threadIdx.x / 32; w < g.nmu * k; w += NW) {
      const int mu = w / k, sl = (w - mu * k) * 32 + lane;
      if (sl >= ns) continue;
      const int64_t b = fbase(d, s0 + sl, mu);
      double u[18];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const double2 v = El::get(d.ptr, b + c * d.s_c);
        u[2 * c] = v.x;
        u[2 * c + 1] = v.y;
      }
      rebuild_row2<MathF64>(u);
#pragma unroll
      for (int c = 0; c < 9; ++c) sm[sl * g.P + mu * 9 + c] = make_double2(u[2 * c], u[2 * c + 1]);
    }
  } else {
    const int rows = g.nmu * g.nc_field * k;
    for (int w0 = threadIdx.x / 32; w0 < rows; w0 += 4 * NW) {
      H v[4];
      int at[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int w = w0 + u * NW, r = w / k, mu = r / g.nc_field, c = r - mu * g.nc_field;
        const int sl = (w - r * k) * 32 + lane;
        at[u] = w < rows && sl < ns ? sl * g.P + mu * g.nc_host + c : -1;
        if (at[u] >= 0) v[u] = El::get(d.ptr, fbase(d, s0 + sl, mu) + c * d.s_c);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (at[u] >= 0) sm[at[u]] = v[u];
    }
  }
  __syncthreads();
  const int64_t base = s0 * g.E;
  const int n = ns * g.E;
  for (int i = threadIdx.x; i < n; i += kTileThreads) {
    const int s = g.E > 1 ? (int)__umulhi((uint32_t)i, g.magic) : i;
    El::store(host, base + i, sm[s * g.P + (i - s * g.E)], g.aligned);
  }
}

static TileGeo tile_geo(const su3s_field* f, int nc_host, const void* host, int host_bytes) {
  TileGeo g;
  g.V = f->V;
  g.Vpad = f->Vpad;
  g.nmu = f->nmu;
  g.nc_host = nc_host;
  g.nc_field = f->ncomp;
  g.E = f->nmu * nc_host;   // 1..72
  g.P = g.E | 1;
  int k = 36 / g.E;
  g.sites = 32 * (k < 1 ? 1 : k > 8 ? 8 : k);
  g.magic = g.E > 1 ? (uint32_t)((1ull << 32) / (uint32_t)g.E + 1) : 0;
  g.aligned = ((uintptr_t)host & (uintptr_t)(host_bytes - 1)) == 0;
  return g;
}

template <class El>
static cudaError_t put_tile(const su3s_field* f, const void* host, int nc_host, cudaStream_t st) {
  using H = typename El::H;
  const TileGeo g = tile_geo(f, nc_host, host, (int)sizeof(H));
  const int64_t nb = (g.Vpad + g.sites - 1) / g.sites;
  if (nb > 0)
    k_put_tile<El><<<(unsigned)nb, kTileThreads, (size_t)g.sites * g.P * sizeof(H), st>>>(f->desc, host, g);
  return cudaGetLastError();
}

template <class El, bool C12>
static cudaError_t get_tile(const su3s_field* f, void* host, int nc_host, cudaStream_t st) {
  using H = typename El::H;
  const TileGeo g = tile_geo(f, nc_host, host, (int)sizeof(H));
  const int64_t nb = (g.V + g.sites - 1) / g.sites;
  if (nb > 0)
    k_get_tile<El, C12><<<(unsigned)nb, kTileThreads, (size_t)g.sites * g.P * sizeof(H), st>>>(f->desc, host, g);
  return cudaGetLastError();
}

static int canon_comp(const su3s_field* f) {
  return f->kind == SU3S_MATRIX ? 9 : f->kind == SU3S_VECTOR ? 3 : 1;
}

cudaError_t launch_pack(const su3s_field* f, const double* canon, cudaStream_t st) {
  const int nc = canon_comp(f);
  if (f->kind == SU3S_REAL) return put_tile<RawElem<double>>(f, canon, nc, st);
  switch (f->prec) {
    case SU3S_F64:
    case SU3S_F64_C12: return put_tile<CanonElem<P_F64>>(f, canon, nc, st);
    case SU3S_F32:
    case SU3S_F32_C12: return put_tile<CanonElem<P_F32>>(f, canon, nc, st);
    case SU3S_BF16: return put_tile<CanonElem<P_BF16>>(f, canon, nc, st);
    default: return put_tile<CanonElem<P_F16>>(f, canon, nc, st);
  }
}

cudaError_t launch_unpack(const su3s_field* f, double* canon, cudaStream_t st) {
  const int nc = canon_comp(f);
  if (f->kind == SU3S_REAL) return get_tile<RawElem<double>, false>(f, canon, nc, st);
  switch (f->prec) {
    case SU3S_F64: return get_tile<CanonElem<P_F64>, false>(f, canon, nc, st);
    case SU3S_F32: return get_tile<CanonElem<P_F32>, false>(f, canon, nc, st);
    case SU3S_BF16: return get_tile<CanonElem<P_BF16>, false>(f, canon, nc, st);
    case SU3S_F16: return get_tile<CanonElem<P_F16>, false>(f, canon, nc, st);
    case SU3S_F64_C12: return get_tile<CanonElem<P_F64>, true>(f, canon, nc, st);
    default: return get_tile<CanonElem<P_F32>, true>(f, canon, nc, st);
  }
}

// Stored-format transfer.  The compact array is site-major like the canonical
// one, but holds per (site, link) only the ncomp stored elements (two rows of a
// C12 matrix), each as the field stores it.
cudaError_t launch_put_stored(const su3s_field* f, const void* src, cudaStream_t st) {
  switch (f->elem_bytes) {
    case 16: return put_tile<RawElem<uint4>>(f, src, f->ncomp, st);
    case 8: return put_tile<RawElem<uint2>>(f, src, f->ncomp, st);
    default: return put_tile<RawElem<uint32_t>>(f, src, f->ncomp, st);
  }
}

cudaError_t launch_get_stored(const su3s_field* f, void* dst, cudaStream_t st) {
  switch (f->elem_bytes) {
    case 16: return get_tile<RawElem<uint4>, false>(f, dst, f->ncomp, st);
    case 8: return get_tile<RawElem<uint2>, false>(f, dst, f->ncomp, st);
    default: return get_tile<RawElem<uint32_t>, false>(f, dst, f->ncomp, st);
  }
}

}  // namespace su3s
