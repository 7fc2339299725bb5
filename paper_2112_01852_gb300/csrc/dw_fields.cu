// Field layout kernels: canonical <-> internal fermion packing, gauge
// conversion with the boundary signs folded in, and precision conversion.
#include "dw_fields.cuh"

namespace dw {

// ---------------------------------------------------------------------------
// Canonical fermion complex128 [rhs][x4][s][spin][col] <-> internal planes.
// Internal real I = half*12 + c*4 + ri*2 + j (chirality half, colour c, re/im
// ri, spin j within the half) holds the canonical real
// ((2*half + j)*3 + c)*2 + ri: each 4-real quad is the spin pair
// (Re j0, Re j1, Im j0, Im j1) of one colour.
//
// Both directions are transposes of one 32-site block and kSC consecutive
// slices per CTA through shared memory: the internal side of the chunk is one
// contiguous run of vecs (coalesced 16-byte accesses, 8-byte at FP16), the
// canonical side is kSC x 12 consecutive complex128 per site (coalesced
// 16-byte accesses).  The staging array holds the canonical complex128 records,
// one row per site padded by one record to an odd count, so the 16-byte accesses of
// both sides are free of bank conflicts.
constexpr int kSC = 4;        // slices per CTA
constexpr int kXposeTPB = 128;
constexpr int kRow = kSC * 12 + 1;  // complex128 records per site row of the staging array

// One quad (spin pair j0, j1 of one colour and chirality half) <-> its two
// canonical complex values.  Spin-pair quads (Re j0, Re j1, Im j0, Im j1);
// interleaved-complex quads (CPLX, the layout ablation) (Re j0, Im j0, Re j1, Im j1).
template <class P>
__device__ __forceinline__ void quad_from_complex(typename P::vec *d, double2 a, double2 b) {
  double r[4];
  if (P::CPLX) {
    r[0] = a.x; r[1] = a.y; r[2] = b.x; r[3] = b.y;
  } else {
    r[0] = a.x; r[1] = b.x; r[2] = a.y; r[3] = b.y;
  }
#pragma unroll
  for (int w = 0; w < 4 / P::R; ++w)
    d[w * kPlaneStride] = narrow_from_f64(r + w * P::R, (typename P::vec *)nullptr);
}
template <class P>
__device__ __forceinline__ void quad_to_complex(double2 &a, double2 &b,
                                                const typename P::vec (&v)[4 / P::R]) {
  typename P::C r[4];
#pragma unroll
  for (int w = 0; w < 4 / P::R; ++w) widen(v[w], r + w * P::R);
  double d[4];
  f64_from_f32(d, r);
  a = P::CPLX ? make_double2(d[0], d[1]) : make_double2(d[0], d[2]);
  b = P::CPLX ? make_double2(d[2], d[3]) : make_double2(d[1], d[3]);
}

template <class P>
__global__ void __launch_bounds__(kXposeTPB) pack_kernel(typename P::vec *dst,
                                                         const double2 *src, int V4, int Ls,
                                                         long long rhs_stride, long long V5) {
  constexpr int NP = 24 / P::R;
  __shared__ double2 sm[32 * kRow];
  const int nch = (Ls + kSC - 1) / kSC;
  const int blk = (int)(blockIdx.x / nch);
  const int s0 = (int)(blockIdx.x % nch) * kSC;
  const int sc = min(kSC, Ls - s0);
  const int rhs = blockIdx.y;
  const int nlane = min(32, V4 - blk * 32);  // padding lanes are never read or written
  // canonical -> staging: consecutive threads read consecutive complex128
  const double2 *sp = src + ((long long)rhs * V5 + (long long)blk * 32 * Ls + s0) * 12;
  if (sc == kSC && nlane == 32) {
    double2 v[32 * kSC * 12 / kXposeTPB];  // all loads of the chunk in flight at once
#pragma unroll
    for (int i = 0; i < 32 * kSC * 12 / kXposeTPB; ++i) {
      const int o = threadIdx.x + i * kXposeTPB;
      const int lane = o / (kSC * 12), rem = o % (kSC * 12);
      v[i] = __ldcs(sp + (long long)lane * Ls * 12 + rem);
    }
#pragma unroll
    for (int i = 0; i < 32 * kSC * 12 / kXposeTPB; ++i) {
      const int o = threadIdx.x + i * kXposeTPB;
      sm[o / (kSC * 12) * kRow + o % (kSC * 12)] = v[i];
    }
  } else {
    for (int o = threadIdx.x; o < nlane * sc * 12; o += kXposeTPB) {
      const int lane = o / (sc * 12), rem = o % (sc * 12);
      sm[lane * kRow + rem] = __ldcs(sp + (long long)lane * Ls * 12 + rem);
    }
  }
  __syncthreads();
  // staging -> internal: the chunk is one contiguous run of sc * NP * 32 vecs; a
  // warp writes one quad of one slice
  typename P::vec *dp = dst + rhs * rhs_stride + ((long long)blk * Ls + s0) * NP * 32;
  const int lane = threadIdx.x & 31;
  if (lane >= nlane) return;
  for (int v = threadIdx.x >> 5; v < sc * 6; v += kXposeTPB / 32) {
    const int q = v % 6, sl = v / 6;  // quad: half * 3 + colour
    const double2 *b = sm + lane * kRow + sl * 12 + (q / 3) * 6 + q % 3;
    quad_from_complex<P>(dp + (sl * 6 + q) * (4 / P::R) * 32 + lane, b[0], b[3]);
  }
}

template <class P>
__global__ void __launch_bounds__(kXposeTPB) unpack_kernel(double2 *dst,
                                                           const typename P::vec *src, int V4,
                                                           int Ls, long long rhs_stride,
                                                           long long V5) {
  constexpr int NP = 24 / P::R;
  __shared__ double2 sm[32 * kRow];
  const int nch = (Ls + kSC - 1) / kSC;
  const int blk = (int)(blockIdx.x / nch);
  const int s0 = (int)(blockIdx.x % nch) * kSC;
  const int sc = min(kSC, Ls - s0);
  const int rhs = blockIdx.y;
  const int nlane = min(32, V4 - blk * 32);
  // internal -> staging: a warp reads one quad of one slice
  const typename P::vec *sp = src + rhs * rhs_stride + ((long long)blk * Ls + s0) * NP * 32;
  const int lane = threadIdx.x & 31;
  if (lane < nlane) {
    constexpr int N = kSC * 6 / (kXposeTPB / 32);
    typename P::vec r[N][4 / P::R];  // all loads of the chunk in flight at once
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int v = (threadIdx.x >> 5) + i * (kXposeTPB / 32);
      if (v < sc * 6) {
#pragma unroll
        for (int w = 0; w < 4 / P::R; ++w) r[i][w] = __ldcs(sp + (v * (4 / P::R) + w) * 32 + lane);
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int v = (threadIdx.x >> 5) + i * (kXposeTPB / 32);
      if (v < sc * 6) {
        const int q = v % 6, sl = v / 6;
        double2 *b = sm + lane * kRow + sl * 12 + (q / 3) * 6 + q % 3;
        quad_to_complex<P>(b[0], b[3], r[i]);
      }
    }
  }
  __syncthreads();
  // staging -> canonical: consecutive threads write consecutive complex128
  double2 *dp = dst + ((long long)rhs * V5 + (long long)blk * 32 * Ls + s0) * 12;
  if (sc == kSC && nlane == 32) {
#pragma unroll
    for (int i = 0; i < 32 * kSC * 12 / kXposeTPB; ++i) {
      const int o = threadIdx.x + i * kXposeTPB;
      const int l = o / (kSC * 12), rem = o % (kSC * 12);
      __stcs(dp + (long long)l * Ls * 12 + rem, sm[l * kRow + rem]);
    }
  } else {
    for (int o = threadIdx.x; o < nlane * sc * 12; o += kXposeTPB) {
      const int l = o / (sc * 12), rem = o % (sc * 12);
      __stcs(dp + (long long)l * Ls * 12 + rem, sm[l * kRow + rem]);
    }
  }
}

template <class P>
static int pack_t(const FieldGeom &g, void *dst, const void *src, int nrhs, cudaStream_t st) {
  const long long nch = (g.Ls + kSC - 1) / kSC;
  dim3 grid((unsigned)(padded_v4(g.V4) / 32 * nch), nrhs);
  pack_kernel<P><<<grid, kXposeTPB, 0, st>>>((typename P::vec *)dst, (const double2 *)src, g.V4,
                                             g.Ls, padded_v4(g.V4) * g.Ls * (24 / P::R), g.V5());
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <class P>
static int unpack_t(const FieldGeom &g, void *dst, const void *src, int nrhs, cudaStream_t st) {
  const long long nch = (g.Ls + kSC - 1) / kSC;
  dim3 grid((unsigned)(padded_v4(g.V4) / 32 * nch), nrhs);
  unpack_kernel<P><<<grid, kXposeTPB, 0, st>>>((double2 *)dst, (const typename P::vec *)src,
                                               g.V4, g.Ls,
                                               padded_v4(g.V4) * g.Ls * (24 / P::R), g.V5());
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int pack_fermion(const FieldGeom &g, int prec, void *dst, const void *src, int nrhs,
                 cudaStream_t st, bool cplx) {
  if (cplx && prec == DW_F32) return pack_t<F32C>(g, dst, src, nrhs, st);
  switch (prec) {
    case DW_F64: return pack_t<F64>(g, dst, src, nrhs, st);
    case DW_F32: return pack_t<F32>(g, dst, src, nrhs, st);
    case DW_F16: return pack_t<F16>(g, dst, src, nrhs, st);
  }
  return -2;
}

int unpack_fermion(const FieldGeom &g, int prec, void *dst, const void *src, int nrhs,
                   cudaStream_t st, bool cplx) {
  if (cplx && prec == DW_F32) return unpack_t<F32C>(g, dst, src, nrhs, st);
  switch (prec) {
    case DW_F64: return unpack_t<F64>(g, dst, src, nrhs, st);
    case DW_F32: return unpack_t<F32>(g, dst, src, nrhs, st);
    case DW_F16: return unpack_t<F16>(g, dst, src, nrhs, st);
  }
  return -2;
}

// ---------------------------------------------------------------------------
// Gauge: canonical complex128 [x4][mu][row][col] -> per precision blocked links
// (link_off): all 18 reals at F64, the first two rows (12 reals) at F32 / F16.
// A link U_mu(x) with x_mu = L_mu - 1 crosses the lattice edge and is
// multiplied by bc[mu].
// One CTA per 32-site block: its 32 x 4 links are 18 KB of consecutive canonical
// memory and one contiguous run of each internal copy, so the block is read with
// coalesced 16-byte loads into shared memory (one padded row of 4 x 18 reals per
// site) and each copy is written with coalesced 16-byte (8-byte at FP16) stores.
constexpr int kGaugeTPB = 128;
constexpr int kGaugeRow = 4 * 9 + 1;  // complex128 records per site row (odd)

// d with its sign bit flipped by f (the boundary factors are +-1)
__device__ __forceinline__ double flip(double d, unsigned f) {
  return __hiloint2double(__double2hiint(d) ^ (int)f, __double2loint(d));
}

template <class P>
__device__ __forceinline__ void store_links(void *gauge, int blk, int nlane, const double2 *sm,
                                            const unsigned (*f)[4]) {
  const int lane = threadIdx.x & 31;
  if (lane >= nlane) return;
  typename P::vec *m = (typename P::vec *)gauge + (long long)blk * 4 * P::NLV * 32;
  for (int v = threadIdx.x >> 5; v < 4 * P::NLV; v += kGaugeTPB / 32) {
    const int mu = v / P::NLV, q = v % P::NLV;
    const double2 *s = sm + lane * kGaugeRow + mu * 9 + q * (P::R / 2);
    const unsigned fm = f[lane][mu];
    double r[P::R];
#pragma unroll
    for (int k = 0; k < P::R / 2; ++k) {
      r[2 * k] = flip(s[k].x, fm);
      r[2 * k + 1] = flip(s[k].y, fm);
    }
    m[v * 32 + lane] = narrow_from_f64(r, (typename P::vec *)nullptr);
  }
}

__global__ void __launch_bounds__(kGaugeTPB)
    gauge_kernel(const double2 *U, int V4, int L0, int L1, int L2, int L3, int bc0, int bc1,
                 int bc2, int bc3, void *g64, void *g32, void *g16) {
  __shared__ double2 sm[32 * kGaugeRow];
  __shared__ unsigned f[32][4];  // sign bit of the boundary factor of (site, mu)
  const int blk = blockIdx.x;
  const int nlane = min(32, V4 - blk * 32);
  if ((int)threadIdx.x < nlane) {
    int rem = blk * 32 + threadIdx.x;
    const int L[4] = {L0, L1, L2, L3};
    const int bc[4] = {bc0, bc1, bc2, bc3};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      f[threadIdx.x][m] = (rem % L[m] == L[m] - 1 && bc[m] < 0) ? 0x80000000u : 0u;
      rem /= L[m];
    }
  }
  const double2 *src = U + (long long)blk * 32 * 36;
  if (nlane == 32) {
    double2 v[32 * 36 / kGaugeTPB];
#pragma unroll
    for (int i = 0; i < 32 * 36 / kGaugeTPB; ++i) v[i] = __ldcs(src + threadIdx.x + i * kGaugeTPB);
#pragma unroll
    for (int i = 0; i < 32 * 36 / kGaugeTPB; ++i) {
      const int o = threadIdx.x + i * kGaugeTPB;
      sm[o / 36 * kGaugeRow + o % 36] = v[i];
    }
  } else {
    for (int o = threadIdx.x; o < nlane * 36; o += kGaugeTPB)
      sm[o / 36 * kGaugeRow + o % 36] = src[o];
  }
  __syncthreads();
  store_links<F64>(g64, blk, nlane, sm, f);
  store_links<F32>(g32, blk, nlane, sm, f);
  store_links<F16>(g16, blk, nlane, sm, f);
}

int load_gauge(const FieldGeom &g, const int bc[4], const void *U, void *const gauge[3],
               cudaStream_t st) {
  gauge_kernel<<<(unsigned)(padded_v4(g.V4) / 32), kGaugeTPB, 0, st>>>(
      (const double2 *)U, g.V4, g.L[0], g.L[1], g.L[2], g.L[3], bc[0], bc[1], bc[2], bc[3],
      gauge[0], gauge[1], gauge[2]);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// Precision conversion between internal fields: one thread per site slot of
// the blocked layout (padding lanes skipped), all 6 quads (a quad is 4 reals:
// plane q of F32/F16, planes 2q and 2q+1 of F64).
template <class PI, class PO>
__global__ void convert_kernel(void *dst, const void *src, long long nslot, int V4, int Ls,
                               long long rhs_in, long long rhs_out) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int rhs = blockIdx.y;
  if (j >= nslot) return;
  const int x4 = (int)((j >> 5) / Ls) * 32 + (int)(j & 31);
  if (x4 >= V4) return;
  const typename PI::vec *s =
      (const typename PI::vec *)((const char *)src + rhs * rhs_in) + (j >> 5) * (24 / PI::R) * 32 + (j & 31);
  typename PO::vec *d =
      (typename PO::vec *)((char *)dst + rhs * rhs_out) + (j >> 5) * (24 / PO::R) * 32 + (j & 31);
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    typename PI::C a[4];
    typename PO::C b[4];
    if (PI::R == 4) {
      load_vec<PI>(a, s + q * 32);
    } else {
      load_vec<PI>(a, s + 2 * q * 32);
      load_vec<PI>(a + 2, s + (2 * q + 1) * 32);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) b[k] = (typename PO::C)a[k];
    if (PO::R == 4) {
      store_vec<PO>(d + q * 32, b);
    } else {
      store_vec<PO>(d + 2 * q * 32, b);
      store_vec<PO>(d + (2 * q + 1) * 32, b + 2);
    }
  }
}

template <class PI, class PO>
static int convert_t(const FieldGeom &g, void *dst, const void *src, int nrhs, cudaStream_t st) {
  const long long nslot = padded_v4(g.V4) * g.Ls;
  const int tpb = 256;
  dim3 grid((unsigned)((nslot + tpb - 1) / tpb), nrhs);
  convert_kernel<PI, PO><<<grid, tpb, 0, st>>>(dst, src, nslot, g.V4, g.Ls, 24 * nslot * PI::RB,
                                               24 * nslot * PO::RB);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <class PI>
static int convert_to(const FieldGeom &g, int po, void *dst, const void *src, int nrhs,
                      cudaStream_t st) {
  switch (po) {
    case DW_F64: return convert_t<PI, F64>(g, dst, src, nrhs, st);
    case DW_F32: return convert_t<PI, F32>(g, dst, src, nrhs, st);
    case DW_F16: return convert_t<PI, F16>(g, dst, src, nrhs, st);
  }
  return -2;
}

int convert_fermion(const FieldGeom &g, int pi, int po, void *dst, const void *src, int nrhs,
                    cudaStream_t st) {
  switch (pi) {
    case DW_F64: return convert_to<F64>(g, po, dst, src, nrhs, st);
    case DW_F32: return convert_to<F32>(g, po, dst, src, nrhs, st);
    case DW_F16: return convert_to<F16>(g, po, dst, src, nrhs, st);
  }
  return -2;
}

}  // namespace dw
