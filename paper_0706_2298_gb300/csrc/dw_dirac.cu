// Wilson-clover operator D (Section 2.1 operator) and its even-odd Schur
// complement A_ee - D_eo A_oo^{-1} D_oe, on packed fields.
//
// One thread per output site; 16-byte structure-of-arrays loads; links
// stored as two rows (third rebuilt in registers); spin projection with the
// chiral-basis (1 -+ gamma_mu) so that only 2x3 complex numbers go through
// each SU(3) multiply.  The kernel is HBM-bound: per site it moves the
// quark field (in + out), 4 links and the clover term once, with the
// neighbour re-reads served by L2 (block-major order keeps them close).
#include "dw_common.cuh"

#include <cstdio>
#include <cstdlib>
#include <mutex>

template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 1) dirac_full_kernel(Geom g, const T* __restrict__ links,
                                                         const T* __restrict__ clov, const T* __restrict__ in,
                                                         T* __restrict__ out) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= g.V) return;
  const size_t V = g.V;
  SiteRef s = decode(g, i);
  cplx<T> psi[12], y[12], acc[12];
  load_site<T, 12>(in, V, i, psi);
  clover_apply(clov, V, i, psi, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  hop_all(g, s, i, links, in, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] -= T(0.5) * acc[k];
  store_site<T, 12>(out, V, i, y);
}

// Multi-RHS D with one thread per (site, right-hand side): the nrhs CTAs of one chunk of 128 sites
// are consecutive in launch order (blockIdx.x = chunk * nrhs + rhs), so the chunk's links and clover
// term come from HBM once and from L2 for the other right-hand sides (fields fstride reals apart).
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 1) dirac_interleaved_kernel(
    Geom g, const T* __restrict__ links, const T* __restrict__ clov, const T* __restrict__ in0, T* __restrict__ out0,
    int nrhs, size_t fstride) {
  const int r = blockIdx.x % nrhs;
  const long long i = (long long)(blockIdx.x / nrhs) * blockDim.x + threadIdx.x;
  if (i >= g.V) return;
  const T* in = in0 + (size_t)r * fstride;
  T* out = out0 + (size_t)r * fstride;
  const size_t V = g.V;
  SiteRef s = decode(g, i);
  cplx<T> psi[12], y[12], acc[12];
  load_site<T, 12>(in, V, i, psi);
  clover_apply(clov, V, i, psi, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  hop_all(g, s, i, links, in, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] -= T(0.5) * acc[k];
  store_site<T, 12>(out, V, i, y);
}

// t_o = A_oo^{-1} D_oe in_e   (odd sites; D_oe = -1/2 * hops)
template <typename T>
__global__ void __launch_bounds__(128) schur_odd_kernel(Geom g, const T* __restrict__ links,
                                                        const T* __restrict__ clovinv, const T* __restrict__ in,
                                                        T* __restrict__ t) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= g.V / 2) return;
  const size_t V = g.V;
  SiteRef s;
  s.b = (int)(tid >> g.lshv);
  s.p = 1;
  s.h = (int)(tid & (g.shv - 1));
  long long i = site_index(g, s.b, 1, s.h);
  cplx<T> acc[12], v[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  hop_all(g, s, i, links, in, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = T(-0.5) * acc[k];
  clover_apply(clovinv, V, i, acc, v);
  store_site<T, 12>(t, V, i, v);
}

// out_e = A_ee in_e - D_eo t_o ; out_o = 0
template <typename T>
__global__ void __launch_bounds__(128) schur_even_kernel(Geom g, const T* __restrict__ links,
                                                         const T* __restrict__ clov, const T* __restrict__ in,
                                                         const T* __restrict__ t, T* __restrict__ out) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= g.V / 2) return;
  const size_t V = g.V;
  SiteRef s;
  s.b = (int)(tid >> g.lshv);
  s.p = 0;
  s.h = (int)(tid & (g.shv - 1));
  long long i = site_index(g, s.b, 0, s.h);
  cplx<T> psi[12], y[12], acc[12];
  load_site<T, 12>(in, V, i, psi);
  clover_apply(clov, V, i, psi, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  hop_all(g, s, i, links, t, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] += T(0.5) * acc[k];
  store_site<T, 12>(out, V, i, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] = {T(0), T(0)};
  store_site<T, 12>(out, V, site_index(g, s.b, 1, s.h), y);
}

// Even-odd preparation and reconstruction of D psi = eta (the Schur complement system
// (A_ee - D_eo A_oo^{-1} D_oe) psi_e = eta_e - D_eo A_oo^{-1} eta_o, psi_o = A_oo^{-1}(eta_o - D_oe psi_e)).
// t_o = A_oo^{-1} in_o on the odd sites
template <typename T>
__global__ void __launch_bounds__(128) clover_inv_odd_kernel(Geom g, const T* __restrict__ clovinv,
                                                             const T* __restrict__ in, T* __restrict__ t) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= g.V / 2) return;
  const size_t V = g.V;
  const int b = (int)(tid >> g.lshv), h = (int)(tid & (g.shv - 1));
  long long i = site_index(g, b, 1, h);
  cplx<T> x[12], y[12];
  load_site<T, 12>(in, V, i, x);
  clover_apply(clovinv, V, i, x, y);
  store_site<T, 12>(t, V, i, y);
}

// out_e = in_e - D_eo t_o = in_e + (1/2) hop(t) on the even sites, out_o = 0
template <typename T>
__global__ void __launch_bounds__(128) eo_rhs_kernel(Geom g, const T* __restrict__ links, const T* __restrict__ in,
                                                     const T* __restrict__ t, T* __restrict__ out) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= g.V / 2) return;
  const size_t V = g.V;
  SiteRef s;
  s.b = (int)(tid >> g.lshv);
  s.p = 0;
  s.h = (int)(tid & (g.shv - 1));
  long long i = site_index(g, s.b, 0, s.h);
  cplx<T> y[12], acc[12];
  load_site<T, 12>(in, V, i, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  hop_all(g, s, i, links, t, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] += T(0.5) * acc[k];
  store_site<T, 12>(out, V, i, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] = {T(0), T(0)};
  store_site<T, 12>(out, V, site_index(g, s.b, 1, s.h), y);
}

// out_o = A_oo^{-1} (in_o - D_oe x_e) = A_oo^{-1} (in_o + (1/2) hop(x)) on the odd sites, out_e = x_e
template <typename T>
__global__ void __launch_bounds__(128) eo_reconstruct_kernel(Geom g, const T* __restrict__ links,
                                                             const T* __restrict__ clovinv, const T* __restrict__ in,
                                                             const T* __restrict__ x, T* __restrict__ out) {
  long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= g.V / 2) return;
  const size_t V = g.V;
  SiteRef s;
  s.b = (int)(tid >> g.lshv);
  s.p = 1;
  s.h = (int)(tid & (g.shv - 1));
  long long io = site_index(g, s.b, 1, s.h), ie = site_index(g, s.b, 0, s.h);
  cplx<T> y[12], acc[12], z[12];
  load_site<T, 12>(in, V, io, y);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  hop_all(g, s, io, links, x, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) y[k] += T(0.5) * acc[k];
  clover_apply(clovinv, V, io, y, z);
  store_site<T, 12>(out, V, io, z);
  load_site<T, 12>(x, V, ie, y);
  store_site<T, 12>(out, V, ie, y);
}

// Multi-RHS D: one thread per site applies D to all right-hand sides (fields stored one after the
// other, stride fstride reals).  RHS are processed R at a time; the links and clover of the site are
// loaded for each group but come from L1/L2 after the first, so HBM sees them once per site.
template <typename T, int R>
__global__ void __launch_bounds__(128) dirac_mrhs_kernel(Geom g, const T* __restrict__ links,
                                                         const T* __restrict__ clov, const T* __restrict__ in,
                                                         T* __restrict__ out, int nrhs, size_t fstride) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= g.V) return;
  const size_t V = g.V;
  SiteRef s = decode(g, i);
  for (int r0 = 0; r0 < nrhs; r0 += R) {
    const int nr = nrhs - r0 < R ? nrhs - r0 : R;
    cplx<T> acc[R][12];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[r][k] = {T(0), T(0)};
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const int mu = d >> 1;
      bool cr;
      const long long j = neighbour(g, s, d, &cr);
      const T sg = time_wrap(g, s, d) ? T(-1) : T(1);
      SU3<T> U;
      load_link(links, V, mu, (d & 1) ? j : i, U);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (r < nr) {
          cplx<T> p[12];
          load_site<T, 12>(in + (size_t)(r0 + r) * fstride, V, j, p);
          switch (d) {
            case 0: hop_acc<0, -1, false>(acc[r], p, U, sg); break;
            case 1: hop_acc<0, +1, true>(acc[r], p, U, sg); break;
            case 2: hop_acc<1, -1, false>(acc[r], p, U, sg); break;
            case 3: hop_acc<1, +1, true>(acc[r], p, U, sg); break;
            case 4: hop_acc<2, -1, false>(acc[r], p, U, sg); break;
            case 5: hop_acc<2, +1, true>(acc[r], p, U, sg); break;
            case 6: hop_acc<3, -1, false>(acc[r], p, U, sg); break;
            default: hop_acc<3, +1, true>(acc[r], p, U, sg); break;
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r < nr) {
        cplx<T> psi[12], y[12];
        load_site<T, 12>(in + (size_t)(r0 + r) * fstride, V, i, psi);
        clover_apply(clov, V, i, psi, y);
#pragma unroll
        for (int k = 0; k < 12; ++k) y[k] -= T(0.5) * acc[r][k];
        store_site<T, 12>(out + (size_t)(r0 + r) * fstride, V, i, y);
      }
    }
  }
}

template <typename T>
void dirac_mrhs(dw_ctx* c, const T* in, T* out, int nrhs, int rgroup, cudaStream_t st) {
  constexpr int P = prec_of<T>();
  unsigned blocks = (unsigned)((c->V + 127) / 128);
  const size_t fs = (size_t)c->V * 24;
  const T* L = (const T*)c->links[P];
  const T* K = (const T*)c->clov[P];
  if (rgroup == 0) {
    const unsigned chunks = (unsigned)((c->V + 127) / 128);
    dirac_interleaved_kernel<T><<<chunks * (unsigned)nrhs, 128, 0, st>>>(c->g, L, K, in, out, nrhs, fs);
    dw_note_launch();
    return;
  }
  if (rgroup >= 3) { dirac_mrhs_kernel<T, 3><<<blocks, 128, 0, st>>>(c->g, L, K, in, out, nrhs, fs); dw_note_launch(); }
  else if (rgroup == 2) { dirac_mrhs_kernel<T, 2><<<blocks, 128, 0, st>>>(c->g, L, K, in, out, nrhs, fs); dw_note_launch(); }
  else { dirac_mrhs_kernel<T, 1><<<blocks, 128, 0, st>>>(c->g, L, K, in, out, nrhs, fs); dw_note_launch(); }
}
template void dirac_mrhs<float>(dw_ctx*, const float*, float*, int, int, cudaStream_t);
template void dirac_mrhs<double>(dw_ctx*, const double*, double*, int, int, cudaStream_t);

template <typename T>
void dirac_full(dw_ctx* c, const T* in, T* out, cudaStream_t st) {
  constexpr int P = prec_of<T>();
  unsigned blocks = (unsigned)((c->V + 127) / 128);
  dirac_full_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], (const T*)c->clov[P], in, out); dw_note_launch();
}
template void dirac_full<float>(dw_ctx*, const float*, float*, cudaStream_t);
template void dirac_full<double>(dw_ctx*, const double*, double*, cudaStream_t);

// D on double-float fields with two threads per site (warps 2m and 2m+1 take the same 32
// sites): thread half q forms the spin-q component of every half-spinor projection, multiplies it
// by the link and adds it to spin q and to the lower spin it feeds; the two halves exchange their
// lower-spin partial sums through shared memory, and each applies rows 3q..3q+2 of both chiral
// clover blocks.  The double-float links are stored with all three rows: rebuilding the third one in
// double-float arithmetic, in both halves, took a third of the operations, and the kernel uses a tenth of
// the memory bandwidth.  The result leaves as FP64, D in or eta - D in.
// Bound: FP32 issue and latency (20 warps per SM).  40x24x16x24, with the conversion of the input: 326 us;
// with a conversion 49 us slower, unrolled over the directions 525 us, also with the third row rebuilt and results
// and residual in passes of their own 745 us; 4 CTAs per SM 3% more, 6 CTAs 10%.
constexpr int DD_BLOCKS = 5;      // CTAs per SM
// s + e = a b for double-float a, b, exact up to the product of the low parts (Dekker's product of
// the leading parts by one FMA); s + e += a b with the leading part added by TwoSum and all errors
// gathered in e (compensated dot product, Ogita, Rump and Oishi 2005)
DW_D void dd2_first(float& s, float& e, dd a, dd b) {
  s = __fmul_rn(a.hi, b.hi);
  e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -s)));
}
DW_D void dd2_acc(float& s, float& e, dd a, dd b) {
  const float h = __fmul_rn(a.hi, b.hi);
  const float l = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -h)));
  const float t = __fadd_rn(s, h);
  const float bb = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(h, bb));
  s = t;
  e = __fadd_rn(e, __fadd_rn(err, l));
}
DW_D float flip(float x, uint32_t m) { return __uint_as_float(__float_as_uint(x) ^ m); }     // m: 0 or the sign bit
DW_D dd flip(dd x, uint32_t m) { return {flip(x.hi, m), flip(x.lo, m)}; }

// One hop of half q of a site, direction d = 2 mu + (1: backward), from the neighbour's spinor at P and the link
// at Lk (unit planes of stride V): au += sign w, and the lower spin that w feeds, own (2 + q) or the other
// one, += its image.  d is a run-time value: unrolled over the eight directions the kernel's code exceeds the
// instruction caches and warps wait for instructions.  Multiplications by +-1 and +-i are sign flips
// and exchanges of real and imaginary parts.
//   v = e_mu-part of the lower spin:  mu 0: -psi_lo, 1: -i psi_lo, 2: (q ? +1 : -1) psi_lo, 3: (q ? +i : -i) psi_lo
//   h = psi_q + S v, S = -1 forward, +1 backward;  w = U h (backward: U^+ h)
//   image of w:                       mu 0: -w, 1: i w, 2: (q ? +1 : -1) w, 3: (q ? -i : +i) w;  times S
DW_D void dd_half_hop(int d, const float4* __restrict__ Lk, const float4* __restrict__ P, size_t V, int q, bool wrap,
                      cplx<dd>* au, cplx<dd>* own, cplx<dd>* oth) {
  constexpr uint32_t SIGN = 0x80000000u;
  const int mu = d >> 1;
  const bool back = d & 1, imag = mu & 1, mine = mu == 0 || mu == 3;      // the lower spin involved: 2 + q or 3 - q
  const int lo = mine ? 2 + q : 3 - q;
  // S v: coefficient +-1 or +-i; i z = (-im, re)
  const bool vneg = ((mu < 2) || !q) != !back;
  const uint32_t vr = (vneg != imag) ? SIGN : 0u, vi = vneg ? SIGN : 0u;
  cplx<dd> h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    cplx<dd> u, l;
    unpack_unit(__ldg(P + (size_t)(3 * q + c) * V), &u);
    unpack_unit(__ldg(P + (size_t)(3 * lo + c) * V), &l);
    const dd a = imag ? l.im : l.re, b = imag ? l.re : l.im;
    h[c] = {u.re + flip(a, vr), u.im + flip(b, vi)};
  }
  // w = U h or U^+ h, each component a compensated sum of its six real products (about 40% fewer FP32
  // operations than product-by-product double-float arithmetic)
  const size_t sa = back ? V : 3 * V, sc = back ? 3 * V : V;               // element (a, c) or (c, a)
  const uint32_t cj = back ? SIGN : 0u;
  const uint32_t sg = wrap ? SIGN : 0u;
  // the image: S (times the wrap sign) and +-1 or +-i
  const bool wneg = (mu == 0 || (mu == 2 && !q) || (mu == 3 && q)) != !back;
  const uint32_t wr = ((wneg != imag) ? SIGN : 0u) ^ sg, wi = (wneg ? SIGN : 0u) ^ sg;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float sr, er, si, ei;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      cplx<dd> u;
      unpack_unit(__ldg(Lk + a * sa + c * sc), &u);
      const dd ui = flip(u.im, cj);
      if (c == 0) {
        dd2_first(sr, er, u.re, h[c].re);
        dd2_first(si, ei, u.re, h[c].im);
      } else {
        dd2_acc(sr, er, u.re, h[c].re);
        dd2_acc(si, ei, u.re, h[c].im);
      }
      dd2_acc(sr, er, -ui, h[c].im);
      dd2_acc(si, ei, ui, h[c].re);
    }
    const dd wre = dd_two_sum(sr, er), wim = dd_two_sum(si, ei);
    au[a] += cplx<dd>{flip(wre, sg), flip(wim, sg)};
    const cplx<dd> l = {flip(imag ? wim : wre, wr), flip(imag ? wre : wim, wi)};
    if (mine) own[a] += l; else oth[a] += l;
  }
}

// rows R0..R0+2 of one packed Hermitian 6x6 chiral block (18 slots at blk, stride V) times x (6
// components): the off-diagonal products of a component as one compensated sum, whose error is that of
// these smaller terms, then the diagonal one in double-float arithmetic
template <int R0>
DW_D void herm6_rows(const float4* __restrict__ blk, size_t V, const cplx<dd>* x, cplx<dd>* y) {
  float sr[3], er[3], si[3], ei[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) sr[r] = er[r] = si[r] = ei[r] = 0.f;
  int k = 3;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
#pragma unroll
    for (int j = i + 1; j < 6; ++j) {
      const bool ri = i >= R0 && i < R0 + 3, rj = j >= R0 && j < R0 + 3;
      if (ri || rj) {
        cplx<dd> m;
        unpack_unit(__ldg(blk + (size_t)k * V), &m);
        if (ri) {                                        // y_i += m x_j
          const int r = i - R0;
          dd2_acc(sr[r], er[r], m.re, x[j].re);
          dd2_acc(si[r], ei[r], m.re, x[j].im);
          dd2_acc(sr[r], er[r], -m.im, x[j].im);
          dd2_acc(si[r], ei[r], m.im, x[j].re);
        }
        if (rj) {                                        // y_j += conj(m) x_i
          const int r = j - R0;
          dd2_acc(sr[r], er[r], m.re, x[i].re);
          dd2_acc(si[r], ei[r], m.re, x[i].im);
          dd2_acc(sr[r], er[r], m.im, x[i].im);
          dd2_acc(si[r], ei[r], -m.im, x[i].re);
        }
      }
      ++k;
    }
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    cplx<dd> d2;
    unpack_unit(__ldg(blk + (size_t)((R0 + r) / 2) * V), &d2);
    const dd d = (R0 + r) % 2 ? d2.im : d2.re;
    y[r] = {dd_two_sum(sr[r], er[r]) + d * x[R0 + r].re, dd_two_sum(si[r], ei[r]) + d * x[R0 + r].im};
  }
}

__global__ void __launch_bounds__(128, DD_BLOCKS) dirac_dd_split_kernel(Geom g, const float4* __restrict__ links,
                                                             const float4* __restrict__ clov,
                                                             const dd* __restrict__ in, const double2* eta,
                                                             double2* out) {
  __shared__ cplx<dd> xch[2][3][64];          // lower-spin partials handed to the other half
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int q = w & 1, grp = w >> 1;           // warp-uniform half
  const int sl = grp * 32 + lane;              // site slot in the CTA (0..63)
  const long long i = (long long)blockIdx.x * 64 + sl;
  const bool valid = i < g.V;
  const size_t V = g.V;
  cplx<dd> au[3], al[3], ao[3];                // upper spin q, lower spins 2 + q and 3 - q
#pragma unroll
  for (int c = 0; c < 3; ++c) { au[c] = {dd(0), dd(0)}; al[c] = au[c]; ao[c] = au[c]; }
  if (valid) {
    const SiteRef s = decode(g, i);
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
      bool cr;
      const long long j = neighbour(g, s, d, &cr);
      dd_half_hop(d, links + (size_t)((d >> 1) * 9) * V + (d & 1 ? j : i), reinterpret_cast<const float4*>(in) + j, V, q,
                  time_wrap(g, s, d), au, al, ao);
    }
  }
  // hand the other lower spin to the partner half
#pragma unroll
  for (int c = 0; c < 3; ++c) xch[q][c][sl] = ao[c];
  __syncthreads();
  if (!valid) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) al[c] += xch[1 - q][c][sl];
  // clover: rows 3q..3q+2 of both chiral blocks (block 0: spins 0, 1; block 1: spins 2, 3)
  cplx<dd> x[6], y[3];
  const float4* P = reinterpret_cast<const float4*>(in);
  const dd hf = dd(0.5f);
  // out spin q (block 0 rows 3q..) and spin 2 + q (block 1 rows 3q..)
#pragma unroll 1
  for (int blk = 0; blk < 2; ++blk) {
#pragma unroll
    for (int k = 0; k < 6; ++k) unpack_unit(__ldg(P + (size_t)(6 * blk + k) * V + i), x + k);
    const float4* cb = clov + (size_t)(18 * blk) * V + i;
    if (q) herm6_rows<3>(cb, V, x, y); else herm6_rows<0>(cb, V, x, y);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cplx<dd> u = y[c] - hf * (blk ? al[c] : au[c]);
      const size_t o = (size_t)(3 * (2 * blk + q) + c) * V + i;
      double2 r = make_double2(widen(u.re.hi) + widen(u.re.lo), widen(u.im.hi) + widen(u.im.lo));
      if (eta) {
        const double2 e = eta[o];
        r = make_double2(e.x - r.x, e.y - r.y);
      }
      out[o] = r;
    }
  }
}

void dirac_full_dd(dw_ctx* c, const dd* in, const double* eta, double* out, cudaStream_t st) {
  unsigned blocks = (unsigned)((c->V + 63) / 64);
  dirac_dd_split_kernel<<<blocks, 128, 0, st>>>(c->g, (const float4*)c->links_dd, (const float4*)c->clov_dd, in,
                                                (const double2*)eta, (double2*)out);
  dw_note_launch();
}

// FP64 fields through double-float arithmetic (nrhs fields, one converted at a time; the converted field comes
// from the context's own memory pool, which keeps it for the next call of whatever stream)
static int dirac_full_f64x(dw_ctx* c, const double* in, double* out, int nrhs, cudaStream_t st) {
  int rc = dw_make_dd(c, st);
  if (rc) return rc;
  const size_t n = (size_t)c->V * 24;
  dd* a = nullptr;
  DW_CUDA(dw_pool_alloc(c, n * sizeof(dd), (void**)&a, st));
  for (int r = 0; r < nrhs; ++r) {
    f64_to_dd(in + r * n, a, n, st);
    dirac_full_dd(c, a, nullptr, out + r * n, st);
  }
  DW_CUDA(cudaFreeAsync(a, st));
  return DW_OK;
}

// bhat_e = eta_e - D_eo A_oo^{-1} eta_o, bhat_o = 0 (t: scratch field)
template <typename T>
void eo_prepare(dw_ctx* c, const T* eta, T* bhat, T* t, cudaStream_t st) {
  constexpr int P = prec_of<T>();
  unsigned blocks = (unsigned)((c->V / 2 + 127) / 128);
  clover_inv_odd_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->clovinv[P], eta, t); dw_note_launch();
  eo_rhs_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], eta, t, bhat); dw_note_launch();
}
// psi_e = x_e, psi_o = A_oo^{-1}(eta_o - D_oe x_e)
template <typename T>
void eo_reconstruct(dw_ctx* c, const T* eta, const T* x, T* psi, cudaStream_t st) {
  constexpr int P = prec_of<T>();
  unsigned blocks = (unsigned)((c->V / 2 + 127) / 128);
  eo_reconstruct_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], (const T*)c->clovinv[P], eta, x,
                                                   psi); dw_note_launch();
}
template void eo_prepare<double>(dw_ctx*, const double*, double*, double*, cudaStream_t);
template void eo_reconstruct<double>(dw_ctx*, const double*, const double*, double*, cudaStream_t);

template <typename T>
int dirac_schur(dw_ctx* c, const T* in, T* out, cudaStream_t st) {
  constexpr int P = prec_of<T>();
  if (!c->sap_d[P]) DW_CUDA(cudaMalloc(&c->sap_d[P], dw_field_bytes(c, P)));
  T* t = (T*)c->sap_d[P];
  unsigned blocks = (unsigned)((c->V / 2 + 127) / 128);
  schur_odd_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], (const T*)c->clovinv[P], in, t); dw_note_launch();
  schur_even_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], (const T*)c->clov[P], in, t, out); dw_note_launch();
  return DW_OK;
}
template int dirac_schur<float>(dw_ctx*, const float*, float*, cudaStream_t);
template int dirac_schur<double>(dw_ctx*, const double*, double*, cudaStream_t);

extern "C" int dw_apply(dw_ctx* c, int prec, int op, int nrhs, const void* in, void* out, void* stream) {
  if (!c || !in || !out || in == out || nrhs < 1 || (prec != DW_F64 && prec != DW_F32 && prec != DW_F64X) ||
      (op != DW_OP_FULL && op != DW_OP_SCHUR) || (prec == DW_F64X && op != DW_OP_FULL)) {
    dw_set_error("dw_apply: bad argument");
    return DW_EINVAL;
  }
  if (int rc = dw_check_device(c, "dw_apply")) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (prec == DW_F64X) {
    int rc = dirac_full_f64x(c, (const double*)in, (double*)out, nrhs, st);
    if (rc) return rc;
    DW_CUDA(cudaGetLastError());
    return DW_OK;
  }
  size_t n = (size_t)c->V * 24;
  if (nrhs > 1 && op == DW_OP_FULL) {   // multi-RHS kernel: links and clover read once per site
    if (prec == DW_F64) dirac_mrhs(c, (const double*)in, (double*)out, nrhs, c->tune_rgroup, st);
    else dirac_mrhs(c, (const float*)in, (float*)out, nrhs, c->tune_rgroup, st);
    DW_CUDA(cudaGetLastError());
    return DW_OK;
  }
  for (int r = 0; r < nrhs; ++r) {
    int rc = DW_OK;
    if (prec == DW_F64) {
      const double* a = (const double*)in + r * n;
      double* b = (double*)out + r * n;
      if (op == DW_OP_FULL) dirac_full(c, a, b, st); else rc = dirac_schur(c, a, b, st);
    } else {
      const float* a = (const float*)in + r * n;
      float* b = (float*)out + r * n;
      if (op == DW_OP_FULL) dirac_full(c, a, b, st); else rc = dirac_schur(c, a, b, st);
    }
    if (rc) return rc;
  }
  DW_CUDA(cudaGetLastError());
  return DW_OK;
}

// ------------------------------------------------------------------ allocation-free Schur operator
// The even-odd Schur complement of dw_apply(DW_OP_SCHUR) with its odd-site intermediate
// A_oo^{-1} D_oe held in a fixed device array of this file instead of memory that the
// library allocates on first use.  For callers that must not allocate device memory at
// the time of the call: cudaMalloc synchronises the device (stalling work queued on other
// streams) and can fail in processes that run with a fixed memory reservation.
//
// The array holds one packed field, so the entry point serves volumes whose packed field
// fits in kSchurStaticBytes; larger ones are rejected with DW_EINVAL.  Every entry of the
// intermediate that is read is written earlier in the same call, so nothing has to start
// at zero.  All calls on one device share the array: calls that overlap in time (issued on
// different streams, or from several host threads without ordering) race on it.
namespace {
constexpr size_t kSchurStaticBytes = size_t(16) << 20;   // 16 MiB: FP64 up to 87381 sites, FP32 up to 174762
constexpr int kMaxDevices = 64;
std::mutex g_schur_static_mu;
void* g_schur_static_ptr[kMaxDevices] = {};
}  // namespace

static __device__ __align__(256) unsigned char g_schur_static[kSchurStaticBytes];

// Address of the array on the current device, looked up once per device (the first call on a
// device does this set-up; make it before any stream capture).
static int schur_static_scratch(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return dw_cuda_fail(e, "dw_apply_schur_static: cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) {
    dw_set_error("dw_apply_schur_static: device ordinal beyond the supported range");
    return DW_EINVAL;
  }
  std::lock_guard<std::mutex> lock(g_schur_static_mu);
  if (!g_schur_static_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_schur_static);
    if (e != cudaSuccess) return dw_cuda_fail(e, "dw_apply_schur_static: cudaGetSymbolAddress");
    g_schur_static_ptr[dev] = p;
  }
  *out = g_schur_static_ptr[dev];
  return DW_OK;
}

template <typename T>
static void schur_static_launch(dw_ctx* c, const T* in, T* out, T* t, cudaStream_t st) {
  constexpr int P = prec_of<T>();
  unsigned blocks = (unsigned)((c->V / 2 + 127) / 128);
  schur_odd_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], (const T*)c->clovinv[P], in, t); dw_note_launch();
  schur_even_kernel<T><<<blocks, 128, 0, st>>>(c->g, (const T*)c->links[P], (const T*)c->clov[P], in, t, out); dw_note_launch();
}

extern "C" int dw_apply_schur_static(dw_ctx* c, int prec, const void* in, void* out, void* stream) {
  if (!c || !in || !out || in == out || (prec != DW_F64 && prec != DW_F32)) {
    dw_set_error("dw_apply_schur_static: bad argument");
    return DW_EINVAL;
  }
  if (int rc = dw_check_device(c, "dw_apply_schur_static")) return rc;
  const size_t need = dw_field_bytes(c, prec);
  if (need > kSchurStaticBytes) {
    char msg[256];
    snprintf(msg, sizeof msg,
             "dw_apply_schur_static: the intermediate field needs %zu bytes, more than the fixed %zu-byte "
             "device array (use dw_apply with DW_OP_SCHUR for this volume and precision)",
             need, kSchurStaticBytes);
    dw_set_error(msg);
    return DW_EINVAL;
  }
  void* t = nullptr;
  int rc = schur_static_scratch(&t);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (prec == DW_F64) schur_static_launch(c, (const double*)in, (double*)out, (double*)t, st);
  else schur_static_launch(c, (const float*)in, (float*)out, (float*)t, st);
  DW_CUDA(cudaGetLastError());
  return DW_OK;
}
