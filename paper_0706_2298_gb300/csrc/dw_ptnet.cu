// Gauge-covariant parallel-transport network (learned subspace generation).
//
// A layer maps C_in channel fields h_c (each a quark field) to C_out fields:
//     h'_{c'}(x) = sum_{d=0..8} sum_c W_d[c' s', c s] (T_d h_c)(x)
// with T_0 = 1, T_{1+2mu} h(x) = U_mu(x) h(x+mu), T_{2+2mu} h(x) = U_mu(x-mu)^+ h(x-mu)
// (fermion links, antiperiodic sign across the time boundary).  W acts on (channel, spin), the
// transports on (site, colour), so the two commute and the adjoint layer
//     g_c(x) = sum_d sum_{c'} W_d^+ (T_d^+ g')(x)
// has the same form with W -> W^+ and T_{+mu} <-> T_{-mu}.  This is the data gradient used in
// back-propagation.  The weight gradient is dW_d = sum_{x, colour} g'(x) (T_d h)(x)^+.
//
// Weights: per layer 9 x (4 C_out) x (4 C_in) complex (FP32), layers stored back to back.
// Channel fields are packed FP32 fields stored one after the other.
#include <algorithm>
#include <cstdlib>
#include <cmath>
#include <vector>

#include "dw_common.cuh"

namespace {

// Every kernel works on tiles of PT_S consecutive sites of one field, a lane per site (V is a multiple of 256:
// Schwarz blocks have at least 16 sites and there are at least 16 of them); the tiles of all fields of a
// batch form one grid.
constexpr int PT_S = 32;
constexpr int PT_THREADS = 256;

// transport of one channel field along PTNet direction d (0 = none) to site s/i; out[4][3]
DW_D void pt_transport(const Geom& g, const float* __restrict__ links, const float* __restrict__ f,
                       const SiteRef& s, long long i, int d, cplx<float> (*o)[3]) {
  const size_t V = g.V;
  cplx<float> p[12];
  if (d == 0) {
    load_site<float, 12>(f, V, i, p);
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int a = 0; a < 3; ++a) o[sp][a] = p[3 * sp + a];
    return;
  }
  const int nd = d - 1, mu = nd >> 1;
  bool cr;
  const long long j = neighbour(g, s, nd, &cr);
  const float sg = time_wrap(g, s, nd) ? -1.f : 1.f;
  SU3<float> U;
  load_link(links, V, mu, (nd & 1) ? j : i, U);
  load_site<float, 12>(f, V, j, p);
#pragma unroll
  for (int sp = 0; sp < 4; ++sp) {
    cplx<float> w[3];
    if (nd & 1) su3_dag_mul(U, p + 3 * sp, w); else su3_mul(U, p + 3 * sp, w);
#pragma unroll
    for (int a = 0; a < 3; ++a) o[sp][a] = sg * w[a];
  }
}

// direction of the adjoint transport: T_{+mu}^+ has the form of T_{-mu} and vice versa
DW_D int pt_reverse(int d) { return d > 0 ? ((d - 1) ^ 1) + 1 : 0; }

struct PtTile {
  size_t field;      // field of the batch
  long long i;       // this lane's site
  SiteRef s;
  DW_D PtTile(const Geom& g, long long tile) {
    const long long per = g.V / PT_S;
    field = (size_t)(tile / per);
    i = (tile % per) * PT_S + (threadIdx.x & 31);
    s = decode(g, i);
  }
};

// NI -> 16 channels: out = sum_d W_d T_d in, or for ADJ the adjoint sum_d W_d^+ T_d^+ in of a layer with NI
// output channels.  A complex matrix product per site and colour: 64 rows (channel, spin) written, 4 NI rows
// read per direction.  Per stage (a direction; all nine for NI = 1) the transported input of the tile's 32
// sites and the weights go to shared memory once, and a thread accumulates 8 rows x 3 colours of its site:
// 96 FMAs per 4 uniform 16-byte and 3 8-byte shared-memory reads.  The sums of a direction are kept apart
// and then added, which keeps the chains of FP32 roundings short.
// Bound: FP32 FMA issue (885 kflop per site for NI = 16).
template <int NI>
struct PtLayer {
  static constexpr int DPS = NI == 1 ? 9 : 1, NST = 9 / DPS, K = DPS * 4 * NI;
  static constexpr int WS = 66;                              // row stride of the staged weights (bank spread)
  static constexpr size_t bytes = (size_t)K * (WS + 3 * PT_S) * sizeof(float2);
};
template <int NI, bool ADJ>
__global__ void __launch_bounds__(PT_THREADS, 2) ptnet_layer_kernel(Geom g, const float* __restrict__ links,
                                                                    const float2* __restrict__ W,
                                                                    const float* __restrict__ in,
                                                                    float* __restrict__ out) {
  using C = PtLayer<NI>;
  extern __shared__ __align__(16) unsigned char pt_smem[];
  float2* sW = reinterpret_cast<float2*>(pt_smem);           // [K][WS]
  cplx<float>* sB = reinterpret_cast<cplx<float>*>(sW + C::K * C::WS);     // [K][3][PT_S]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const PtTile tl(g, blockIdx.x);
  const size_t fs = (size_t)g.V * 24;
  const float* fin = in + tl.field * NI * fs;
  cplx<float> acc[8][3];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[r][a] = {0.f, 0.f};
  for (int st = 0; st < C::NST; ++st) {
    __syncthreads();
    // weights as [k][row]: forward W_d [64][4 NI], adjoint W_d^+ of W_d [4 NI][64]
    for (int e = t; e < C::K * 64; e += PT_THREADS) {
      int k, r;
      float2 w;
      if (ADJ) {
        k = e >> 6; r = e & 63;
        w = W[(size_t)st * C::K * 64 + e];
        w.y = -w.y;
      } else {
        const int d = e / (256 * NI), q = e % (256 * NI);      // within the stage
        r = q / (4 * NI); k = d * 4 * NI + q % (4 * NI);
        w = W[(size_t)st * C::K * 64 + e];
      }
      sW[k * C::WS + r] = w;
    }
    for (int it = warp; it < C::DPS * NI; it += PT_THREADS / 32) {
      const int d = NI == 1 ? it : st, c = NI == 1 ? 0 : it;
      cplx<float> th[4][3];
      pt_transport(g, links, fin + (size_t)c * fs, tl.s, tl.i, ADJ ? pt_reverse(d) : d, th);
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int a = 0; a < 3; ++a) sB[((4 * it + sp) * 3 + a) * PT_S + lane] = th[sp][a];
    }
    __syncthreads();
    cplx<float> part[8][3];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int a = 0; a < 3; ++a) part[r][a] = {0.f, 0.f};
#pragma unroll 2
    for (int k = 0; k < C::K; ++k) {
      cplx<float> w[8], b[3];
      const float4* wp = reinterpret_cast<const float4*>(sW + k * C::WS + 8 * warp);
#pragma unroll
      for (int q = 0; q < 4; ++q) unpack_unit(wp[q], w + 2 * q);
#pragma unroll
      for (int a = 0; a < 3; ++a) b[a] = sB[(k * 3 + a) * PT_S + lane];
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int a = 0; a < 3; ++a) cmac(part[r][a], w[r], b[a]);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int a = 0; a < 3; ++a) acc[r][a] += part[r][a];
  }
  // rows 8 warp .. are the two channels 2 warp, 2 warp + 1
#pragma unroll
  for (int q = 0; q < 2; ++q)
    store_site<float, 12>(out + (tl.field * 16 + 2 * warp + q) * fs, g.V, tl.i, &acc[4 * q][0]);
}

// 16 -> 1 channel layer, first half: the weights act on (channel, spin) and the transports on (site,
// colour), so the channels are contracted before the transport: z_d = W_d h, nine fields, each
// transported once, instead of 16 x 9 transports per site.  Rows (d, spin): 36, a warp takes two
// directions; cols and staging as above.
constexpr int PT_ZW = 5;                                     // warps of the contraction
constexpr size_t PT_Z_BYTES = (size_t)64 * (40 + 3 * PT_S) * sizeof(float2);
__global__ void __launch_bounds__(32 * PT_ZW) ptnet_contract_kernel(Geom g, const float2* __restrict__ W,
                                                                    const float* __restrict__ in,
                                                                    float* __restrict__ z) {
  extern __shared__ __align__(16) unsigned char pt_smem[];
  float2* sW = reinterpret_cast<float2*>(pt_smem);           // [64][40]
  cplx<float>* sB = reinterpret_cast<cplx<float>*>(sW + 64 * 40);          // [64][3][PT_S]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const PtTile tl(g, blockIdx.x);
  const size_t fs = (size_t)g.V * 24;
  for (int e = t; e < 64 * 40; e += 32 * PT_ZW) {
    const int r = e >> 6, k = e & 63;                        // row (d, spin) of W [9][4][64]
    sW[k * 40 + r] = r < 36 ? W[r * 64 + k] : make_float2(0.f, 0.f);
  }
  for (int c = warp; c < 16; c += PT_ZW) {
    cplx<float> p[12];
    load_site<float, 12>(in + (tl.field * 16 + c) * fs, g.V, tl.i, p);
#pragma unroll
    for (int k = 0; k < 12; ++k) sB[((4 * c + k / 3) * 3 + k % 3) * PT_S + lane] = p[k];
  }
  __syncthreads();
  cplx<float> acc[8][3];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[r][a] = {0.f, 0.f};
#pragma unroll 2
  for (int k = 0; k < 64; ++k) {
    cplx<float> w[8], b[3];
    const float4* wp = reinterpret_cast<const float4*>(sW + k * 40 + 8 * warp);
#pragma unroll
    for (int q = 0; q < 4; ++q) unpack_unit(wp[q], w + 2 * q);
#pragma unroll
    for (int a = 0; a < 3; ++a) b[a] = sB[(k * 3 + a) * PT_S + lane];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int a = 0; a < 3; ++a) cmac(acc[r][a], w[r], b[a]);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (2 * warp + q < 9)
      store_site<float, 12>(z + (tl.field * 9 + 2 * warp + q) * fs, g.V, tl.i, &acc[4 * q][0]);
}
// second half: out = sum_d T_d z_d; a thread per site
__global__ void __launch_bounds__(128) ptnet_collect_kernel(Geom g, const float* __restrict__ links,
                                                            const float* __restrict__ z, float* __restrict__ out) {
  const long long t = blockIdx.x * 128LL + threadIdx.x;
  const size_t f = (size_t)(t / g.V), fs = (size_t)g.V * 24;   // V is a multiple of 128
  const long long i = t % g.V;
  const SiteRef s = decode(g, i);
  cplx<float> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {0.f, 0.f};
#pragma unroll
  for (int d = 0; d < 9; ++d) {
    cplx<float> th[4][3];
    pt_transport(g, links, z + (f * 9 + d) * fs, s, i, d, th);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] += th[k / 3][k % 3];
  }
  store_site<float, 12>(out + f * fs, g.V, i, acc);
}

// Partial weight gradients dW_d = sum_{x, colour} g(x) (T_d h)(x)^+ over a chunk of tiles.  A CTA forms
// A B^+ with A: 64 rows (16 channels x spin) of a field taken where it stands, B: transported rows.
//   MODE 0 (16 -> 16): A = g, B = T_d h of direction d = blockIdx.y (64 rows)
//   MODE 1 (1 -> 16):  A = g, B = (T_0 h .. T_8 h) of the single input channel (36 rows)
//   MODE 2 (16 -> 1):  A = h, B = (T_0^+ g .. T_8^+ g) of the single output channel (36 rows); the sum over
//                      sites moved by the transport, g (T_d h)^+ = (T_d^+ g) h^+, so that one field is
//                      transported instead of 16; the entries are conjugated and transposed
// A thread owns 4 x 4 entries.  Per entry the sum of 8 sites (24 products) is formed in FP32 and folded into
// a compensated (Kahan) FP32 accumulator, so that the error of a chunk's sum does not grow with the number
// of sites it covers.
constexpr int PT_K = 3 * PT_S;                               // (site, colour) per tile
constexpr int PT_AS = 66;
template <int MODE>
struct PtDw {
  static constexpr int N = MODE == 0 ? 64 : 36, BS = N + 2;
  static constexpr size_t bytes = (size_t)PT_K * (PT_AS + BS) * sizeof(float2);
};
template <int MODE>
__global__ void __launch_bounds__(PT_THREADS, 2) ptnet_dw_kernel(Geom g, const float* __restrict__ links,
                                                                 const float* __restrict__ local,
                                                                 const float* __restrict__ moved, float2* partial,
                                                                 long long ntiles) {
  using C = PtDw<MODE>;
  constexpr int NC = C::N / 4;                               // column groups
  extern __shared__ __align__(16) unsigned char pt_smem[];
  cplx<float>* sA = reinterpret_cast<cplx<float>*>(pt_smem); // [PT_K][PT_AS]
  cplx<float>* sB = sA + PT_K * PT_AS;                       // [PT_K][BS]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int tr = t / NC, tc = t - tr * NC;
  const bool active = tr < 16;
  const size_t fs = (size_t)g.V * 24;
  cplx<float> acc[4][4], cmp[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) { acc[r][c] = {0.f, 0.f}; cmp[r][c] = {0.f, 0.f}; }
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const PtTile tl(g, tile);
    __syncthreads();
    for (int c = warp; c < 16; c += PT_THREADS / 32) {
      cplx<float> p[12];
      load_site<float, 12>(local + (tl.field * 16 + c) * fs, g.V, tl.i, p);
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int sp = 0; sp < 4; sp += 2) {
          const cplx<float> v[2] = {p[3 * sp + a], p[3 * (sp + 1) + a]};
          *reinterpret_cast<float4*>(sA + (3 * lane + a) * PT_AS + 4 * c + sp) = pack_unit(v);
        }
    }
    for (int it = warp; it < NC; it += PT_THREADS / 32) {    // it: channel (MODE 0) or direction
      const int d = MODE == 0 ? (int)blockIdx.y : MODE == 1 ? it : pt_reverse(it);
      const float* f = moved + (MODE == 0 ? tl.field * 16 + it : tl.field) * fs;
      cplx<float> th[4][3];
      pt_transport(g, links, f, tl.s, tl.i, d, th);
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int sp = 0; sp < 4; sp += 2) {
          const cplx<float> v[2] = {th[sp][a], th[sp + 1][a]};
          *reinterpret_cast<float4*>(sB + (3 * lane + a) * C::BS + 4 * it + sp) = pack_unit(v);
        }
    }
    __syncthreads();
    if (active) {
      for (int k0 = 0; k0 < PT_K; k0 += 24) {
        cplx<float> part[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) part[r][c] = {0.f, 0.f};
#pragma unroll 4
        for (int k = k0; k < k0 + 24; ++k) {
          cplx<float> av[4], bv[4];
          const float4* ap = reinterpret_cast<const float4*>(sA + k * PT_AS + 4 * tr);
          const float4* bp = reinterpret_cast<const float4*>(sB + k * C::BS + 4 * tc);
          unpack_unit(ap[0], av);
          unpack_unit(ap[1], av + 2);
          unpack_unit(bp[0], bv);
          unpack_unit(bp[1], bv + 2);
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) cmacc(part[r][c], bv[c], av[r]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float yr = part[r][c].re - cmp[r][c].re, yi = part[r][c].im - cmp[r][c].im;
            const float sr = acc[r][c].re + yr, si = acc[r][c].im + yi;
            cmp[r][c] = {(sr - acc[r][c].re) - yr, (si - acc[r][c].im) - yi};
            acc[r][c] = {sr, si};
          }
      }
    }
  }
  if (!active) return;
  // [chunk][d][entry], entries as in the weights
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int row = 4 * tr + r;
      const float2 v = make_float2(acc[r][c].re, MODE == 2 ? -acc[r][c].im : acc[r][c].im);
      if (MODE == 0) partial[((size_t)blockIdx.x * 9 + blockIdx.y) * 4096 + row * 64 + 4 * tc + c] = v;
      else if (MODE == 1) partial[((size_t)blockIdx.x * 9 + tc) * 256 + row * 4 + c] = v;
      else partial[((size_t)blockIdx.x * 9 + tc) * 256 + c * 64 + row] = v;
    }
}

// grad[d][e] = scale * sum over chunks (fixed order)
__global__ void ptnet_dw_reduce_kernel(const float2* __restrict__ partial, int nchunk, int E, float scale,
                                       float2* grad) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 9 * E) return;
  double re = 0, im = 0;
  for (int c = 0; c < nchunk; ++c) {
    float2 v = partial[(size_t)c * 9 * E + t];
    re += v.x;
    im += v.y;
  }
  grad[t] = make_float2((float)(scale * re), (float)(scale * im));
}

// Adam on real and imaginary parts
__global__ void ptnet_adam_kernel(size_t n, float* w, const float* gr, float* m, float* v, float lr, float b1,
                                  float b2, float eps, float c1, float c2) {
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float g = gr[t];
  const float mt = b1 * m[t] + (1.f - b1) * g;
  const float vt = b2 * v[t] + (1.f - b2) * g * g;
  m[t] = mt;
  v[t] = vt;
  w[t] -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
}

// nf fields: NI channels each in, 16 out (ADJ: the adjoint of a 16 -> NI layer)
template <int NI, bool ADJ>
cudaError_t launch_layer(dw_ctx* c, const float2* W, const float* in, float* out, int nf, cudaStream_t st) {
  if (const cudaError_t e = dw_smem_limit<ptnet_layer_kernel<NI, ADJ>>(PtLayer<NI>::bytes)) return e;
  const unsigned tiles = (unsigned)(c->V / PT_S * nf);
  ptnet_layer_kernel<NI, ADJ><<<tiles, PT_THREADS, PtLayer<NI>::bytes, st>>>(c->g, (const float*)c->links[DW_F32], W,
                                                                             in, out);
  dw_note_launch();
  return cudaGetLastError();
}
// 16 channels in, 1 out; z: 9 scratch fields per field
cudaError_t launch_layer_last(dw_ctx* c, const float2* W, const float* in, float* z, float* out, int nf,
                              cudaStream_t st) {
  if (const cudaError_t e = dw_smem_limit<ptnet_contract_kernel>(PT_Z_BYTES)) return e;
  ptnet_contract_kernel<<<(unsigned)(c->V / PT_S * nf), 32 * PT_ZW, PT_Z_BYTES, st>>>(c->g, W, in, z);
  dw_note_launch();
  ptnet_collect_kernel<<<(unsigned)(c->V / 128 * nf), 128, 0, st>>>(c->g, (const float*)c->links[DW_F32], z, out);
  dw_note_launch();
  return cudaGetLastError();
}
// CTAs over the tiles of a weight gradient: two waves of the resident CTAs (two per SM) in all directions
int pt_chunks(const dw_ctx* c, long long tiles, int ndir) {
  return (int)std::min<long long>(tiles, std::max(1, 4 * c->sms / ndir));
}
template <int MODE>
cudaError_t launch_dw(dw_ctx* c, const float* local, const float* moved, float2* partial, float2* grad, int nf,
                      cudaStream_t st) {
  if (const cudaError_t e = dw_smem_limit<ptnet_dw_kernel<MODE>>(PtDw<MODE>::bytes)) return e;
  constexpr int E = MODE == 0 ? 4096 : 256, ND = MODE == 0 ? 9 : 1;
  const long long tiles = c->V / PT_S * nf;
  const int nc = pt_chunks(c, tiles, ND);
  ptnet_dw_kernel<MODE><<<dim3(nc, ND), PT_THREADS, PtDw<MODE>::bytes, st>>>(c->g, (const float*)c->links[DW_F32],
                                                                             local, moved, partial, tiles);
  dw_note_launch();
  ptnet_dw_reduce_kernel<<<(unsigned)((9 * E + 255) / 256), 256, 0, st>>>(partial, nc, E, 2.f, grad);
  dw_note_launch();
  return cudaGetLastError();
}
// fields worked on together: enough for a full GPU, at most 2^19 sites (about 3.7 GB of training workspace); fewer
// where the memory is taken
int pt_group(const dw_ctx* c, int nf) {
  return (int)std::min<long long>(nf, std::max<long long>(1, (1LL << 19) / c->V));
}

// ------------------------------------------------------------------ tensor-core 16 -> 16 layer
// The 16-channel layer is a dense complex contraction per site and colour: out = sum_d W_d (T_d h)
// with W_d a 64 x 64 complex matrix on (channel, spin).  In real form it is one GEMM per CTA tile:
//   D[128 x 192] += A_d[128 x 128] B_d[128 x 192],  d = 0..8
// A_d = [[Re W_d, -Im W_d], [Im W_d, Re W_d]] (rows: output (channel, spin) x (re, im)), B_d the
// transported input of 64 sites x 3 colours (columns) by (channel, spin) x (re, im) (rows), BF16
// operands in shared memory, the FP32 accumulator in tensor memory (tcgen05.mma, kind::f16, one
// elected thread issues).  A_d is staged by a bulk copy from a pre-arranged image; B_d is built by
// all threads (parallel transport on the CUDA cores, rounded to BF16).  Two stages: the
// transports of direction d + 1 overlap the MMAs of direction d.  Operands are K-major without
// swizzle: 8 x 16-byte core matrices, K-adjacent ones 128 bytes apart (leading byte offset),
// 8-row groups 2048 bytes apart (stride byte offset).
constexpr int TC_M = 128, TC_K = 128;
constexpr int TC_THREADS = 256;
constexpr int TC_A_BYTES = TC_M * TC_K * 2;    // 32 KB
// per tile of S sites (S = 64: one CTA per SM; S = 32: two, for more warps hiding the transports)
template <int S>
struct TcTile {
  static constexpr int N = 3 * S;                              // columns: (site, colour)
  static constexpr int B_BYTES = N * TC_K * 2;                 // 48 KB / 24 KB
  static constexpr uint32_t TMEM_COLS = N <= 128 ? 128u : 256u;
  static constexpr int STAGE_LD = N + 1;                       // FP32 staging row stride (bank-conflict free)
  static constexpr size_t SMEM = 2 * TC_A_BYTES + 2 * B_BYTES + 128;   // two per SM fit at S = 32
  static constexpr int MIN_BLOCKS = S <= 32 ? 2 : 1;
  // instruction descriptor, kind::f16: D FP32, A and B BF16, both K-major, N = 3S, M = 128
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
                                    ((uint32_t)(TC_M >> 4) << 24);
};

// byte offset of element (row, k) in a K-major no-swizzle operand with K = 128
DW_HD uint32_t tc_off(int row, int k) {
  return (uint32_t)((row >> 3) * 2048 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}
DW_D uint64_t tc_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;             // leading byte offset: next core matrix along K
  d |= (uint64_t)(2048 >> 4) << 32;            // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                      // descriptor version of tcgen05; no swizzle
  return d;
}

DW_D void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
DW_D void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
DW_D void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
DW_D void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// the load and its wait in one statement: the registers are undefined before the wait, and a compiler may copy them
DW_D void tc_ld16(uint32_t taddr, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(taddr)
      : "memory");
}

// A_d images of one 16 -> 16 layer (ADJ: of W_d^+), BF16 in the core-matrix layout
template <bool ADJ>
__global__ void ptnet_tc_pack_kernel(const float2* __restrict__ W, __nv_bfloat16* A) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 9 * TC_M * TC_K) return;
  const int d = t / (TC_M * TC_K), e = t % (TC_M * TC_K), r = e / TC_K, k = e % TC_K;
  const int ro = r & 63, ko = k & 63;
  const float2* Wd = W + (size_t)d * 64 * 64;
  float2 w = ADJ ? Wd[ko * 64 + ro] : Wd[ro * 64 + ko];
  if (ADJ) w.y = -w.y;
  const float val = r < 64 ? (k < 64 ? w.x : -w.y) : (k < 64 ? w.y : w.x);
  A[(size_t)d * TC_M * TC_K + tc_off(r, k) / 2] = __float2bfloat16_rn(val);
}

template <bool ADJ, int S>
__global__ void __launch_bounds__(TC_THREADS, TcTile<S>::MIN_BLOCKS) ptnet_tc_layer_kernel(Geom g, const float* __restrict__ links,
                                                                       const __nv_bfloat16* __restrict__ Apack,
                                                                       const float* __restrict__ in,
                                                                       float* __restrict__ out, int* err) {
  using TT = TcTile<S>;
  extern __shared__ uint8_t tc_raw[];
  __shared__ uint64_t bar_tma[2], bar_mma[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  const uint32_t raw = smem_u32(tc_raw);
  uint8_t* sb = tc_raw + (((raw + 127u) & ~127u) - raw);         // 128-byte aligned operand area
  uint8_t* abuf[2] = {sb, sb + TC_A_BYTES};
  uint8_t* bbuf[2] = {sb + 2 * TC_A_BYTES, sb + 2 * TC_A_BYTES + TT::B_BYTES};
  float* stage = reinterpret_cast<float*>(sb);                   // epilogue: [128][TT::STAGE_LD] FP32
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    mbar_init(&bar_tma[0], 1);
    mbar_init(&bar_tma[1], 1);
    mbar_init(&bar_mma[0], 1);
    mbar_init(&bar_mma[1], 1);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(TT::TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const size_t V = g.V, fs = V * 24;
  const long long ntiles = ((long long)V + S - 1) / S;
  uint32_t use[2] = {0, 0};
  int gc = 0;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long i0 = tile * S;
    for (int d = 0; d < 9; ++d) {
      const int b = gc & 1;
      // the MMAs that last read stage b must be complete before it is refilled
      if (use[b] > 0 && !mbar_wait(&bar_mma[b], (use[b] - 1) & 1, err)) fail = 1;
      __syncthreads();
      if (fail) break;
      if (tid == 0) {
        mbar_expect_tx(&bar_tma[b], TC_A_BYTES);
        bulk_load(abuf[b], Apack + (size_t)d * TC_M * TC_K, TC_A_BYTES, &bar_tma[b]);
      }
      // B_d: item (site q, input channel c) -> rows (4c .. 4c+3) re and (64 + 4c ..) im, columns 3q + colour
      const int dt = (ADJ && d > 0) ? (((d - 1) ^ 1) + 1) : d;
      for (int it = tid; it < S * 16; it += TC_THREADS) {
        const int q = it & (S - 1), c = it / S;
        const long long i = i0 + q;
        cplx<float> th[4][3];
        if (i < (long long)V) {
          const SiteRef s = decode(g, i);
          pt_transport(g, links, in + (size_t)c * fs, s, i, dt, th);
        } else {
#pragma unroll
          for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int a = 0; a < 3; ++a) th[sp][a] = {0.f, 0.f};
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int n = 3 * q + a;
          __nv_bfloat162 re01 = __floats2bfloat162_rn(th[0][a].re, th[1][a].re);
          __nv_bfloat162 re23 = __floats2bfloat162_rn(th[2][a].re, th[3][a].re);
          __nv_bfloat162 im01 = __floats2bfloat162_rn(th[0][a].im, th[1][a].im);
          __nv_bfloat162 im23 = __floats2bfloat162_rn(th[2][a].im, th[3][a].im);
          uint2 vr, vi;
          vr.x = *reinterpret_cast<uint32_t*>(&re01);
          vr.y = *reinterpret_cast<uint32_t*>(&re23);
          vi.x = *reinterpret_cast<uint32_t*>(&im01);
          vi.y = *reinterpret_cast<uint32_t*>(&im23);
          *reinterpret_cast<uint2*>(bbuf[b] + tc_off(n, 4 * c)) = vr;
          *reinterpret_cast<uint2*>(bbuf[b] + tc_off(n, 64 + 4 * c)) = vi;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");    // generic-proxy writes -> tensor core
      tc_fence_before();
      __syncthreads();
      if (tid == 0) {
        tc_fence_after();
        if (mbar_wait(&bar_tma[b], use[b] & 1, err)) {
          const uint32_t a0 = smem_u32(abuf[b]), b0 = smem_u32(bbuf[b]);
#pragma unroll
          for (int kk = 0; kk < TC_K / 16; ++kk)
            tc_mma(tmem, tc_desc(a0 + kk * 256), tc_desc(b0 + kk * 256), TT::IDESC, (d > 0 || kk > 0) ? 1u : 0u);
          tc_commit(&bar_mma[b]);
        } else {
          fail = 1;
        }
      }
      ++use[b];
      ++gc;
    }
    __syncthreads();
    if (fail) break;
    // epilogue: all MMAs of the tile complete -> TMEM rows to shared memory -> output fields
    const int bl = (gc - 1) & 1;
    if (!mbar_wait(&bar_mma[bl], (use[bl] - 1) & 1, err)) fail = 1;
    __syncthreads();
    if (fail) break;
    tc_fence_after();
    {
      const int row = 32 * (warp & 3) + lane, half = warp >> 2;
#pragma unroll
      for (int j = 0; j < TT::N / 2 / 16; ++j) {
        const int col = half * (TT::N / 2) + 16 * j;
        float v[16];
        tc_ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)col, v);
#pragma unroll
        for (int e = 0; e < 16; ++e) stage[row * TT::STAGE_LD + col + e] = v[e];
      }
    }
    tc_fence_before();
    __syncthreads();
    for (int it = tid; it < S * 16; it += TC_THREADS) {
      const int q = it & (S - 1), c = it / S;
      const long long i = i0 + q;
      if (i >= (long long)V) continue;
      cplx<float> o[12];
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int m = 4 * c + sp, n = 3 * q + a;
          o[3 * sp + a] = {stage[m * TT::STAGE_LD + n], stage[(m + 64) * TT::STAGE_LD + n]};
        }
      store_site<float, 12>(out + (size_t)c * fs, V, i, o);
    }
    __syncthreads();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TT::TMEM_COLS) : "memory");
}

// one 16 -> 16 layer (adjoint: W_d^+ and reversed transports) on the tensor cores
template <bool ADJ, int S>
static int launch_tc(dw_ctx* c, const __nv_bfloat16* A, const float* in, float* out, int* err, cudaStream_t st) {
  using TT = TcTile<S>;
  DW_CUDA((dw_smem_limit<ptnet_tc_layer_kernel<ADJ, S>>(TT::SMEM)));
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long ntiles = (c->V + S - 1) / S;
  const unsigned grid = (unsigned)std::min<long long>(ntiles, (long long)sms * TT::MIN_BLOCKS);
  ptnet_tc_layer_kernel<ADJ, S><<<grid, TC_THREADS, TT::SMEM, st>>>(c->g, (const float*)c->links[DW_F32], A, in, out, err);
  dw_note_launch();
  return DW_OK;
}

// one 16 -> 16 layer (adjoint: W_d^+ and reversed transports) on the tensor cores; tiles of 64 sites
// (one CTA per SM) or, with DW_TC_TILE=32, of 32 sites (two CTAs per SM)
int tc_layer16(dw_ctx* c, const float2* W, int adjoint, const float* in, float* out, cudaStream_t st) {
  __nv_bfloat16* A = nullptr;
  int* err = nullptr;
  DW_CUDA(cudaMallocAsync((void**)&A, (size_t)9 * TC_A_BYTES, st));
  DW_CUDA(cudaMallocAsync((void**)&err, sizeof(int), st));
  DW_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
  const int n = 9 * TC_M * TC_K;
  const char* te = getenv("DW_TC_TILE");
  const bool small = te && atoi(te) == 32;
  int rc;
  if (adjoint) {
    ptnet_tc_pack_kernel<true><<<(n + 255) / 256, 256, 0, st>>>(W, A); dw_note_launch();
    rc = small ? launch_tc<true, 32>(c, A, in, out, err, st) : launch_tc<true, 64>(c, A, in, out, err, st);
  } else {
    ptnet_tc_pack_kernel<false><<<(n + 255) / 256, 256, 0, st>>>(W, A); dw_note_launch();
    rc = small ? launch_tc<false, 32>(c, A, in, out, err, st) : launch_tc<false, 64>(c, A, in, out, err, st);
  }
  if (rc) return rc;
  DW_CUDA(cudaGetLastError());
  int herr = 0;
  DW_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  DW_CUDA(cudaStreamSynchronize(st));
  cudaFreeAsync(A, st);
  cudaFreeAsync(err, st);
  if (herr) { dw_set_error("ptnet tensor-core layer: a wait on the tensor core or bulk copy timed out"); return DW_ECUDA; }
  return DW_OK;
}

}  // namespace

extern "C" size_t ptnet_weight_count(int C) {
  return (size_t)9 * 16 * (C + C * C + C);   // complex numbers, layers 1 -> C -> C -> 1
}

static bool ptnet_ok(int C) { return C == 16; }

// y = N(x) for nf fields (one batch); h1, h2: 16 fields per field, z: 9 per field (h1 where it is not needed later)
static cudaError_t ptnet_forward_impl(dw_ctx* c, const float2* W, const float* x, float* y, float* h1, float* h2,
                                      float* z, int nf, cudaStream_t st) {
  const size_t w1 = 9 * 16 * 16, w2 = w1 * 16;
  cudaError_t e = launch_layer<1, false>(c, W, x, h1, nf, st);
  if (e == cudaSuccess) e = launch_layer<16, false>(c, W + w1, h1, h2, nf, st);
  if (e == cudaSuccess) e = launch_layer_last(c, W + w1 + w2, h2, z, y, nf, st);
  return e;
}

extern "C" int ptnet_forward(dw_ctx* c, int C, const void* W, int nf, const void* x, void* y, void* stream) {
  if (!c || !W || !x || !y || x == y || nf < 1 || !ptnet_ok(C)) {
    dw_set_error("ptnet_forward: bad argument (C must be 16)");
    return DW_EINVAL;
  }
  const size_t fs = (size_t)c->V * 24;
  int ng = pt_group(c, nf);
  float* acts = nullptr;
  cudaError_t e = fit_group(ng, cudaErrorMemoryAllocation, [&](int n) {
    const cudaError_t m = cudaMalloc(&acts, 2 * C * fs * n * sizeof(float));
    if (m != cudaSuccess) cudaGetLastError();
    return m;
  });
  if (e != cudaSuccess) return dw_cuda_fail(e, "ptnet_forward");
  for (int f = 0; f < nf && e == cudaSuccess; f += ng) {
    const int n = std::min(ng, nf - f);
    e = ptnet_forward_impl(c, (const float2*)W, (const float*)x + f * fs, (float*)y + f * fs, acts,
                           acts + (size_t)C * fs * ng, acts, n, (cudaStream_t)stream);
  }
  const cudaError_t es = cudaStreamSynchronize((cudaStream_t)stream);
  cudaFree(acts);
  if (e == cudaSuccess) e = es;
  return e == cudaSuccess ? DW_OK : dw_cuda_fail(e, "ptnet_forward");
}

// One 16 -> 16 layer on a set of 16 channel fields: out = sum_d W_d T_d in (adjoint:
// sum_d W_d^+ T_d^+ in), on the tensor cores (BF16 operands, FP32 accumulation) or the CUDA cores (FP32).
extern "C" int ptnet_layer16(dw_ctx* c, const void* W, int adjoint, int tensor_cores, const void* in, void* out,
                             void* stream) {
  if (!c || !W || !in || !out || in == out) { dw_set_error("ptnet_layer16: bad argument"); return DW_EINVAL; }
  if (int rc = dw_check_device(c, "ptnet_layer16")) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (tensor_cores) return tc_layer16(c, (const float2*)W, adjoint, (const float*)in, (float*)out, st);
  DW_CUDA(adjoint ? (launch_layer<16, true>(c, (const float2*)W, (const float*)in, (float*)out, 1, st))
                  : (launch_layer<16, false>(c, (const float2*)W, (const float*)in, (float*)out, 1, st)));
  DW_CUDA(cudaStreamSynchronize(st));
  return DW_OK;
}

// The network with its 16 -> 16 layer on the tensor cores (the 1 -> 16 and 16 -> 1 layers, 16x fewer
// flops, on the CUDA cores).
extern "C" int ptnet_forward_tc(dw_ctx* c, int C, const void* Wv, int nf, const void* x, void* y, void* stream) {
  if (!c || !Wv || !x || !y || x == y || nf < 1 || !ptnet_ok(C)) {
    dw_set_error("ptnet_forward_tc: bad argument (C must be 16)");
    return DW_EINVAL;
  }
  if (int rc = dw_check_device(c, "ptnet_forward_tc")) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const float2* W = (const float2*)Wv;
  const size_t fs = (size_t)c->V * 24, w1 = 9 * 16 * C, w2 = 9 * 16 * C * C;
  float* acts = nullptr;
  DW_CUDA(cudaMalloc(&acts, 2 * C * fs * sizeof(float)));
  float* h1 = acts;
  float* h2 = acts + (size_t)C * fs;
  int rc = DW_OK;
  for (int f = 0; f < nf && rc == DW_OK; ++f) {
    cudaError_t e = launch_layer<1, false>(c, W, (const float*)x + f * fs, h1, 1, st);
    if (e == cudaSuccess) {
      rc = tc_layer16(c, W + w1, 0, h1, h2, st);
      if (rc == DW_OK) e = launch_layer_last(c, W + w1 + w2, h2, h1, (float*)y + f * fs, 1, st);
    }
    if (e != cudaSuccess) rc = dw_cuda_fail(e, "ptnet_forward_tc");
  }
  cudaStreamSynchronize(st);
  cudaFree(acts);
  if (rc == DW_OK) DW_CUDA(cudaGetLastError());
  return rc;
}

// loss = sum_f |N(x_f) - y_f|^2 / sum_f |y_f|^2 and its gradient dL/dRe W + i dL/dIm W
extern "C" int ptnet_loss_grad(dw_ctx* c, int C, const void* Wv, int nf, const void* xv, const void* yv,
                               void* gradv, double* loss, void* stream) {
  if (!c || !Wv || !xv || !yv || !gradv || nf < 1 || !ptnet_ok(C)) {
    dw_set_error("ptnet_loss_grad: bad argument (C must be 16)");
    return DW_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const float2* W = (const float2*)Wv;
  const size_t fs = (size_t)c->V * 24, n = (size_t)c->V * 12;
  const size_t w1 = 9 * 16 * C, w2 = 9 * 16 * C * C, w3 = 9 * 16 * C, nw = w1 + w2 + w3;
  int ng = pt_group(c, nf);
  // the workspace stays in the context up to 8 GB: h1, h2, g2, g1 (16 fields each), the output, the gradients
  WsArena& ar = c->ws_solve[4];
  float *ws = nullptr, *gw = nullptr;
  const cudaError_t em = fit_group(ng, cudaErrorMemoryAllocation, [&](int n) {
    const size_t np = (size_t)std::max(pt_chunks(c, c->V / PT_S * n, 9) * 9 * 4096,
                                       pt_chunks(c, c->V / PT_S * n, 1) * 9 * 256);
    ar.rewind();
    cudaError_t m = ar.get((4 * C + 1) * fs * n * sizeof(float), (void**)&ws);
    if (m == cudaSuccess) m = ar.get((np + 2 * nw) * sizeof(float2), (void**)&gw);
    if (m != cudaSuccess) {
      ar.release();
      cudaGetLastError();
    }
    return m;
  });
  if (em != cudaSuccess) return dw_cuda_fail(em, "ptnet_loss_grad");
  struct Keep {
    WsArena& a;
    bool keep;
    ~Keep() { if (!keep) a.release(); }
  } guard{ar, (4 * C + 1) * fs * ng * sizeof(float) <= (size_t)8 << 30};
  float* h1 = ws;
  float* h2 = h1 + (size_t)C * fs * ng;
  float* g2 = h2 + (size_t)C * fs * ng;
  float* g1 = g2 + (size_t)C * fs * ng;
  float* out = g1 + (size_t)C * fs * ng;
  float2* gacc = reinterpret_cast<float2*>(gw);
  float2* gtmp = gacc + nw;
  float2* partial = gtmp + nw;
  DW_CUDA(cudaMemsetAsync(gacc, 0, nw * sizeof(float2), st));
  double num = 0, den = 0;
  double* dres = c->d_red + 65536 + 12288;
  for (int f = 0; f < nf; f += ng) {
    const int m = std::min(ng, nf - f);
    const float* x = (const float*)xv + f * fs;
    const float* y = (const float*)yv + f * fs;
    cudaError_t e = ptnet_forward_impl(c, W, x, out, h1, h2, g1, m, st);
    if (e != cudaSuccess) return dw_cuda_fail(e, "ptnet_loss_grad");
    // e = out - y ; loss numerator |e|^2, denominator |y|^2 (the fields of the group are contiguous)
    blas_axpy<float>(y, out, -1.0, 0.0, n * m, st);
    blas_dot<float>(c, out, out, n * m, dres, st);
    blas_dot<float>(c, y, y, n * m, dres + 3, st);
    // back-propagation: gradient of |e|^2 wrt the output is 2 e (the factor is in the reductions)
    if ((e = launch_dw<2>(c, h2, out, partial, gtmp + w1 + w2, m, st)) != cudaSuccess ||
        (e = launch_layer<1, true>(c, W + w1 + w2, out, g2, m, st)) != cudaSuccess ||
        (e = launch_dw<0>(c, g2, h1, partial, gtmp + w1, m, st)) != cudaSuccess ||
        (e = launch_layer<16, true>(c, W + w1, g2, g1, m, st)) != cudaSuccess ||
        (e = launch_dw<1>(c, g1, x, partial, gtmp, m, st)) != cudaSuccess)
      return dw_cuda_fail(e, "ptnet_loss_grad");
    blas_axpy<float>((const float*)gtmp, (float*)gacc, 1.0, 0.0, nw, st);
    DW_CUDA(cudaMemcpyAsync(c->h_red, dres, 6 * sizeof(double), cudaMemcpyDeviceToHost, st));
    DW_CUDA(cudaStreamSynchronize(st));
    num += c->h_red[2];
    den += c->h_red[5];
  }
  // normalise by sum |y|^2
  blas_scale<float>((float*)gacc, den > 0 ? 1.0 / den : 0.0, 0.0, nw, st);
  DW_CUDA(cudaMemcpyAsync(gradv, gacc, nw * sizeof(float2), cudaMemcpyDeviceToDevice, st));
  DW_CUDA(cudaStreamSynchronize(st));
  if (loss) *loss = den > 0 ? num / den : 0.0;
  return DW_OK;
}

extern "C" int ptnet_adam(size_t ncomplex, void* W, const void* grad, void* m, void* v, int step, double lr,
                          void* stream) {
  if (!W || !grad || !m || !v || step < 1) { dw_set_error("ptnet_adam: bad argument"); return DW_EINVAL; }
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  const size_t n = 2 * ncomplex;
  ptnet_adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      n, (float*)W, (const float*)grad, (float*)m, (float*)v, (float)lr, b1, b2, 1e-8f, c1, c2); dw_note_launch();
  DW_CUDA(cudaGetLastError());
  return DW_OK;
}

// the plain procedure (5.1) on nf packed FP32 fields in place: nsteps x (psi <- M_sap psi / |.|)
extern "C" int dfl_inverse_iteration(dw_ctx* c, int ncy, int nmr, int nsteps, int nf, void* fields, void* stream) {
  if (!c || !fields || nf < 1 || nsteps < 0) { dw_set_error("dfl_inverse_iteration: bad argument"); return DW_EINVAL; }
  cudaStream_t st = (cudaStream_t)stream;
  const size_t fs = (size_t)c->V * 24, n = (size_t)c->V * 12;
  float* tmp = nullptr;
  DW_CUDA(cudaMalloc(&tmp, fs * nf * sizeof(float)));
  float* f = (float*)fields;
  double* dres = c->d_red + 65536 + 16384;
  int rc = DW_OK;
  for (int it = 0; it < nsteps && rc == DW_OK; ++it) {
    rc = nf > 1 ? sap_apply_mrhs(c, ncy, nmr, f, tmp, nf, st) : sap_apply<float>(c, ncy, nmr, f, tmp, st);
    if (rc) break;
    for (int l = 0; l < nf; ++l) blas_dot<float>(c, tmp + l * fs, tmp + l * fs, n, dres + 3 * l, st);
    cudaError_t e = cudaMemcpyAsync(c->h_red, dres, 3 * nf * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { rc = dw_cuda_fail(e, "dfl_inverse_iteration"); break; }
    for (int l = 0; l < nf; ++l) blas_convert<float, float>(tmp + l * fs, f + l * fs, 1.0 / sqrt(c->h_red[3 * l + 2]), n, st);
  }
  cudaStreamSynchronize(st);
  cudaFree(tmp);
  return rc;
}
