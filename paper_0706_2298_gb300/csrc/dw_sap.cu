// Schwarz alternating procedure M_sap (Section 6.1; Section 5.3 uses it as
// the approximate inverse of the inverse iteration (5.1)).
//
//   xi = 0, r = rho; ncy times, for colour in (black, white):
//     for every block L of the colour: delta_L = MR_nmr(D^_L) applied to r|_L
//     xi += delta, r = rho - D xi
//
// GPU form.  One CTA per block of the current colour (blocks of one colour
// never touch).  The CTA keeps the block's even-odd MR iteration on chip:
//   * residual r|_L is read once; its boundary sites first receive the
//     change caused by the other colour's last correction (halo hops of
//     delta from the neighbouring blocks), so r = rho - D xi is maintained
//     exactly without a global operator application;
//   * r^_e = b_e - D_eo A_oo^{-1} b_o, then nmr MR steps
//         p = (A_ee - D_eo A_oo^{-1} D_oe) r^_e,  alpha = (p, r^)/|p|^2  (block reduction),
//         x_e += alpha r^_e,  r^_e -= alpha p
//     with r^_e and the odd intermediate in shared memory;
//   * odd reconstruction x_o = A_oo^{-1}(b_o - D_oe x_e);
//   * the new block residual is (r^_e, 0) exactly; it, the correction delta
//     and xi += delta are written back.
// Links and the clover term are read through the read-only cache.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <tuple>
#include <type_traits>

#include "dw_common.cuh"

namespace {

template <int MU, typename T, int SHV>
DW_D void inblock_dir(const Geom& g, const SiteRef& s, long long i, const uint16_t* nbe,
                      const T* __restrict__ links, const cplx<T>* sm, cplx<T>* acc) {
  const size_t V = g.V;
  SU3<T> U;
  cplx<T> p[12];
  uint16_t e = nbe[2 * MU];
  if (!(e >> 15)) {
    int hn = e & 0x7fff;
    load_link(links, V, MU, i, U);
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = sm[k * SHV + hn];
    hop_acc<MU, -1, false>(acc, p, U, T(1));
  }
  e = nbe[2 * MU + 1];
  if (!(e >> 15)) {
    int hn = e & 0x7fff;
    load_link(links, V, MU, site_index(g, s.b, 1 - s.p, hn), U);
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = sm[k * SHV + hn];
    hop_acc<MU, +1, true>(acc, p, U, T(1));
  }
}
template <typename T, int SHV>
DW_D void inblock_hops(const Geom& g, const SiteRef& s, long long i, const uint16_t* nbe,
                       const T* __restrict__ links, const cplx<T>* sm, cplx<T>* acc) {
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  inblock_dir<0, T, SHV>(g, s, i, nbe, links, sm, acc);
  inblock_dir<1, T, SHV>(g, s, i, nbe, links, sm, acc);
  inblock_dir<2, T, SHV>(g, s, i, nbe, links, sm, acc);
  inblock_dir<3, T, SHV>(g, s, i, nbe, links, sm, acc);
}

// acc += hops of a global field that cross the block boundary
template <int MU, typename T>
DW_D void halo_dir(const Geom& g, const SiteRef& s, long long i, const uint16_t* nbe,
                   const T* __restrict__ links, const T* __restrict__ f, cplx<T>* acc) {
  const size_t V = g.V;
  SU3<T> U;
  cplx<T> p[12];
  bool cr;
  if (nbe[2 * MU] >> 15) {
    long long j = neighbour(g, s, 2 * MU, &cr);
    T sg = time_wrap(g, s, 2 * MU) ? T(-1) : T(1);
    load_link(links, V, MU, i, U);
    load_site_rw<T, 12>(f, V, j, p);
    hop_acc<MU, -1, false>(acc, p, U, sg);
  }
  if (nbe[2 * MU + 1] >> 15) {
    long long j = neighbour(g, s, 2 * MU + 1, &cr);
    T sg = time_wrap(g, s, 2 * MU + 1) ? T(-1) : T(1);
    load_link(links, V, MU, j, U);
    load_site_rw<T, 12>(f, V, j, p);
    hop_acc<MU, +1, true>(acc, p, U, sg);
  }
}
template <typename T>
DW_D void halo_add(const Geom& g, const SiteRef& s, long long i, const uint16_t* nbe, const T* __restrict__ links,
                   const T* __restrict__ f, cplx<T>* b) {
  cplx<T> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {T(0), T(0)};
  halo_dir<0>(g, s, i, nbe, links, f, acc);
  halo_dir<1>(g, s, i, nbe, links, f, acc);
  halo_dir<2>(g, s, i, nbe, links, f, acc);
  halo_dir<3>(g, s, i, nbe, links, f, acc);
  // r - D delta on the boundary: D contributes -1/2 * hops
#pragma unroll
  for (int k = 0; k < 12; ++k) b[k] += T(0.5) * acc[k];
}

// sum over the lanes of a warp that hold block threads (SHV < 32: only SHV lanes exist)
template <int SHV>
DW_D double warp_sum(double v) {
  constexpr unsigned mask = SHV >= 32 ? 0xffffffffu : ((1u << SHV) - 1u);
#pragma unroll
  for (int o = (SHV >= 32 ? 16 : SHV / 2); o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  return v;
}

template <typename T, int SHV>
__global__ void __launch_bounds__(SHV) sap_block_kernel(Geom g, const T* __restrict__ links,
                                                        const T* __restrict__ clov, const T* __restrict__ clovinv,
                                                        const int* __restrict__ blocks, const T* rsrc, T* rdst,
                                                        const T* dprev, T* dout, T* xi, int first, int nmr) {
  constexpr int NW = (SHV + 31) / 32;
  extern __shared__ __align__(16) unsigned char sap_smem[];
  cplx<T>* s_r = reinterpret_cast<cplx<T>*>(sap_smem);   // r^_e
  cplx<T>* s_t = s_r + 12 * SHV;                          // odd intermediate, later x_e
  cplx<T>* s_b = s_t + 12 * SHV;                          // b_o (source on odd sites)
  __shared__ double s_red[3][NW];
  const size_t V = g.V;
  const int h = threadIdx.x;
  const int b = blocks[blockIdx.x];
  SiteRef se = {b, 0, h}, so = {b, 1, h};
  const long long ie = site_index(g, b, 0, h), io = site_index(g, b, 1, h);
  uint16_t nbe_e[8], nbe_o[8];
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    nbe_e[d] = __ldg(g.nbtab + (h << 3) + d);
    nbe_o[d] = __ldg(g.nbtab + ((SHV + h) << 3) + d);
  }
  cplx<T> v[12], w[12], acc[12];
  // ---- residual with halo correction
  load_site_rw<T, 12>(rsrc, V, io, v);
  if (dprev) halo_add(g, so, io, nbe_o, links, dprev, v);
#pragma unroll
  for (int k = 0; k < 12; ++k) s_b[k * SHV + h] = v[k];
  clover_apply(clovinv, V, io, v, w);                       // A_oo^{-1} b_o
#pragma unroll
  for (int k = 0; k < 12; ++k) s_t[k * SHV + h] = w[k];
  load_site_rw<T, 12>(rsrc, V, ie, v);
  if (dprev) halo_add(g, se, ie, nbe_e, links, dprev, v);
  __syncthreads();
  inblock_hops<T, SHV>(g, se, ie, nbe_e, links, s_t, acc);  // r^_e = b_e - D_eo A^{-1} b_o
  cplx<T> x[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    v[k] += T(0.5) * acc[k];
    s_r[k * SHV + h] = v[k];
    x[k] = {T(0), T(0)};
  }
  __syncthreads();
  // ---- minimal residual steps on the even-odd block operator
  for (int it = 0; it < nmr; ++it) {
    inblock_hops<T, SHV>(g, so, io, nbe_o, links, s_r, acc);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = T(-0.5) * acc[k];
    clover_apply(clovinv, V, io, acc, w);                   // A_oo^{-1} D_oe r^_e
    __syncthreads();                                        // all reads of s_t from the last step done
#pragma unroll
    for (int k = 0; k < 12; ++k) s_t[k * SHV + h] = w[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = s_r[k * SHV + h];
    clover_apply(clov, V, ie, v, w);                        // A_ee r^_e
    inblock_hops<T, SHV>(g, se, ie, nbe_e, links, s_t, acc);
    double pr = 0, pi = 0, pp = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      w[k] += T(0.5) * acc[k];                              // p = D^ r^
      pr += (double)w[k].re * v[k].re + (double)w[k].im * v[k].im;
      pi += (double)w[k].re * v[k].im - (double)w[k].im * v[k].re;
      pp += (double)w[k].re * w[k].re + (double)w[k].im * w[k].im;
    }
    pr = warp_sum<SHV>(pr); pi = warp_sum<SHV>(pi); pp = warp_sum<SHV>(pp);
    if ((h & 31) == 0) { s_red[0][h >> 5] = pr; s_red[1][h >> 5] = pi; s_red[2][h >> 5] = pp; }
    __syncthreads();
    pr = 0; pi = 0; pp = 0;
#pragma unroll
    for (int j = 0; j < NW; ++j) { pr += s_red[0][j]; pi += s_red[1][j]; pp += s_red[2][j]; }
    cplx<T> alpha = {T(0), T(0)};
    if (pp > 0) alpha = {(T)(pr / pp), (T)(pi / pp)};
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cmac(x[k], alpha, v[k]);
      cmsub(v[k], alpha, w[k]);
      s_r[k * SHV + h] = v[k];
    }
    __syncthreads();                                        // s_red reused, s_r complete
  }
  // ---- odd reconstruction x_o = A_oo^{-1}(b_o - D_oe x_e)
#pragma unroll
  for (int k = 0; k < 12; ++k) s_t[k * SHV + h] = x[k];
  __syncthreads();
  inblock_hops<T, SHV>(g, so, io, nbe_o, links, s_t, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = s_b[k * SHV + h] + T(0.5) * acc[k];
  clover_apply(clovinv, V, io, acc, w);                     // x_o
  // ---- outputs
  if (dout) {
    store_site<T, 12>(dout, V, ie, x);
    store_site<T, 12>(dout, V, io, w);
  }
  if (rdst) {
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = s_r[k * SHV + h];
    store_site<T, 12>(rdst, V, ie, v);
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = {T(0), T(0)};
    store_site<T, 12>(rdst, V, io, v);
  }
  if (!first) {
    load_site_rw<T, 12>(xi, V, ie, v);
#pragma unroll
    for (int k = 0; k < 12; ++k) x[k] += v[k];
    load_site_rw<T, 12>(xi, V, io, v);
#pragma unroll
    for (int k = 0; k < 12; ++k) w[k] += v[k];
  }
  store_site<T, 12>(xi, V, ie, x);
  store_site<T, 12>(xi, V, io, w);
}

// ============================================================================ staged FP32 kernel
// Same algorithm as sap_block_kernel, one thread per site of the block (thread t = site t: the even
// sites first, then the odd ones).  Every link product is done by the thread that owns the link:
//   * forward term of a hop: the destination x reads psi(x + mu) from shared memory and multiplies it
//     by its own U_mu(x);
//   * backward term: the source y forms U_mu(y)^+ (1 + gamma_mu) psi(y) from its own registers and
//     hands the half-spinor to y + mu through shared memory.
// So both parities work in each hop, and a link and a clover block are read by one thread only: they
// need not be in shared memory.  Blocks of 128 and 256 sites keep the links (72 reals per thread) and
// one chiral block of A_ee / A_oo^{-1} (36 reals) in tensor memory, used as a second register file
// (tcgen05.st / tcgen05.ld 32x32b: a thread's columns of its lane), the other chiral block, the vector,
// the half-spinors and x_e / b_o in shared memory: a block solve reads nothing from L2 between its first
// and last access.  Smaller blocks keep the links in shared memory and read the clover term from L2.
// While the odd sites apply A_oo^{-1}, the even ones apply A_ee.  The diagonal of the clover term, the largest part
// of the block operator, is added to each sum last: 1.1e-7 from FP64 (4 cycles of 4 steps), 1.5e-7 with the hops added to
// A_ee r^, at the same speed.
// Bound: instruction issue and latency (16 warps per SM at 128 registers and 98 KB, issue slots 57% busy);
// the rest is the two parities waiting for each other and tensor-memory loads.  48x24^3 on 4^4 blocks, 4
// cycles of 4 steps: 1.40 ms (22 TFLOP/s); links in shared memory and the whole clover term in tensor
// memory 1.60 ms; pulling both hop terms from shared memory with one thread per (site pair, spin) 1.78 ms.
template <int SHV>
struct SapCfg {
  static constexpr int NS = 2 * SHV;
  static constexpr bool TM = SHV >= 64;
  DW_HD static constexpr uint32_t tcols() { return SHV >= 128 ? 256 : 128; }   // columns of a CTA: 128 per warp of a lane quarter
  static constexpr int FIXED = TM ? NS * 144 : NS * 288;      // clover block 1, or the links
  static constexpr size_t bytes = (size_t)FIXED + (size_t)SHV * (12 + 6 + 12) * 16;
};

DW_D void tm_st16(uint32_t a, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
DW_D void tm_st2(uint32_t a, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(a), "r"(__float_as_uint(v[0])),
               "r"(__float_as_uint(v[1])) : "memory");
}
DW_D void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Loads from tensor memory and the wait for them in one statement: their registers are undefined until the wait, and a
// compiler may move or copy a value between two statements.
// 2 x 18 consecutive columns
DW_D void tm_ld36(uint32_t a, float* u, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%36];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%16,%17}, [%37];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33}, [%38];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%34,%35}, [%39];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(u[0]), "=f"(u[1]), "=f"(u[2]), "=f"(u[3]), "=f"(u[4]), "=f"(u[5]), "=f"(u[6]), "=f"(u[7]), "=f"(u[8]),
        "=f"(u[9]), "=f"(u[10]), "=f"(u[11]), "=f"(u[12]), "=f"(u[13]), "=f"(u[14]), "=f"(u[15]), "=f"(u[16]), "=f"(u[17]),
        "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]), "=f"(v[17])
      : "r"(a), "r"(a + 16), "r"(a + 18), "r"(a + 34));
}
// 30 and 6 consecutive columns
DW_D void tm_ld30(uint32_t a, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%30];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%31];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%28,%29}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]),
        "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]),
        "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29])
      : "r"(a), "r"(a + 16), "r"(a + 24), "r"(a + 28));
}
DW_D void tm_ld6(uint32_t a, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%6];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%4,%5}, [%7];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5])
      : "r"(a), "r"(a + 4));
}
// 18 consecutive columns, and while they are on their way the spinor at shared address s (6 units, SHV apart)
template <int SHV>
DW_D void tm_ld18_spinor(uint32_t a, uint32_t s, float* v, float* p) {
  constexpr int B = 16 * SHV;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%42];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%16,%17}, [%43];\n\t"
      "ld.shared.v4.f32 {%18,%19,%20,%21}, [%44];\n\t"
      "ld.shared.v4.f32 {%22,%23,%24,%25}, [%44+%45];\n\t"
      "ld.shared.v4.f32 {%26,%27,%28,%29}, [%44+%46];\n\t"
      "ld.shared.v4.f32 {%30,%31,%32,%33}, [%44+%47];\n\t"
      "ld.shared.v4.f32 {%34,%35,%36,%37}, [%44+%48];\n\t"
      "ld.shared.v4.f32 {%38,%39,%40,%41}, [%44+%49];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]), "=f"(v[17]),
        "=f"(p[0]), "=f"(p[1]), "=f"(p[2]), "=f"(p[3]), "=f"(p[4]), "=f"(p[5]), "=f"(p[6]), "=f"(p[7]), "=f"(p[8]),
        "=f"(p[9]), "=f"(p[10]), "=f"(p[11]), "=f"(p[12]), "=f"(p[13]), "=f"(p[14]), "=f"(p[15]), "=f"(p[16]), "=f"(p[17]),
        "=f"(p[18]), "=f"(p[19]), "=f"(p[20]), "=f"(p[21]), "=f"(p[22]), "=f"(p[23])
      : "r"(a), "r"(a + 16), "r"(s), "n"(B), "n"(2 * B), "n"(3 * B), "n"(4 * B), "n"(5 * B)
      : "memory");
}

// CTA barriers of a subset: wait for, or only announce, the arrival of n threads at barrier id
DW_D void bar_wait(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
DW_D void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// the block's data as thread t sees it
template <int SHV>
struct SapBlock {
  using Cfg = SapCfg<SHV>;
  static constexpr int NS = 2 * SHV;
  float4* fix4;     // TM: clover block 1, [9 units][NS]; else the links' complex 0..7, [4 mu][4 units][NS]
  float2* fix2;     // else: complex 8 of the links, [4 mu][NS]
  float4* half;     // [4 mu][3 units][SHV]  half-spinors of the backward terms, at the source's index
  float4* vec;      // [6 units][SHV]        r_e, t_o or x_e
  float4* xb;       // [6 units][NS]         x_e on the even sites, b_o on the odd ones
  uint32_t tm;      // this thread's tensor-memory address
  const float* cl;  // else: A_oo^{-1} (odd t) or A_ee (even t) in global memory
  int t;

  DW_D void set(unsigned char* p, int thread) {
    t = thread;
    fix4 = reinterpret_cast<float4*>(p);
    fix2 = reinterpret_cast<float2*>(p + (size_t)NS * 256);
    half = reinterpret_cast<float4*>(p + Cfg::FIXED);
    vec = half + 12 * SHV;
    xb = vec + 6 * SHV;
  }
  DW_D void stage(const float* __restrict__ links, const float* __restrict__ clover, size_t V, long long i) {
    cl = clover;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      SU3<float> U;
      load_link(links, V, mu, i, U);
      if constexpr (Cfg::TM) {
        tm_st16(tm + mu * 18, &U.m[0][0].re);
        tm_st2(tm + mu * 18 + 16, &U.m[2][2].re);
      } else {
        const cplx<float>* m = &U.m[0][0];
#pragma unroll
        for (int k = 0; k < 4; ++k) fix4[(mu * 4 + k) * NS + t] = pack_unit(m + 2 * k);
        fix2[mu * NS + t] = make_float2(m[8].re, m[8].im);
      }
    }
    if constexpr (Cfg::TM) {
      cplx<float> s[18];
      load_site<float, 18>(clover, V, i, s);
      tm_st16(tm + 72, &s[0].re);
      tm_st2(tm + 88, &s[8].re);
      tm_st16(tm + 90, &s[9].re);
      tm_st2(tm + 106, &s[17].re);
      const float4* q = reinterpret_cast<const float4*>(clover + 36 * V);
#pragma unroll
      for (int k = 0; k < 9; ++k) fix4[k * NS + t] = __ldg(q + (size_t)k * V + i);
      tm_wait_st();
    }
  }
  // the links of directions mu and mu + 1; whole warps only (tensor memory)
  DW_D void link_pair(int mu, SU3<float>& U, SU3<float>& N) const {
    if constexpr (Cfg::TM) {
      tm_ld36(tm + mu * 18, &U.m[0][0].re, &N.m[0][0].re);
    } else {
      link(mu, U);
      link(mu + 1, N);
    }
  }
  // a link and the spinor of vec at site `at`; whole warps only (tensor memory)
  DW_D void link_spinor(int mu, int at, SU3<float>& U, cplx<float>* f) const {
    if constexpr (Cfg::TM) {
      tm_ld18_spinor<SHV>(tm + mu * 18, smem_u32(vec + at), &U.m[0][0].re, &f[0].re);
    } else {
      link(mu, U);
      get(vec, SHV, at, f);
    }
  }
  // from shared memory
  DW_D void link(int mu, SU3<float>& U) const {
    cplx<float>* m = &U.m[0][0];
#pragma unroll
    for (int k = 0; k < 4; ++k) unpack_unit(fix4[(mu * 4 + k) * NS + t], m + 2 * k);
    const float2 l = fix2[mu * NS + t];
    m[8] = {l.x, l.y};
  }
  // The clover term, A_oo^{-1} (odd) or A_ee (even), in two parts, so that the diagonal products, the largest, can be
  // added last: y = its off-diagonal part times x, and its diagonal d[12]
  DW_D void clover_off(size_t V, long long i, const cplx<float>* x, cplx<float>* y) const {
    cplx<float> s[16];                                    // s[0]: the last diagonal pair, unused
    if constexpr (Cfg::TM) {
      tm_ld30(tm + 78, &s[1].re);
      herm6_off(s + 1, x, y);
#pragma unroll
      for (int k = 0; k < 8; ++k) unpack_unit(fix4[(k + 1) * NS + t], s + 2 * k);
      herm6_off(s + 1, x + 6, y + 6);
    } else {
      const float4* q = reinterpret_cast<const float4*>(cl) + i;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
#pragma unroll
        for (int k = 0; k < 8; ++k) unpack_unit(__ldg(q + (size_t)(9 * b + k + 1) * V), s + 2 * k);
        herm6_off(s + 1, x + 6 * b, y + 6 * b);
      }
    }
  }
  DW_D void clover_diag(size_t V, long long i, float* d) const {
    float4 u[2];
    if constexpr (Cfg::TM) {
      tm_ld6(tm + 72, d);
      u[0] = fix4[t];
      u[1] = fix4[NS + t];
    } else {
      const float4* q = reinterpret_cast<const float4*>(cl) + i;
      u[0] = __ldg(q);
      u[1] = __ldg(q + V);
      d[0] = u[0].x; d[1] = u[0].y; d[2] = u[0].z; d[3] = u[0].w; d[4] = u[1].x; d[5] = u[1].y;
      u[0] = __ldg(q + 9 * V);
      u[1] = __ldg(q + 10 * V);
    }
    d[6] = u[0].x; d[7] = u[0].y; d[8] = u[0].z; d[9] = u[0].w; d[10] = u[1].x; d[11] = u[1].y;
  }
  DW_D void put(float4* a, int stride, int at, const cplx<float>* f) const {
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k * stride + at] = pack_unit(f + 2 * k);
  }
  DW_D void get(const float4* a, int stride, int at, cplx<float>* f) const {
#pragma unroll
    for (int k = 0; k < 6; ++k) unpack_unit(a[k * stride + at], f + 2 * k);
  }
};

// the eight neighbour-table entries of a site (direction 2 mu forward, 2 mu + 1 backward)
struct SapNb {
  uint32_t w[4];
  DW_D bool in(int d) const { return !((w[d >> 1] >> ((d & 1) * 16 + 15)) & 1u); }
  DW_D int at(int d) const { return (int)((w[d >> 1] >> ((d & 1) * 16)) & 0x7fffu); }
};

// half-spinor w = W (1 + S gamma_mu) psi, W = U or U^+
template <int MU, int S, bool DAG>
DW_D void half_spinor(const cplx<float>* psi, const SU3<float>& U, cplx<float>* w) {
  cplx<float> hs[2][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    cplx<float> v0, v1;
    e_mul<MU>(psi[6 + c], psi[9 + c], v0, v1);
    if (S > 0) { hs[0][c] = psi[c] + v0; hs[1][c] = psi[3 + c] + v1; }
    else       { hs[0][c] = psi[c] - v0; hs[1][c] = psi[3 + c] - v1; }
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    if (DAG) su3_dag_mul(U, hs[a], w + 3 * a); else su3_mul(U, hs[a], w + 3 * a);
  }
}
// acc += the spinor [w ; S e_mu^+ w] of a half-spinor
template <int MU, int S>
DW_D void add_half(const cplx<float>* w, cplx<float>* acc) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    cplx<float> l0, l1;
    edag_mul<MU>(w[c], w[3 + c], l0, l1);
    acc[c] += w[c];
    acc[3 + c] += w[3 + c];
    if (S > 0) { acc[6 + c] += l0; acc[9 + c] += l1; }
    else       { acc[6 + c] -= l0; acc[9 + c] -= l1; }
  }
}

// acc += (1 - gamma_mu) U_mu(x) psi(x + mu), psi in the shared vector
template <int MU, int SHV>
DW_D void sap_forward(const SapBlock<SHV>& sb, const SapNb& nb, cplx<float>* acc) {
  SU3<float> U;
  cplx<float> p[12], w[6];
  sb.link_spinor(MU, nb.at(2 * MU), U, p);     // some site of the block where the hop leaves it
  if (nb.in(2 * MU)) {
    half_spinor<MU, -1, false>(p, U, w);
    add_half<MU, -1>(w, acc);
  }
}
// half-spinor U_mu(y)^+ (1 + gamma_mu) psi(y) of the owner's spinor
template <int MU, int SHV>
DW_D void sap_push(const SapBlock<SHV>& sb, const SapNb& nb, int h, const cplx<float>* psi, const SU3<float>& U) {
  if (nb.in(2 * MU)) {
    cplx<float> w[6];
    half_spinor<MU, +1, true>(psi, U, w);
#pragma unroll
    for (int k = 0; k < 3; ++k) sb.half[(MU * 3 + k) * SHV + h] = pack_unit(w + 2 * k);
  }
}
// acc += the backward term of direction mu, from the half-spinor of x - mu
template <int MU, int SHV>
DW_D void sap_gather(const SapBlock<SHV>& sb, const SapNb& nb, cplx<float>* acc) {
  if (nb.in(2 * MU + 1)) {
    const int hn = nb.at(2 * MU + 1);
    cplx<float> w[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) unpack_unit(sb.half[(MU * 3 + k) * SHV + hn], w + 2 * k);
    add_half<MU, +1>(w, acc);
  }
}

// Halo of a block: the hops of the neighbouring blocks' last correction f into the block's boundary
// sites.  One thread per (face, site of the face) forms the half-spinor, so that no lane idles on
// interior sites; the boundary sites then collect them from shared memory ([3 units][items], in the
// space of half, vec and xb, which is large enough for every block of 2 SHV sites).
struct SapFaces {
  uint32_t pos, wid;               // bytes: bit position and width of coordinate mu in the local index
  int off[9];                      // first item of each face (constant subscripts only)
  DW_D explicit SapFaces(const Geom& g) : pos(0), wid(0) {
    int at = 0;
#pragma unroll
    for (int mu = 3; mu >= 0; --mu) {
      const int w = 31 - __clz(g.sb[mu]);
      pos |= (uint32_t)at << (8 * mu);
      wid |= (uint32_t)w << (8 * mu);
      at += w;
    }
    off[0] = 0;
#pragma unroll
    for (int d = 0; d < 8; ++d) off[d + 1] = off[d] + (g.svol >> width(d >> 1));
  }
  DW_D int shift(int mu) const { return (int)((pos >> (8 * mu)) & 255u); }
  DW_D int width(int mu) const { return (int)((wid >> (8 * mu)) & 255u); }
  // local lexicographic index of face site j of direction d (forward: the last coordinate, backward: 0)
  DW_D int lex(int d, int j) const {
    const int s = shift(d >> 1), w = width(d >> 1), lo = j & ((1 << s) - 1);
    return ((j - lo) << w) | (((d & 1) ? 0 : (1 << w) - 1) << s) | lo;
  }
  DW_D int face(int d, int lx) const {
    const int s = shift(d >> 1), lo = lx & ((1 << s) - 1);
    return ((lx >> (s + width(d >> 1))) << s) | lo;
  }
  DW_D int parity(int lx) const { return ((lx >> shift(0)) ^ (lx >> shift(1)) ^ (lx >> shift(2)) ^ lx) & 1; }
};

template <int D>
DW_D void halo_item(const Geom& g, const SiteRef& s, long long i, const float* __restrict__ links, const float* f,
                    cplx<float>* w) {
  bool cr;
  const long long j = neighbour(g, s, D, &cr);
  SU3<float> U;
  cplx<float> p[12];
  load_link(links, (size_t)g.V, D >> 1, (D & 1) ? j : i, U);
  load_site_rw<float, 12>(f, (size_t)g.V, j, p);
  half_spinor<(D >> 1), (D & 1) ? +1 : -1, (D & 1) != 0>(p, U, w);
}

template <int D, int SHV>
DW_D void halo_gather(const SapFaces& fc, const float4* buf, const SapNb& nb, int lx, bool wrap, cplx<float>* acc) {
  if (nb.in(D)) return;
  const int at = fc.off[D] + fc.face(D, lx), n = fc.off[8];
  cplx<float> w[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) unpack_unit(buf[k * n + at], w + 2 * k);
  if (wrap) {
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = -w[k];
  }
  add_half<(D >> 1), (D & 1) ? +1 : -1>(w, acc);
}

// b += 1/2 hops of f across the block boundary (r - D delta on the boundary); all threads, with barriers
template <int SHV>
DW_D void sap_halo(const Geom& g, const SapBlock<SHV>& sb, const SapNb& nb, int b, const float* __restrict__ links,
                   const float* f, cplx<float>* v) {
  const SapFaces fc(g);
  float4* buf = sb.half;
  const int n = fc.off[8], t = sb.t;
  for (int it = t; it < n; it += 2 * SHV) {
    int d = 0, o = 0;
#pragma unroll
    for (int q = 1; q < 8; ++q)
      if (it >= fc.off[q]) { d = q; o = fc.off[q]; }
    const int lx = fc.lex(d, it - o);
    const SiteRef s = {b, fc.parity(lx), lx >> 1};
    const long long i = site_index(g, b, s.p, s.h);
    cplx<float> w[6];
    switch (d) {
      case 0: halo_item<0>(g, s, i, links, f, w); break;
      case 1: halo_item<1>(g, s, i, links, f, w); break;
      case 2: halo_item<2>(g, s, i, links, f, w); break;
      case 3: halo_item<3>(g, s, i, links, f, w); break;
      case 4: halo_item<4>(g, s, i, links, f, w); break;
      case 5: halo_item<5>(g, s, i, links, f, w); break;
      case 6: halo_item<6>(g, s, i, links, f, w); break;
      default: halo_item<7>(g, s, i, links, f, w); break;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) buf[k * n + it] = pack_unit(w + 2 * k);
  }
  __syncthreads();
  const int p = t >= SHV ? 1 : 0, h = t - p * SHV;
  int lx = 2 * h;
  lx |= fc.parity(lx) ^ p;
  const SiteRef s = {b, p, h};
  cplx<float> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {0.f, 0.f};
  halo_gather<0, SHV>(fc, buf, nb, lx, time_wrap(g, s, 0), acc);
  halo_gather<1, SHV>(fc, buf, nb, lx, time_wrap(g, s, 1), acc);
  halo_gather<2, SHV>(fc, buf, nb, lx, false, acc);
  halo_gather<3, SHV>(fc, buf, nb, lx, false, acc);
  halo_gather<4, SHV>(fc, buf, nb, lx, false, acc);
  halo_gather<5, SHV>(fc, buf, nb, lx, false, acc);
  halo_gather<6, SHV>(fc, buf, nb, lx, false, acc);
  halo_gather<7, SHV>(fc, buf, nb, lx, false, acc);
#pragma unroll
  for (int k = 0; k < 12; ++k) v[k] += 0.5f * acc[k];
  __syncthreads();
}

// right-hand sides rpc blockIdx.y .. of the blocks of one colour
template <int SHV>
__global__ void __launch_bounds__(2 * SHV, 256 / SHV) sap_staged_kernel(
    Geom g, const float* __restrict__ links, const float* __restrict__ clov, const float* __restrict__ clovinv,
    const int* __restrict__ blocks, const float* rsrc0, float* rdst0, const float* dprev0, float* dout0, float* xi0,
    int first, int nmr, int nrhs, int rpc, size_t fstride) {
  using Cfg = SapCfg<SHV>;
  constexpr int NW = SHV > 32 ? SHV / 32 : 1, NS = 2 * SHV;     // NW: warps of even sites
  extern __shared__ __align__(16) unsigned char sap_smem[];
  __shared__ float s_red[3][NW];
  __shared__ uint32_t s_tm;
  const size_t V = g.V;
  const int t = threadIdx.x, p = t >= SHV ? 1 : 0, h = t - p * SHV;
  const int b = blocks[blockIdx.x];
  const long long i = ((long long)b << g.lsvol) + t;
  SapBlock<SHV> sb;
  sb.set(sap_smem, t);
  if constexpr (Cfg::TM) {
    if (t < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tm)),
                   "r"(Cfg::tcols()) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int w = t >> 5;        // warp w reads lanes 32 (w mod 4) .. and the columns of its group of four warps
    sb.tm = s_tm + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(w >> 2) * 128u;
  }
  sb.stage(links, p ? clovinv : clov, V, i);
  SapNb nb;
  {
    const uint4 e = __ldg(reinterpret_cast<const uint4*>(g.nbtab) + t);
    nb.w[0] = e.x; nb.w[1] = e.y; nb.w[2] = e.z; nb.w[3] = e.w;
  }
  const int rhs1 = min(nrhs, (int)(blockIdx.y + 1) * rpc);
  for (int rhs = blockIdx.y * rpc; rhs < rhs1; ++rhs) {
    const size_t fo = (size_t)rhs * fstride;
    // f: the field this thread's site contributes to hops (t_o; r^_e, finally x_e); a: hop sums
    cplx<float> f[12], a[12];
    load_site_rw<float, 12>(rsrc0 + fo, V, i, f);
    if (dprev0) sap_halo<SHV>(g, sb, nb, b, links, dprev0 + fo, f);
#pragma unroll
    for (int k = 0; k < 12; ++k) a[k] = {0.f, 0.f};
    if (p) {                                  // b_o aside, t_o = A_oo^{-1} b_o
      sb.put(sb.xb, NS, t, f);
      float d[12];
      sb.clover_off(V, i, f, a);
      sb.clover_diag(V, i, d);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        f[k] = {fmaf(d[k], f[k].re, a[k].re), fmaf(d[k], f[k].im, a[k].im)};
        a[k] = {0.f, 0.f};
      }
      sb.put(sb.vec, SHV, h, f);
    } else {
      sb.put(sb.xb, NS, t, a);                // x_e = 0
    }
    __syncthreads();
    // half steps: s even: r^_e (s = 0) or D^ r^_e from t_o; s odd: t_o from r^_e (last: x_o from x_e)
    const int last = 2 * nmr + 1;
    for (int s = 0; s <= last; ++s) {
      const int dst = s & 1;
      if (p == dst) {
        sap_forward<0>(sb, nb, a);
        sap_forward<1>(sb, nb, a);
        sap_forward<2>(sb, nb, a);
        sap_forward<3>(sb, nb, a);
      } else {
        SU3<float> U, N;
        sb.link_pair(0, U, N);
        sap_push<0>(sb, nb, h, f, U);
        sap_push<1>(sb, nb, h, f, N);
        sb.link_pair(2, U, N);
        sap_push<2>(sb, nb, h, f, U);
        sap_push<3>(sb, nb, h, f, N);
      }
      // the half-spinors are complete; their writers need not wait
      if (SHV < 32) __syncthreads();
      else if (p == dst) bar_wait(1, NS);
      else bar_arrive(1, NS);
      if (p == dst) {
        sap_gather<0>(sb, nb, a);
        sap_gather<1>(sb, nb, a);
        sap_gather<2>(sb, nb, a);
        sap_gather<3>(sb, nb, a);
      }
      if (dst) {
        // odd: t_o = -1/2 A_oo^{-1} hops, or at the end x_o = A_oo^{-1}(b_o + 1/2 hops);
        // even: the off-diagonal part of 2 A_ee r^ (doubled: the hops added to it are halved below)
        cplx<float> y[12];
        if (p) {
          if (s == last) sb.get(sb.xb, NS, t, f);
#pragma unroll
          for (int k = 0; k < 12; ++k) f[k] = s == last ? f[k] + 0.5f * a[k] : -0.5f * a[k];
        }
        if (p || s < last) {
          sb.clover_off(V, i, f, y);
          if (p) {
            float d[12];
            sb.clover_diag(V, i, d);
#pragma unroll
            for (int k = 0; k < 12; ++k) {
              f[k] = {fmaf(d[k], f[k].re, y[k].re), fmaf(d[k], f[k].im, y[k].im)};
              a[k] = {0.f, 0.f};
            }
          } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) a[k] = 2.f * y[k];
          }
        }
        if (s == last) break;
        if (p) sb.put(sb.vec, SHV, h, f);
      } else {
        if (s == 0) {                         // r^_e = b_e - D_eo t_o = b_e + 1/2 hops
          if (!p) {
#pragma unroll
            for (int k = 0; k < 12; ++k) f[k] += 0.5f * a[k];
          }
        } else {                              // minimal-residual step with p = A_ee r^ - D_eo t_o = a / 2
          float pr = 0.f, pi = 0.f, pp = 0.f;
          if (!p) {
            float d[12];
            sb.clover_diag(V, i, d);
#pragma unroll
            for (int k = 0; k < 12; ++k) {                // the largest term of p, d r^, is added last
              a[k] = {fmaf(d[k], f[k].re, 0.5f * a[k].re), fmaf(d[k], f[k].im, 0.5f * a[k].im)};
              pr += a[k].re * f[k].re + a[k].im * f[k].im;
              pi += a[k].re * f[k].im - a[k].im * f[k].re;
              pp += a[k].re * a[k].re + a[k].im * a[k].im;
            }
          }
          // sum over the even sites: their warps only (one warp holds both parities when SHV = 16)
          if (SHV < 32 || !p) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
              pr += __shfl_xor_sync(0xffffffffu, pr, o);
              pi += __shfl_xor_sync(0xffffffffu, pi, o);
              pp += __shfl_xor_sync(0xffffffffu, pp, o);
            }
            if constexpr (NW > 1) {
              if ((t & 31) == 0) { s_red[0][t >> 5] = pr; s_red[1][t >> 5] = pi; s_red[2][t >> 5] = pp; }
              bar_wait(2, SHV);
              pr = 0.f; pi = 0.f; pp = 0.f;
#pragma unroll
              for (int j = 0; j < NW; ++j) { pr += s_red[0][j]; pi += s_red[1][j]; pp += s_red[2][j]; }
            }
          }
          if (!p) {
            cplx<float> al = {0.f, 0.f};
            if (pp > 0.f) al = {pr / pp, pi / pp};
#pragma unroll
            for (int k = 0; k < 6; ++k) {
              cplx<float> x[2];
              unpack_unit(sb.xb[k * NS + t], x);
              cmac(x[0], al, f[2 * k]);
              cmac(x[1], al, f[2 * k + 1]);
              sb.xb[k * NS + t] = pack_unit(x);
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) cmsub(f[k], al, a[k]);
          }
        }
        if (!p) {
          if (s + 1 == last) {                // the new residual on the even sites; x_e goes on
            if (rdst0) store_site<float, 12>(rdst0 + fo, V, i, f);
            sb.get(sb.xb, NS, t, f);
          }
          sb.put(sb.vec, SHV, h, f);
        }
      }
      __syncthreads();
    }
    // f = x_e, x_o; the new residual vanishes on the odd sites
    if (rdst0 && p) {
#pragma unroll
      for (int k = 0; k < 12; ++k) a[k] = {0.f, 0.f};
      store_site<float, 12>(rdst0 + fo, V, i, a);
    }
    if (dout0) store_site<float, 12>(dout0 + fo, V, i, f);
    if (!first) {
      load_site_rw<float, 12>(xi0 + fo, V, i, a);
#pragma unroll
      for (int k = 0; k < 12; ++k) f[k] += a[k];
    }
    store_site<float, 12>(xi0 + fo, V, i, f);
    __syncthreads();             // the next right-hand side writes half, vec and xb
  }
  if constexpr (Cfg::TM) {
    // every warp's tensor-memory accesses come before the columns are given back
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (t < 32)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tm), "r"(Cfg::tcols())
                   : "memory");
  }
}

// Right-hand sides per CTA of a batch.  A CTA that takes several stages the block once for all of them,
// but too few CTAs leave SMs idle: the number of waves times the work of a CTA is made smallest (staging
// costs about 0.1 of a block solve).  20 fields at 24x16^3 (192 blocks of a colour, 304 CTAs resident):
// 3.35 ms; one CTA for all fields of a block 6.86 ms with the kernel this one replaced.
inline int sap_rhs_per_cta(int nblocks, int nrhs, int slots) {
  int best = nrhs;
  double best_t = 1e300;
  for (int g = 1; g <= nrhs; ++g) {
    const int rpc = (nrhs + g - 1) / g;
    const long long ctas = (long long)nblocks * ((nrhs + rpc - 1) / rpc);
    const double t = (double)((ctas + slots - 1) / slots) * (rpc + 0.1);
    if (t < best_t * 0.999) { best_t = t; best = rpc; }
  }
  return best;
}

template <int SHV>
bool launch_sap_staged(dw_ctx* c, int colour, const float* rsrc, float* rdst, const float* dprev, float* dout,
                       float* xi, int first, int nmr, cudaStream_t st, int nrhs = 1) {
  constexpr size_t smem = SapCfg<SHV>::bytes;
  if (dw_smem_limit<sap_staged_kernel<SHV>>(smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const int* list = c->d_colour_list + (colour ? c->ncolour[0] : 0);
  const int slots = c->sms * (256 / SHV);                                // resident CTAs (launch bounds)
  const int rpc = sap_rhs_per_cta(c->ncolour[colour], nrhs, slots);
  const dim3 grid((unsigned)c->ncolour[colour], (unsigned)((nrhs + rpc - 1) / rpc));
  sap_staged_kernel<SHV><<<grid, 2 * SHV, smem, st>>>(c->g, (const float*)c->links[DW_F32],
                                                      (const float*)c->clov[DW_F32],
                                                      (const float*)c->clovinv[DW_F32], list, rsrc,
                                                      rdst, dprev, dout, xi, first, nmr, nrhs, rpc,
                                                      (size_t)c->V * 24); dw_note_launch();
  return true;
}

template <typename T, int SHV>
void launch_sap(dw_ctx* c, int colour, const T* rsrc, T* rdst, const T* dprev, T* dout, T* xi, int first, int nmr,
                cudaStream_t st) {
  constexpr int P = prec_of<T>();
  const int* list = c->d_colour_list + (colour ? c->ncolour[0] : 0);
  constexpr size_t smem = 3 * 12 * SHV * sizeof(cplx<T>);
  dw_smem_limit<sap_block_kernel<T, SHV>>(smem);         // a failure shows at the launch
  sap_block_kernel<T, SHV><<<c->ncolour[colour], SHV, smem, st>>>(c->g, (const T*)c->links[P], (const T*)c->clov[P],
                                                              (const T*)c->clovinv[P], list, rsrc, rdst, dprev,
                                                              dout, xi, first, nmr); dw_note_launch();
}

}  // namespace

static dw_ctx* g_tune_ctx = nullptr;   // context whose autotuned choice applies to the current call
static bool use_staged() {
  const char* e = getenv("DW_SAP_STAGED");
  if (e) return e[0] != '0';
  return g_tune_ctx ? g_tune_ctx->tune_sap_staged != 0 : true;
}

template <typename T>
int sap_apply(dw_ctx* c, int ncy, int nmr, const T* rho, T* xi, cudaStream_t st) {
  g_tune_ctx = c;
  constexpr int P = prec_of<T>();
  size_t bytes = dw_field_bytes(c, P);
  if (!c->sap_r[P]) DW_CUDA(cudaMalloc(&c->sap_r[P], bytes * (P == DW_F32 && c->sap_cap > 1 ? c->sap_cap : 1)));
  if (!c->sap_d[P]) DW_CUDA(cudaMalloc(&c->sap_d[P], bytes * (P == DW_F32 && c->sap_cap > 1 ? c->sap_cap : 1)));
  if (ncy <= 0) {
    DW_CUDA(cudaMemsetAsync(xi, 0, bytes, st));
    return DW_OK;
  }
  T* r = (T*)c->sap_r[P];
  T* d = (T*)c->sap_d[P];
  for (int cy = 0; cy < ncy; ++cy)
    for (int col = 0; col < 2; ++col) {
      bool last = (cy == ncy - 1 && col == 1);
      const T* rsrc = cy == 0 ? rho : r;
      T* rdst = last ? nullptr : r;
      const T* dprev = (cy == 0 && col == 0) ? nullptr : d;
      T* dout = last ? nullptr : d;
      int first = cy == 0;
      if (std::is_same<T, float>::value && use_staged()) {
        bool ok = false;
        const float* rs = (const float*)rsrc; float* rd = (float*)rdst; const float* dp = (const float*)dprev;
        float* dd = (float*)dout; float* xx = (float*)xi;
        switch (c->g.shv) {
          case 16: ok = launch_sap_staged<16>(c, col, rs, rd, dp, dd, xx, first, nmr, st); break;
          case 32: ok = launch_sap_staged<32>(c, col, rs, rd, dp, dd, xx, first, nmr, st); break;
          case 64: ok = launch_sap_staged<64>(c, col, rs, rd, dp, dd, xx, first, nmr, st); break;
          case 128: ok = launch_sap_staged<128>(c, col, rs, rd, dp, dd, xx, first, nmr, st); break;
          default: break;
        }
        if (ok) continue;
      }
      switch (c->g.shv) {
        case 8: launch_sap<T, 8>(c, col, rsrc, rdst, dprev, dout, xi, first, nmr, st); break;
        case 16: launch_sap<T, 16>(c, col, rsrc, rdst, dprev, dout, xi, first, nmr, st); break;
        case 32: launch_sap<T, 32>(c, col, rsrc, rdst, dprev, dout, xi, first, nmr, st); break;
        case 64: launch_sap<T, 64>(c, col, rsrc, rdst, dprev, dout, xi, first, nmr, st); break;
        case 128: launch_sap<T, 128>(c, col, rsrc, rdst, dprev, dout, xi, first, nmr, st); break;
        default:
          dw_set_error("sap_precondition: unsupported Schwarz block volume");
          return DW_EINVAL;
      }
    }
  DW_CUDA(cudaGetLastError());
  return DW_OK;
}
// M_sap on nrhs FP32 fields at once (staged kernel; falls back to one field at a time)
int sap_apply_mrhs(dw_ctx* c, int ncy, int nmr, const float* rho, float* xi, int nrhs, cudaStream_t st) {
  g_tune_ctx = c;
  const size_t fb = dw_field_bytes(c, DW_F32);
  if (c->sap_cap < nrhs) {
    sap_graphs_free(c);   // captured graphs refer to the old workspace
    for (int P = 0; P < 2; ++P) {
      if (c->sap_r[P]) { cudaFree(c->sap_r[P]); c->sap_r[P] = nullptr; }
      if (c->sap_d[P]) { cudaFree(c->sap_d[P]); c->sap_d[P] = nullptr; }
    }
    DW_CUDA(cudaMalloc(&c->sap_r[DW_F32], fb * nrhs));
    DW_CUDA(cudaMalloc(&c->sap_d[DW_F32], fb * nrhs));
    c->sap_cap = nrhs;
  }
  const size_t fs = (size_t)c->V * 24;
  if (ncy <= 0) {
    DW_CUDA(cudaMemsetAsync(xi, 0, fb * nrhs, st));
    return DW_OK;
  }
  if (!use_staged() || c->g.shv < 16 || c->g.shv > 128) {
    for (int r = 0; r < nrhs; ++r) {
      int rc = sap_apply<float>(c, ncy, nmr, rho + r * fs, xi + r * fs, st);
      if (rc) return rc;
    }
    return DW_OK;
  }
  float* r = (float*)c->sap_r[DW_F32];
  float* d = (float*)c->sap_d[DW_F32];
  for (int cy = 0; cy < ncy; ++cy)
    for (int col = 0; col < 2; ++col) {
      bool last = (cy == ncy - 1 && col == 1);
      const float* rsrc = cy == 0 ? rho : r;
      float* rdst = last ? nullptr : r;
      const float* dprev = (cy == 0 && col == 0) ? nullptr : d;
      float* dout = last ? nullptr : d;
      bool ok = false;
      switch (c->g.shv) {
        case 16: ok = launch_sap_staged<16>(c, col, rsrc, rdst, dprev, dout, xi, cy == 0, nmr, st, nrhs); break;
        case 32: ok = launch_sap_staged<32>(c, col, rsrc, rdst, dprev, dout, xi, cy == 0, nmr, st, nrhs); break;
        case 64: ok = launch_sap_staged<64>(c, col, rsrc, rdst, dprev, dout, xi, cy == 0, nmr, st, nrhs); break;
        case 128: ok = launch_sap_staged<128>(c, col, rsrc, rdst, dprev, dout, xi, cy == 0, nmr, st, nrhs); break;
        default: break;
      }
      if (!ok) {
        dw_set_error("sap_apply_mrhs: staged kernel unavailable");
        return DW_EINVAL;
      }
    }
  DW_CUDA(cudaGetLastError());
  return DW_OK;
}

// ---------------------------------------------------------------- CUDA graphs of M_sap
struct SapGraph {
  int uses = 0;
  cudaGraphExec_t exec = nullptr;
  int nodes = 0;
};
using SapKey = std::tuple<const void*, void*, int, int, int>;
using SapGraphMap = std::map<SapKey, SapGraph>;

void sap_graphs_free(dw_ctx* c) {
  if (!c->graph_cache) return;
  auto* m = static_cast<SapGraphMap*>(c->graph_cache);
  for (auto& kv : *m)
    if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
  delete m;
  c->graph_cache = nullptr;
}

static bool graphs_enabled() {
  const char* e = getenv("DW_GRAPH");
  return !(e && e[0] == '0');
}

int sap_apply_mrhs_graph(dw_ctx* c, int ncy, int nmr, const float* rho, float* xi, int nrhs, cudaStream_t st) {
  if (!graphs_enabled() || c->sap_cap < nrhs) return sap_apply_mrhs(c, ncy, nmr, rho, xi, nrhs, st);
  if (!c->graph_cache) c->graph_cache = new SapGraphMap();
  auto& m = *static_cast<SapGraphMap*>(c->graph_cache);
  SapGraph& gph = m[SapKey(rho, xi, nrhs, ncy, nmr)];
  if (!gph.exec) {
    if (gph.uses++ == 0) return sap_apply_mrhs(c, ncy, nmr, rho, xi, nrhs, st);   // first use: run directly
    if (!c->cap_stream) DW_CUDA(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
    cudaGraph_t graph;
    const long long n0 = dw_launch_count();
    DW_CUDA(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
    int rc = sap_apply_mrhs(c, ncy, nmr, rho, xi, nrhs, c->cap_stream);
    cudaError_t e = cudaStreamEndCapture(c->cap_stream, &graph);
    if (rc) return rc;
    if (e != cudaSuccess) return dw_cuda_fail(e, "cudaStreamEndCapture");
    gph.nodes = (int)(dw_launch_count() - n0);
    e = cudaGraphInstantiate(&gph.exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) { gph.exec = nullptr; return dw_cuda_fail(e, "cudaGraphInstantiate"); }
  }
  DW_CUDA(cudaGraphLaunch(gph.exec, st));
  for (int i = 0; i < gph.nodes; ++i) dw_note_launch();   // the graph's kernels
  return DW_OK;
}

// ---------------------------------------------------------------- autotuner
// Times the candidate launch shapes on this lattice with CUDA events (median of 5 after 2 warm-ups)
// and keeps the fastest: the multi-RHS D as one thread per (site, right-hand side) with the chunks
// interleaved, or one thread per site with 1, 2 or 3 right-hand sides per pass; the staged or
// generic FP32 Schwarz kernel.
extern "C" int dw_autotune(dw_ctx* c, int nrhs, char* report, size_t report_len) {
  if (!c || nrhs < 1 || nrhs > 64) { dw_set_error("dw_autotune: bad argument"); return DW_EINVAL; }
  const size_t fb = dw_field_bytes(c, DW_F32);
  float *x = nullptr, *y = nullptr;
  DW_CUDA(cudaMalloc(&x, fb * nrhs));
  cudaError_t e = cudaMalloc(&y, fb * nrhs);
  if (e != cudaSuccess) { cudaFree(x); return dw_cuda_fail(e, "cudaMalloc"); }
  cudaMemset(x, 0, fb * nrhs);
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  auto time_it = [&](auto fn) {
    std::vector<float> ts;
    for (int it = 0; it < 7; ++it) {
      cudaEventRecord(a, 0);
      fn();
      cudaEventRecord(b, 0);
      cudaEventSynchronize(b);
      float ms = 0;
      cudaEventElapsedTime(&ms, a, b);
      if (it >= 2) ts.push_back(ms);
    }
    std::sort(ts.begin(), ts.end());
    return ts[ts.size() / 2];
  };
  float td[4] = {0, 0, 0, 0};
  int best_r = 0;
  for (int rg = 0; rg <= 3; ++rg) {     // 0: one thread per (site, right-hand side), chunk-interleaved
    td[rg] = time_it([&] { dirac_mrhs<float>(c, x, y, nrhs, rg, 0); });
    if (td[rg] < td[best_r]) best_r = rg;
  }
  c->tune_rgroup = best_r;
  float ts[2] = {0, 0};
  const char* env = getenv("DW_SAP_STAGED");
  for (int st = 0; st < 2; ++st) {
    c->tune_sap_staged = st;
    if (!env) ts[st] = time_it([&] { sap_apply<float>(c, 1, 4, x, y, 0); });
  }
  c->tune_sap_staged = (env || ts[1] <= ts[0]) ? 1 : 0;
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(x);
  cudaFree(y);
  if (report && report_len) {
    snprintf(report, report_len,
             "{\"nrhs\": %d, \"dirac_mrhs_ms\": {\"interleaved\": %.4f, \"1\": %.4f, \"2\": %.4f, \"3\": %.4f}, "
             "\"rgroup\": %d, "
             "\"sap_pass_ms\": {\"generic\": %.4f, \"staged\": %.4f}, \"sap_staged\": %d}",
             nrhs, td[0], td[1], td[2], td[3], best_r, ts[0], ts[1], c->tune_sap_staged);
  }
  DW_CUDA(cudaGetLastError());
  return DW_OK;
}

template int sap_apply<float>(dw_ctx*, int, int, const float*, float*, cudaStream_t);
template int sap_apply<double>(dw_ctx*, int, int, const double*, double*, cudaStream_t);

extern "C" int sap_precondition(dw_ctx* c, int prec, int ncy, int nmr, int nrhs, const void* rho, void* xi,
                                void* stream) {
  if (!c || !rho || !xi || rho == xi || nrhs < 1 || nmr < 0 || (prec != DW_F64 && prec != DW_F32)) {
    dw_set_error("sap_precondition: bad argument");
    return DW_EINVAL;
  }
  if (int rc = dw_check_device(c, "sap_precondition")) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  size_t n = (size_t)c->V * 24;
  if (prec == DW_F32 && nrhs > 1) return sap_apply_mrhs(c, ncy, nmr, (const float*)rho, (float*)xi, nrhs, st);
  for (int r = 0; r < nrhs; ++r) {
    int rc = prec == DW_F64 ? sap_apply(c, ncy, nmr, (const double*)rho + r * n, (double*)xi + r * n, st)
                            : sap_apply(c, ncy, nmr, (const float*)rho + r * n, (float*)xi + r * n, st);
    if (rc) return rc;
  }
  return DW_OK;
}
