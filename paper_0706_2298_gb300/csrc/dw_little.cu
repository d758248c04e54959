// FP32 little GCR (Appendix A.2-A.4) of one system: one persistent CTA of 16 warps per SM, cooperative
// launch.  Every CTA owns a range of block rows of both parities.
//
// A hop is a list of tasks (block row q, direction d): a warp reads the Ns x Ns complex block with
// ceil(Ns^2 / 64) fully coalesced 16-byte loads per lane (lane = position in the column-major block, so a
// lane holds two rows of every G-th column) straight into registers, one task ahead of the products, and
// the first block of the next hop is on its way while the CTA passes the grid barrier and the reductions
// between the hops.  The products take the vector from shared memory, the G column groups meet by
// shuffles and the eight directions in shared memory.
// The CTA's slices of g, B^ g and chi'_j stay in shared memory (where they fit), so the inner products and
// updates of a step touch no L2.
// Bound: latency and instruction issue of short phases at 4 warps per scheduler (16 warps of 128 registers;
// L2 would deliver the 75 MB of an iteration in 4 us).  Time per iteration: Nb = 2592, Ns = 20: 23.7 us, with
// a shared-memory ring of bulk copies and 8 warps 34.8 us; Nb = 384: 16.7 (20.5) us; Nb = 32, Ns = 16: 14.6
// (18.7) us.  Two blocks in registers per warp spill and cost 3.7 us more, 8 warps with two blocks 2.6 us; blocks
// kept in tensor memory or staged in shared memory save L2 reads that are not the bound (6.5 us more: the code for
// several sources of blocks costs more issue slots).
// A step has three grid barriers: between its hops, after c = B^ rho_k, where (g_l, c), (chi'_j, c) and the CTA
// shares of |rho_k|^2 are reduced, and after chi'_k is formed, where (chi'_k, rho_k), |chi'_k|^2 and (B^ g_l, chi'_k)
// are summed from chi'_k itself.  The coefficients of P~_L c on chi'_j follow from (chi'_j, c) and the stored
// (B^ g_l, chi'_j).  The last barrier also publishes chi'_k, so that the residual of a step needs none of its own:
// the next odd hop forms rho_{k+1} = rho_k - alpha chi'_k from the two vectors as it gathers them.
// Reductions: FP64 atomics into one of three rotating accumulator sets, one grid barrier, then every CTA
// reads the totals.  A value has four accumulators (a quarter of the CTAs each): the atomics on one address
// are served one after the other, and 132 values of 152 CTAs take 3.5 us with one accumulator, 2.1 us with
// four, 2.6 us with 16 (barrier alone 1.3 us; one flag per CTA polled by all 2.7 us).
#include "dw_little.cuh"

#include <algorithm>
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace {

using cf = cplx<float>;
constexpr int LT = 512, LW = LT / 32, LROW = LW / 8;      // LROW: rows worked on at once
constexpr int LCH = 16;               // block rows per hop chunk
constexpr int LPART = 8;              // threads that share a row of a small matrix-vector product

template <int NS>
struct Lay {
  static constexpr int HR = NS / 2;                       // 16-byte units per column
  static constexpr int G = 32 / HR;                       // columns per pass of a warp
  static constexpr int U = NS * HR;                       // units per block
  static constexpr int P = (U + G * HR - 1) / (G * HR);   // passes
};

struct LShared {
  float ws[LW][4];
  float cta[LITTLE_NV];      // this CTA's share of the values being reduced
  float res[LITTLE_NV];      // grid-wide sums
  float c2[LITTLE_NKV];      // |chi'_j|^2
  cf al[LITTLE_NKV];         // (chi'_j, rho_j)
  cf beta[LITTLE_NKV];       // solution coefficients
  cf be[LITTLE_NKV][LITTLE_NKV];   // [j][k]: (chi'_j, P~_L c_k) / |chi'_j|^2
  cf tg[LITTLE_NKV][32];     // (B^ g_l, chi'_j) of the current cycle
  cf z[32];                  // A~^{-1} g^+ c
  cf ainv[32 * 32];          // A~^{-1}, row-major
  cf ac;                     // alpha_{k-1}
  float rr;                  // this CTA's share of |rho_k|^2 (folded into the next reduction)
  int phase;
};

DW_D cf ldcg(const cf* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
DW_D float wsum(float y) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
  return y;
}

// one block in registers
template <int NS>
struct Block {
  float4 m[Lay<NS>::P];
  DW_D void load(const float4* __restrict__ b, int lane) {
    using L = Lay<NS>;
#pragma unroll
    for (int p = 0; p < L::P; ++p) {
      const int u = p * L::G * L::HR + lane;
      m[p] = lane < L::G * L::HR && u < L::U ? __ldg(b + u) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  // rows 2r, 2r+1 of block times x (on lanes r < HR)
  DW_D float4 mv(const cf* x, int lane) const {
    using L = Lay<NS>;
    const int g = lane / L::HR;
    cf a0 = {0.f, 0.f}, a1 = {0.f, 0.f};
#pragma unroll
    for (int p = 0; p < L::P; ++p) {
      const int c = p * L::G + g;
      const cf xc = x[c < NS ? c : NS - 1];               // blocks are zero past the last column
      cmac(a0, cf{m[p].x, m[p].y}, xc);
      cmac(a1, cf{m[p].z, m[p].w}, xc);
    }
    float4 s = make_float4(a0.re, a0.im, a1.re, a1.im);
#pragma unroll
    for (int q = 1; q < L::G; ++q) {
      const int src = (lane + q * L::HR) & 31;
      s.x += __shfl_sync(0xffffffffu, a0.re, src);
      s.y += __shfl_sync(0xffffffffu, a0.im, src);
      s.z += __shfl_sync(0xffffffffu, a1.re, src);
      s.w += __shfl_sync(0xffffffffu, a1.im, src);
    }
    return s;
  }
};

// this CTA's rows of one parity
struct Rows {
  int first, n;
  const int* L;      // shared: block of each row
  const int* J;      // shared: neighbours' positions, [row][8]
};

template <int NS>
DW_D void preload(Block<NS>& buf, const float4* M, const Rows& r, int w, int lane) {
  if ((w >> 3) < r.n) buf.load(M + ((size_t)r.L[w >> 3] * 8 + (w & 7)) * Lay<NS>::U, lane);
}

// f(entry, sum) for every entry of this CTA's rows, sum = sum_d M[row][d] (src - cs corr)[neighbour d]
// (corr may be null); buf holds the warp's first block and is left with that of `next`.  Ends with a CTA
// barrier.
template <int NS, typename F>
DW_D void hop(Block<NS>& buf, const float4* M, const Rows& rows, const Rows& next, const cf* src, const cf* corr,
              cf cs, cf* xs, cf* hp, F&& f) {
  const int t = threadIdx.x, w = t >> 5, lane = t & 31, d = w & 7, qo = w >> 3;
  for (int r0 = 0; r0 < rows.n; r0 += LCH) {
    const int nc = min(LCH, rows.n - r0), ne = nc * 8 * NS;
    for (int e0 = t; e0 < ne; e0 += 4 * LT) {            // the gathers of a chunk are in flight together
      cf x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * LT;
        if (e < ne) {
          const int task = e / NS;
          const size_t at = (size_t)rows.J[r0 * 8 + task] * NS + (e - task * NS);
          x[u] = ldcg(src + at);
          if (corr) y[u] = ldcg(corr + at);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * LT;
        if (e < ne) {
          if (corr) cmsub(x[u], cs, y[u]);
          xs[e] = x[u];
        }
      }
    }
    __syncthreads();
    for (int q = qo; q < nc; q += LROW) {
      const float4 s = buf.mv(xs + (q * 8 + d) * NS, lane);
      const int qn = r0 + q + LROW;
      if (qn < rows.n) buf.load(M + ((size_t)rows.L[qn] * 8 + d) * Lay<NS>::U, lane);
      if (lane < Lay<NS>::HR) reinterpret_cast<float4*>(hp + (q * 8 + d) * NS)[lane] = s;
    }
    __syncthreads();
    for (int e = t; e < nc * NS; e += LT) {
      const int q = e / NS, k = e - q * NS;
      cf sum = hp[q * 8 * NS + k];
#pragma unroll
      for (int dd = 1; dd < 8; ++dd) sum += hp[(q * 8 + dd) * NS + k];
      f(r0 * NS + e, sum);
    }
    if (r0 + LCH < rows.n) __syncthreads();
  }
  preload<NS>(buf, M, next, w, lane);
  __syncthreads();
}

DW_D void grid_barrier(cg::grid_group& grid) {
  __syncthreads();
  grid.sync();
  __syncthreads();
}

// sh.cta[0..nv) summed over all CTAs into sh.res
DW_D void reduce(cg::grid_group& grid, LShared& sh, int nv, double* acc_base) {
  constexpr int SET = LITTLE_COPIES * LITTLE_NV;
  __syncthreads();
  const int t = threadIdx.x;
  double* acc = acc_base + (size_t)(sh.phase % 3) * SET;
  if (t < nv) atomicAdd(acc + (blockIdx.x % LITTLE_COPIES) * LITTLE_NV + t, (double)sh.cta[t]);
  grid_barrier(grid);
  if (t < nv) {
    double x[LITTLE_COPIES];
#pragma unroll
    for (int c = 0; c < LITTLE_COPIES; ++c) x[c] = __ldcg(acc + c * LITTLE_NV + t);
    sh.res[t] = (float)((x[0] + x[1]) + (x[2] + x[3]));
  }
  // the set used two reductions ahead was last read before this barrier
  if (blockIdx.x < LITTLE_COPIES && t < LITTLE_NV)
    acc_base[(size_t)((sh.phase + 2) % 3) * SET + blockIdx.x * LITTLE_NV + t] = 0.0;
  __syncthreads();
  if (t == 0) sh.phase += 1;
  __syncthreads();
}

// x[0..NV) summed over the CTA into sh.cta[0..NV)
template <int NV>
DW_D void cta_sum(LShared& sh, float (&x)[NV]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const float y = wsum(x[j]);
    if (lane == 0) sh.ws[w][j] = y;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    float y = 0;
#pragma unroll
    for (int q = 0; q < LW; ++q) y += sh.ws[q][threadIdx.x];
    sh.cta[threadIdx.x] = y;
  }
}

// sh.cta[off + 2v], + 1 = this CTA's share of (X_v, y); X_v = A + v as for v < na, B + (v - na) bs beyond
DW_D void dots(LShared& sh, const cf* A, size_t as, int na, const cf* B, size_t bs, int nvec, const cf* y, int n,
               int off) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int v0 = w; v0 < nvec; v0 += 4 * LW) {
    const cf* xp[4];
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int nu = min(4, (nvec - v0 + LW - 1) / LW);                 // warp-uniform
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int v = min(v0 + u * LW, nvec - 1);
      xp[u] = v < na ? A + v * as : B + (v - na) * bs;
    }
#pragma unroll 2
    for (int i = lane; i < n; i += 32) {
      const cf q = y[i];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) {
          const cf p = xp[u][i];
          acc[2 * u] = fmaf(p.im, q.im, fmaf(p.re, q.re, acc[2 * u]));
          acc[2 * u + 1] = fmaf(-p.im, q.re, fmaf(p.re, q.im, acc[2 * u + 1]));
        }
    }
    // eight values over the lanes by recursive halving: lane holds value m of acc
    int m = 0;
#pragma unroll
    for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int j = 0; j < h; ++j) {
        const float send = up ? acc[j] : acc[j + h];
        acc[j] = (up ? acc[j + h] : acc[j]) + __shfl_xor_sync(0xffffffffu, send, o);
      }
      if (up) m += h;
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    const int v = v0 + (m >> 1) * LW;
    if ((lane & 3) == 0 && v < nvec) sh.cta[off + 2 * v + (m & 1)] = acc[0];
  }
}

// sum over the LPART threads of a row
DW_D cf part_sum(cf s) {
#pragma unroll
  for (int o = LPART / 2; o > 0; o >>= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
  }
  return s;
}
// f(row, part) for `rows` rows with LPART threads each, whole warps at a time (f is also called for rows past
// the end, to keep the shuffles of a warp complete)
template <typename F>
DW_D void small_rows(int rows, F&& f) {
  for (int b = threadIdx.x & ~31; b < rows * LPART; b += LT) {
    const int e = b + (threadIdx.x & 31);
    f(e / LPART, e % LPART);
  }
}
// sh.z = A~^{-1} u, u = sh.res[0..2 NS); LPART threads per row (whole warps: NS LPART is a multiple of 32)
template <int NS>
DW_D void coarse(LShared& sh, const float* u) {
  small_rows(NS, [&](int r, int part) {
    cf s = {0.f, 0.f};
    if (r < NS)
      for (int q = part; q < NS; q += LPART) cmac(s, sh.ainv[r * NS + q], cf{u[2 * q], u[2 * q + 1]});
    s = part_sum(s);
    if (part == 0 && r < NS) sh.z[r] = s;
  });
}

// shared memory after the static part: hop tables, gathered vectors and direction sums of a chunk, the slices
// of chi_k and rho_k, and (VS) the slices of g, B^ g and chi'_j
template <int NS>
size_t dyn_bytes(int rows, int nkv, bool vs) {
  size_t b = (size_t)2 * 9 * rows * sizeof(int);
  b = (b + 15) / 16 * 16;
  b += (size_t)2 * std::min(rows, LCH) * 8 * NS * sizeof(cf) + (size_t)2 * rows * NS * sizeof(cf);
  if (vs) b += (size_t)(2 * NS + nkv) * rows * NS * sizeof(cf);
  return b;
}
constexpr size_t DYN_MAX = 194 * 1024;      // with the static part (21 KB) below 227 KB

template <int NS, bool VS>
__global__ void __launch_bounds__(LT, 1) little_gcr_warp_kernel(LittleArgs a) {
  __shared__ LShared sh;
  extern __shared__ __align__(16) unsigned char dyn[];
  const int t = threadIdx.x;
  const size_t n = (size_t)a.Ne * NS;
  const int Rmax = (max(a.Ne, a.No) + gridDim.x - 1) / gridDim.x;
  int* tab = reinterpret_cast<int*>(dyn);
  auto rows_of = [&](int nrow, int* L) {
    const int R = (nrow + gridDim.x - 1) / gridDim.x, rb = min(nrow, (int)blockIdx.x * R);
    return Rows{rb, min(nrow, rb + R) - rb, L, L + Rmax};
  };
  const Rows even = rows_of(a.Ne, tab), odd = rows_of(a.No, tab + 9 * Rmax);
  const int CR = min(Rmax, LCH);
  cf* xs = reinterpret_cast<cf*>(dyn + ((size_t)18 * Rmax * sizeof(int) + 15) / 16 * 16);
  cf* hp = xs + CR * 8 * NS;
  cf* ckS = hp + CR * 8 * NS;                            // c = B^ rho_k, then chi'_k; rho_k; (VS) g, B^ g, chi'_j
  cf* rkS = ckS + Rmax * NS;
  const int len = even.n * NS;                           // entries of this CTA
  const size_t s0 = (size_t)even.first * NS;             // first of them in the global vectors
  for (int e = t; e < even.n; e += LT) tab[e] = a.list_e[even.first + e];
  for (int e = t; e < even.n * 8; e += LT) tab[Rmax + e] = a.lnb_e[even.first * 8 + e];
  for (int e = t; e < odd.n; e += LT) tab[9 * Rmax + e] = a.list_o[odd.first + e];
  for (int e = t; e < odd.n * 8; e += LT) tab[10 * Rmax + e] = a.lnb_o[odd.first * 8 + e];
  const cf* gg = reinterpret_cast<const cf*>(a.g);
  const cf* gb = reinterpret_cast<const cf*>(a.Bg);
  cf* W = reinterpret_cast<cf*>(a.work);
  const int nkv = a.nkv;
  auto chi = [&](int k) { return W + (size_t)k * n; };   // chi'_k, unnormalised (norm c_k)
  auto xi = [&](int k) { return W + (size_t)(nkv + k) * n + s0; };
  cf* rhob[2] = {W + (size_t)2 * nkv * n, W + (size_t)(2 * nkv + 1) * n};
  cf* tmpo = W + (size_t)(2 * nkv + 2) * n;
  cf* rhsd = W + (size_t)(2 * nkv + 4) * n + s0;
  const cf* b = reinterpret_cast<const cf*>(a.b) + s0;
  cf* v = reinterpret_cast<cf*>(a.v);
  // the vectors of the inner products and updates: entry i of vector j at [j vn + i]
  const size_t vn = VS ? (size_t)Rmax * NS : n;
  cf* sl = rkS + Rmax * NS;
  const cf* gV = VS ? sl : gg + s0;
  const cf* bgV = VS ? sl + NS * vn : gb + s0;
  cf* chiV = VS ? sl + 2 * NS * vn : W + s0;
  cg::grid_group grid = cg::this_grid();
  if (t == 0) sh.phase = 0;
  if (a.a3) {
    const cf* Ai = reinterpret_cast<const cf*>(a.Ainv);
    for (int e = t; e < NS * NS; e += LT) sh.ainv[e] = Ai[e];
    if (VS)
      for (int e = t; e < NS * len; e += LT) {
        const int l = e / len, i = e - l * len;
        sl[l * vn + i] = gg[l * n + s0 + i];
        sl[(NS + l) * vn + i] = gb[l * n + s0 + i];
      }
  }
  __syncthreads();
  const float4* M = reinterpret_cast<const float4*>(a.M);
  Block<NS> buf;
  const int nd = a.a3 ? NS : 0;                          // deflation vectors
  const cf zero = {0.f, 0.f};
  auto each = [&](auto&& f) {
    for (int i = t; i < len; i += LT) f(i);
  };
  // y -= sum_l z_l X_l on this CTA's entries (sign +: add), two threads per entry
  auto project = [&](cf* y, const cf* X, float sign) {
    for (int e0 = t & ~31; e0 < 2 * len; e0 += LT) {     // whole warps
      const int e = e0 + (t & 31), i = min(e, 2 * len - 1) >> 1;
      cf s = zero;
      for (int l = e & 1; l < NS; l += 2) cmac(s, sh.z[l], X[l * vn + i]);
      s.re += __shfl_xor_sync(0xffffffffu, s.re, 1);
      s.im += __shfl_xor_sync(0xffffffffu, s.im, 1);
      if (e < 2 * len && !(e & 1)) { y[i].re += sign * s.re; y[i].im += sign * s.im; }
    }
  };
  // ckS = B^ x (x published; its own slice at x + s0)
  auto bhat = [&](const cf* x) {
    hop<NS>(buf, M, odd, even, x, nullptr, zero, xs, hp,
            [&](int e, cf s) { tmpo[(size_t)odd.first * NS + e] = s; });
    grid_barrier(grid);
    hop<NS>(buf, M, even, odd, tmpo, nullptr, zero, xs, hp, [&](int e, cf s) { ckS[e] = x[s0 + e] - s; });
  };
  // ckS = P~_L ckS
  auto PL = [&] {
    dots(sh, gV, vn, NS, nullptr, 0, NS, ckS, len, 0);
    reduce(grid, sh, 2 * NS, a.acc);
    coarse<NS>(sh, sh.res);
    __syncthreads();
    project(ckS, bgV, -1.f);
    __syncthreads();
  };
  // rho in ckS: published as rho_0 of a cycle; |rho|^2 reduced
  auto start_cycle = [&](cf* out, float* norm) {
    float s1[1] = {0.f};
    each([&](int i) {
      const cf x = ckS[i];
      rkS[i] = x;
      out[i] = x;
      s1[0] += norm2(x);
    });
    cta_sum<1>(sh, s1);
    if (t == 0) sh.rr = sh.cta[0];
    reduce(grid, sh, 1, a.acc);
    *norm = sqrtf(sh.res[0]);
  };

  // rhsd = P~_L b, rho = rhsd, v = 0
  preload<NS>(buf, M, odd, t >> 5, t & 31);
  each([&](int i) { ckS[i] = b[i]; });
  __syncthreads();
  if (a.a3) PL();
  each([&](int i) {
    rhsd[i] = ckS[i];
    v[s0 + i] = zero;
  });
  float bn = 0.f;
  start_cycle(rhob[0] + s0, &bn);
  float rn = bn;
  int total = 0, cur = 0;                                // rhob[cur]: rho_k on this CTA's rows
  const float stop = __double2float_rd(a.tol * (double)bn);
  while (bn > 0 && rn > stop && total < a.maxit) {
    int k = 0;
    for (; k < nkv && total < a.maxit; ++k) {
      cf* ck = chi(k) + s0;
      cf* xk = xi(k);
      each([&](int i) { xk[i] = rkS[i]; });              // xi_k = rho_k
      // the odd hop reads rho_k of other CTAs as rho_{k-1} - alpha chi'_{k-1}: both were written before the last
      // reduction's grid barrier
      const cf acs = k > 0 ? sh.ac : zero;
      hop<NS>(buf, M, odd, even, k > 0 ? rhob[cur ^ 1] : rhob[cur], k > 0 ? chi(k - 1) : nullptr, acs, xs, hp,
              [&](int e, cf s) { tmpo[(size_t)odd.first * NS + e] = s; });
      grid_barrier(grid);
      hop<NS>(buf, M, even, odd, tmpo, nullptr, zero, xs, hp, [&](int e, cf s) { ckS[e] = rkS[e] - s; });
      // first reduction: |rho_k|^2, (g_l, c), (chi'_j, c)
      dots(sh, gV, vn, nd, chiV, vn, nd + k, ckS, len, 1);
      if (t == 0) sh.cta[0] = sh.rr;
      reduce(grid, sh, 1 + 2 * (nd + k), a.acc);
      const float rn2 = sh.res[0];
      rn = sqrtf(rn2);
      if (rn <= stop) break;                             // rho_k already converged: c unused
      // z = A~^{-1} (g, c)
      const float* re = sh.res + 1 + 2 * nd;
      if (a.a3) coarse<NS>(sh, sh.res + 1);
      __syncthreads();
      // beta_j = (chi'_j, P~_L c) / |chi'_j|^2, (chi'_j, P~_L c) = (chi'_j, c) - sum_l z_l (chi'_j, B^ g_l)
      small_rows(k, [&](int j, int part) {
        cf s = zero;
        if (j < k)
          for (int l = part; l < nd; l += LPART) cmac(s, sh.z[l], conjg(sh.tg[j][l]));
        s = part_sum(s);
        if (part == 0 && j < k) {
          const float ic = 1.f / sh.c2[j];
          sh.be[j][k] = {(re[2 * j] - s.re) * ic, (re[2 * j + 1] - s.im) * ic};
        }
      });
      __syncthreads();
      // chi'_k = P~_L c - sum_j beta_j chi'_j
      float s3[3] = {0.f, 0.f, 0.f};
      for (int e0 = t & ~31; e0 < 2 * len; e0 += LT) {   // two threads per entry, whole warps
        const int e = e0 + (t & 31), i = min(e, 2 * len - 1) >> 1;
        cf s = zero;
        if (a.a3) {
#pragma unroll
          for (int l = 0; l < NS; l += 2) cmac(s, sh.z[l + (e & 1)], bgV[(l + (e & 1)) * vn + i]);
        }
#pragma unroll 4
        for (int j = e & 1; j < k; j += 2) cmac(s, sh.be[j][k], chiV[j * vn + i]);
        s.re += __shfl_xor_sync(0xffffffffu, s.re, 1);
        s.im += __shfl_xor_sync(0xffffffffu, s.im, 1);
        if (e < 2 * len && !(e & 1)) {
          const cf y = ckS[i] - s, r = rkS[i];
          ck[i] = y;
          if (VS) chiV[(size_t)k * vn + i] = y;
          ckS[i] = y;
          s3[0] += y.re * r.re + y.im * r.im;
          s3[1] += y.re * r.im - y.im * r.re;
          s3[2] += norm2(y);
        }
      }
      // second reduction: (chi'_k, rho_k), |chi'_k|^2, (B^ g_l, chi'_k); its grid barrier publishes chi'_k, which the
      // next odd hop gathers
      cta_sum<3>(sh, s3);
      dots(sh, bgV, vn, nd, nullptr, 0, nd, ckS, len, 3);
      reduce(grid, sh, 3 + 2 * nd, a.acc);
      const float c2 = sh.res[2];
      const cf ar = {sh.res[0], sh.res[1]};
      if (!(c2 > 0.f)) break;                            // the step is not used (zero or not a number)
      // rho_{k+1} = rho_k - alpha chi'_k
      const cf alpha = {ar.re / c2, ar.im / c2};
      cf* rn1 = rhob[cur ^ 1] + s0;
      float s1[1] = {0.f};
      each([&](int i) {
        cf r = rkS[i];
        cmsub(r, alpha, ckS[i]);
        rkS[i] = r;
        rn1[i] = r;
        s1[0] += norm2(r);
      });
      if (t < nd) sh.tg[k][t] = {sh.res[3 + 2 * t], sh.res[4 + 2 * t]};
      cta_sum<1>(sh, s1);
      if (t == 0) {
        sh.rr = sh.cta[0];
        sh.ac = alpha;
        sh.c2[k] = c2;
        sh.al[k] = ar;
      }
      __syncthreads();
      cur ^= 1;
      ++total;
      // |rho_{k+1}|^2 = |rho_k|^2 - |(chi'_k, rho_k)|^2 / |chi'_k|^2 (one step from the exact |rho_k|^2)
      const float est = rn2 - norm2(ar) / c2;
      rn = est <= 0.f ? 0.f : sqrtf(est);                // not a number stays one, and is not converged
      if (rn <= stop) { ++k; break; }
    }
    // v += sum_j y_j xi_j with y_j = alpha_j - sum_{i > j} beta_ji y_i: warp 0, lane i holds row i
    if (t < 32) {
      cf x = zero;
      if (t < k) x = {sh.al[t].re / sh.c2[t], sh.al[t].im / sh.c2[t]};
      for (int j = k - 1; j >= 0; --j) {
        const cf y = {__shfl_sync(0xffffffffu, x.re, j), __shfl_sync(0xffffffffu, x.im, j)};
        if (t < j) cmsub(x, sh.be[t][j], y);
      }
      if (t < k) sh.beta[t] = x;
    }
    __syncthreads();
    each([&](int i) {
      cf x = v[s0 + i];
#pragma unroll 4
      for (int j = 0; j < k; ++j) cmac(x, sh.beta[j], xi(j)[i]);
      v[s0 + i] = x;
    });
    grid_barrier(grid);
    if (k == 0) break;
    // true residual of the deflated system
    bhat(v);
    if (a.a3) PL();
    each([&](int i) { ckS[i] = rhsd[i] - ckS[i]; });
    __syncthreads();
    start_cycle(rhob[cur] + s0, &rn);
  }
  if (a.a3) {
    // v = chi + g A~^{-1} g^+ (b - B^ chi)
    grid_barrier(grid);
    bhat(v);
    each([&](int i) { ckS[i] = b[i] - ckS[i]; });
    __syncthreads();
    dots(sh, gV, vn, NS, nullptr, 0, NS, ckS, len, 0);
    reduce(grid, sh, 2 * NS, a.acc);
    coarse<NS>(sh, sh.res);
    __syncthreads();
    project(v + s0, gV, 1.f);
  }
  if (blockIdx.x == 0 && t == 0) {
    a.out[0] = total;
    a.out[1] = bn > 0 ? (double)rn / (double)bn : 0.0;
  }
}

template <int NS>
bool ready(int grid, int sms) {
  int b = 0;
  if (cudaFuncSetAttribute(little_gcr_warp_kernel<NS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)DYN_MAX) != cudaSuccess ||
      cudaFuncSetAttribute(little_gcr_warp_kernel<NS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)DYN_MAX) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, little_gcr_warp_kernel<NS, true>, LT, DYN_MAX) != cudaSuccess ||
      b < 1 ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, little_gcr_warp_kernel<NS, false>, LT, DYN_MAX) != cudaSuccess)
    return false;
  return b > 0 && grid <= sms;
}
template <int NS>
cudaError_t launch(const LittleArgs& a, int grid, cudaStream_t s) {
  const int rows = (std::max(a.Ne, a.No) + grid - 1) / grid;
  const bool vs = dyn_bytes<NS>(rows, a.nkv, true) <= DYN_MAX;
  const size_t dyn = dyn_bytes<NS>(rows, a.nkv, vs);
  if (dyn > DYN_MAX) return cudaErrorInvalidConfiguration;
  LittleArgs arg = a;
  void* p[] = {&arg};
  return cudaLaunchCooperativeKernel(vs ? (void*)little_gcr_warp_kernel<NS, true>
                                        : (void*)little_gcr_warp_kernel<NS, false>, grid, LT, p, dyn, s);
}

}  // namespace

#define LITTLE_NS(NSRT, EXPR, OTHER)  \
  switch (NSRT) {                     \
    case 8: { constexpr int NSV = 8; return EXPR; }   \
    case 12: { constexpr int NSV = 12; return EXPR; } \
    case 16: { constexpr int NSV = 16; return EXPR; } \
    case 20: { constexpr int NSV = 20; return EXPR; } \
    case 24: { constexpr int NSV = 24; return EXPR; } \
    case 32: { constexpr int NSV = 32; return EXPR; } \
    default: return OTHER;            \
  }

bool little_warp_ready(int Ns, int rows, int grid, int sms) {
  LITTLE_NS(Ns, (dyn_bytes<NSV>(rows, LITTLE_NKV, false) <= DYN_MAX && ready<NSV>(grid, sms)), false)
}
cudaError_t little_warp_launch(const LittleArgs& a, int Ns, int grid, cudaStream_t s) {
  LITTLE_NS(Ns, (launch<NSV>(a, grid, s)), cudaErrorInvalidValue)
}
