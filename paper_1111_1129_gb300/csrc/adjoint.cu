// Reverse mode (adjoint) of the sweep, for gradients of the mean axial
// velocity J = (1/N) sum_n u_axis,n of the collision of step K with respect
// to the body force F and a per-cell Brinkman damping alpha_n.
//
// Forward: f_0 given; for t = 1..K: g_t = S f_{t-1} (pull through the
// adjacency list), f_t = C(g_t; F, alpha) (TRT collision).  Reverse:
//   lam_g_K = dJ/dg_K,  lam_f_{t-1} = S^T lam_g_t,
//   lam_g_t = C'(g_t)^T lam_f_t  (t = K-1 .. 1),
// with dJ/dF and dJ/dalpha accumulated from every step.
//
// C'^T is applied in closed form.  Writing the collision as
//   f*_q = L(g)_q + E_q(rho, u) + S_q(u),
//   L(g)_q = (1 - (w+ + w-)/2) g_q + ((w- - w+)/2) g_opp(q),
//   E_q = w+ w_q (rho + 4.5 (c_q.u)^2 - 1.5 u.u) + 3 w- w_q c_q.u,
//   S_q = (1 - w-/2) 3 w_q c_q.(F - alpha u),
// with drho/dg_r = 1 and du/dg_r = s c_r (s = 1/(1 + alpha/2)), one gets
//   lam_g_r = L^T(lam)_r + w+ M0 + s c_r.G,
//   G = 9 w+ M2 u - 3 w+ M0 u + 3 (w- - alpha (1 - w-/2)) M1,
//   dJ/dF     += (s/2) G + 3 (1 - w-/2) M1,
//   dJ/dalpha += -(s/2) G.u - 3 (1 - w-/2) M1.u,
// where M0 = sum w_q lam_q, M1 = sum w_q lam_q c_q, M2 = sum w_q lam_q c_q c_q^T.
//
// The reverse step needs g_t only through the velocity u of its collision,
// three values a cell in place of 19 pulled ones.  So a forward step keeps u
// (3 rows) rather than f (19 rows): within the memory of a checkpoint every
// `stride` steps and one segment of `stride` states (stride ~ sqrt(K), as
// lbm_adjoint_create is asked), U velocity fields cover the last U steps
// outright, and a few checkpoints of f the rest, recomputed in segments of at
// most U steps.  Up to K ~ 160 nothing is recomputed in FP32.
//
// lambda is kept with its rows reversed: row r holds the adjoint of direction
// opp(r).  The reader of slot (q, m) is m + c_q, the upwind neighbour of m in
// direction opp(q), or m itself bounced back -- what the links of direction
// opp(q) name in row opp(q).  With that, S^T is the pull S itself, through the
// same links.
//
// The reverse steps are bound by bytes: 222 per cell in FP32 (38 links, 12 u,
// 76 + 76 lambda, 16 dJ/dalpha, 4 alpha; none of the 16 where dJ/dalpha is not
// asked for) against 320 with g_t pulled from 19 rows through 32-bit links,
// FP64 storage 398 against 560.  Damped 128^3 bed (1.03 M cells), against that
// version: 200 steps and their gradient 26.6 -> 16.8 ms in FP32 shifted;
// reverse pass of 2000 steps (a quarter of them kept) 178 -> 133 ms in FP32
// shifted, 373 -> 302 in FP64 storage, 1,294 -> 1,031 in IEEE FP64, which is
// bound by its arithmetic and no longer forms u a second time.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "double_single.cuh"
#include "lbm_kernels.cuh"

struct lbm_adjoint {
  uint32_t magic;
  const lbm_state* st;
  cudaStream_t stream;   // the state's stream, kept so that freeing needs no state
  int32_t K;
  // Steps 1..M (M = K - 1) advance f.  u holds the velocities of the last
  // min(M, slots) steps after a forward pass; the steps before them form n_seg
  // segments of seg_len steps (the last one may be shorter), each with a
  // checkpoint of the f it starts from.
  int32_t slots, n_seg, seg_len;
  void* ckpt;       // n_seg states of 19 rows of ld storage elements
  void* f[2];       // the two states steps alternate between
  void* u;          // slots fields of 3 rows of ld, in the arithmetic precision
  const void* last; // f_M
  void* lam[2];     // 19 rows of ld arithmetic-precision adjoints
  bool fresh;       // lam[0], part, dalpha, u and last are as the forward pass left them
  double* part;     // [nblocks][4]: dJ/dF_x, dJ/dF_y, dJ/dF_z, sum u_axis
  double* dalpha;   // [N]
  double* red_host; // [4], pinned, written by final_sum_kernel
  cudaEvent_t done;
  int have_forward;
  double wp, wm, F[3];
  int32_t axis;
};

namespace lbm {
namespace {

// Coefficients of the reverse step, for its two forms (adjoint_step_kernel):
// the weighted form, and the pair form, which carries the weighted moments
// M of the adjoint as M' = 36 M (w0 = 12/36, w1 = 2/36, w2 = 1/36) with the
// 1/36 in the coefficients that multiply them.
template <class C>
struct AdjCoef {
  C wp, one_m_wp;  // w+, 1 - w+
  C k1, k2;        // 1 - (w+ + w-)/2, (w- - w+)/2
  C wm, src;       // w-, 1 - w-/2
  C hp, hm;        // (1 - w+)/2, (1 - w-)/2: the pair form of L^T
  C wp36, wp12, wp4;   // w+/36 (base), 3 w+/36, 9 w+/36 (G)
  C wm12, src12;   // beta/36 = w-/12 - alpha src/12
  C inv_n;         // 1 / N
};

template <class C>
AdjCoef<C> make_adj_coef(double wp, double wm, int64_t n) {
  AdjCoef<C> a;
  a.wp = (C)wp;
  a.one_m_wp = (C)(1.0 - wp);
  a.k1 = (C)(1.0 - 0.5 * (wp + wm));
  a.k2 = (C)(0.5 * (wm - wp));
  a.wm = (C)wm;
  a.src = (C)(1.0 - 0.5 * wm);
  a.hp = (C)(0.5 * (1.0 - wp));
  a.hm = (C)(0.5 * (1.0 - wm));
  a.wp36 = (C)(wp / 36.0);
  a.wp12 = (C)(wp / 12.0);
  a.wp4 = (C)(0.25 * wp);
  a.wm12 = (C)(wm / 12.0);
  a.src12 = (C)((1.0 - 0.5 * wm) / 12.0);
  a.inv_n = (C)(n > 0 ? 1.0 / (double)n : 0.0);
  return a;
}

// Velocity of the collision of the pulled values g (same arithmetic as the
// collision) and s = 1 / (1 + alpha/2).
template <class C, bool DAMPED>
__device__ __forceinline__ void velocity(const C g[19], const Coef<C>& k, C alpha, C u[3], C& s) {
  C d[9];
#pragma unroll
  for (int p = 0; p < 9; ++p) d[p] = g[2 * p + 1] - g[2 * p + 2];
  const C jx = ((d[0] + d[3]) + (d[4] + d[5])) + d[6];
  const C jy = ((d[1] + d[3]) - (d[4] - d[7])) + d[8];
  const C jz = ((d[2] + d[5]) - (d[6] - d[7])) - d[8];
  s = DAMPED ? C(1) / (C(1) + C(0.5) * alpha) : C(1);
  u[0] = (jx + k.hF[0]) * s;
  u[1] = (jy + k.hF[1]) * s;
  u[2] = (jz + k.hF[2]) * s;
}

__device__ __forceinline__ int axis_component(int q, int axis) {
  return axis == 0 ? cx(q) : (axis == 1 ? cy(q) : cz(q));
}

// Block-sum 4 values and add them to acc[4] (each block owns its slot;
// launches on one stream are ordered, so the accumulation is race free).
// The warp level sums in the arithmetic precision T of the values: FP64
// adds issue at 1/64 of the FP32 rate on GB300, and a shuffle tree costs
// every lane 20 of them per cell, most of an FP32 adjoint step.  Warp sums
// then accumulate in FP64.
template <class T>
__device__ __forceinline__ void block_accumulate4(T v[4], double* acc, bool assign) {
  __shared__ double sm[kSweepThreads / 32][4];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += __shfl_down_sync(0xffffffffu, v[j], o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int j = 0; j < 4; ++j) sm[warp][j] = (double)v[j];
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kSweepThreads / 32; ++w) s += sm[w][threadIdx.x];
    acc[threadIdx.x] = assign ? s : acc[threadIdx.x] + s;
  }
}

// Seed: lam_g_K = dJ/dg_K from f_{K-1}; initialises dJ/dF, dJ/dalpha and
// the sum of u_axis (J = sum / N).  Cells, PDFs, lambda: rows of ld.
template <int PREC, bool DAMPED, bool SHORT>
__global__ void __launch_bounds__(kSweepThreads)
    adjoint_seed_kernel(const typename Form<PREC>::S* __restrict__ f_prev, Links links, int32_t n,
                        int32_t ld, Coef<typename Form<PREC>::C> k,
                        AdjCoef<typename Form<PREC>::C> a,
                        const typename Form<PREC>::C* __restrict__ alpha, int axis,
                        typename Form<PREC>::C* __restrict__ lam_out, double* __restrict__ part,
                        double* __restrict__ dalpha) {
  using C = typename Form<PREC>::C;
  // A chained launch waits for the previous kernel here.  The zero it returns
  // offsets every index and pointer, so no access can be scheduled earlier.
  const int32_t z = prior_step_done();
  const int32_t i = blockIdx.x * kSweepThreads + threadIdx.x + z;
  double red[4] = {0.0, 0.0, 0.0, 0.0};
  int32_t idx[18];
  load_links<SHORT>(links, n, ld, i, idx);
  if (i < n) {
    C g[19];
    pull<PREC>(f_prev, idx, i, k.inv_scale, g);
    C u[3], s;
    const C al = DAMPED ? alpha[i] : C(0);
    velocity<C, DAMPED>(g, k, al, u, s);
    const C seed = s * a.inv_n;
#pragma unroll
    for (int q = 0; q < 19; ++q) lam_out[opp(q) * ld + i] = C(axis_component(q, axis)) * seed;
    red[axis] = 0.5 * (double)seed;
    red[3] = (double)u[axis];
    dalpha[i] = -0.5 * (double)seed * (double)u[axis];
  }
  block_accumulate4(red, part + z + 4 * (int64_t)blockIdx.x, true);
}

__device__ __forceinline__ float2 ld_nc(const float2* p) {
  float2 v;
  asm volatile("ld.global.nc" LBM_LD_HINT ".v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}

// The 19 pulled adjoints of cell i, lf[q] that of direction q.
template <class T>
__device__ __forceinline__ void pull_adjoint(const T* __restrict__ lam_in, const int32_t idx[18],
                                             int32_t i, T lf[19]) {
  lf[0] = ld_nc(lam_in + i);
#pragma unroll
  for (int q = 1; q < 19; ++q) lf[opp(q)] = ld_nc(lam_in + idx[q - 1]);
}

// The reverse step of one cell in FP32 arithmetic: lf the pulled adjoints, out
// the new ones in reversed rows, red its terms of dJ/dF.  Returns its term of
// dJ/dalpha.
template <class C, bool DAMPED>
__device__ __forceinline__ C reverse_cell(const C lf[19], const C u[3], C al, const AdjCoef<C>& a,
                                          C out[19], C red[4]) {
  const C s = DAMPED ? C(1) / (C(1) + C(0.5) * al) : C(1);
  C S[9], D[9];
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    S[p] = lf[2 * p + 1] + lf[2 * p + 2];
    D[p] = lf[2 * p + 1] - lf[2 * p + 2];
  }
  // weighted moments of the adjoint
  const C w0 = C(1.0 / 3.0), w1 = C(1.0 / 18.0), w2 = C(1.0 / 36.0);
  const C M0 = w0 * lf[0] + w1 * (S[0] + S[1] + S[2]) +
               w2 * (((S[3] + S[4]) + (S[5] + S[6])) + (S[7] + S[8]));
  const C M1x = w1 * D[0] + w2 * ((D[3] + D[4]) + (D[5] + D[6]));
  const C M1y = w1 * D[1] + w2 * ((D[3] - D[4]) + (D[7] + D[8]));
  const C M1z = w1 * D[2] + w2 * ((D[5] - D[6]) + (D[7] - D[8]));
  const C Mxx = w1 * S[0] + w2 * ((S[3] + S[4]) + (S[5] + S[6]));
  const C Myy = w1 * S[1] + w2 * ((S[3] + S[4]) + (S[7] + S[8]));
  const C Mzz = w1 * S[2] + w2 * ((S[5] + S[6]) + (S[7] + S[8]));
  const C Mxy = w2 * (S[3] - S[4]);
  const C Mxz = w2 * (S[5] - S[6]);
  const C Myz = w2 * (S[7] - S[8]);
  const C nine_wp = C(9) * a.wp, three_wp_m0 = C(3) * a.wp * M0;
  const C beta = C(3) * (a.wm - al * a.src);
  // G = nine_wp (M2 u) - three_wp_m0 u + beta M1, each rounding written out:
  // left to the compiler, the sums contract differently from one
  // instantiation of this kernel to the next
  const auto G = [&](C q, C uj, C m1) {
    return __fmaf_rn(beta, m1, __fmaf_rn(nine_wp, q, -__fmul_rn(three_wp_m0, uj)));
  };
  const C Gx = G(__fmaf_rn(Mxz, u[2], __fmaf_rn(Mxx, u[0], __fmul_rn(Mxy, u[1]))), u[0], M1x);
  const C Gy = G(__fmaf_rn(Myz, u[2], __fmaf_rn(Myy, u[1], __fmul_rn(Mxy, u[0]))), u[1], M1y);
  const C Gz = G(__fmaf_rn(Mzz, u[2], __fmaf_rn(Mxz, u[0], __fmul_rn(Myz, u[1]))), u[2], M1z);
  const C base = a.wp * M0;
  out[0] = a.one_m_wp * lf[0] + base;
#define LBM_ADJ_PAIR(P, CG)                                                    \
  {                                                                            \
    const C sg_ = s * (CG);                                                    \
    out[2 * P + 2] = a.k1 * lf[2 * P + 1] + a.k2 * lf[2 * P + 2] + base + sg_; \
    out[2 * P + 1] = a.k1 * lf[2 * P + 2] + a.k2 * lf[2 * P + 1] + base - sg_; \
  }
  LBM_ADJ_PAIR(0, Gx)
  LBM_ADJ_PAIR(1, Gy)
  LBM_ADJ_PAIR(2, Gz)
  LBM_ADJ_PAIR(3, Gx + Gy)
  LBM_ADJ_PAIR(4, Gx - Gy)
  LBM_ADJ_PAIR(5, Gx + Gz)
  LBM_ADJ_PAIR(6, Gx - Gz)
  LBM_ADJ_PAIR(7, Gy + Gz)
  LBM_ADJ_PAIR(8, Gy - Gz)
#undef LBM_ADJ_PAIR
  const C hs = C(0.5) * s, three_src = C(3) * a.src;
  red[0] = hs * Gx + three_src * M1x;
  red[1] = hs * Gy + three_src * M1y;
  red[2] = hs * Gz + three_src * M1z;
  const C Gu = Gx * u[0] + Gy * u[1] + Gz * u[2];
  const C M1u = M1x * u[0] + M1y * u[1] + M1z * u[2];
  return -hs * Gu - three_src * M1u;
}

// One reverse step t: lam_f_t = S^T lam_g_{t+1} (pulled), then
// lam_g_t = C'(g_t)^T lam_f_t with the velocity u of that collision, rows of
// ld.  dalpha may be null (dJ/dalpha not wanted).
// FP32, lists with 32-bit links, at 5 resident blocks (48 registers): reverse
// pass of 200 damped steps on 29,479 cells 0.757 ms (at 4 and 6 blocks 0.783 and
// 0.777), on a box of 305,184 cells 2.20 (2.32, 2.34), of 20 steps on 15.9
// million cells with a slit plate 11.1 (11.7, 11.3); on 200,704 cells 1.69, and
// 1.66 at 6.
#ifndef LBM_ADJ_MIN_BLOCKS
#define LBM_ADJ_MIN_BLOCKS 5
#endif
template <class C, bool DAMPED, bool SHORT>
__global__ void __launch_bounds__(kSweepThreads, sizeof(C) == 4 ? LBM_ADJ_MIN_BLOCKS : 1)
    adjoint_step_kernel(const C* __restrict__ u_in, Links links, int32_t n, int32_t ld,
                        AdjCoef<C> a, const C* __restrict__ alpha, const C* __restrict__ lam_in,
                        C* __restrict__ lam_out, double* __restrict__ part,
                        double* __restrict__ dalpha) {
  const int32_t z = prior_step_done();  // as in adjoint_seed_kernel
  const int32_t i = blockIdx.x * kSweepThreads + threadIdx.x + z;
  C red[4] = {C(0), C(0), C(0), C(0)};
  int32_t idx[18];
  load_links<SHORT>(links, n, ld, i, idx);
  if (i < n) {
    C lf[19], u[3];
    pull_adjoint(lam_in, idx, i, lf);
#pragma unroll
    for (int j = 0; j < 3; ++j) u[j] = ld_nc(u_in + j * ld + i);
    const C al = DAMPED ? ld_nc(alpha + i) : C(0);
    // Two forms of the same update.  FP64 arithmetic takes the pair form:
    // the outputs of pair (a, b) are e +- o, e = (1 - w+)/2 S + base and
    // o = (1 - w-)/2 D + s G (L^T's k1 la + k2 lb and k1 lb + k2 la have sum
    // (1 - w+) S and difference (1 - w-) D), with the moments carried as
    // 36 M.  It issues about a quarter fewer FP64 instructions: on the damped
    // 128^3 bed the IEEE reverse step took 371 us against 448 and the
    // reverse pass 1,297 ms against 1,450.  FP32 arithmetic keeps the
    // weighted form: there the pair form took 40 registers instead of 48,
    // ran 6 blocks per SM instead of 5, and was slower, 57.6 us against 53.2
    // (DRAM 65% against 71%; reverse pass 187 ms against 178).
    if constexpr (sizeof(C) == 8) {
      const C s = DAMPED ? C(1) / (C(1) + C(0.5) * al) : C(1);
      C S[9], D[9];
#pragma unroll
      for (int p = 0; p < 9; ++p) {
        S[p] = lf[2 * p + 1] + lf[2 * p + 2];
        D[p] = lf[2 * p + 1] - lf[2 * p + 2];
      }
      const C s34 = S[3] + S[4], s56 = S[5] + S[6], s78 = S[7] + S[8];
      const C M0 = C(12) * lf[0] + C(2) * ((S[0] + S[1]) + S[2]) + ((s34 + s56) + s78);
      const C M1x = C(2) * D[0] + ((D[3] + D[4]) + (D[5] + D[6]));
      const C M1y = C(2) * D[1] + ((D[3] - D[4]) + (D[7] + D[8]));
      const C M1z = C(2) * D[2] + ((D[5] - D[6]) + (D[7] - D[8]));
      const C Mxx = C(2) * S[0] + (s34 + s56);
      const C Myy = C(2) * S[1] + (s34 + s78);
      const C Mzz = C(2) * S[2] + (s56 + s78);
      const C Mxy = S[3] - S[4], Mxz = S[5] - S[6], Myz = S[7] - S[8];
      // G = 9 w+ M2 u - 3 w+ M0 u + beta M1, beta = 3 (w- - alpha (1 - w-/2))
      const C m0 = a.wp12 * M0;
      const C beta = a.wm12 - al * a.src12;
      const C Gx = a.wp4 * (Mxx * u[0] + Mxy * u[1] + Mxz * u[2]) - m0 * u[0] + beta * M1x;
      const C Gy = a.wp4 * (Mxy * u[0] + Myy * u[1] + Myz * u[2]) - m0 * u[1] + beta * M1y;
      const C Gz = a.wp4 * (Mxz * u[0] + Myz * u[1] + Mzz * u[2]) - m0 * u[2] + beta * M1z;
      const C base = a.wp36 * M0;
      lam_out[i] = a.one_m_wp * lf[0] + base;
#define LBM_ADJ_PAIR(P, CG)                                                    \
  {                                                                            \
    const C e_ = a.hp * S[P] + base;                                           \
    const C o_ = a.hm * D[P] + s * (CG);                                       \
    lam_out[(2 * P + 2) * ld + i] = e_ + o_;                                    \
    lam_out[(2 * P + 1) * ld + i] = e_ - o_;                                    \
  }
      LBM_ADJ_PAIR(0, Gx)
      LBM_ADJ_PAIR(1, Gy)
      LBM_ADJ_PAIR(2, Gz)
      LBM_ADJ_PAIR(3, Gx + Gy)
      LBM_ADJ_PAIR(4, Gx - Gy)
      LBM_ADJ_PAIR(5, Gx + Gz)
      LBM_ADJ_PAIR(6, Gx - Gz)
      LBM_ADJ_PAIR(7, Gy + Gz)
      LBM_ADJ_PAIR(8, Gy - Gz)
#undef LBM_ADJ_PAIR
      // dJ/dF += (s/2) G + 3 (1 - w-/2) M1; dJ/dalpha += -(s/2) G.u - 3 (1 - w-/2) M1.u
      const C hs = C(0.5) * s;
      red[0] = hs * Gx + a.src12 * M1x;
      red[1] = hs * Gy + a.src12 * M1y;
      red[2] = hs * Gz + a.src12 * M1z;
      const C Gu = Gx * u[0] + Gy * u[1] + Gz * u[2];
      const C M1u = M1x * u[0] + M1y * u[1] + M1z * u[2];
      if (dalpha) dalpha[i] += (double)(-hs * Gu - a.src12 * M1u);
    } else {
      C out[19];
      const C da = reverse_cell<C, DAMPED>(lf, u, al, a, out, red);
#pragma unroll
      for (int q = 0; q < 19; ++q) lam_out[q * ld + i] = out[q];
      if (dalpha) dalpha[i] += (double)da;
    }
  }
  block_accumulate4(red, part + z + 4 * (int64_t)blockIdx.x, false);
}

// The same for lists with short links, two adjacent cells a thread as in
// sweep_pair32_kernel: a warp takes one tile of links, a block of 128 threads
// the 256 cells of a block above.  Its sums are formed in the same order: the
// halves of a warp are the two warps above, and the last level of their tree
// adds a thread's two cells.  Bound by latency and bytes (65% of the DRAM rate
// in a launch of 40 us, 24 warps per SM); with 18 instead of 36 link loads for
// two cells and twice the pulls in flight per thread, 200 steps and their
// gradient on the damped 128^3 bed took 17.39 -> 16.83 ms, 40 steps on a
// 151x141x201 bed 6.33 -> 6.04, 100 undamped steps of 128^3 7.62 -> 7.45.
// Damped at 6 blocks per SM (80 registers), 17.1 ms at 5 and 17.9 at 7;
// undamped at 5 (7.92 at 6, which spills).  Links loaded before the wait for
// the previous step: 17.0.
#ifndef LBM_ADJ_PAIR_MIN_BLOCKS
#define LBM_ADJ_PAIR_MIN_BLOCKS 6
#endif
template <bool DAMPED>
__global__ void __launch_bounds__(kSweepThreads / 2, DAMPED ? LBM_ADJ_PAIR_MIN_BLOCKS : 5)
    adjoint_pair_kernel(const float* __restrict__ u_in, Links links, int32_t n, int32_t ld,
                        AdjCoef<float> a, const float* __restrict__ alpha,
                        const float* __restrict__ lam_in, float* __restrict__ lam_out,
                        double* __restrict__ part, double* __restrict__ dalpha) {
  const int32_t z = prior_step_done();  // as in adjoint_seed_kernel
  const int32_t i = 2 * (int32_t)(blockIdx.x * (kSweepThreads / 2) + threadIdx.x) + z;
  const bool two = i + 1 < n;
  float r[2][4] = {};
  if (i < ld) {   // whole warps
    uint32_t word[18];
    int32_t entry;
    load_pair_links(links, ld, i, word, entry);
    float lf[2][19];
    if (i < n) lf[0][0] = ld_nc(lam_in + i);
    if (two) lf[1][0] = ld_nc(lam_in + i + 1);
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      const int32_t m0 = short_slot(q, ld, entry, word[q - 1]);
      const int32_t m1 = short_slot(q, ld, entry, word[q - 1] >> 16);
      if (i < n) lf[0][opp(q)] = ld_nc(lam_in + m0);
      if (two) lf[1][opp(q)] = ld_nc(lam_in + m1);
    }
    if (i < n) {
      // past the end of an odd list: the padding of the rows of ld
      float2 u[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) u[j] = ld_nc(reinterpret_cast<const float2*>(u_in + j * ld + i));
      const float al0 = DAMPED ? ld_nc(alpha + i) : 0.f;
      const float al1 = DAMPED && two ? ld_nc(alpha + i + 1) : 0.f;
      float out[19];
      const float u0[3] = {u[0].x, u[1].x, u[2].x}, u1[3] = {u[0].y, u[1].y, u[2].y};
      const float d0 = reverse_cell<float, DAMPED>(lf[0], u0, al0, a, out, r[0]);
      if (two) {
        float out1[19];
        const float d1 = reverse_cell<float, DAMPED>(lf[1], u1, al1, a, out1, r[1]);
#pragma unroll
        for (int q = 0; q < 19; ++q)
          *reinterpret_cast<float2*>(lam_out + q * ld + i) = make_float2(out[q], out1[q]);
        if (dalpha) {
          double2* at = reinterpret_cast<double2*>(dalpha + i);
          const double2 v = *at;
          *at = make_double2(v.x + (double)d0, v.y + (double)d1);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 19; ++q) lam_out[q * ld + i] = out[q];
        if (dalpha) dalpha[i] += (double)d0;
      }
    }
  }
  // block_accumulate4 of 256 cells
  __shared__ double sm[kSweepThreads / 32][4];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      r[0][j] += __shfl_down_sync(0xffffffffu, r[0][j], o);
      r[1][j] += __shfl_down_sync(0xffffffffu, r[1][j], o);
    }
  if ((threadIdx.x & 15) == 0)
#pragma unroll
    for (int j = 0; j < 3; ++j) sm[threadIdx.x >> 4][j] = (double)(r[0][j] + r[1][j]);
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kSweepThreads / 32; ++w) s += sm[w][threadIdx.x];
    part[z + 4 * (int64_t)blockIdx.x + threadIdx.x] += s;
  }
}

// ---- FP64-storage adjoint in double-single arithmetic --------------------------
// For LBM_F64X the reverse step keeps FP64-level accuracy without FP64
// instructions on its common path.  lambda is stored as a pair of FP32
// values (hi, lo) whose unevaluated sum carries ~48 significant bits
// (double_single.cuh).  The forward velocity is the one of the fixed-point
// sweep (exact in units 2^-58), kept as a pair.
// Coefficients of the reverse step as pairs (those of AdjCoef).
struct AdjCoefDS {
  ds one_m_wp, hp, hm, wp36, wp12, wp4, wm12, src12;
};

AdjCoefDS make_adj_coef_ds(double wp, double wm) {
  AdjCoefDS a;
  a.one_m_wp = ds_from_double(1.0 - wp);
  a.hp = ds_from_double(0.5 * (1.0 - wp));
  a.hm = ds_from_double(0.5 * (1.0 - wm));
  a.wp36 = ds_from_double(wp / 36.0);
  a.wp12 = ds_from_double(wp / 12.0);
  a.wp4 = ds_from_double(0.25 * wp);
  a.wm12 = ds_from_double(wm / 12.0);
  a.src12 = ds_from_double((1.0 - 0.5 * wm) / 12.0);
  return a;
}

// Block sums of four pairs, added to acc[4] in FP64 (as block_accumulate4).
__device__ __forceinline__ void block_accumulate4_ds(ds v[4], double* acc, bool assign) {
  __shared__ double sm[kSweepThreads / 32][4];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const ds w = {__shfl_down_sync(0xffffffffu, v[j].hi, o),
                    __shfl_down_sync(0xffffffffu, v[j].lo, o)};
      v[j] = ds_add(v[j], w);
    }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int j = 0; j < 4; ++j) sm[warp][j] = ds_to_double(v[j]);
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kSweepThreads / 32; ++w) t += sm[w][threadIdx.x];
    acc[threadIdx.x] = assign ? t : acc[threadIdx.x] + t;
  }
}

// Seed of the FP64-storage adjoint: as adjoint_seed_kernel, lambda written
// as pairs (float2, 19 rows of ld).
template <bool DAMPED, bool SHORT>
__global__ void __launch_bounds__(kSweepThreads)
    adjoint_seed_ds_kernel(const double* __restrict__ f_prev, Links links, int32_t n, int32_t ld,
                           Coef<double> k, AdjCoef<double> a, const double* __restrict__ alpha,
                           int axis, float2* __restrict__ lam_out, double* __restrict__ part,
                           double* __restrict__ dalpha) {
  const int32_t z = prior_step_done();  // as in adjoint_seed_kernel
  const int32_t i = blockIdx.x * kSweepThreads + threadIdx.x + z;
  double red[4] = {0.0, 0.0, 0.0, 0.0};
  int32_t idx[18];
  load_links<SHORT>(links, n, ld, i, idx);
  if (i < n) {
    double g[19];
    pull<LBM_F64>(f_prev, idx, i, 1.0, g);
    double u[3], s;
    const double al = DAMPED ? alpha[i] : 0.0;
    velocity<double, DAMPED>(g, k, al, u, s);
    const double seed = s * a.inv_n;
#pragma unroll
    for (int q = 0; q < 19; ++q) {
      const ds v = ds_from_double((double)axis_component(q, axis) * seed);
      lam_out[opp(q) * ld + i] = make_float2(v.hi, v.lo);
    }
    red[axis] = 0.5 * seed;
    red[3] = u[axis];
    dalpha[i] = -0.5 * seed * u[axis];
  }
  block_accumulate4(red, part + z + 4 * (int64_t)blockIdx.x, true);
}

// One reverse step of the FP64-storage adjoint (adjoint_step_kernel's
// formulas) in double-single arithmetic.
// 3 resident blocks (80 registers): 60 steps and their gradient on a damped
// 91x83x117 bed 5.12 ms, 5.16 at 4 and 5.95 at 2.
#ifndef LBM_ADJ_DS_MIN_BLOCKS
#define LBM_ADJ_DS_MIN_BLOCKS 3
#endif
template <bool DAMPED, bool SHORT>
__global__ void __launch_bounds__(kSweepThreads, LBM_ADJ_DS_MIN_BLOCKS)
    adjoint_step_ds_kernel(const float2* __restrict__ u_in, Links links, int32_t n, int32_t ld,
                           AdjCoefDS a, const double* __restrict__ alpha,
                           const int64_t* __restrict__ alpha_fx,
                           const float2* __restrict__ lam_in, float2* __restrict__ lam_out,
                           double* __restrict__ part, double* __restrict__ dalpha) {
  const int32_t z = prior_step_done();  // as in adjoint_seed_kernel
  const int32_t i = blockIdx.x * kSweepThreads + threadIdx.x + z;
  ds red[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  int32_t idx[18];
  load_links<SHORT>(links, n, ld, i, idx);
  if (i < n) {
    float2 l2[19];
    pull_adjoint(lam_in, idx, i, l2);
    ds u[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2 v = ld_nc(u_in + j * ld + i);
      u[j] = {v.x, v.y};
    }
    // s = 1/(1 + alpha/2) = 1 - e, and alpha, from their fixed-point values
    // where alpha lies in [0, 1/2)
    ds s = {1.f, 0.f}, al = {0.f, 0.f};
    if constexpr (DAMPED) {
      const int64_t A = __ldg(alpha_fx + i);
      if (A >= 0) {
        s = ds_sub(s, ds_from_fixed(__ldg(alpha_fx + n + i), 63));
        al = ds_from_fixed(A, 63);
      } else {
        s = ds_from_double(1.0 / (1.0 + 0.5 * alpha[i]));
        al = ds_from_double(alpha[i]);
      }
    }
    ds lf[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) lf[q] = {l2[q].x, l2[q].y};
    // moments carried as 36 M, as in adjoint_step_kernel; the scalings by
    // 2, 4 and 8 are exact
    ds S[9], D[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
      S[p] = ds_add(lf[2 * p + 1], lf[2 * p + 2]);
      D[p] = ds_sub(lf[2 * p + 1], lf[2 * p + 2]);
    }
    const ds s34 = ds_add(S[3], S[4]), s56 = ds_add(S[5], S[6]), s78 = ds_add(S[7], S[8]);
    const ds M0 = ds_add(ds_add(ds_add(ds_scale_pow2(lf[0], 8.f), ds_scale_pow2(lf[0], 4.f)),
                                ds_scale_pow2(ds_add(ds_add(S[0], S[1]), S[2]), 2.f)),
                         ds_add(ds_add(s34, s56), s78));
    const ds M1x = ds_add(ds_scale_pow2(D[0], 2.f), ds_add(ds_add(D[3], D[4]), ds_add(D[5], D[6])));
    const ds M1y = ds_add(ds_scale_pow2(D[1], 2.f), ds_add(ds_sub(D[3], D[4]), ds_add(D[7], D[8])));
    const ds M1z = ds_add(ds_scale_pow2(D[2], 2.f), ds_add(ds_sub(D[5], D[6]), ds_sub(D[7], D[8])));
    const ds Mxx = ds_add(ds_scale_pow2(S[0], 2.f), ds_add(s34, s56));
    const ds Myy = ds_add(ds_scale_pow2(S[1], 2.f), ds_add(s34, s78));
    const ds Mzz = ds_add(ds_scale_pow2(S[2], 2.f), ds_add(s56, s78));
    const ds Mxy = ds_sub(S[3], S[4]);
    const ds Mxz = ds_sub(S[5], S[6]);
    const ds Myz = ds_sub(S[7], S[8]);
    const ds m0 = ds_mul(a.wp12, M0);
    // beta/36 = w-/12 - alpha src/12
    ds beta = a.wm12;
    if constexpr (DAMPED) beta = ds_sub(beta, ds_mul(a.src12, al));
    const ds Gx = ds_add(ds_sub(ds_mul(a.wp4, ds_add(ds_add(ds_mul(Mxx, u[0]), ds_mul(Mxy, u[1])), ds_mul(Mxz, u[2]))),
                                ds_mul(m0, u[0])), ds_mul(beta, M1x));
    const ds Gy = ds_add(ds_sub(ds_mul(a.wp4, ds_add(ds_add(ds_mul(Mxy, u[0]), ds_mul(Myy, u[1])), ds_mul(Myz, u[2]))),
                                ds_mul(m0, u[1])), ds_mul(beta, M1y));
    const ds Gz = ds_add(ds_sub(ds_mul(a.wp4, ds_add(ds_add(ds_mul(Mxz, u[0]), ds_mul(Myz, u[1])), ds_mul(Mzz, u[2]))),
                                ds_mul(m0, u[2])), ds_mul(beta, M1z));
    const ds base = ds_mul(a.wp36, M0);
    {
      const ds v = ds_add(ds_mul(a.one_m_wp, lf[0]), base);
      lam_out[i] = make_float2(v.hi, v.lo);
    }
#define LBM_ADJ_DS_PAIR(P, CG)                                                                  \
  {                                                                                             \
    const ds e_ = ds_add(ds_mul(a.hp, S[P]), base);                                             \
    const ds o_ = ds_add(ds_mul(a.hm, D[P]), ds_mul(s, (CG)));                                  \
    const ds va_ = ds_add(e_, o_);                                                              \
    const ds vb_ = ds_sub(e_, o_);                                                              \
    lam_out[(2 * P + 2) * ld + i] = make_float2(va_.hi, va_.lo);                                \
    lam_out[(2 * P + 1) * ld + i] = make_float2(vb_.hi, vb_.lo);                                \
  }
    LBM_ADJ_DS_PAIR(0, Gx)
    LBM_ADJ_DS_PAIR(1, Gy)
    LBM_ADJ_DS_PAIR(2, Gz)
    LBM_ADJ_DS_PAIR(3, ds_add(Gx, Gy))
    LBM_ADJ_DS_PAIR(4, ds_sub(Gx, Gy))
    LBM_ADJ_DS_PAIR(5, ds_add(Gx, Gz))
    LBM_ADJ_DS_PAIR(6, ds_sub(Gx, Gz))
    LBM_ADJ_DS_PAIR(7, ds_add(Gy, Gz))
    LBM_ADJ_DS_PAIR(8, ds_sub(Gy, Gz))
#undef LBM_ADJ_DS_PAIR
    const ds hs = ds_scale_pow2(s, 0.5f);
    red[0] = ds_add(ds_mul(hs, Gx), ds_mul(a.src12, M1x));
    red[1] = ds_add(ds_mul(hs, Gy), ds_mul(a.src12, M1y));
    red[2] = ds_add(ds_mul(hs, Gz), ds_mul(a.src12, M1z));
    const ds Gu = ds_add(ds_add(ds_mul(Gx, u[0]), ds_mul(Gy, u[1])), ds_mul(Gz, u[2]));
    const ds M1u = ds_add(ds_add(ds_mul(M1x, u[0]), ds_mul(M1y, u[1])), ds_mul(M1z, u[2]));
    if (dalpha) dalpha[i] += ds_to_double(ds_neg(ds_add(ds_mul(hs, Gu), ds_mul(a.src12, M1u))));
  }
  block_accumulate4_ds(red, part + z + 4 * (int64_t)blockIdx.x, false);
}

// lam_f_0 = S^T lam_g_1 (gradient with respect to the initial PDFs, [19][n]).
__device__ __forceinline__ double as_double(double v) { return v; }
__device__ __forceinline__ double as_double(float v) { return (double)v; }
__device__ __forceinline__ double as_double(float2 v) { return (double)v.x + (double)v.y; }
template <class T, bool SHORT>
__global__ void __launch_bounds__(kSweepThreads)
    adjoint_initial_kernel(Links links, int32_t n, int32_t ld, const T* __restrict__ lam_in,
                           double* __restrict__ out) {
  const int32_t i = blockIdx.x * kSweepThreads + threadIdx.x;
  int32_t idx[18];
  load_links<SHORT>(links, n, ld, i, idx);
  if (i >= n) return;
  T lf[19];
  pull_adjoint(lam_in, idx, i, lf);
#pragma unroll
  for (int q = 0; q < 19; ++q) out[q * (int64_t)n + i] = as_double(lf[q]);
}

// ---- host orchestration -------------------------------------------------------

template <int PREC>
struct Runner {
  using S = typename Form<PREC>::S;
  using C = typename Form<PREC>::C;
  // an element of lambda and of the kept velocities
  using E = std::conditional_t<PREC == LBM_F64X, float2, C>;
  lbm_adjoint* ad;
  const lbm_state* st;
  int32_t n, ld, M;
  cudaStream_t stream;
  unsigned grid;
  Links links;
  Coef<C> k;
  AdjCoef<C> a;
  AdjCoefDS ads;   // LBM_F64X: the reverse step in double-single arithmetic
  // Kernels after the first of a forward or backward pass are chained
  // (programmatic dependent launch; the kernels wait for their predecessor),
  // except in FP64 arithmetic, which chaining slows down.
  static constexpr bool kChain = PREC != LBM_F64;
  bool chained = false;
  cudaError_t err = cudaSuccess;

  Runner(lbm_adjoint* ad_) : ad(ad_), st(ad_->st) {
    n = (int32_t)st->sp->n;
    ld = (int32_t)st->sp->ld;
    M = ad->K - 1;
    stream = st->sp->stream;
    grid = (unsigned)st->nblocks;
    links = state_links(st->sp);
    k = make_coef<C>(ad->wp, ad->wm, ad->F, st->scale_exp);
    a = make_adj_coef<C>(ad->wp, ad->wm, n);
    if constexpr (PREC == LBM_F64X) ads = make_adj_coef_ds(ad->wp, ad->wm);
  }
  S* ckpt(int j) const { return (S*)ad->ckpt + (size_t)j * 19 * ld; }
  E* u(int slot) const { return (E*)ad->u + (size_t)slot * 3 * ld; }
  E* lam(int i) const { return (E*)ad->lam[i]; }

  template <class... P, class... A>
  void launch_threads(void (*kernel)(P...), unsigned threads, A... args) {
    const cudaError_t e = launch_chained(kernel, grid, threads, stream, kChain && chained, args...);
    if (err == cudaSuccess) err = e;
    chained = true;
  }
  template <class... P, class... A>
  void launch(void (*kernel)(P...), A... args) {
    launch_threads(kernel, (unsigned)kSweepThreads, args...);
  }
  void step(const void* src, void* dst, E* u_out) {
    const cudaError_t e = launch_plain_step(st, src, dst, u_out, ad->wp, ad->wm, ad->F, stream,
                                            kChain && chained);
    if (err == cudaSuccess) err = e;
    chained = true;
  }
  template <bool DA, bool SH>
  void seed_form(const S* f_prev) {
    const C* alpha = (const C*)st->alpha;
    if constexpr (PREC == LBM_F64X)
      launch(adjoint_seed_ds_kernel<DA, SH>, f_prev, links, n, ld, k, a, alpha, ad->axis, lam(0),
             ad->part, ad->dalpha);
    else
      launch(adjoint_seed_kernel<PREC, DA, SH>, f_prev, links, n, ld, k, a, alpha, ad->axis,
             lam(0), ad->part, ad->dalpha);
  }
  void seed() {
    const S* f_prev = (const S*)ad->last;
    if (links.wide) st->alpha ? seed_form<true, false>(f_prev) : seed_form<false, false>(f_prev);
    else st->alpha ? seed_form<true, true>(f_prev) : seed_form<false, true>(f_prev);
  }
  template <bool DA, bool SH>
  void reverse_form(const E* u_in, int in, double* dalpha) {
    const C* alpha = (const C*)st->alpha;
    if constexpr (PREC == LBM_F64X)
      launch(adjoint_step_ds_kernel<DA, SH>, u_in, links, n, ld, ads, alpha,
             (const int64_t*)st->alpha_fx, (const float2*)lam(in), lam(in ^ 1), ad->part, dalpha);
    else if constexpr (SH && sizeof(C) == 4)
      launch_threads(adjoint_pair_kernel<DA>, (unsigned)kSweepThreads / 2, u_in, links, n, ld, a, alpha,
                     (const C*)lam(in), lam(in ^ 1), ad->part, dalpha);
    else
      launch(adjoint_step_kernel<C, DA, SH>, u_in, links, n, ld, a, alpha, (const C*)lam(in),
             lam(in ^ 1), ad->part, dalpha);
  }
  void reverse(const E* u_in, int in, double* dalpha) {
    if (links.wide)
      st->alpha ? reverse_form<true, false>(u_in, in, dalpha) : reverse_form<false, false>(u_in, in, dalpha);
    else
      st->alpha ? reverse_form<true, true>(u_in, in, dalpha) : reverse_form<false, true>(u_in, in, dalpha);
  }

  // First step of segment j (j = n_seg: of the last steps, whose velocities
  // the forward pass keeps).
  int32_t first(int j) const {
    return j < ad->n_seg ? j * ad->seg_len + 1 : M - std::min(M, ad->slots) + 1;
  }

  // Steps t0..t1 from f_{t0-1} = cur, keeping the velocities of those from
  // `keep` on in slots 0, 1, ...; with `checkpoints`, the f a segment starts
  // from goes to its checkpoint.  Returns f_{t1}.
  const void* advance(const void* cur, int32_t t0, int32_t t1, int32_t keep, bool checkpoints) {
    int j = 1;
    for (int32_t t = t0; t <= t1; ++t) {
      while (j < ad->n_seg && first(j) <= t) ++j;
      void* dst = checkpoints && j < ad->n_seg && first(j) == t + 1 ? (void*)ckpt(j)
                  : cur == ad->f[0]                                 ? ad->f[1]
                                                                    : ad->f[0];
      step(cur, dst, t >= keep ? u(t - keep) : nullptr);
      cur = dst;
    }
    return cur;
  }

  // Forward pass from the state's current PDFs.
  int forward() {
    const size_t bytes = 19 * (size_t)ld * sizeof(S);
    const void* cur = st->buf[st->cur];
    // the PDFs a later reverse pass starts over from
    void* copy = ad->n_seg > 0 ? ad->ckpt : (M == 0 ? ad->f[0] : nullptr);
    if (copy) {
      LBM_CUDA_TRY(cudaMemcpyAsync(copy, cur, bytes, cudaMemcpyDeviceToDevice, stream));
      cur = copy;
    }
    chained = false;
    ad->last = advance(cur, 1, M, first(ad->n_seg), true);
    seed();
    ad->fresh = true;
    return LBM_OK;
  }

  int backward(double* dJdf0, double* dalpha) {
    const int32_t kept = first(ad->n_seg);
    chained = false;
    if (!ad->fresh) {   // a second reverse pass: everything the first one overwrote
      if (ad->n_seg > 0)
        ad->last = advance(ckpt(ad->n_seg - 1), first(ad->n_seg - 1), M, kept, false);
      seed();
    }
    ad->fresh = false;
    int in = 0;
    for (int32_t t = M; t >= kept; --t, in ^= 1) reverse(u(t - kept), in, dalpha);
    for (int j = ad->n_seg - 1; j >= 0; --j) {
      const int32_t t0 = first(j), t1 = first(j + 1) - 1;
      advance(ckpt(j), t0, t1, t0, false);
      for (int32_t t = t1; t >= t0; --t, in ^= 1) reverse(u(t - t0), in, dalpha);
    }
    if (dJdf0) {
      if (links.wide)
        adjoint_initial_kernel<E, false><<<grid, kSweepThreads, 0, stream>>>(links, n, ld, (const E*)lam(in), dJdf0);
      else
        adjoint_initial_kernel<E, true><<<grid, kSweepThreads, 0, stream>>>(links, n, ld, (const E*)lam(in), dJdf0);
    }
    LBM_CUDA_TRY(err);
    LBM_CUDA_TRY(cudaGetLastError());
    return LBM_OK;
  }
};

template <int PREC>
int run_forward(lbm_adjoint* ad) {
  Runner<PREC> r(ad);
  if (r.n == 0) return LBM_OK;
  ad->fresh = false;
  const int rc = r.forward();
  if (rc != LBM_OK) return rc;
  if (r.err != cudaSuccess) ad->fresh = false;
  LBM_CUDA_TRY(r.err);
  LBM_CUDA_TRY(cudaGetLastError());
  return LBM_OK;
}

template <int PREC>
int run_backward(lbm_adjoint* ad, double* dJdf0, double* dalpha) {
  Runner<PREC> r(ad);
  if (r.n == 0) return LBM_OK;
  return r.backward(dJdf0, dalpha);
}

#define LBM_ADJ_DISPATCH(prec, fn, ...)                      \
  switch (prec) {                                            \
    case LBM_F64: return fn<LBM_F64>(__VA_ARGS__);           \
    case LBM_F64X: return fn<LBM_F64X>(__VA_ARGS__);         \
    case LBM_F32: return fn<LBM_F32>(__VA_ARGS__);           \
    case LBM_F32S: return fn<LBM_F32S>(__VA_ARGS__);         \
    case LBM_F16S: return fn<LBM_F16S>(__VA_ARGS__);         \
    default: return fn<LBM_BF16S>(__VA_ARGS__);              \
  }

int dispatch_forward(lbm_adjoint* ad) { LBM_ADJ_DISPATCH(ad->st->precision, run_forward, ad) }
int dispatch_backward(lbm_adjoint* ad, double* dJdf0, double* dalpha) {
  LBM_ADJ_DISPATCH(ad->st->precision, run_backward, ad, dJdf0, dalpha)
}

bool valid_adjoint(const lbm_adjoint* ad) { return ad && ad->magic == kMagicAdjoint; }

// Final sums of the per-block accumulators into red_host.
int finish_sums(lbm_adjoint* ad) {
  const cudaStream_t stream = ad->st->sp->stream;
  if (ad->st->sp->n == 0) {
    for (int j = 0; j < 4; ++j) ad->red_host[j] = 0.0;
    return LBM_OK;
  }
  final_sum_kernel<<<1, 1024, 0, stream>>>(ad->part, ad->st->nblocks, ad->red_host);
  LBM_CUDA_TRY(cudaGetLastError());
  return wait_event(ad->done, stream, 0.0);
}

}  // namespace

void free_adjoint(lbm_adjoint* ad) {
  if (!ad) return;
  // the state may already be released (a garbage collector may free the two
  // in either order): only the stream kept here is used
  const cudaStream_t s = ad->stream;
  cudaStreamSynchronize(s);
  for (void* p : {ad->ckpt, ad->f[0], ad->f[1], ad->u, ad->lam[0], ad->lam[1], (void*)ad->part,
                  (void*)ad->dalpha})
    dev_free(p, s, false);
  if (ad->red_host) cudaFreeHost(ad->red_host);
  if (ad->done) cudaEventDestroy(ad->done);
  ad->magic = 0;
  delete ad;
}

}  // namespace lbm

using namespace lbm;

extern "C" int lbm_adjoint_create(const lbm_state* st, int32_t n_steps, int32_t stride,
                                  lbm_adjoint** out) {
  clear_error();
  if (!out) return fail(LBM_EINVAL, "out is NULL");
  *out = nullptr;
  if (!valid_state(st)) return fail(LBM_EINVAL, "not a state handle");
  if (st->batch) return fail(LBM_EINVAL, "the adjoint is not available on a batched state");
  if (n_steps < 1) return fail(LBM_EINVAL, "n_steps = %d must be >= 1", n_steps);
  if (stride < 0) return fail(LBM_EINVAL, "checkpoint stride %d < 0", stride);
  if (stride == 0) stride = (int32_t)std::ceil(std::sqrt((double)n_steps));
  if (stride > n_steps) stride = n_steps;
  lbm_adjoint* ad = new lbm_adjoint{};
  ad->magic = kMagicAdjoint;
  ad->st = st;
  ad->stream = st->sp->stream;
  ad->K = n_steps;
  const size_t n = (size_t)(st->sp->n > 0 ? st->sp->n : 1);
  const size_t ld = (size_t)(st->sp->ld > 0 ? st->sp->ld : 1);
  const size_t srow = storage_bytes(st->precision) * ld, crow = compute_bytes(st->precision) * ld;
  // The memory asked for: a checkpoint every `stride` steps and a segment of
  // `stride` states, in rows.  Two states and n_seg checkpoints leave the rest
  // to velocities; the fewest segments none of which is longer than those.
  const int64_t M = n_steps - 1;
  const int64_t states = M / stride + 1 + std::max(stride, 2);
  const int64_t per_slot = 3 * (int64_t)(crow / srow);
  int64_t seg = 0, slots = 0;
  for (;; ++seg) {
    slots = std::min(M, (19 * (states - 2 - seg)) / per_slot);
    if (slots * (seg + 1) >= M) break;
  }
  ad->slots = (int32_t)slots;
  ad->n_seg = (int32_t)seg;
  ad->seg_len = seg > 0 ? (int32_t)((M - slots + seg - 1) / seg) : 0;
  if (seg > 0) ad->n_seg = (int32_t)((M - slots + ad->seg_len - 1) / ad->seg_len);
  const cudaStream_t s = st->sp->stream;
  const auto rows = [&](void** p, size_t count, size_t row) {
    return count == 0 || dev_alloc(p, count * row, s, false) == cudaSuccess;
  };
  bool ok = rows(&ad->ckpt, 19 * (size_t)ad->n_seg, srow) && rows(&ad->f[0], 19, srow) &&
            rows(&ad->f[1], M > 1 ? 19 : 0, srow) && rows(&ad->u, 3 * (size_t)ad->slots, crow) &&
            rows(&ad->lam[0], 19, crow) && rows(&ad->lam[1], 19, crow) &&
            dev_alloc(&ad->part, sizeof(double) * 4 * st->nblocks, s, false) == cudaSuccess &&
            dev_alloc(&ad->dalpha, sizeof(double) * n, s, false) == cudaSuccess &&
            cudaMallocHost(&ad->red_host, sizeof(double) * 4) == cudaSuccess &&
            cudaEventCreateWithFlags(&ad->done, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    const int32_t ad_seg = ad->n_seg;
    free_adjoint(ad);
    return fail(LBM_ENOMEM,
                "adjoint allocation failed (%d checkpoints of %zu bytes, %d velocity fields of %zu)",
                (int)ad_seg, 19 * srow, (int)slots, 3 * crow);
  }
  *out = ad;
  return LBM_OK;
}

extern "C" int lbm_adjoint_forward(lbm_adjoint* ad, double omega_plus, double omega_minus,
                                   const double force[3], int32_t axis, double* J_out) {
  clear_error();
  if (!valid_adjoint(ad)) return fail(LBM_EINVAL, "not an adjoint handle");
  if (!valid_state(ad->st)) return fail(LBM_EINVAL, "the adjoint's state was released");
  if (axis < 0 || axis > 2) return fail(LBM_EINVAL, "axis %d outside {0,1,2}", axis);
  if (!(omega_plus > 0.0 && omega_plus < 2.0) || !(omega_minus > 0.0 && omega_minus < 2.0))
    return fail(LBM_EINVAL, "relaxation rates must lie in (0, 2): %g, %g", omega_plus, omega_minus);
  if (!force) return fail(LBM_EINVAL, "force is NULL");
  for (int d = 0; d < 3; ++d)
    if (!std::isfinite(force[d])) return fail(LBM_EINVAL, "force[%d] is not finite", d);
  ad->wp = omega_plus;
  ad->wm = omega_minus;
  for (int d = 0; d < 3; ++d) ad->F[d] = force[d];
  ad->axis = axis;
  int rc = dispatch_forward(ad);
  if (rc != LBM_OK) return rc;
  rc = finish_sums(ad);
  if (rc != LBM_OK) return rc;
  const int64_t n = ad->st->sp->n;
  const double J = n > 0 ? ad->red_host[3] / (double)n : 0.0;
  if (!std::isfinite(J)) return fail(LBM_ENONFINITE, "objective is not finite");
  ad->have_forward = 1;
  if (J_out) *J_out = J;
  return LBM_OK;
}

extern "C" int lbm_adjoint_backward(lbm_adjoint* ad, double dJdF_out[3], double* dJdalpha_dev,
                                    double* dJdf0_dev) {
  clear_error();
  if (!valid_adjoint(ad)) return fail(LBM_EINVAL, "not an adjoint handle");
  if (!valid_state(ad->st)) return fail(LBM_EINVAL, "the adjoint's state was released");
  if (!ad->have_forward) return fail(LBM_EINVAL, "lbm_adjoint_forward has not run");
  int rc = dispatch_backward(ad, dJdf0_dev, dJdalpha_dev ? ad->dalpha : nullptr);
  if (rc != LBM_OK) return rc;
  const cudaStream_t stream = ad->st->sp->stream;
  const int64_t n = ad->st->sp->n;
  if (dJdalpha_dev && n > 0)
    LBM_CUDA_TRY(cudaMemcpyAsync(dJdalpha_dev, ad->dalpha, sizeof(double) * n,
                                 cudaMemcpyDeviceToDevice, stream));
  rc = finish_sums(ad);
  if (rc != LBM_OK) return rc;
  for (int d = 0; d < 3; ++d)
    if (!std::isfinite(ad->red_host[d])) return fail(LBM_ENONFINITE, "dJ/dF is not finite");
  if (dJdF_out)
    for (int d = 0; d < 3; ++d) dJdF_out[d] = ad->red_host[d];
  return LBM_OK;
}

extern "C" int lbm_adjoint_step(lbm_state* st, lbm_adjoint* ad, int32_t n_steps,
                                double omega_plus, double omega_minus, const double force[3],
                                int32_t axis, double* J_out, double dJdF_out[3],
                                double* dJdalpha_dev) {
  clear_error();
  if (!valid_adjoint(ad)) return fail(LBM_EINVAL, "not an adjoint handle");
  if (ad->st != st) return fail(LBM_EINVAL, "the adjoint was created for another state");
  if (n_steps != ad->K)
    return fail(LBM_EINVAL, "the adjoint was created for %d steps, not %d", ad->K, n_steps);
  int rc = lbm_adjoint_forward(ad, omega_plus, omega_minus, force, axis, J_out);
  if (rc != LBM_OK) return rc;
  return lbm_adjoint_backward(ad, dJdF_out, dJdalpha_dev, nullptr);
}
