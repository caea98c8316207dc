// Adjoint of the WD WENO 2x zoom (arXiv 2312.00229, Sec. 3), FP32.
//
// For one blend point u = sum_k omega_k p_k with omega_k = alpha_k / sum alpha
// and alpha_k = D_k^-beta (Eqs. alpha, IzrazOmega2d, 2dKombinacija and the
// phase-2 forms), the local adjoints of an incoming u_bar are
//     p_bar_k = u_bar omega_k
//     D_bar_k = -u_bar beta omega_k (p_k - u) / D_k .
// D_k = SI_k(c) + w sum_{nbr} SI_k(c + delta) (Eqs. 2DsmoothnessFinal, tezine),
// so SI_bar_k(c) = D_bar_k(c) + w sum of D_bar_k over the points whose D
// reads c.  With SI = g^2 + kappa^2 s^2 + eps', g = N1 - N0,
// s = N0 - 2 N1 + N2 and p = 3/8 N0 + 3/4 N1 - 1/8 N2 (Eq. p), a stencil
// sends to its nodes
//     N0: 3/8 p_bar + (-2 g + 2 kappa^2 s) SI_bar
//     N1: 3/4 p_bar + ( 2 g - 4 kappa^2 s) SI_bar
//     N2: -1/8 p_bar + 2 kappa^2 s SI_bar .
//
// Two row-sweep kernels, each CTA one plane x one strip of columns x one band
// of rows, sweeping its band top to bottom one coarse row per step with one
// barrier per step; a stage at step s works on row s - L for its own lag L.
//
//   k_bwd_plus   recomputes the forward pass (phase-1 indicators and values,
//                phase-2 indicators) and runs the phase-2 adjoint: p_bar,
//                D_bar of every E and S point, their SI_bar and the node
//                coefficients, gathered onto the x points (X_bar, plus the
//                x-point output gradient) and onto the input samples (plus
//                the sample-point output gradient).  Writes X_bar and that
//                partial A_bar on the grid extended by 2 cells per side.
//   k_bwd_cross  recomputes the phase-1 indicators, runs the phase-1 adjoint
//                from X_bar, gathers the node coefficients onto the samples,
//                adds the partial A_bar and folds the clamp-to-edge
//                extension back onto the edge pixels (its adjoint).
//
// What bounds them: shared-memory wavefronts (one a cycle and SM).  Read from
// four-row float4 rings, the five terms of every D and SI_bar cost 20
// wavefronts a point, and a warp's step took 172 of them in k_bwd_plus and 93
// in k_bwd_cross, 80% of the time.  So values of a thread's own column stay
// in registers, and what a neighbour needs is published once, summed over the
// two rows it reads (one float4 read a point instead of five):
//     VS(r) = SIS(r-1) + SIS(r), VE(r) likewise, for the D of E(r), S(r-1);
//     VDS(r), VDE(r): the same sums of D_bar for the SI_bar of E(r), S(r-1);
//     x points: the column's sum of three rows in registers, and the
//     indicators (D_bar) of the two side columns.
// The stencil data of a "+" point (second and first differences) wait in
// shared memory for its two later stages instead of being formed again.
// Scatters are gathers: a contribution to a thread's own column is added to
// a short register ring of row accumulators, contributions to other columns
// are published per row in shared memory and gathered one step later.
// In the middle of a band the steps run in groups of four with every ring
// slot a compile-time constant and no stage guards (sweep_band); the global
// values a step needs are copied to shared memory asynchronously three steps
// before it (copy_async).
//
// 32x3x512x512, both kernels: 1078 us with the four-row rings and register
// prefetch; 1001 with the row-pair sums, own-column registers and kept
// stencils; 883 with the asynchronous copies; 856 with a forward and a
// backward thread per column in k_bwd_plus; 816 with the forward threads also
// requesting the gradients that the backward threads use, and strides read
// from the constant bank (2x3x1024x1024: 276, 248, 238, 233; 3x256x256: 49, 45, 44,
// 36, the last with the shapes of pick_shape).  Now 140 and 56 wavefronts a
// warp's step, LSU pipe 78% and 63% busy, 377 and 176 M warp instructions
// (455 and 233 before).  Two to five CTAs per SM in k_bwd_cross measure the same.
#include "wd_bwd.h"

#include <atomic>
#include <cmath>

#include "wd_packed.cuh"

namespace wdweno {

namespace {

// ---- shared-memory rings ------------------------------------------------------
constexpr int PAD = 2;  // ring columns before / after the CTA's threads

// k_bwd_plus: thread t owns column c = b0 - HL1 + t of a strip whose outputs
// are columns [b0, b0 + NT - HL1 - HR1) of the extended grid.
constexpr int HL1 = 6, HR1 = 7;
// k_bwd_cross: the strip's outputs are image columns [b0, b0 + NT - HL2 - HR2)
// plus, at the image edges, the ghost columns folded onto them.
constexpr int HL2 = 10, HR2 = 10;
// CTA widths built for both sweeps (the host picks one per image width)
constexpr int NT_NARROW = 128, NT_WIDE = 192;
constexpr int GA = 5;  // ghost rows / columns of A_bar (nonzero up to 4)
// A request made in step s is used in step s + AHEAD + 1; AHEAD + 1 groups of
// copies are in flight.
constexpr int AHEAD = 2;

// Stencil data of a point: what its blend and its adjoint need once the
// indicators are formed.  Opposite directions share their first difference
// (g of direction 1 is -g01, of direction 3 -g23).
struct Sten {
  float4 s;     // N0 - 2 N1 + N2 per direction
  float2 g;     // N1 - N0 of directions 0 and 2
  float M0, M1; // N0 + N1 of the direction pairs (0,1) and (2,3)
};

// Rings of the two-role sweep (slot = row mod depth).
template <int NT>
struct RingsPlus {
  static constexpr int W = NT + 2 * PAD;
  float4 SIX[2][W];   // phase-1 indicators (4 directions)
  float4 VS[2][W];    // S-point indicators of rows r-1 and r summed
  float4 VE[2][W];    // E-point indicators of rows r-1 and r summed
  float4 VDS[2][W];   // 2 D_bar of the S points of rows r-1 and r summed
  float4 VDE[2][W];   // 2 D_bar of the E points of rows r-1 and r summed
  float EY[4][W];     // second difference of input row r centred at c
  float SY[4][W];     // second difference of x row r centred at c
  float A[8][W];      // input rows
  float X[2][W];      // phase-1 values
  // Row stencils' node contributions pre-summed by target column, one array
  // per target so that each gather reads a scalar per thread (no strided
  // component reads of a vector array)
  float EH[3][2][W];  // E along row r: to sample columns c-1, c+1, c+2
  float SH[3][2][W];  // S along row r: to x columns c-2, c-1, c+1
  // From the forward thread of a column to its backward thread: own-column
  // parts of the D of E(r), S(r-1); column second differences of the two
  // vertical directions, first differences, (M1 - M0) / 2 of E(r), S(r)
  float4 DE[2][NT], DS[2][NT];
  float2 EZ[4][NT], SZ[4][NT], EG[4][NT], SG[4][NT];
  float EM[4][NT], SM[4][NT];
  // Output gradients: fine rows 2r, columns
  // 2c, 2c + 1 (samples, E points), and 2r + 1 (S, x points)
  float2 GE[4][NT], GS[4][NT];
};

template <int NT>
struct RingsCross {
  static constexpr int W = NT + 2 * PAD;
  float4 SIX[2][W];
  float4 DX[2][W];    // x 2 D_bar
  float2 C1[2][W];    // contributions to column c+1: rows a, a+1
  float2 C2[2][W];    // to column c+2: rows a+2, a-1
  float2 CM[2][W];    // to column c-1: rows a-1, a+2
  float XB[4][W];     // X_bar and partial A_bar of the column (thread-private)
  float AB[4][W];
  float A[8][W];      // input rows
  float AF[2][W];     // row-folded A_bar of the row emitted in the previous step
};

// ---- the method's per-point quantities ---------------------------------------
__device__ __forceinline__ float diff2(float n0, float n1, float n2) {
  return fmaf(-2.f, n1, n0 + n2);
}

// x point X(a,b) (fine (2a+1, 2b+1)).  Directions: 0 (1,1): A(a,b),
// A(a+1,b+1), A(a+2,b+2); 1 (-1,-1): A(a+1,b+1), A(a,b), A(a-1,b-1);
// 2 (1,-1): A(a,b+1), A(a+1,b), A(a+2,b-1); 3 (-1,1): A(a+1,b), A(a,b+1),
// A(a-1,b+2).  am1..a2: rows a-1 .. a+2 at column b.
__device__ __forceinline__ Sten sten_x(const float* am1, const float* a0, const float* a1,
                                       const float* a2) {
  const float n00 = a0[0], n01 = a0[1], n10 = a1[0], n11 = a1[1];
  Sten q;
  q.g = make_float2(n11 - n00, n10 - n01);
  q.s = make_float4(diff2(n00, n11, a2[2]), diff2(n11, n00, am1[-1]), diff2(n01, n10, a2[-1]),
                    diff2(n10, n01, am1[2]));
  q.M0 = n00 + n11;
  q.M1 = n01 + n10;
  return q;
}

// The helpers below work on the direction pairs (0, 1) and (2, 3) with the
// packed two-lane FP32 instructions of wd_packed.cuh.
__device__ __forceinline__ f2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ f2 hi2(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 cat4(f2 a, f2 b) { return make_float4(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ float4 zero4() { return make_float4(0.f, 0.f, 0.f, 0.f); }

__device__ __forceinline__ float4 add4(const float4& a, const float4& b) {
  return cat4(pk_add(lo2(a), lo2(b)), pk_add(hi2(a), hi2(b)));
}

// a + w b
__device__ __forceinline__ float4 fma4(float w, const float4& b, const float4& a) {
  return cat4(pk_fma(pk_bc(w), lo2(b), lo2(a)), pk_fma(pk_bc(w), hi2(b), hi2(a)));
}

// SI_k = g_k^2 + (kappa s_k)^2 + eps
__device__ __forceinline__ float4 indicators(const float4& s, const float2& g, float kap,
                                             float eps) {
  const f2 k01 = pk_mul(pk_bc(kap), lo2(s)), k23 = pk_mul(pk_bc(kap), hi2(s));
  const f2 e01 = pk_fma(k01, k01, pk_bc(eps)), e23 = pk_fma(k23, k23, pk_bc(eps));
  return make_float4(fmaf(g.x, g.x, e01.x), fmaf(g.x, g.x, e01.y), fmaf(g.y, g.y, e23.x),
                     fmaf(g.y, g.y, e23.y));
}

// Normalised weights omega_k from D_k (Eqs. alpha, IzrazOmega2d), and 1/D_k.
template <int BMODE>
__device__ __forceinline__ void weights(const float4& D, float beta, f2 (&om)[2], f2 (&rd)[2]) {
  f2 al[2];
  rd[0] = pk_rcp(lo2(D));
  rd[1] = pk_rcp(hi2(D));
  if (BMODE == B0) {
    al[0] = al[1] = pk_bc(1.f);
  } else {
    const f2 dmin = pk_bc(fminf(fminf(D.x, D.y), fminf(D.z, D.w)));
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const f2 r = pk_mul(dmin, rd[p]);
      if (BMODE == B2) {
        al[p] = pk_mul(r, r);
      } else {
        const f2 l = pk_mul(pk_bc(beta), make_float2(lg2_approx(r.x), lg2_approx(r.y)));
        al[p] = make_float2(ex2_approx(l.x), ex2_approx(l.y));
      }
    }
  }
  // the largest alpha is 1, so the sum lies in [1, 4]
  const f2 inv = pk_bc(rcp_approx((al[0].x + al[0].y) + (al[1].x + al[1].y)));
  om[0] = pk_mul(al[0], inv);
  om[1] = pk_mul(al[1], inv);
}

// u = sum_k omega_k p_k with p_k = (N0 + N1)/2 - s_k/8 (Eq. p)
template <int BMODE>
__device__ __forceinline__ float blend(const float4& D, float M0, float M1, const float4& s,
                                       float beta) {
  f2 om[2], rd[2];
  weights<BMODE>(D, beta, om, rd);
  const f2 p01 = pk_fma(pk_bc(-0.125f), lo2(s), pk_bc(0.5f * M0));
  const f2 p23 = pk_fma(pk_bc(-0.125f), hi2(s), pk_bc(0.5f * M1));
  return fmaf(om[1].y, p23.y, fmaf(om[1].x, p23.x, fmaf(om[0].y, p01.y, om[0].x * p01.x)));
}

// p_bar and 2 D_bar of one blend point given its D and stencil data (D_bar
// is carried doubled: the node coefficients' factors of 2 fold into it).
// s: second differences; hM = (M1 - M0) / 2.
template <int BMODE>
__device__ __forceinline__ void point_adjoint(const float4& s, float hM, const float4& D,
                                              float beta, float ub, float4& pb4, float4& db4) {
  f2 om[2], rd[2];
  weights<BMODE>(D, beta, om, rd);
  // p_k - u from differences of the stencil data, so that no two O(1)
  // values cancel: d_k = p_k - p_0 = (M_k - M_0)/2 - (s_k - s_0)/8 and
  // u - p_0 = sum_l omega_l d_l, so p_k - u = d_k - sum_l omega_l d_l.
  const float d1 = -0.125f * (s.y - s.x);
  const float d2 = fmaf(-0.125f, s.z - s.x, hM);
  const float d3 = fmaf(-0.125f, s.w - s.x, hM);
  const float v = fmaf(om[0].y, d1, fmaf(om[1].x, d2, om[1].y * d3));
  const f2 pu[2] = {make_float2(-v, d1 - v), pk_sub(make_float2(d2, d3), pk_bc(v))};
  const float ubb = -ub * (2.f * beta);
  f2 pb[2], db[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    pb[p] = pk_mul(pk_bc(ub), om[p]);
    db[p] = BMODE == B0 ? pk_bc(0.f)
                        : pk_mul(pk_mul(pk_mul(pk_bc(ubb), om[p]), pu[p]), rd[p]);
  }
  pb4 = cat4(pb[0], pb[1]);
  db4 = cat4(db[0], db[1]);
}

// Contributions of one direction pair to its nodes, opposite directions
// summed: the nodes are d (N2 of the second direction), a (N0 of the first,
// N1 of the second), b (N1 and N0) and c (N2 of the first), in a line.
// pb, s, sb2 (2 SI_bar): the pair's lanes; g: N1 - N0 of the first direction.
struct Nodes {
  float d, a, b, c;
};
__device__ __forceinline__ Nodes node_coefs(f2 pb, f2 s, float g, f2 sb2, float k2) {
  const f2 s2 = pk_mul(pk_mul(pk_bc(k2), s), sb2);
  const f2 h = pk_mul(pk_bc(0.375f), pb);
  const f2 t = pk_add(h, s2);                       // 3/8 p_bar + s2 (N0)
  const f2 y = pk_sub(h, s2);                       // 2 y = 3/4 p_bar - 2 s2 (N1)
  const f2 e = pk_fma(pk_bc(-0.125f), pb, s2);      // N2
  const float G = g * (sb2.x + sb2.y);
  Nodes n;
  n.a = fmaf(2.f, y.y, t.x) - G;
  n.b = fmaf(2.f, y.x, t.y) + G;
  n.c = e.x;
  n.d = e.y;
  return n;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) {
  return v < lo ? lo : (v > hi ? hi : v);
}

// Asynchronous copy of SIZE bytes to shared memory.  Global values a later
// step needs are requested this way and not loaded to registers: a load in
// flight holds one of a warp's six scoreboards, which the shared loads,
// reciprocals and other global loads of the steps in between share, so each
// wait for one of those waited for the youngest load too (long-scoreboard
// stalls of 1.4 an issued instruction in k_bwd_cross).
template <int SIZE>
__device__ __forceinline__ void copy_async(void* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "n"(SIZE)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Waits until at most the AHEAD youngest groups of this thread are in flight.
template <int AHEAD>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD) : "memory");
}

// ---- ring addressing of one step ---------------------------------------------
// A step at row s reads ring rows s - L for lags L known at compile time.
// RowsRT computes every slot from s at run time (slot = row mod depth);
// RowsCT<PH> serves the steps s = 4 G + PH of a four-step group: the rows of
// the 8-row ring fall into two groups of four consecutive slots, whose
// addresses (RingGroups) are formed once per group of steps, and row s - L
// lies in group (G - j) mod 2 at position p with j and p compile-time
// constants; the 4- and 2-row rings' slots are constants.
template <int W>
struct RowsRT {
  float* A;  // row slot 0 of the 8-row ring, at the thread's column
  int s;
  template <int L>
  __device__ __forceinline__ float* a() const { return A + ((s - L) & 7) * W; }
  template <int L>
  __device__ __forceinline__ int m4() const { return (s - L) & 3; }
  template <int L>
  __device__ __forceinline__ int m2() const { return (s - L) & 1; }
};

template <int W>
struct RingGroups {
  float* A[2];  // A[j]: first slot of ring group (G - j) mod 2, G = s >> 2
  __device__ __forceinline__ RingGroups(float* a, int s) {
    const int G = s >> 2;
    A[0] = a + 4 * (G & 1) * W;
    A[1] = a + 4 * ((G - 1) & 1) * W;
  }
};

template <int W, int PH>
struct RowsCT {
  const RingGroups<W>& g;
  template <int L>
  static constexpr int J = PH >= L ? -((PH - L) / 4) : (L - PH + 3) / 4;  // groups back
  template <int L>
  static constexpr int P = PH - L + 4 * J<L>;  // position inside the group
  template <int L>
  __device__ __forceinline__ float* a() const { return g.A[J<L> & 1] + P<L> * W; }
  template <int L>
  __device__ static constexpr int m4() { return (PH - L) & 3; }
  template <int L>
  __device__ static constexpr int m2() { return (PH - L) & 1; }
};

// Runs a band's steps s_begin .. s_end: four-step groups of FULL steps
// (every stage live, compile-time slots, no guards) where s is a multiple of
// 4 and the group lies inside [s_lo, s_hi], generic steps (run-time slots,
// stage guards) elsewhere.  One instance of each step form.
template <class SW>
__device__ __forceinline__ void sweep_band(SW& sw, float* ringA, int s_begin, int s_end,
                                           int s_lo, int s_hi) {
  constexpr int W = SW::W;
  int s = s_begin;
#pragma unroll 1
  while (s <= s_end) {
    if ((s & 3) == 0 && s >= s_lo && s + 3 <= s_hi) {
      const RingGroups<W> g(ringA, s);
      sw.template step<true>(s, RowsCT<W, 0>{g});
      sw.template step<true>(s + 1, RowsCT<W, 1>{g});
      sw.template step<true>(s + 2, RowsCT<W, 2>{g});
      sw.template step<true>(s + 3, RowsCT<W, 3>{g});
      s += 4;
    } else {
      sw.template step<false>(s, RowsRT<W>{ringA, s});
      ++s;
    }
  }
}

__device__ __forceinline__ bool any_nonzero(const float4& v, const float4& s) {
  return (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f) ||
         (s.x != 0.f || s.y != 0.f || s.z != 0.f || s.w != 0.f);
}

// ---- k_bwd_plus ----------------------------------------------------------------
// Two roles of NT threads each, a forward and a backward thread per column,
// half of the warps each.  All stages of a step read what earlier steps
// published, so the roles' stages of one step run side by side: twice the
// warps a scheduler can pick from, each with half of the step's dependent
// chain and half of its registers (80 instead of 168), for the own-column
// values handed over through shared memory.
// Lags (row = s - L at step s): input row 0, x indicators 3, x values 4, "+"
// indicators 5 (forward); E adjoints 6, S adjoints 7, "+" coefficients 8; the
// partial A_bar of row s - 9 and X_bar of row s - 10 are complete at step s
// (backward).
__device__ __forceinline__ void sync_cta() { asm volatile("bar.sync 0;" ::: "memory"); }

template <int BMODE, int NT1>
struct PlusForward {
  static constexpr int W = RingsPlus<NT1>::W;
  RingsPlus<NT1>& R;
  const BwdArgs& a;       // (kernel parameters: read from the constant bank)
  const MethodConsts& k;
  int t, u, n, a0, a1;
  const float* xin;  // input row s + 2 (clamped) of the column, in step s
  // output gradients of the fine columns 2c (samples, S points) and 2c + 1
  // (E and x points), which the column's backward thread reads
  const float* gp;       // fine row 2 (s - 3), column 2c, in step s
  bool g_pair, g_one0, g_one1;  // both columns inside and one aligned pair; else each
  // carried from step to step
  float4 six1, six2;          // phase-1 indicators of rows s-4, s-5
  float4 xs;                  // x stencils of row s-4: second differences
  float xM0, xM1;             // and node sums
  float x1, x2;               // phase-1 values of the column, rows s-5, s-6
  float ac1;                  // input row s-4 of the column
  float sxv, sav;             // column second differences centred at X(s-6), A(s-5)
  float4 sie1, sis1;          // "+" indicators of row s-6

  __device__ __forceinline__ PlusForward(RingsPlus<NT1>& R_, const BwdArgs& a_,
                                         const MethodConsts& k_, int thread, int c, int a0_,
                                         int a1_)
      : R(R_), a(a_), k(k_), t(thread), u(thread + PAD), n((int)a_.n), a0(a0_), a1(a1_) {
    // the first request is that of step a0 - 6 - (AHEAD + 1)
    xin = a.x + (int64_t)blockIdx.z * a.x_sc + (int64_t)clampi(c, 0, (int)a.m - 1) * a.x_sw +
          (int64_t)clampi(a0 - 6 - (AHEAD + 1) + 2, 0, n - 1) * a.x_sh;
    const int64_t Q = 2 * (int64_t)c;
    const bool inside = Q >= 0 && Q < a.ocols;
    g_pair = a.g_vec && inside && Q + 1 < a.ocols;
    g_one0 = inside && !g_pair;
    g_one1 = inside && Q + 1 < a.ocols && !g_pair;
    const int s0 = a0 - 6;  // first step (requests start AHEAD + 1 steps before it)
    gp = a.gout + (int64_t)blockIdx.z * a.g_sc + (inside ? Q : 0) * a.g_sw +
         2 * (int64_t)(s0 - (AHEAD + 1) - 3) * a.g_sh;
    six1 = six2 = xs = sie1 = sis1 = zero4();
    xM0 = xM1 = x1 = x2 = ac1 = sxv = sav = 0.f;
  }

  // Requests columns 2c, 2c + 1 of output-gradient row `row`, at q (FULL steps
  // request rows known to lie inside the output; columns outside it stay zero
  // from the rings' start).
  template <bool FULL>
  __device__ __forceinline__ void request_grad(float2* dst, const float* q, int row) const {
    if (!FULL && (row < 0 || row >= (int)a.orows)) {
      *dst = make_float2(0.f, 0.f);
      return;
    }
    if (g_pair) copy_async<8>(dst, q);
    if (g_one0) {
      copy_async<4>(&dst->x, q);
      if (g_one1) copy_async<4>(&dst->y, q + a.g_sw);
    }
  }

  // Step s's requests: input row s + 2 (to the ring; first read in step
  // s + 3) and the output gradients that step s + 3 uses.
  template <bool FULL, class SL>
  __device__ __forceinline__ void request(const int s, const SL& sl) {
    copy_async<4>(sl.template a<-2>(), xin);
    if (s + 2 >= 0 && s + 2 < n - 1) xin += a.x_sh;
    request_grad<FULL>(&R.GE[sl.template m4<3>()][t], gp, 2 * (s - 3));
    request_grad<FULL>(&R.GS[sl.template m4<4>()][t], gp - a.g_sh, 2 * (s - 4) + 1);
    copy_commit();
    gp += 2 * a.g_sh;
  }

  // Each stage runs only on the rows the band's outputs need (the guards are
  // uniform): the pipeline's fill and drain steps do just the stages that
  // have work.
  template <bool FULL, class SL>
  __device__ __forceinline__ void step(const int s, const SL& sl) {
    copy_wait<AHEAD>();
    sync_cta();
    request<FULL>(s, sl);
    // ---- x indicators, row s-3 ----
    const float ac = sl.template a<3>()[0];
    float4 six = zero4();
    Sten q;
    q.s = zero4();
    q.M0 = q.M1 = 0.f;
    if (FULL || (s - 3 >= a0 - 5 && s - 3 <= a1 + 4)) {
      q = sten_x(sl.template a<4>(), sl.template a<3>(), sl.template a<2>(), sl.template a<1>());
      six = indicators(q.s, q.g, k.kappa1, k.eps1);
      R.SIX[sl.template m2<3>()][u] = six;
    }
    // ---- x values, row s-4 ----
    float x0 = 0.f;
    if (FULL || (s - 4 >= a0 - 4 && s - 4 <= a1 + 3)) {
      const float4 l = R.SIX[sl.template m2<4>()][u - 1], r = R.SIX[sl.template m2<4>()][u + 1];
      const float4 D = fma4(k.w, add4(add4(six2, six), add4(l, r)), six1);
      x0 = blend<BMODE>(D, xM0, xM1, xs, k.beta);
      R.X[sl.template m2<4>()][u] = x0;
    }
    six2 = six1;
    six1 = six;
    xs = q.s; xM0 = q.M0; xM1 = q.M1;
    // ---- "+" indicators, row r = s-5 ----
    if (FULL || (s - 5 >= a0 - 4 && s - 5 <= a1 + 2)) {
      // E(r,c) (fine (2r, 2c+1)).  0 (0,1): A(r,c), A(r,c+1), A(r,c+2);
      // 1 (0,-1): A(r,c+1), A(r,c), A(r,c-1); 2 (1,0): X(r-1,c), X(r,c),
      // X(r+1,c); 3 (-1,0): X(r,c), X(r-1,c), X(r-2,c).
      const float* ar = sl.template a<5>();
      const float am = ar[-1], a_0 = ar[0], ap = ar[1], app = ar[2];
      const float sxn = diff2(x2, x1, x0);  // centred at X(r)
      const float4 es = make_float4(diff2(a_0, ap, app), diff2(ap, a_0, am), sxn, sxv);
      const float2 eg = make_float2(ap - a_0, x1 - x2);
      const float4 sie = indicators(es, eg, k.kappa2, k.eps2);
      R.EY[sl.template m4<5>()][u] = es.y;  // es.x is column c+1's
      R.EZ[sl.template m4<5>()][t] = make_float2(sxn, sxv);
      R.EG[sl.template m4<5>()][t] = eg;
      R.EM[sl.template m4<5>()][t] = 0.5f * ((x2 + x1) - (a_0 + ap));
      // S(r,c) (fine (2r+1, 2c)).  0 (0,1): X(r,c-1), X(r,c), X(r,c+1);
      // 1 (0,-1): X(r,c), X(r,c-1), X(r,c-2); 2 (1,0): A(r,c), A(r+1,c),
      // A(r+2,c); 3 (-1,0): A(r+1,c), A(r,c), A(r-1,c).
      const float* xr = R.X[sl.template m2<5>()] + u;
      const float xm = xr[-1], xmm = xr[-2], xp = xr[1];
      const float san = diff2(a_0, ac1, ac);  // centred at A(r+1)
      const float4 ss = make_float4(diff2(xm, x1, xp), diff2(x1, xm, xmm), san, sav);
      const float2 sg = make_float2(x1 - xm, ac1 - a_0);
      const float4 sis = indicators(ss, sg, k.kappa2, k.eps2);
      R.SY[sl.template m4<5>()][u] = ss.x;  // ss.y is column c-1's
      R.SZ[sl.template m4<5>()][t] = make_float2(san, sav);
      R.SG[sl.template m4<5>()][t] = sg;
      R.SM[sl.template m4<5>()][t] = 0.5f * ((a_0 + ac1) - (xm + x1));
      const float4 vs = add4(sis1, sis), ve = add4(sie1, sie);
      R.VS[sl.template m2<5>()][u] = vs;
      R.VE[sl.template m2<5>()][u] = ve;
      R.DE[sl.template m2<5>()][t] = fma4(k.w, vs, sie);
      R.DS[sl.template m2<5>()][t] = fma4(k.w, ve, sis1);
      sie1 = sie; sis1 = sis;
      sxv = sxn; sav = san;
    }
    x2 = x1; x1 = x0;
    ac1 = ac;
  }
};

template <int BMODE, int NT1>
struct PlusBackward {
  static constexpr int W = RingsPlus<NT1>::W;
  RingsPlus<NT1>& R;
  const BwdArgs& a;       // (kernel parameters: read from the constant bank)
  const MethodConsts& k;
  float k2;
  int t, u, a0, a1;
  float* wxb;            // X_bar row s - 10 of the column
  bool col_out;
  // carried from step to step
  float4 pe1, pe2, ps1;       // p_bar of E rows s-7, s-8 and of S row s-8
  float4 de1, ds1;            // 2 D_bar of E row s-7, S row s-8
  float4 sbE, sbS;            // own-column part of 2 SI_bar of E, S row s-8
  float xacc[4], aacc[4];     // X_bar rows s-10 .. s-7 and A_bar rows s-9 .. s-6

  __device__ __forceinline__ PlusBackward(RingsPlus<NT1>& R_, const BwdArgs& a_,
                                          const MethodConsts& k_, int thread, int c, int b0,
                                          int b1, int a0_, int a1_)
      : R(R_), a(a_), k(k_), k2(k_.kappa2 * k_.kappa2), t(thread), u(thread + PAD), a0(a0_),
        a1(a1_) {
    col_out = c >= b0 && c < b1;
    const int s0 = a0 - 6;  // first step
    wxb = a.ws + (int64_t)blockIdx.z * 2 * a.ws_cells +
          (int64_t)(s0 - 10 + BWD_GHOST) * a.ws_ld + (c + BWD_GHOST);
    pe1 = pe2 = ps1 = de1 = ds1 = sbE = sbS = zero4();
#pragma unroll
    for (int j = 0; j < 4; ++j) xacc[j] = aacc[j] = 0.f;
  }

  // Guarded steps skip the work of points whose incoming adjoints are all
  // zero (a sparse output gradient); FULL steps do it, with the same result.
  template <bool FULL, class SL>
  __device__ __forceinline__ void step(const int s, const SL& sl) {
    sync_cta();
    const float2 gE = R.GE[sl.template m4<6>()][t], gS = R.GS[sl.template m4<7>()][t];
    // the accumulators' newest rows start from the output gradient there
    aacc[3] = gE.x;  // sample (s-6, c)
    xacc[3] = gS.y;  // x point (s-7, c)

    // ---- row stencils' contributions of row s-9 ----
    {
      const int sp = sl.template m2<9>();
      xacc[1] += R.SH[0][sp][u + 2] + R.SH[1][sp][u + 1] + R.SH[2][sp][u - 1];
      aacc[0] += R.EH[0][sp][u + 1] + R.EH[1][sp][u - 1] + R.EH[2][sp][u - 2];
    }
    // ---- "+" coefficients, row r = s-8 ----
    if (FULL || (s - 8 >= a0 - 2 && s - 8 <= a1 + 1)) {
      {
        // E(r,c) is read by S(r,c), S(r,c+1), S(r-1,c), S(r-1,c+1)
        const float4 sb = fma4(k.w, R.VDS[sl.template m2<8>()][u + 1], sbE);
        float eh[3] = {0.f, 0.f, 0.f};
        if (FULL || any_nonzero(pe2, sb)) {
          const float* y = R.EY[sl.template m4<8>()] + u;
          const float2 z = R.EZ[sl.template m4<8>()][t], g = R.EG[sl.template m4<8>()][t];
          // along row r (samples): columns c-1, c, c+1, c+2
          const Nodes h = node_coefs(lo2(pe2), make_float2(y[1], y[0]), g.x, lo2(sb), k2);
          eh[0] = h.d; eh[1] = h.b; eh[2] = h.c;
          aacc[1] += h.a;
          // along column c (x values): rows r-2 .. r+1
          const Nodes v = node_coefs(hi2(pe2), z, g.y, hi2(sb), k2);
          xacc[0] += v.d; xacc[1] += v.a; xacc[2] += v.b; xacc[3] += v.c;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) R.EH[j][sl.template m2<8>()][u] = eh[j];
      }
      {
        // S(r,c) is read by E(r,c), E(r+1,c), E(r,c-1), E(r+1,c-1)
        const float4 sb = fma4(k.w, R.VDE[sl.template m2<7>()][u - 1], sbS);
        float sh[3] = {0.f, 0.f, 0.f};
        if (FULL || any_nonzero(ps1, sb)) {
          const float* y = R.SY[sl.template m4<8>()] + u;
          const float2 z = R.SZ[sl.template m4<8>()][t], g = R.SG[sl.template m4<8>()][t];
          // along row r (x values): columns c-2, c-1, c, c+1
          const Nodes h = node_coefs(lo2(ps1), make_float2(y[0], y[-1]), g.x, lo2(sb), k2);
          sh[0] = h.d; sh[1] = h.a; sh[2] = h.c;
          xacc[2] += h.b;
          // along column c (samples): rows r-1 .. r+2
          const Nodes v = node_coefs(hi2(ps1), z, g.y, hi2(sb), k2);
          aacc[0] += v.d; aacc[1] += v.a; aacc[2] += v.b; aacc[3] += v.c;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) R.SH[j][sl.template m2<8>()][u] = sh[j];
      }
    }
    // ---- X_bar of row s-10 and the partial A_bar of row s-9 are complete ----
    if (col_out && (FULL || (s - 10 >= a0 && s - 10 < a1))) *wxb = xacc[0];
    if (col_out && (FULL || (s - 9 >= a0 && s - 9 < a1))) wxb[a.ws_cells + a.ws_ld] = aacc[0];
    wxb += a.ws_ld;  // (A_bar row s-9 lies ws_cells + ws_ld behind X_bar row s-10)
    xacc[0] = xacc[1]; xacc[1] = xacc[2]; xacc[2] = xacc[3];
    aacc[0] = aacc[1]; aacc[1] = aacc[2]; aacc[2] = aacc[3];

    // ---- "+" adjoints: E row s-6, S row s-7 ----
    if (FULL || s - 6 >= a0 - 2) {
      float4 pe0 = zero4(), de = pe0, ps0 = pe0, ds = pe0;
      if (FULL || (s - 6 <= a1 + 1 && gE.y != 0.f)) {
        // E(r,c): D reads S at (r-1,c), (r,c), (r-1,c+1), (r,c+1)
        const float4 D =
            fma4(k.w, R.VS[sl.template m2<6>()][u + 1], R.DE[sl.template m2<6>()][t]);
        const float* y = R.EY[sl.template m4<6>()] + u;
        const float2 z = R.EZ[sl.template m4<6>()][t];
        point_adjoint<BMODE>(make_float4(y[1], y[0], z.x, z.y), R.EM[sl.template m4<6>()][t], D,
                             k.beta, gE.y, pe0, de);
      }
      if (FULL || (s - 7 >= a0 - 2 && s - 7 <= a1 + 1 && gS.x != 0.f)) {
        // S(r,c): D reads E at (r,c-1), (r,c), (r+1,c-1), (r+1,c)
        const float4 D =
            fma4(k.w, R.VE[sl.template m2<6>()][u - 1], R.DS[sl.template m2<6>()][t]);
        const float* y = R.SY[sl.template m4<7>()] + u;
        const float2 z = R.SZ[sl.template m4<7>()][t];
        point_adjoint<BMODE>(make_float4(y[0], y[-1], z.x, z.y), R.SM[sl.template m4<7>()][t], D,
                             k.beta, gS.x, ps0, ds);
      }
      const float4 vde = add4(de1, de), vds = add4(ds1, ds);  // rows s-7, s-6; s-8, s-7
      R.VDE[sl.template m2<6>()][u] = vde;
      R.VDS[sl.template m2<7>()][u] = vds;
      sbE = fma4(k.w, vds, de1);
      sbS = fma4(k.w, vde, ds);
      de1 = de; ds1 = ds;
      pe2 = pe1; pe1 = pe0; ps1 = ps0;
    }
  }
};

template <int BMODE, int NT1>
__global__ void __launch_bounds__(2 * NT1, NT1 == NT_NARROW ? 3 : 2)
    k_bwd_plus(const __grid_constant__ BwdArgs a, const __grid_constant__ MethodConsts k,
               int rows) {
  extern __shared__ __align__(16) unsigned char smem[];
  RingsPlus<NT1>& R = *reinterpret_cast<RingsPlus<NT1>*>(smem);
  {
    float* z = reinterpret_cast<float*>(smem);
    for (int i = threadIdx.x; i < (int)(sizeof(RingsPlus<NT1>) / sizeof(float)); i += 2 * NT1)
      z[i] = 0.f;
  }
  __syncthreads();  // the rings are zero before the first copies land in them
  constexpr int TW1 = NT1 - HL1 - HR1;
  const int n = (int)a.n, m = (int)a.m, orows = (int)a.orows;
  const int b0 = -BWD_GHOST + (int)blockIdx.x * TW1, b1 = min(b0 + TW1, m + BWD_GHOST);
  const int a0 = -BWD_GHOST + (int)blockIdx.y * rows, a1 = min(a0 + rows, n + BWD_GHOST);
  const int s_begin = a0 - 6, s_end = a1 - 1 + 10;
  // FULL steps: every stage live and every output row written (s in
  // [a0 + 10, a1 + 7]), and the output-gradient rows a step requests inside
  // the output (2 (s - 4) + 1 >= 0, 2 (s - 3) < orows)
  const int s_lo = max(a0 + 10, 4);
  const int s_hi = min(a1 + 7, (orows - 1) / 2 + 3);
  const bool forward = threadIdx.x < NT1;  // whole warps
  const int t = (int)threadIdx.x - (forward ? 0 : NT1);
  const int c = b0 - HL1 + t;
  if (forward) {
    PlusForward<BMODE, NT1> sw(R, a, k, t, c, a0, a1);
    float* ringA = &R.A[0][sw.u];
#pragma unroll 1
    for (int s = s_begin - (AHEAD + 1); s < s_begin; ++s)
      sw.template request<false>(s, RowsRT<RingsPlus<NT1>::W>{ringA, s});
    sweep_band(sw, ringA, s_begin, s_end, s_lo, s_hi);
    copy_wait<0>();  // no copy lands in shared memory after the CTA
  } else {
    PlusBackward<BMODE, NT1> sw(R, a, k, t, c, b0, b1, a0, a1);
    sweep_band(sw, &R.A[0][sw.u], s_begin, s_end, s_lo, s_hi);
  }
}

// ---- k_bwd_cross ---------------------------------------------------------------
// Lags: input row 0, x indicators 3, x adjoints 4, x coefficients 5; A_bar
// of row s - 7 is complete at step s and written (column-folded) at s + 1.
template <int BMODE, int NT2>
struct CrossSweep {
  static constexpr int W = RingsCross<NT2>::W;
  RingsCross<NT2>& R;
  const MethodConsts k;
  float w, k1;
  int u, n, a0, a1;
  const float* xin;  // input row s + 2 (clamped) of the column, in step s
  int64_t x_sh;
  bool cg;  // column on the workspace grid
  const float* wxb;      // X_bar row s - 1 of the column, in step s
  int64_t ws_ld, ws_ab;  // workspace row stride; from X_bar row r to A_bar row r - 3
  // the thread writes grad_in column c; columns 0 and m-1 also sum the ghost
  // columns folded onto them
  bool emit_col, fold_left, fold_right;
  float* gin;  // grad_in column c, row 0
  int64_t gi_sh;
  // carried from step to step
  float4 six1, six2;        // indicators of rows s-4, s-5
  Sten q1;                  // x stencils of row s-4
  float4 q2s;               // second and first differences of row s-5
  float2 q2g;
  float4 px1, dx1, dx2;     // p_bar of row s-5, 2 D_bar of rows s-5, s-6
  float acc[4];             // A_bar rows s-7 .. s-4 of this column
  float rowsum;             // ghost rows folded onto an edge row
  int emitted;              // grad_in row published in the previous step (-1: none)

  __device__ __forceinline__ CrossSweep(RingsCross<NT2>& R_, const BwdArgs& a,
                                        const MethodConsts& k_, int rows)
      : R(R_), k(k_) {
    constexpr int TW2 = NT2 - HL2 - HR2;
    const int t = threadIdx.x;
    const int64_t plane = blockIdx.z;
    n = (int)a.n;
    const int m = (int)a.m;
    const int nby = (int)gridDim.y;
    const int b0 = (int)blockIdx.x * TW2;
    const int b1 = min(b0 + TW2, m);
    const int c = b0 - HL2 + t;
    // A_bar rows of this band: image rows [r0, r1) plus the ghost rows that
    // fold onto row 0 (first band) and row n-1 (last band)
    const int r0 = (int)blockIdx.y * rows, r1 = min(r0 + rows, n);
    a0 = blockIdx.y == 0 ? -GA : r0;
    a1 = (int)blockIdx.y == nby - 1 ? n + GA : r1;
    x_sh = a.x_sh;
    // the first request is that of step a0 - 5 - (AHEAD + 1)
    xin = a.x + plane * a.x_sc + (int64_t)clampi(c, 0, m - 1) * a.x_sw +
          (int64_t)clampi(a0 - 5 - (AHEAD + 1) + 2, 0, n - 1) * x_sh;
    cg = c >= -BWD_GHOST && c < m + BWD_GHOST;
    ws_ld = a.ws_ld;
    const int64_t cells = a.ws_cells;
    ws_ab = cells - 3 * ws_ld;
    const int s0 = a0 - 5;  // first step (requests start AHEAD + 1 steps before it)
    wxb = a.ws + plane * 2 * cells + (int64_t)(s0 - (AHEAD + 1) - 1 + BWD_GHOST) * ws_ld + (c + BWD_GHOST);
    emit_col = c >= b0 && c < b1;
    fold_left = c == 0;
    fold_right = c == m - 1;
    gin = a.gin + plane * a.gi_sc + (int64_t)(emit_col ? c : 0) * a.gi_sw;
    gi_sh = a.gi_sh;
    w = k.w;
    k1 = k.kappa1 * k.kappa1;
    u = t + PAD;
  }

  // FULL steps request workspace rows known to lie on the workspace grid;
  // columns off the grid stay zero from the rings' start.
  template <bool FULL>
  __device__ __forceinline__ void request_ws(float* dst, const float* p, int r) const {
    if (!FULL && (r < -BWD_GHOST || r >= n + BWD_GHOST))
      *dst = 0.f;
    else if (cg)
      copy_async<4>(dst, p);
  }

  // Step s's requests: input row s + 2 (to the ring; first read in step
  // s + 3) and the workspace values that step s + 3 uses.
  template <bool FULL, class SL>
  __device__ __forceinline__ void request(const int s, const SL& sl) {
    copy_async<4>(sl.template a<-2>(), xin);
    if (s + 2 >= 0 && s + 2 < n - 1) xin += x_sh;
    request_ws<FULL>(&R.XB[sl.template m4<1>()][u], wxb, s - 1);
    request_ws<FULL>(&R.AB[sl.template m4<4>()][u], wxb + ws_ab, s - 4);
    copy_commit();
    wxb += ws_ld;
  }

  template <bool FULL, class SL>
  __device__ __forceinline__ void step(const int s, const SL& sl) {
    copy_wait<AHEAD>();
    __syncthreads();
    request<FULL>(s, sl);
    const float xb_s = R.XB[sl.template m4<4>()][u], ab_s = R.AB[sl.template m4<7>()][u];

    // ---- grad_in row published in the previous step: fold the ghost columns ----
    if ((FULL || emitted >= 0) && emit_col) {
      const float* af = R.AF[sl.template m2<1>()] + u;
      float v = af[0];
      if (fold_left) v += (af[-5] + af[-4]) + (af[-3] + af[-2]) + af[-1];
      if (fold_right) v += (af[1] + af[2]) + (af[3] + af[4]) + af[5];
      gin[(int64_t)(FULL ? s - 8 : emitted) * gi_sh] = v;
    }

    // Stages run only on the rows the band's outputs need (uniform guards).
    // ---- contributions of x row s-6 from the neighbouring columns ----
    if (FULL || (s - 6 >= a0 - 2 && s - 6 <= a1)) {
      const int sp = sl.template m2<6>();
      const float2 c1 = R.C1[sp][u - 1];  // from column c-1: rows s-6, s-5
      const float2 c2 = R.C2[sp][u - 2];  // from column c-2: rows s-4, s-7
      const float2 cm = R.CM[sp][u + 1];  // from column c+1: rows s-7, s-4
      acc[0] += c2.y + cm.x;
      acc[1] += c1.x;
      acc[2] += c1.y;
      acc[3] += c2.x + cm.y;
    }
    // ---- A_bar of row q = s-7 is complete ----
    {
      const int q = s - 7;
      const float v = acc[0] + ab_s;
      if (FULL) {
        // an interior row: no ghost rows to fold (rowsum is 0 here)
        R.AF[sl.template m2<0>()][u] = v;
        emitted = q;
      } else {
        emitted = -1;
        if (q >= a0 && q < a1) {
          rowsum += v;
          // rows -GA..0 fold onto row 0, rows n-1..n+GA-1 onto row n-1
          if (q >= 0 && (q < n - 1 || q == n - 1 + GA)) {
            emitted = min(q, n - 1);
            R.AF[sl.template m2<0>()][u] = rowsum;
            rowsum = 0.f;
          }
        }
      }
    }
    // ---- x indicators, row s-3 ----
    float4 six = zero4();
    Sten q;
    q.s = zero4();
    q.g = make_float2(0.f, 0.f);
    q.M0 = q.M1 = 0.f;
    if (FULL || (s - 3 >= a0 - 4 && s - 3 <= a1 + 2)) {
      q = sten_x(sl.template a<4>(), sl.template a<3>(), sl.template a<2>(), sl.template a<1>());
      six = indicators(q.s, q.g, k.kappa1, k.eps1);
      R.SIX[sl.template m2<3>()][u] = six;
    }
    // ---- x adjoints, row s-4 ----
    float4 px = zero4(), dx = px;
    if (FULL || (s - 4 >= a0 - 3 && s - 4 <= a1 + 1)) {
      if (FULL || xb_s != 0.f) {
        const float4 l = R.SIX[sl.template m2<4>()][u - 1], r = R.SIX[sl.template m2<4>()][u + 1];
        const float4 D = fma4(w, add4(add4(six2, six), add4(l, r)), six1);
        point_adjoint<BMODE>(q1.s, 0.5f * (q1.M1 - q1.M0), D, k.beta, xb_s, px, dx);
      }
      R.DX[sl.template m2<4>()][u] = dx;
    }
    // ---- x coefficients, row s-5 ----
    if (FULL || (s - 5 >= a0 - 2 && s - 5 <= a1)) {
      const float4 l = R.DX[sl.template m2<5>()][u - 1], r = R.DX[sl.template m2<5>()][u + 1];
      const float4 sb = fma4(w, add4(add4(dx2, dx), add4(l, r)), dx1);  // 2 SI_bar
      float2 c1 = make_float2(0.f, 0.f), c2 = c1, cm = c1;
      if (FULL || any_nonzero(px1, sb)) {
        // (row, column) offsets: the (1,1) line d (-1,-1), a (0,0), b (1,1),
        // c (2,2); the (1,-1) line d (-1,2), a (0,1), b (1,0), c (2,-1)
        const Nodes e = node_coefs(lo2(px1), lo2(q2s), q2g.x, lo2(sb), k1);
        const Nodes f = node_coefs(hi2(px1), hi2(q2s), q2g.y, hi2(sb), k1);
        acc[2] += e.a;  // row s-5
        acc[3] += f.b;  // row s-4
        c1 = make_float2(f.a, e.b);
        c2 = make_float2(e.c, f.d);
        cm = make_float2(e.d, f.c);
      }
      R.C1[sl.template m2<5>()][u] = c1;
      R.C2[sl.template m2<5>()][u] = c2;
      R.CM[sl.template m2<5>()][u] = cm;
    }
    dx2 = dx1;
    dx1 = dx;
    px1 = px;
    six2 = six1;
    six1 = six;
    q2s = q1.s;
    q2g = q1.g;
    q1 = q;
    acc[0] = acc[1]; acc[1] = acc[2]; acc[2] = acc[3]; acc[3] = 0.f;
  }
};

template <int BMODE, int NT2>
__global__ void __launch_bounds__(NT2, NT2 == NT_NARROW ? 4 : 2)
    k_bwd_cross(BwdArgs a, MethodConsts k, int rows) {
  extern __shared__ __align__(16) unsigned char smem[];
  RingsCross<NT2>& R = *reinterpret_cast<RingsCross<NT2>*>(smem);
  {
    float* z = reinterpret_cast<float*>(smem);
    for (int i = threadIdx.x; i < (int)(sizeof(RingsCross<NT2>) / sizeof(float)); i += NT2)
      z[i] = 0.f;
  }
  CrossSweep<BMODE, NT2> sw(R, a, k, rows);
  const int s_begin = sw.a0 - 5, s_end = sw.a1 - 1 + 8;
  __syncthreads();  // the rings are zero before the first copies land in them
#pragma unroll 1
  for (int s = s_begin - (AHEAD + 1); s < s_begin; ++s)
    sw.template request<false>(s, RowsRT<CrossSweep<BMODE, NT2>::W>{&R.A[0][sw.u], s});
  sw.six1 = sw.six2 = sw.q1.s = sw.q2s = sw.px1 = sw.dx1 = sw.dx2 = zero4();
  sw.q1.g = sw.q2g = make_float2(0.f, 0.f);
  sw.q1.M0 = sw.q1.M1 = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) sw.acc[j] = 0.f;
  sw.rowsum = 0.f;
  sw.emitted = -1;
  // FULL steps: every stage live (s in [a0 + 8, a1 + 5]), the previous and
  // the current A_bar rows interior ones (s - 8 >= max(a0, 0),
  // s - 7 < min(a1, n - 1)) and the workspace rows a step requests on the
  // workspace grid (s - 1 < n + 2)
  const int s_lo = max(sw.a0, 0) + 8;
  const int s_hi = min(sw.a1 + 5, sw.n + 2);
  sweep_band(sw, &R.A[0][sw.u], s_begin, s_end, s_lo, s_hi);
  copy_wait<0>();  // no copy lands in shared memory after the CTA
}

// Resident CTAs per SM of a kernel with `smem` bytes of dynamic shared memory,
// which this also allows it: a function of the kernel and the device, asked
// once per pair (the two queries took 6 us of host time a kernel and call).
template <class K>
cudaError_t resident_ctas(K kern, int threads, size_t smem, int dev, std::atomic<int>* known,
                          int* occ) {
  const int i = dev >= 0 && dev < 64 ? dev : -1;
  *occ = i >= 0 ? known[i].load(std::memory_order_acquire) : 0;
  if (*occ > 0) return cudaSuccess;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, threads, smem);
  if (e == cudaSuccess && i >= 0 && *occ > 0) known[i].store(*occ, std::memory_order_release);
  return e;
}

// Time model of a sweep (as wd_fwd_model.h): a band of `rows` rows takes
// rows + fill steps, and a step, with k CTAs on an SM,
// sqrt(lat^2 + (k issue)^2) us.
struct SweepModel {
  float lat, issue[2];  // (narrow, wide)
  float fill;
};
// The step times follow the full-size runs (1.1 and 0.49 us with the CTAs
// resident), the others short bands on an idle GPU; latencies of 0.5 to 0.75
// and 0.3 to 0.5 us and fills 25% off choose shapes within 2% of each other.
// Bands of at least 16 rows, the rule before, left small images on a few CTAs:
// 3x64x64 39.5 -> 23.0 us, 3x256x256 43.3 -> 40.5 (then 20.8 and 35.9 with the
// requests moved).
constexpr SweepModel PLUS_MODEL = {0.50f, {0.31f, 0.46f}, 13.f};
constexpr SweepModel CROSS_MODEL = {0.30f, {0.133f, 0.20f}, 10.f};

struct SweepShape {
  int wide, strips, rows;
  int64_t bands;
};

// The CTA width and band height of least modelled time.
SweepShape pick_shape(const SweepModel& model, const int (&occ)[2], const int (&tw)[2], int sms,
                      int64_t rows_total, int64_t cols_total, int64_t planes) {
  SweepShape best{0, 1, (int)rows_total, 1};
  double best_us = 1e300;
  for (int i = 0; i < 2; ++i) {
    if (occ[i] < 1) continue;
    const int64_t strips = (cols_total + tw[i] - 1) / tw[i], slots = (int64_t)occ[i] * sms;
    auto step = [&](int64_t k) {
      const double q = double(k) * model.issue[i];
      return std::sqrt(double(model.lat) * model.lat + q * q);
    };
    const double full = step(occ[i]);
    int64_t last = -1;
    for (int64_t b = 1; b <= rows_total && b <= 4096; ++b) {
      const int64_t rows = (rows_total + b - 1) / b;
      if (rows == last) continue;
      // bands below 16 rows only where they still find idle CTA slots
      if (b > 1 && (rows < 2 || (rows < 16 && strips * planes * b > slots))) break;
      last = rows;
      const int64_t bands = (rows_total + rows - 1) / rows, ctas = strips * planes * bands;
      const int64_t rest = ctas % slots;
      double us = double(ctas / slots) * full;
      if (rest) us += step((rest + sms - 1) / sms);
      us *= double(rows) + model.fill;
      if (us < best_us - 1e-9) {
        best_us = us;
        best = SweepShape{i, (int)strips, (int)rows, bands};
      }
    }
  }
  return best;
}

template <int BMODE>
cudaError_t launch_all(const BwdArgs& a, const MethodConsts& k, cudaStream_t st) {
  static std::atomic<int> known[4][64], known_sms[64];
  constexpr size_t plus_n = sizeof(RingsPlus<NT_NARROW>), plus_w = sizeof(RingsPlus<NT_WIDE>);
  constexpr size_t cross_n = sizeof(RingsCross<NT_NARROW>), cross_w = sizeof(RingsCross<NT_WIDE>);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int sms = dev >= 0 && dev < 64 ? known_sms[dev].load(std::memory_order_relaxed) : 0;
  if (sms <= 0) {
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
    if (dev >= 0 && dev < 64) known_sms[dev].store(sms, std::memory_order_relaxed);
  }
  int occ1[2], occ2[2];
  if ((e = resident_ctas(k_bwd_plus<BMODE, NT_NARROW>, 2 * NT_NARROW, plus_n, dev, known[0],
                         &occ1[0])) != cudaSuccess ||
      (e = resident_ctas(k_bwd_plus<BMODE, NT_WIDE>, 2 * NT_WIDE, plus_w, dev, known[1],
                         &occ1[1])) != cudaSuccess ||
      (e = resident_ctas(k_bwd_cross<BMODE, NT_NARROW>, NT_NARROW, cross_n, dev, known[2],
                         &occ2[0])) != cudaSuccess ||
      (e = resident_ctas(k_bwd_cross<BMODE, NT_WIDE>, NT_WIDE, cross_w, dev, known[3],
                         &occ2[1])) != cudaSuccess)
    return e;
  if ((occ1[0] < 1 && occ1[1] < 1) || (occ2[0] < 1 && occ2[1] < 1))
    return cudaErrorInvalidConfiguration;
  // k_bwd_plus: the extended grid, rows and columns [-2, n+2) x [-2, m+2)
  const SweepShape s1 =
      pick_shape(PLUS_MODEL, occ1, {NT_NARROW - HL1 - HR1, NT_WIDE - HL1 - HR1}, sms,
                 a.n + 2 * BWD_GHOST, a.m + 2 * BWD_GHOST, a.planes);
  const dim3 g1((unsigned)s1.strips, (unsigned)s1.bands, (unsigned)a.planes);
  if (s1.wide)
    k_bwd_plus<BMODE, NT_WIDE><<<g1, 2 * NT_WIDE, plus_w, st>>>(a, k, s1.rows);
  else
    k_bwd_plus<BMODE, NT_NARROW><<<g1, 2 * NT_NARROW, plus_n, st>>>(a, k, s1.rows);
  // k_bwd_cross: image rows and columns, ghosts folded at the edges
  const SweepShape s2 = pick_shape(CROSS_MODEL, occ2, {NT_NARROW - HL2 - HR2, NT_WIDE - HL2 - HR2},
                                   sms, a.n, a.m, a.planes);
  const dim3 g2((unsigned)s2.strips, (unsigned)s2.bands, (unsigned)a.planes);
  if (s2.wide)
    k_bwd_cross<BMODE, NT_WIDE><<<g2, NT_WIDE, cross_w, st>>>(a, k, s2.rows);
  else
    k_bwd_cross<BMODE, NT_NARROW><<<g2, NT_NARROW, cross_n, st>>>(a, k, s2.rows);
  return cudaGetLastError();
}

}  // namespace

size_t bwd_workspace_bytes(int64_t n, int64_t m, int64_t planes) {
  // X_bar and the partial A_bar on the grid extended by BWD_GHOST cells
  return sizeof(float) * 2 * (size_t)(n + 2 * BWD_GHOST) * (size_t)(m + 2 * BWD_GHOST) *
         (size_t)planes;
}

cudaError_t launch_zoom2x_bwd(const BwdArgs& args, const MethodConsts& k, int bmode,
                              cudaStream_t stream) {
  BwdArgs a = args;
  a.ws_ld = a.m + 2 * BWD_GHOST;
  a.ws_cells = (a.n + 2 * BWD_GHOST) * a.ws_ld;
  switch (bmode) {
    case B2: return launch_all<B2>(a, k, stream);
    case B0: return launch_all<B0>(a, k, stream);
    default: return launch_all<BGEN>(a, k, stream);
  }
}

}  // namespace wdweno
