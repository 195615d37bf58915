// agcm_adjoint.cuh — hand-written adjoint (vector-Jacobian product) of the
// spatial operator T at a state x, in gather form: every element of the
// result is formed by the one thread that owns it, as the sum over the
// tendency terms whose stencil reads it.  No two threads write the same
// element, so there are no atomics and the result does not depend on the
// order in which threads run (bit-identical from run to run).
//
//   k_colstate    (agcm_phases.cuh) phase A at x: m = pi~ + pi, P = sqrt(m) and
//                 its U/V-point values and reciprocals.
//   k_adj_col     one row segment per block, rows staged in shared memory, a
//                 walk down and one up the levels: phase B at x (the
//                 leap divergence D_k of Eq. 6, its column sum C, the sigma
//                 mass flux W_h = sh_h C - sum_{k<h} ds_k D_k of Alg. 1 /
//                 Alg. 2, the Omega~ factor S_k and the hydrostatic psi)
//                 together with its transpose: the adjoints of W and psi
//                 gathered from the tendencies that read them, the
//                 transposed prefix / suffix scans and the adjoint Dbar_k of
//                 D_k.
//   k_adj_rows    one row segment per block, levels in a loop over rows staged
//                 in shared memory: the adjoints of the mass fluxes F = P^u U,
//                 P^v V, of G = U / P^u, V / P^v, Phi / P and of U, V through
//                 the Coriolis pair, each gathered from the tendency points
//                 that read it, then the chain F = P U, G = F / P back to U, V,
//                 Phi and the level sums of the adjoints of the 2-D factors.
//                 k_adj_gather does the same through L1 for the rows whose
//                 strides reach past a row segment's halo.
//   k_adj_colstate  m^u, m^v are stride-1 means of m: the adjoint of pi.
//
// The transposed stencil.  Every advection term is a face flux Z times the
// value G at the far end of a pair of points (x, x + M):  the tendency at x
// holds + Z G(x + M) and the tendency at x + M holds - Z G(x), both with the
// same face flux (Z at x + M/2; the skew form of the advection).  With
// hb(x) = dT(x) / d(hor)(x) * ybar(x) the adjoint of the face flux is
// hb(x) G(x + M) - hb(x + M) G(x), and the adjoint of G(x) is
// hb(x - M) Z(x - M/2) - hb(x + M) Z(x + M/2): the leap offsets of the
// forward stencil mirrored.  A face flux is a mean of one or two mass fluxes
// F, so F's adjoint sums the adjoints of the faces that average it.  The same
// holds meridionally (pairs of rows j, j + 1) and vertically (levels k, k + 1,
// face flux W).  The Coriolis pair and the pressure gradient are read at
// fixed neighbours and transposed the same way.
//
// Output: out = (accumulate ? out : 0) + scale * J(x)^T ybar, and optionally
// sum += scale * J(x)^T ybar in the same pass (the stage accumulation).
#pragma once
#include "agcm_common.cuh"
#include "agcm_phases.cuh"
#include "agcm_row.cuh"

namespace agcm {

// Outputs of k_adj_col (the inputs of the gather kernels).
template <class T>
struct AdjCol {
  T* W;      // (K+1)*J*I: the sigma mass flux at the half levels h = 1..K-1
  T* psi;    // K*J*I: hydrostatic psi
  T* Db;     // K*J*I: adjoint of the divergence D_k
  T* aPhi;   // K*J*I: adjoint of Phi through psi and the Omega~ term
  T* arP;    // J*I: adjoint of 1/P through the Omega~ term
  T* aPiD;   // J*I: adjoint of pi through the surface term of psi
};

// Phase B and its transpose.  Forward (per column):
//   D_k  = (F^u[i+(M-1)/2] - F^u[i-(M+1)/2]) rdx + (sv_j F^v_j - sv_{j-1} F^v_{j-1}) rdy
//   C    = sum_k ds_k D_k;  dpi/dt = -C
//   W_h  = sh_h C - sum_{k<h} ds_k D_k  =  sum_{k>=h} ds_k D_k - (1 - sh_h) C
//   G_k  = Phi_k / P;  c_k = 1 (+ rho_k G_k with the delta kappa Phi/P term)
//   B_k  = G_k c_k;  psi_k = Hkk_k B_k + sum_{k'>k} hk_k' B_k' + R T~_s pi / pi~
//   S_k  = Hkk_k D_k + hk_k / ds_k sum_{k'<k} ds_k' D_k';  Omega~ tendency -c_k S_k / P
//   (H carries the level coefficient beta of its source level)
// Transposed: the adjoint of psi_k (gathered from the pressure-gradient terms
// of the U and V points that read it) runs a prefix scan to the adjoint of
// B_k, hence of Phi_k and 1/P; the adjoint of W_h (gathered from the
// vertical advection of the levels h-1, h at the points whose face means hold
// W(j, i)) and of -C give Cbar and the suffix sums that form Dbar_k.
//
// The sums run in the state's precision: FP64 issues at 1/64 of the FP32 rate
// on this GPU, and per level and column they would be the bulk of the pass.
//   k_adj_col    a row segment per block, rows staged in shared memory, one
//                walk down and one up the levels, each level's D (and adjoint
//                of W) kept in shared memory between them;
//   k_adj_col_w  so many levels that shared memory holds few such blocks or
//                none: 32 columns and kColG groups of levels per block, stencil
//                read through L1.
constexpr int kColG = 2;

// Level tables: ds, Hkk, hk, hk_rds, r2ds, 1 - sh, rho.
enum { kLds, kLHkk, kLhk, kLhkr, kLr2ds, kLoms, kLrho, kLN = 8 };
template <class T>
__device__ __forceinline__ void col_tables(const Geom<T>& g, T* lt, int tid, int nthreads) {
  for (int k = tid; k < g.K; k += nthreads) {
    T* L = lt + kLN * k;
    L[kLds] = g.ds[k];
    L[kLHkk] = g.Hkk[k];
    L[kLhk] = g.hk[k];
    L[kLhkr] = g.hk_rds[k];
    L[kLr2ds] = g.r2ds[k];
    L[kLoms] = g.oms[k];
    L[kLrho] = g.nl ? g.rho[k] : T(0);
    L[7] = T(0);
  }
}
// The per-column pieces of k_adj_col_w.
template <class T>
struct ColCtx {
  const Geom<T>& g;
  const T *U, *V, *Phi, *yU, *yV, *yPhi;
  // element offsets fit 32 bits: nlon * nlat * nlev <= 4e9
  unsigned plane, vplane, r2;
  int ic, ue, uw, im;
  bool hasS, hasN, nl;
  T rdx, rdy, rady, svS, svN, Pue, Puw, rPc, rPui, rPum, PvS, PvN, rPvS, rPvN;

  __device__ T tab(int k, int f) const {
    const T* p = f == kLds ? g.ds : f == kLHkk ? g.Hkk : f == kLhk ? g.hk : f == kLhkr ? g.hk_rds
               : f == kLr2ds ? g.r2ds : f == kLoms ? g.oms : g.rho;
    return ldg(p + k);
  }
  __device__ ColCtx(const Geom<T>& g_, const T* U_, const T* V_, const T* Phi_,
                    const ColState<T>& cs, const T* yU_, const T* yV_, const T* yPhi_, int i, int j)
      : g(g_), U(U_), V(V_), Phi(Phi_), yU(yU_), yV(yV_), yPhi(yPhi_) {
    const int I = g.I, J = g.J;
    plane = (unsigned)J * (unsigned)I;
    vplane = (unsigned)(J - 1) * (unsigned)I;
    r2 = (unsigned)j * (unsigned)I;
    ic = i;
    hasS = j < J - 1;
    hasN = j > 0;
    nl = g.nl != 0;
    const int M = ldg(g.Mu + j);
    ue = wrapi(ic + (M - 1) / 2, I);
    uw = wrapi(ic - (M + 1) / 2, I);
    im = wrapi(ic - 1, I);
    rdx = ldg(g.rdx + j);
    rdy = ldg(g.rdy + j);
    rady = g.rady;
    svS = hasS ? ldg(g.sv + j) : T(0);
    svN = hasN ? ldg(g.sv + j - 1) : T(0);
    const unsigned n = r2 + ic;
    Pue = ldg(cs.Pu + r2 + ue);
    Puw = ldg(cs.Pu + r2 + uw);
    rPc = ldg(cs.rP + n);
    rPui = ldg(cs.rPu + n);
    rPum = ldg(cs.rPu + r2 + im);
    PvS = hasS ? ldg(cs.Pv + n) : T(0);
    PvN = hasN ? ldg(cs.Pv + n - I) : T(0);
    rPvS = hasS ? ldg(cs.rPv + n) : T(0);
    rPvN = hasN ? ldg(cs.rPv + n - I) : T(0);
  }
  // the values of one level: D, the adjoint of psi, Phi, ybar_Phi and the
  // products y / P, x / P of the five points whose vertical advection holds
  // W(j, i): Phi (j, i), U (j, i-1), U (j, i), V (j-1, i), V (j, i)
  struct Lev {
    T D, pb, ph, yx, q[5], x[5];
  };
  __device__ void level(int k, Lev& v) const {
    const int I = g.I;
    const unsigned o3 = (unsigned)k * plane + r2, ov = (unsigned)k * vplane + r2;
    const T* u = U + o3;
    const T* yu = yU + o3;
    const T* vv = V + ov;
    const T* yvv = yV + ov;
    const T VS = hasS ? ldg(vv + ic) : T(0), VN = hasN ? ldg(vv - I + ic) : T(0);
    const T yVS = hasS ? ldg(yvv + ic) : T(0), yVN = hasN ? ldg(yvv - I + ic) : T(0);
    v.D = (Pue * ldg(u + ue) - Puw * ldg(u + uw)) * rdx + (svS * PvS * VS - svN * PvN * VN) * rdy;
    // the pressure-gradient terms of the U points i - (M+1)/2, i + (M-1)/2
    // and the V points (j-1, i), (j, i) read psi(j, i)
    v.pb = rdx * (ldg(yu + ue) * Pue - ldg(yu + uw) * Puw) + rady * (yVS * PvS - yVN * PvN);
    v.ph = ldg(Phi + o3 + ic);
    v.yx = ldg(yPhi + o3 + ic);
    v.q[0] = v.yx * rPc;
    v.x[0] = v.ph * rPc;
    v.q[1] = ldg(yu + im) * rPum;
    v.x[1] = ldg(u + im) * rPum;
    v.q[2] = ldg(yu + ic) * rPui;
    v.x[2] = ldg(u + ic) * rPui;
    v.q[3] = yVN * rPvN;
    v.x[3] = VN * rPvN;
    v.q[4] = yVS * rPvS;
    v.x[4] = VS * rPvS;
  }
  // adjoint of W_k: vb(k-1) G(k) - vb(k) G(k-1) at the five points,
  // vb = -y r2ds / P (the U and V points hold W(j, i) in a face mean, weight 1/2)
  __device__ T adj_w(int k, const Lev& c, const Lev& p) const {
    const T r = tab(k, kLr2ds), rm = tab(k - 1, kLr2ds);
    const T aw = r * c.q[0] * p.x[0] - rm * p.q[0] * c.x[0];
    T h = 0;
#pragma unroll
    for (int q = 1; q < 5; ++q) h += r * c.q[q] * p.x[q] - rm * p.q[q] * c.x[q];
    return aw + T(0.5) * h;
  }
  __device__ T Bk(int k, T ph) const {
    T B = rPc * ph;
    if (nl) B *= T(1) + tab(k, kLrho) * B;
    return B;
  }
  // Omega~ carries c_k: its D-dependence is that of -c_k S_k / P
  __device__ T xbk(int k, T ph, T yx) const { return nl ? yx * (T(1) + tab(k, kLrho) * rPc * ph) : yx; }
  // the prefix quantities of level k: the adjoint of Phi, and arp += the
  // adjoint of 1/P (Q, pre: the prefix sums before level k)
  __device__ T adj_phi(int k, T D, T pb, T ph, T yx, T Q, T pre, T& arp) const {
    const T Hkk = tab(k, kLHkk);
    const T Sk = Hkk * D + tab(k, kLhkr) * Q;
    const T Bb = Hkk * pb + tab(k, kLhk) * pre;
    if (!nl) {
      arp += Bb * ph - yx * Sk;
      return Bb * rPc;
    }
    const T rho = tab(k, kLrho), G = rPc * ph;
    const T Gb = Bb * (T(1) + T(2) * rho * G) - yx * rPc * rho * Sk;  // dB/dG = 1 + 2 rho G
    arp += Gb * ph - yx * (T(1) + rho * G) * Sk;
    return Gb * rPc;
  }
};

// Group sums of one column: sum ds D, sum pb, sum sh aW, sum aW, sum hk B, sum hk_rds xb.
template <class T>
struct ColSums {
  T Q, pre, C, Cb, psum, Rs, Ss, SXs, SWs;
};
template <class T>
__device__ __forceinline__ ColSums<T> col_exchange(T* red, int G, int gy, int lane, const T s[6]) {
  // red: [6][G][32]
#pragma unroll
  for (int q = 0; q < 6; ++q) red[(q * G + gy) * 32 + lane] = s[q];
  __syncthreads();
  ColSums<T> r{};
  for (int q = 0; q < G; ++q) {
    const T d = red[(0 * G + q) * 32 + lane], p = red[(1 * G + q) * 32 + lane];
    r.C += d;
    r.Cb += red[(2 * G + q) * 32 + lane];
    r.psum += p;
    if (q < gy) {
      r.Q += d;
      r.pre += p;
    } else if (q > gy) {
      r.Rs += d;
      r.SWs += red[(3 * G + q) * 32 + lane];
      r.Ss += red[(4 * G + q) * 32 + lane];
      r.SXs += red[(5 * G + q) * 32 + lane];
    }
  }
  return r;
}

// The suffix quantities of level k: W_k, psi_k, Dbar_k.  q*: this group's
// sums up to level k (qD before it, the others including it), s*: this
// group's totals, r: the other groups' offsets.
template <class T>
__device__ __forceinline__ void col_suffix(const ColCtx<T>& c, const AdjCol<T>& o, int k, unsigned q3, T D, T B,
                                           T xb, T qD, T qB, T qX, T qA, T sD, T sB, T sX, T sA,
                                           const ColSums<T>& r, T ps) {
  const T ds = c.tab(k, kLds), Hkk = c.tab(k, kLHkk);
  if (k > 0) o.W[q3] = r.Rs + (sD - qD) - c.tab(k, kLoms) * r.C;  // sum_{k' >= k} ds D - (1 - sh_k) C
  o.psi[q3] = Hkk * B + (r.Ss + (sB - qB)) + ps;
  const T SW = r.SWs + (sA - qA), SX = r.SXs + (sX - qX);
  o.Db[q3] = ds * (r.Cb - SW) - c.rPc * (Hkk * xb + ds * SX);
}

// One row segment per block, one thread per column.  The rows of U, ybar_U,
// V and ybar_V (V rows j-1, j), Phi and ybar_Phi arrive level by level in a
// ring of shared-memory slots, two 16-byte copies a thread, on the way down;
// that walk forms D, the gathered adjoints of psi and W, the prefix sums and
// with them the adjoint of Phi, and keeps D and the adjoint of W (kKeep 1: that
// in Dbar's place); the walk up forms W, psi and Dbar from the suffix sums,
// reading Phi and ybar_Phi once more (from L2).  Rows whose divergence pair lies
// outside the halo (kind 1) read the pair from global memory a level ahead.
// Bound by load latency (16 warps an SM, 106 registers) in FP32 and by the FP64
// pipe in FP64.  Per launch of the reverse pass, before (32 columns and four
// groups of eight levels per block, stencil through L1) and now: 720 x 360 x 30
// FP32 108 -> 82 us (7.8 M points, 40 B a point at the copy rate 46 us), FP64
// 1503 -> 1108; 256 x 128 x 30 FP64 201 -> 193, FP32 20 either way; 128 x 64 x
// 16 FP32 13.5 -> 11.1, FP64 39 -> 48 (one warp a scheduler: its levels are one
// chain of FP64 issue); 128 x 64 x 120 FP32 71 -> 42, FP64 368 -> 313.  Ring of
// two slots 107, three 90 (five blocks 82, but 256 x 128 and 405 x 203 4 to 7 %
// slower); groups of six levels 83.  FP64 keeps the adjoint of W in Dbar's place
// instead of shared memory: 80 KB a block would hold two blocks (1209); so does
// FP32 where three blocks an SM would not hold both.
constexpr int kColRaw = 8;  // U, yU, V j-1, V j, yV j-1, yV j, Phi, yPhi
constexpr int kColPad = 64;  // before the ring: a halo column's pair reaches at most H <= 32 to the west of it
constexpr int kColB = 8;  // levels of a partial sum
template <class T>
struct ColRing {
  static constexpr int R = sizeof(T) == 4 ? 4 : 2;      // slots
  static constexpr int kCtas = sizeof(T) == 4 ? 4 : 3;  // blocks per SM
};
// keep: the arrays kept over the levels in shared memory, D alone or D and the adjoint of W
template <class T>
constexpr size_t adj_col_smem(int K, int keep) {
  return sizeof(T) * (kColPad + (size_t)kRowB * (ColRing<T>::R * kColRaw + keep * K) + (size_t)kLN * K);
}
// Halo of row j's column pass: the divergence pair and the column to the west.
__host__ __device__ inline int adj_col_halo(int M) { return ((M + 1) / 2 + 3) & ~3; }
template <class T>
struct AdjColArgs {
  const T *U, *V, *Phi, *pi;        // x
  const T *yU, *yV, *yPhi, *ypi;    // ybar
  const int4* items;                // kind << 24 | row j, first own column, own columns, halo
  int vec;                          // 1: every row is 16-byte aligned
};
template <class T, int kKeep>
__global__ void __launch_bounds__(kRowB, ColRing<T>::kCtas)
    k_adj_col(const __grid_constant__ Geom<T> g, const __grid_constant__ ColState<T> cs,
              const __grid_constant__ AdjColArgs<T> a, const __grid_constant__ AdjCol<T> o) {
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_launch();
  constexpr int R = ColRing<T>::R, NTP = kRowB;
  const int I = g.I, J = g.J, K = g.K;
  const int4 item = a.items[blockIdx.x];
  const bool wide = item.x >> 24;
  const int j = item.x & 0xffffff, c0 = item.y, own = item.z, H = item.w;
  const bool hasS = j < J - 1, hasN = j > 0, nl = g.nl != 0;
  const int M = g.Mu[j];
  const int NT = own + 2 * H, NTW = (NT + 31) & ~31;
  const int t = threadIdx.x;
  if (t >= NTW) leave();
  const bool owner = t >= H && t < H + own;
  int cstart = c0 - H;
  while (cstart < 0) cstart += I;
  int c = cstart + t;
  while (c >= I) c -= I;
  T* const ring = reinterpret_cast<T*>(smem) + kColPad;
  T* const kept = ring + (size_t)R * kColRaw * NTP + t;          // D, the adjoint of W of every level
  T* const lt = ring + (size_t)(R * kColRaw + kKeep * K) * NTP;  // level tables
  col_tables(g, lt, t, NTW);
  // element offsets fit 32 bits: nlon * nlat * nlev <= 4e9
  const unsigned plane = (unsigned)J * (unsigned)I, vplane = (unsigned)(J - 1) * (unsigned)I;
  const unsigned r2 = (unsigned)j * (unsigned)I;
  // a quarter of the threads each: four columns of two rows, as the stage
  // kernel stages them (next to each other, or tr apart where rows are not aligned)
  const int tr = NTW >> 2, cr = t / tr, cc = (a.vec ? 4 : 1) * (t - cr * tr);
  int c4 = cstart + cc;
  while (c4 >= I) c4 -= I;
  const unsigned turns = a.vec ? 0u : row_turns(c4, tr, I);
  const bool vr = cr == 1 || cr == 2;  // V, yV; quarters 0 and 3: U, yU and Phi, yPhi
  const bool in = cc < NT, ok0 = in && (!vr || hasN), ok1 = in && (!vr || hasS);
  const T* const f0 = cr == 0 ? a.U : (cr == 1 ? a.V : (cr == 2 ? a.yV : a.Phi));
  const T* const f1 = cr == 0 ? a.yU : (cr == 1 ? a.V : (cr == 2 ? a.yV : a.yPhi));
  const unsigned so = r2 + (unsigned)c4;
  const unsigned o0 = vr ? (ok0 ? so - I : 0u) : so, o1 = vr ? (ok1 ? so : 0u) : so;
  const unsigned ring_s = smem_addr(ring) + (unsigned)((2 * cr * NTP + cc) * (int)sizeof(T));
  auto issue_level = [&](int k, int s) __attribute__((always_inline)) {
    const unsigned p = (unsigned)k * (vr ? vplane : plane), d = ring_s + (unsigned)(s * kColRaw * NTP * (int)sizeof(T));
    if (a.vec) {
#pragma unroll
      for (int e = 0; e < 4; e += 16 / (int)sizeof(T)) {
        copy16_g2s(d + e * sizeof(T), f0 + (p + o0 + e), true, ok0);
        copy16_g2s(d + (NTP + e) * sizeof(T), f1 + (p + o1 + e), true, ok1);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned x = e * tr - (turns >> 8 * e & 255u) * I, de = d + (unsigned)(e * tr * (int)sizeof(T));
        copy_elem_g2s<sizeof(T)>(de, f0 + (p + (ok0 ? o0 + x : 0u)), true, ok0);
        copy_elem_g2s<sizeof(T)>(de + NTP * sizeof(T), f1 + (p + (ok1 ? o1 + x : 0u)), true, ok1);
      }
    }
  };
  pdl_wait();  // the launches before this one have written the P family and ybar
  for (int s = 0; s < R; ++s) {
    if (s < K) issue_level(s, s);
    copy_commit();
  }
  // ---- the factors of the column
  const int de = (M - 1) / 2, dw = -(M + 1) / 2;
  const unsigned n = r2 + (unsigned)c;
  int ue = c + de, uw = c + dw;
  ue = ue >= I ? ue - I : ue;
  uw = uw < 0 ? uw + I : uw;
  const T rdx = g.rdx[j], rdy = g.rdy[j], rady = g.rady;
  const T svS = hasS ? ldg(g.sv + j) : T(0), svN = hasN ? ldg(g.sv + j - 1) : T(0);
  const T PuE = cs.Pu[r2 + ue], PuW = cs.Pu[r2 + uw];
  const T PvS = hasS ? cs.Pv[n] : T(0), PvN = hasN ? cs.Pv[n - I] : T(0);
  const T bS = svS * PvS, bN = svN * PvN;
  const T rPc = cs.rP[n], rPu = cs.rPu[n], rPm = cs.rPu[r2 + (c > 0 ? c - 1 : I - 1)];
  const T rPvS = hasS ? cs.rPv[n] : T(0), rPvN = hasN ? cs.rPv[n - I] : T(0);
  const T ps = ldg(g.rt0pit + n) * a.pi[n], rt = ldg(g.rt0pit + n), yp = a.ypi[n];
  T wu[4] = {0, 0, 0, 0};  // wide rows: U, yU at the pair, a level ahead
  if (wide) {
    wu[0] = a.U[r2 + ue];
    wu[1] = a.U[r2 + uw];
    wu[2] = a.yU[r2 + ue];
    wu[3] = a.yU[r2 + uw];
  }
  // ---- down: D, the adjoints of psi and W, prefix sums
  // sums over the levels in groups of kColB, each in two parts (whole groups,
  // the group so far): one chain of K roundings would be less exact
  T Q0 = 0, Q1 = 0, pre0 = 0, pre1 = 0, Cb0 = 0, Cb1 = 0, arp0 = 0, arp = 0;
  T r0 = 0;  // 1 / (2 dsigma) of the level above
  T pq[5] = {0, 0, 0, 0, 0}, px[5] = {0, 0, 0, 0, 0};  // y / P, x / P of the level above
  copy_wait<R - 1>();
  row_sync(NTW);
  int slot = 0;
  for (int k = 0; k < K; ++k) {
    const T* const raw = ring + (size_t)slot * (kColRaw * NTP) + t;
    const T* const L = lt + kLN * k;
    T Ue, Uw, ye, yw;
    if (wide) {
      Ue = wu[0];
      Uw = wu[1];
      ye = wu[2];
      yw = wu[3];
      if (k + 1 < K) {
        const unsigned q = (unsigned)(k + 1) * plane + r2;
        wu[0] = a.U[q + ue];
        wu[1] = a.U[q + uw];
        wu[2] = a.yU[q + ue];
        wu[3] = a.yU[q + uw];
      }
    } else {
      Ue = raw[de];
      Uw = raw[dw];
      ye = raw[NTP + de];
      yw = raw[NTP + dw];
    }
    const T VN = raw[2 * NTP], VS = raw[3 * NTP], yVN = raw[4 * NTP], yVS = raw[5 * NTP];
    const T ph = raw[6 * NTP], yx = raw[7 * NTP];
    // metric factors outside: folded into P they would put one rounding of
    // each into the sum over all levels
    const T D = rdx * (PuE * Ue - PuW * Uw) + rdy * (bS * VS - bN * VN);
    const T pb = rdx * (PuE * ye - PuW * yw) + rady * (PvS * yVS - PvN * yVN);
    // the points whose vertical advection holds W(j, i): Phi (j, i), and in a
    // face mean (weight 1/2, in q) U (j, i-1), U (j, i), V (j-1, i), V (j, i)
    const T q[5] = {yx * rPc, raw[NTP - 1] * (T(0.5) * rPm), raw[NTP] * (T(0.5) * rPu), yVN * (T(0.5) * rPvN),
                    yVS * (T(0.5) * rPvS)};
    const T x[5] = {ph * rPc, raw[-1] * rPm, raw[0] * rPu, VN * rPvN, VS * rPvS};
    T u = 0, d = 0;
#pragma unroll
    for (int e = 0; e < 5; ++e) {
      u += q[e] * px[e];
      d += pq[e] * x[e];
      pq[e] = q[e];
      px[e] = x[e];
    }
    const T r1 = L[kLr2ds], aw = r1 * u - r0 * d;  // the adjoint of W_k (0 at k = 0)
    r0 = r1;
    kept[(size_t)k * NTP] = D;
    if (kKeep > 1)
      kept[(size_t)(K + k) * NTP] = aw;
    else if (owner)
      o.Db[(unsigned)k * plane + n] = aw;  // read back below
    Cb1 += (T(1) - L[kLoms]) * aw;
    const T Q = Q0 + Q1, pre = pre0 + pre1;
    // the prefix quantities: the adjoints of Phi and 1/P
    const T Hkk = L[kLHkk], Sk = Hkk * D + L[kLhkr] * Q, Bb = Hkk * pb + L[kLhk] * pre;
    T ap = Bb;
    if (!nl) {
      arp += Bb * ph - yx * Sk;
    } else {
      const T rho = L[kLrho], G = rPc * ph;
      ap = Bb * (T(1) + T(2) * rho * G) - yx * rPc * rho * Sk;  // dB/dG = 1 + 2 rho G
      arp += ap * ph - yx * (T(1) + rho * G) * Sk;
    }
    if (owner) o.aPhi[(unsigned)k * plane + n] = ap * rPc;
    Q1 += L[kLds] * D;
    pre1 += pb;
    if (k % kColB == kColB - 1) {
      Q0 += Q1;
      pre0 += pre1;
      Cb0 += Cb1;
      arp0 += arp;
      Q1 = pre1 = Cb1 = arp = T(0);
    }
    copy_wait<R - 2>();
    row_sync(NTW);
    if (k + R < K) issue_level(k + R, slot);
    copy_commit();
    slot = slot + 1 == R ? 0 : slot + 1;
  }
  if (!owner) return;
  // ---- up: W, psi, Dbar from the suffix sums
  o.arP[n] = arp0 + arp;
  o.aPiD[n] = (pre0 + pre1) * rt;
  const T C = Q0 + Q1, Cb = (Cb0 + Cb1) - yp;
  T SD0 = 0, S0 = 0, SW0 = 0, SX0 = 0;
  constexpr int B = kColB;  // Phi and ybar_Phi of a group are loaded together
  for (int kt = K - 1; kt >= 0; kt -= B) {
    T ph[B], yx[B], kA[B];
#pragma unroll
    for (int e = 0; e < B; ++e) {
      const unsigned q = (unsigned)max(kt - e, 0) * plane + n;
      ph[e] = a.Phi[q];
      yx[e] = a.yPhi[q];
      if (kKeep == 1) kA[e] = o.Db[q];
    }
    T SD = 0, S = 0, SW = 0, SX = 0;  // of this group
#pragma unroll
    for (int e = 0; e < B; ++e) {
      const int k = kt - e;
      if (k >= 0) {
        const T* const L = lt + kLN * k;
        const unsigned q = (unsigned)k * plane + n;
        const T D = kept[(size_t)k * NTP], aw = kKeep > 1 ? kept[(size_t)(K + k) * NTP] : kA[e];
        const T ds = L[kLds], Hkk = L[kLHkk];
        const T f = nl ? T(1) + L[kLrho] * (rPc * ph[e]) : T(1), Bk = rPc * ph[e] * f, xb = yx[e] * f;
        SD += ds * D;
        if (k > 0) o.W[q] = (SD0 + SD) - L[kLoms] * C;
        o.psi[q] = Hkk * Bk + (S0 + S) + ps;
        o.Db[q] = ds * (Cb - (SW0 + SW)) - rPc * (Hkk * xb + ds * (SX0 + SX));
        S += L[kLhk] * Bk;
        SW += aw;
        SX += L[kLhkr] * xb;
      }
    }
    SD0 += SD;
    S0 += S;
    SW0 += SW;
    SX0 += SX;
  }
}

// Any K: kColG groups of L = ceil(K / kColG) levels; walk 2 re-forms each level.
template <class T>
__global__ void __launch_bounds__(32 * kColG) k_adj_col_w(Geom<T> g, const T* __restrict__ U, const T* __restrict__ V,
                                                          const T* __restrict__ Phi, const T* __restrict__ pi,
                                                          ColState<T> cs, const T* __restrict__ yU,
                                                          const T* __restrict__ yV, const T* __restrict__ yPhi,
                                                          const T* __restrict__ ypi, AdjCol<T> o) {
  __shared__ T red[7 * kColG * 32];
  const int I = g.I, K = g.K;
  const int lane = threadIdx.x, gy = threadIdx.y;
  const int i = blockIdx.x * 32 + lane, j = blockIdx.y;
  const bool col = i < I;
  const ColCtx<T> c(g, U, V, Phi, cs, yU, yV, yPhi, col ? i : 0, j);
  const int L = (K + kColG - 1) / kColG;
  const int kb = min(K, gy * L), ke = min(K, kb + L);
  const unsigned n = c.r2 + c.ic;
  T s[6] = {0, 0, 0, 0, 0, 0};
  typename ColCtx<T>::Lev cv{}, pv{};
  if (kb < ke) {
    if (kb > 0) c.level(kb - 1, pv);
    for (int k = kb; k < ke; ++k) {
      c.level(k, cv);
      const T aw = k > 0 ? c.adj_w(k, cv, pv) : T(0);
      s[0] += ldg(g.ds + k) * cv.D;
      s[1] += cv.pb;
      s[2] += (T(1) - ldg(g.oms + k)) * aw;
      s[3] += aw;
      s[4] += ldg(g.hk + k) * c.Bk(k, cv.ph);
      s[5] += ldg(g.hk_rds + k) * c.xbk(k, cv.ph, cv.yx);
      pv = cv;
    }
  }
  ColSums<T> r = col_exchange(red, kColG, gy, lane, s);
  T arp = 0;
  if (col && kb < ke) {
    r.Cb -= ldg(ypi + n);
    const T ps = ldg(g.rt0pit + n) * ldg(pi + n);
    T qD = 0, qB = 0, qX = 0, qA = 0, Q = r.Q, pre = r.pre;
    if (kb > 0) c.level(kb - 1, pv);
    for (int k = kb; k < ke; ++k) {
      c.level(k, cv);
      const unsigned q3 = (unsigned)k * c.plane + n;
      o.aPhi[q3] = c.adj_phi(k, cv.D, cv.pb, cv.ph, cv.yx, Q, pre, arp);
      Q += ldg(g.ds + k) * cv.D;
      pre += cv.pb;
      const T B = c.Bk(k, cv.ph), xb = c.xbk(k, cv.ph, cv.yx);
      const T qD0 = qD;
      qD += ldg(g.ds + k) * cv.D;
      qB += ldg(g.hk + k) * B;
      qX += ldg(g.hk_rds + k) * xb;
      if (k > 0) qA += c.adj_w(k, cv, pv);
      col_suffix(c, o, k, q3, cv.D, B, xb, qD0, qB, qX, qA, s[0], s[4], s[5], s[3], r, ps);
      pv = cv;
    }
  }
  T* const rarp = red + 6 * kColG * 32;
  rarp[gy * 32 + lane] = arp;
  __syncthreads();
  if (gy == 0 && col) {
    T a = 0;
    for (int q = 0; q < kColG; ++q) a += rarp[q * 32 + lane];
    o.arP[n] = a;
    o.aPiD[n] = r.psum * ldg(g.rt0pit + n);
  }
}

// Output of the adjoint product and the optional stage accumulation.
template <class T>
struct AdjOut {
  T *oU, *oV, *oPhi, *opi;  // out = (accumulate ? out : 0) + scale * J^T ybar
  T *sU, *sV, *sPhi, *spi;  // sum = sum_in + scale * J^T ybar (when sU != nullptr)
  const T *rU, *rV, *rPhi, *rpi;  // sum_in: the sum itself, or another array
  T scale;
  int accumulate;
};

// Adjoints of the 2-D factors, summed over the levels by k_adj_gather.
template <class T>
struct AdjM {
  T *mub, *mvb, *mcb;
};

constexpr int kAdjTileX = 32, kAdjTileY = 4;

// An empty asm that the compiler must assume changes p: loads through the
// result cannot be hoisted out of the loop that calls it.
template <class P>
__device__ __forceinline__ P* opaque(P* p) {
  asm volatile("" : "+l"(p));
  return p;
}

// The gathered adjoint of one column (j, i) at the levels of one chunk of
// lev levels (blockIdx.z): the U point (j, i), the Phi point (j, i)
// and, for j < J-1, the V point (j, i).  Each neighbour value is read through
// L1.  This is the general form for any stride; k_adj_rows below takes the
// rows whose strides are small, and this kernel the nrows rows in `rows`.
// The level sums of the 2-D factors' adjoints are written per chunk to
// part[3][nchunks][nrows][I] and added in chunk order by k_adj_fold.  Chunks of
// one level where the blocks are few: the more the shorter the launch
// (256x128x30: 282 against 297 us a reverse step with 4); up to four levels
// where that leaves four blocks an SM, since the fold reads a value a chunk and
// a block's set-up is that of many levels (strides of 75 in every row, FP32: the
// gather of a reverse step at 720x360x30 2696 -> 2282 us, 256x128x30 327 -> 265).
// Offsets in row j (stride M = Mu_j):  a0 = i - (M-1)/2, b0 = i + (M+1)/2 =
// a0 + M (the pair whose face flux is F^u(i) for a Phi point, one of the two
// for a U point), a1 = i - (M+1)/2, b1 = i + (M-1)/2 = a1 + M (the other U
// pair), iW = i - M, iE = i + M.
template <class T>
__global__ void __launch_bounds__(kAdjTileX* kAdjTileY, 4) k_adj_gather(
    Geom<T> g, const T* __restrict__ U, const T* __restrict__ V, const T* __restrict__ Phi, ColState<T> cs,
    const T* __restrict__ W, const T* __restrict__ psi, const T* __restrict__ Db, const T* __restrict__ aPhi,
    const T* __restrict__ arPcol, const T* __restrict__ yU, const T* __restrict__ yV, const T* __restrict__ yPhi,
    const int* __restrict__ rows, int nrows, int lev, T* __restrict__ part, AdjOut<T> o) {
  const int I = g.I, J = g.J, K = g.K;
  const int i = blockIdx.x * kAdjTileX + (int)(threadIdx.x % kAdjTileX);
  const int jq = blockIdx.y * kAdjTileY + (int)(threadIdx.x / kAdjTileX);
  if (i >= I || jq >= nrows) return;
  const int j = ldg(rows + jq);
  const int kb = blockIdx.z * lev, ke = min(K, kb + lev);
  const size_t plane = (size_t)J * I, vplane = (size_t)(J - 1) * I;
  const bool hasS = j < J - 1, hasN = j > 0, hasSS = j + 1 < J - 1;
  const int M = ldg(g.Mu + j);
  const int a0 = wrapi(i - (M - 1) / 2, I), b0 = wrapi(i + (M + 1) / 2, I);
  const int a1 = wrapi(i - (M + 1) / 2, I), b1 = wrapi(i + (M - 1) / 2, I);
  const int iE = wrapi(i + M, I), iW = wrapi(i - M, I), ip = wrapi(i + 1, I), im = wrapi(i - 1, I);
  const T zf = ldg(g.zf + j), r2A = ldg(g.r2A + j), rdx = ldg(g.rdx + j), f0 = ldg(g.f0 + j),
          cota = ldg(g.cota + j);
  const T r2AN = hasN ? ldg(g.r2A + j - 1) : T(0), r2AS = hasS ? ldg(g.r2A + j + 1) : T(0);
  const T yvS = hasS ? ldg(g.yv + j) : T(0), yvN = hasN ? ldg(g.yv + j - 1) : T(0),
          yvSS = hasSS ? ldg(g.yv + j + 1) : T(0);
  const T cnS = hasS ? ldg(g.cn + j) : T(0), csN = hasN ? ldg(g.cs + j - 1) : T(0);
  // V row j (stride Mv_j) and V row j-1 (stride Mv_{j-1})
  int cS = i, dS = i, vE = i, vW = i, fEv = i, fWv = i, cN = i, dN = i;
  T zfvS = 0, r2AvS = 0, r2AvSS = 0, r2AvN = 0, zfvN = 0, svS = 0, rdyS = 0, rdyS1 = 0, f0S = 0, cotaS = 0;
  if (hasS) {
    const int Mv = ldg(g.Mv + j);
    cS = wrapi(i - (Mv - 1) / 2, I);
    dS = wrapi(i + (Mv + 1) / 2, I);
    vE = wrapi(i + Mv, I);
    vW = wrapi(i - Mv, I);
    fEv = wrapi(i + (Mv - 1) / 2, I);
    fWv = wrapi(i - (Mv + 1) / 2, I);
    zfvS = ldg(g.zfv + j);
    r2AvS = ldg(g.r2Av + j);
    svS = ldg(g.sv + j);
    rdyS = ldg(g.rdy + j);
    rdyS1 = ldg(g.rdy + j + 1);
    f0S = ldg(g.f0 + j + 1);
    cotaS = ldg(g.cota + j + 1);
    if (hasSS) r2AvSS = ldg(g.r2Av + j + 1);
  }
  if (hasN) {
    const int Mv = ldg(g.Mv + j - 1);
    cN = wrapi(i - (Mv - 1) / 2, I);
    dN = wrapi(i + (Mv + 1) / 2, I);
    zfvN = ldg(g.zfv + j - 1);
    r2AvN = ldg(g.r2Av + j - 1);
  }
  const T rady = g.rady;
  const size_t r2 = (size_t)j * I, r2n = r2 - I, r2s = r2 + I;
  const T rPc = ldg(cs.rP + r2 + i), rPuc = ldg(cs.rPu + r2 + i), Puc = ldg(cs.Pu + r2 + i);
  const T rPvc = hasS ? ldg(cs.rPv + r2 + i) : T(0), Pvc = hasS ? ldg(cs.Pv + r2 + i) : T(0);
  // pointwise factors: hb = -ybar r2A / P (horizontal), G = x / P, F = P x
  auto hbP = [&](size_t r3x, size_t r2x, T r2Ax, int ii) { return -ldg(yPhi + r3x + ii) * r2Ax * ldg(cs.rP + r2x + ii); };
  auto hbU = [&](size_t r3x, size_t r2x, T r2Ax, int ii) { return -ldg(yU + r3x + ii) * r2Ax * ldg(cs.rPu + r2x + ii); };
  auto hbV = [&](size_t rvx, size_t r2x, T r2Ax, int ii) { return -ldg(yV + rvx + ii) * r2Ax * ldg(cs.rPv + r2x + ii); };
  auto Gs = [&](size_t r3x, size_t r2x, int ii) { return ldg(Phi + r3x + ii) * ldg(cs.rP + r2x + ii); };
  auto Gu = [&](size_t r3x, size_t r2x, int ii) { return ldg(U + r3x + ii) * ldg(cs.rPu + r2x + ii); };
  auto Gv = [&](size_t rvx, size_t r2x, int ii) { return ldg(V + rvx + ii) * ldg(cs.rPv + r2x + ii); };
  auto Fl = [&](size_t r3x, size_t r2x, int ii) { return ldg(cs.Pu + r2x + ii) * ldg(U + r3x + ii); };
  auto Ft = [&](size_t rvx, size_t r2x, int ii) { return ldg(cs.Pv + r2x + ii) * ldg(V + rvx + ii); };
  T aPu = 0, arPu = 0, aPv = 0, arPv = 0, arP = blockIdx.z == 0 ? ldg(arPcol + r2 + i) : T(0);
  for (int k = kb; k < ke; ++k) {
    // the 2-D factors are re-read at every level (L1 hits) rather than held
    // in registers across the loop: the pointers are made opaque per level
    cs.rP = opaque(cs.rP);
    cs.rPu = opaque(cs.rPu);
    cs.Pu = opaque(cs.Pu);
    cs.rPv = opaque(cs.rPv);
    cs.Pv = opaque(cs.Pv);
    const size_t r3 = (size_t)k * plane + r2, r3n = r3 - I, r3s = r3 + I;
    const size_t rv = (size_t)k * vplane + r2, rvn = rv - I, rvs = rv + I;
    const T r2ds = ldg(g.r2ds + k);
    const T r2dsU = k > 0 ? ldg(g.r2ds + k - 1) : T(0), r2dsD = k < K - 1 ? ldg(g.r2ds + k + 1) : T(0);
    const T Wt = k > 0 ? ldg(W + r3 + i) : T(0), Wb = k < K - 1 ? ldg(W + r3 + plane + i) : T(0);
    // ---------------- U point (j, i) and the zonal mass flux F^u(j, i)
    const T Fla0 = Fl(r3, r2, a0), Flb0 = Fl(r3, r2, b0), Fla1 = Fl(r3, r2, a1), Flb1 = Fl(r3, r2, b1);
    const T FtS = hasS ? Ft(rv, r2, i) : T(0), FtSp = hasS ? Ft(rv, r2, ip) : T(0);
    const T FtN = hasN ? Ft(rvn, r2n, i) : T(0), FtNp = hasN ? Ft(rvn, r2n, ip) : T(0);
    // adjoint of F^u(j, i): the Phi pair (a0, b0), the U pairs (a0, b0) and
    // (a1, b1), the V pairs of rows j and j-1 whose face means hold it, and
    // the divergence of the scalar points a0 and b0
    T aFl = zf * (hbP(r3, r2, r2A, a0) * Gs(r3, r2, b0) - hbP(r3, r2, r2A, b0) * Gs(r3, r2, a0));
    aFl += T(0.5) * zf *
           ((hbU(r3, r2, r2A, a0) * Gu(r3, r2, b0) - hbU(r3, r2, r2A, b0) * Gu(r3, r2, a0)) +
            (hbU(r3, r2, r2A, a1) * Gu(r3, r2, b1) - hbU(r3, r2, r2A, b1) * Gu(r3, r2, a1)));
    if (hasS) aFl += T(0.5) * zfvS * (hbV(rv, r2, r2AvS, cS) * Gv(rv, r2, dS) - hbV(rv, r2, r2AvS, dS) * Gv(rv, r2, cS));
    if (hasN)
      aFl += T(0.5) * zfvN * (hbV(rvn, r2n, r2AvN, cN) * Gv(rvn, r2n, dN) - hbV(rvn, r2n, r2AvN, dN) * Gv(rvn, r2n, cN));
    aFl += rdx * (ldg(Db + r3 + a0) - ldg(Db + r3 + b0));
    // adjoint of G^u(j, i): zonal pairs (i - M, i), (i, i + M), meridional
    // pairs with rows j-1 and j+1, vertical pairs with levels k-1 and k+1,
    // and the Coriolis terms of the U point itself and of the V points
    // (j, i), (j, i+1), (j-1, i), (j-1, i+1)
    const T ZEu = T(0.5) * zf * (Flb1 + Flb0), ZWu = T(0.5) * zf * (Fla1 + Fla0);
    const T YSu = T(0.5) * yvS * (FtS + FtSp), YNu = T(0.5) * yvN * (FtN + FtNp);
    const T WTu = k > 0 ? T(0.5) * (Wt + ldg(W + r3 + ip)) : T(0);
    const T WBu = k < K - 1 ? T(0.5) * (Wb + ldg(W + r3 + plane + ip)) : T(0);
    const T yUc = ldg(yU + r3 + i), Uc = ldg(U + r3 + i);
    const T yVS0 = hasS ? ldg(yV + rv + i) : T(0), yVS1 = hasS ? ldg(yV + rv + ip) : T(0);
    const T yVN0 = hasN ? ldg(yV + rvn + i) : T(0), yVN1 = hasN ? ldg(yV + rvn + ip) : T(0);
    const T VS0 = hasS ? ldg(V + rv + i) : T(0), VS1 = hasS ? ldg(V + rv + ip) : T(0);
    const T VN0 = hasN ? ldg(V + rvn + i) : T(0), VN1 = hasN ? ldg(V + rvn + ip) : T(0);
    const T Cu = cnS * (yVS0 + yVS1) + csN * (yVN0 + yVN1);
    T aGu = hbU(r3, r2, r2A, iW) * ZWu - hbU(r3, r2, r2A, iE) * ZEu;
    if (hasN) aGu += hbU(r3n, r2n, r2AN, i) * YNu;
    if (hasS) aGu -= hbU(r3s, r2s, r2AS, i) * YSu;
    if (k > 0) aGu -= ldg(yU + r3 - plane + i) * r2dsU * rPuc * WTu;
    if (k < K - 1) aGu += ldg(yU + r3 + plane + i) * r2dsD * rPuc * WBu;
    aGu += (T(-0.25) * yUc * (VN0 + VN1 + VS0 + VS1) + Cu * Uc) * cota;
    const T Guc = Uc * rPuc;
    const T aU = Cu * (f0 + Guc * cota);
    // the U point's own tendency: its factors 1/P^u and P^u
    T horU = ZEu * Gu(r3, r2, iE) - ZWu * Gu(r3, r2, iW);
    if (hasS) horU += YSu * Gu(r3s, r2s, i);
    if (hasN) horU -= YNu * Gu(r3n, r2n, i);
    T verU = 0;
    if (k < K - 1) verU += WBu * ldg(U + r3 + plane + i) * rPuc;
    if (k > 0) verU -= WTu * ldg(U + r3 - plane + i) * rPuc;
    const T tRPu = -yUc * (horU * r2A + verU * r2ds);
    const T tPu = -yUc * (ldg(psi + r3 + b0) - ldg(psi + r3 + a0)) * rdx;
    // F^u = P^u U, G^u = U / P^u
    const T bu = aU + aFl * Puc + aGu * rPuc;
    aPu += aFl * Uc + tPu;
    arPu += aGu * Uc + tRPu;
    {
      const size_t q = r3 + i;
      const T v = o.scale * bu;
      o.oU[q] = (o.accumulate ? o.oU[q] : T(0)) + v;
      if (o.sU) o.sU[q] = o.rU[q] + v;
    }
    // ---------------- Phi point (j, i)
    // adjoint of G^s(j, i): zonal pairs (i - M, i), (i, i + M) with face
    // fluxes F^u(a1), F^u(b1), meridional pairs, vertical pairs
    const T yPc = ldg(yPhi + r3 + i), Phc = ldg(Phi + r3 + i);
    T aGs = zf * (hbP(r3, r2, r2A, iW) * Fla1 - hbP(r3, r2, r2A, iE) * Flb1);
    if (hasN) aGs += hbP(r3n, r2n, r2AN, i) * yvN * FtN;
    if (hasS) aGs -= hbP(r3s, r2s, r2AS, i) * yvS * FtS;
    if (k > 0) aGs -= ldg(yPhi + r3 - plane + i) * r2dsU * rPc * Wt;
    if (k < K - 1) aGs += ldg(yPhi + r3 + plane + i) * r2dsD * rPc * Wb;
    // the Phi point's own tendency: its factor 1/P
    T horP = zf * (Flb1 * Gs(r3, r2, iE) - Fla1 * Gs(r3, r2, iW));
    if (hasS) horP += yvS * FtS * Gs(r3s, r2s, i);
    if (hasN) horP -= yvN * FtN * Gs(r3n, r2n, i);
    T verP = 0;
    if (k < K - 1) verP += Wb * ldg(Phi + r3 + plane + i) * rPc;
    if (k > 0) verP -= Wt * ldg(Phi + r3 - plane + i) * rPc;
    const T tRP = -yPc * (horP * r2A + verP * r2ds);
    const T bp = ldg(aPhi + r3 + i) + aGs * rPc;
    arP += aGs * Phc + tRP;
    {
      const size_t q = r3 + i;
      const T v = o.scale * bp;
      o.oPhi[q] = (o.accumulate ? o.oPhi[q] : T(0)) + v;
      if (o.sU) o.sPhi[q] = o.rPhi[q] + v;
    }
    // ---------------- V point (j, i)
    if (hasS) {
      const T yVc = yVS0, Vc = VS0;
      const T FtSS = hasSS ? Ft(rvs, r2s, i) : T(0);
      // adjoint of F^v(j, i): the Phi pair and the U pairs (i-1, i) of rows
      // (j, j+1), the V pairs (j-1, j) and (j, j+1), the divergence of the
      // scalar points (j, i) and (j+1, i)
      const T hbVc = -yVc * r2AvS * rPvc;
      const T GvS = Gv(rv, r2, i);
      const T aYP = hbP(r3, r2, r2A, i) * Gs(r3s, r2s, i) - hbP(r3s, r2s, r2AS, i) * Gs(r3, r2, i);
      const T aYU = (hbU(r3, r2, r2A, i) * Gu(r3s, r2s, i) - hbU(r3s, r2s, r2AS, i) * Gu(r3, r2, i)) +
                    (hbU(r3, r2, r2A, im) * Gu(r3s, r2s, im) - hbU(r3s, r2s, r2AS, im) * Gu(r3, r2, im));
      T aYV = 0;
      if (hasSS) aYV += hbVc * Gv(rvs, r2s, i) - hbV(rvs, r2s, r2AvSS, i) * GvS;
      if (hasN) aYV += hbV(rvn, r2n, r2AvN, i) * GvS - hbVc * Gv(rvn, r2n, i);
      T aFt = yvS * aYP + T(0.5) * yvS * (aYU + aYV);
      aFt += svS * (rdyS * ldg(Db + r3 + i) - rdyS1 * ldg(Db + r3s + i));
      // adjoint of G^v(j, i): zonal pairs (i - Mv, i), (i, i + Mv) with face
      // fluxes the means of F^u over rows j, j+1; meridional and vertical pairs
      const T ZEv = T(0.5) * zfvS * (Fl(r3, r2, fEv) + Fl(r3s, r2s, fEv));
      const T ZWv = T(0.5) * zfvS * (Fl(r3, r2, fWv) + Fl(r3s, r2s, fWv));
      const T YSv = hasSS ? T(0.5) * (yvS * FtS + yvSS * FtSS) : T(0);
      const T YNv = hasN ? T(0.5) * (yvN * FtN + yvS * FtS) : T(0);
      const T WTv = k > 0 ? T(0.5) * (Wt + ldg(W + r3s + i)) : T(0);
      const T WBv = k < K - 1 ? T(0.5) * (Wb + ldg(W + r3s + plane + i)) : T(0);
      T aGv = hbV(rv, r2, r2AvS, vW) * ZWv - hbV(rv, r2, r2AvS, vE) * ZEv;
      if (hasN) aGv += hbV(rvn, r2n, r2AvN, i) * YNv;
      if (hasSS) aGv -= hbV(rvs, r2s, r2AvSS, i) * YSv;
      if (k > 0) aGv -= ldg(yV + rv - vplane + i) * r2dsU * rPvc * WTv;
      if (k < K - 1) aGv += ldg(yV + rv + vplane + i) * r2dsD * rPvc * WBv;
      // adjoint of V(j, i): the Coriolis terms of the U points (j, i-1),
      // (j, i), (j+1, i-1), (j+1, i)
      const T aV = T(-0.25) * (ldg(yU + r3 + im) * (f0 + Gu(r3, r2, im) * cota) + yUc * (f0 + Guc * cota) +
                               ldg(yU + r3s + im) * (f0S + Gu(r3s, r2s, im) * cotaS) +
                               ldg(yU + r3s + i) * (f0S + Gu(r3s, r2s, i) * cotaS));
      // the V point's own tendency: its factors 1/P^v and P^v
      T horV = ZEv * Gv(rv, r2, vE) - ZWv * Gv(rv, r2, vW);
      if (hasSS) horV += YSv * Gv(rvs, r2s, i);
      if (hasN) horV -= YNv * Gv(rvn, r2n, i);
      T verV = 0;
      if (k < K - 1) verV += WBv * ldg(V + rv + vplane + i) * rPvc;
      if (k > 0) verV -= WTv * ldg(V + rv - vplane + i) * rPvc;
      const T tRPv = -yVc * (horV * r2AvS + verV * r2ds);
      const T tPv = -yVc * (ldg(psi + r3s + i) - ldg(psi + r3 + i)) * rady;
      const T bv = aV + aFt * Pvc + aGv * rPvc;
      aPv += aFt * Vc + tPv;
      arPv += aGv * Vc + tRPv;
      const size_t q = rv + i;
      const T v = o.scale * bv;
      o.oV[q] = (o.accumulate ? o.oV[q] : T(0)) + v;
      if (o.sU) o.sV[q] = o.rV[q] + v;
    }
  }
  // P^u = sqrt(m^u): dP^u/dm^u = 1/(2 P^u), d(1/P^u)/dm^u = -1/(2 P^u^3)
  const size_t cstride = (size_t)gridDim.z * nrows * I;
  const size_t n = ((size_t)blockIdx.z * nrows + jq) * I + i;
  part[n] = aPu * T(0.5) * rPuc - arPu * T(0.5) * rPuc * rPuc * rPuc;
  part[cstride + n] = hasS ? aPv * T(0.5) * rPvc - arPv * T(0.5) * rPvc * rPvc * rPvc : T(0);
  part[2 * cstride + n] = -arP * T(0.5) * rPc * rPc * rPc;
}

// The level-chunk partial sums of k_adj_gather, added in chunk order into
// the adjoints of m^u, m^v, m for its rows.
template <class T>
__global__ void __launch_bounds__(256) k_adj_fold(Geom<T> g, const int* __restrict__ rows, int nrows, int nchunks,
                                                  const T* __restrict__ part, AdjM<T> m) {
  const int I = g.I;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nrows * I) return;
  const int jq = q / I, i = q - jq * I;
  const size_t cstride = (size_t)nchunks * nrows * I;
  T su = 0, sv = 0, sc = 0;
  for (int c = 0; c < nchunks; ++c) {
    const size_t n = ((size_t)c * nrows + jq) * I + i;
    su += part[n];
    sv += part[cstride + n];
    sc += part[2 * cstride + n];
  }
  const size_t n = (size_t)ldg(rows + jq) * I + i;
  m.mub[n] = su;
  m.mvb[n] = sv;
  m.mcb[n] = sc;
}

// ---------------------------------------------------------------------------
// Row-segment form of k_adj_gather.  A CTA of at most kRowB threads takes one
// row j and a segment of own columns with a halo of H columns on each side (H
// no less than the widest offset at which the row's transposed stencil reads:
// max(M_j, Mv_j, (Mv_{j-1} + 1) / 2)), and streams the levels from the top.
// Per level, 28 rows arrive in a ring of shared-memory slots by asynchronous
// copies issued a ring's length ahead, seven a thread: x and ybar (U, Phi, V
// at j-1, j, j+1), psi, Dbar and W at j, j+1, the adjoint of Phi from the
// column pass, and the stage sum (of the level above, which this level
// completes).  Every thread forms the pointwise factors of its column, h =
// -ybar / (2 A P), G = x / P and the face fluxes, and publishes the sixteen
// that its neighbours read; after one barrier the columns gather the
// transposed stencil from there.  The vertical pairs of a level need h and G
// of the level below: its own column's terms are added one iteration later,
// when the level is written.
//
// As in the forward kernel the areas are multiplied out: the face fluxes carry
// their face lengths, h the area (and for the U and V points the half of
// their face means), so a face sum is a plain chain of multiply-adds, about
// 150 operations a point and level where the terms formed one by one took
// 240.  M1: all strides of the row are 1, which makes half of the partner
// reads the own or an already read value.
//
// Bound by shared-memory reads (their pipe is busy half of the cycles) and the
// latency left at 12 warps an SM: 181 us a launch at 720x360x30 FP32 (ncu,
// cold caches), 396 instructions a point, against 250 us and 810 for
// 256-thread CTAs that loaded their rows into registers a level ahead; 200 at
// two ring slots, 215 with four CTAs an SM at 128 registers.  FP64: 3.0 ms.
enum AdjRowArr {
  kpHP, kpGs, kpHU, kpGu, kpFL, kpHV, kpGv, kpFT,  // row j, V row j
  kpFLs, kpHVm, kpGvm, kpFTm,                       // F^u of row j+1, V row j-1
  kpYC, kpVs, kpCU, kpEU,                           // Coriolis combinations; U pairs of rows j, j+1
  kAdjPub
};
constexpr int kAdjRaw = 28;
template <class T, int B>
struct AdjRing {
  static constexpr int R = sizeof(T) == 4 ? 4 : 2;
};

// Halo of row j's adjoint stencil (Mv = 0 without a V row j, Mvm = 0 without
// a V row j-1), a multiple of four columns.
__host__ __device__ inline int adj_row_halo(int M, int Mv, int Mvm) {
  int h = M > Mv ? M : Mv;
  const int hm = (Mvm + 1) / 2;
  if (hm > h) h = hm;
  return (h + 3) & ~3;
}
template <class T, int B = kRowB>
constexpr size_t adj_row_smem(int K) {
  return sizeof(T) * ((size_t)B * (AdjRing<T, B>::R * kAdjRaw + 2 * kAdjPub) + K + 64);
}

template <class T>
struct AdjRowArgs {
  const T *U, *V, *Phi;      // x
  const T *yU, *yV, *yPhi;   // ybar
  const T *W, *psi, *Db, *aPhi, *arPcol;
  const T *rU, *rV, *rPhi;   // the array added to: stage sum or the output itself; null: none
  const int4* items;         // row j, first own column, own columns, halo
  int vec;                   // 1: every row is 16-byte aligned
};

// VEC: as in row_segment.
template <class T, bool M1, int VEC = -1, int NTP = kRowB>
__device__ __forceinline__ void adj_row(const Geom<T>& g, const ColState<T>& cs, const AdjRowArgs<T>& a,
                                        const AdjM<T>& m, const AdjOut<T>& o, const int4 item, unsigned char* smem) {
  constexpr int R = AdjRing<T, NTP>::R;
  const int I = g.I, J = g.J, K = g.K;
  const int j = item.x & 0xffffff, c0 = item.y, own = item.z, H = item.w;
  const bool hasS = M1 || j < J - 1, hasN = M1 || j > 0;
  const int M = M1 ? 1 : g.Mu[j], Mv = M1 ? 1 : (hasS ? g.Mv[j] : 1), Mvm = M1 ? 1 : (hasN ? g.Mv[j - 1] : 1);
  const int NT = own + 2 * H, NTW = (NT + 31) & ~31;
  const int t = threadIdx.x;
  if (t >= NTW) leave();  // whole warps past the segment
  const bool owner = t >= H && t < H + own;
  int cstart = c0 - H;
  while (cstart < 0) cstart += I;
  int c = cstart + t;
  while (c >= I) c -= I;
  T* const ring = reinterpret_cast<T*>(smem);
  T* const pub = ring + (size_t)R * kAdjRaw * NTP;
  T* const s_rds = pub + (size_t)2 * kAdjPub * NTP;  // 1 / dsigma_k
  for (int k = t; k < K; k += NTW) s_rds[k] = T(2) * g.r2ds[k];
  // element offsets fit 32 bits: nlon * nlat * nlev <= 4e9
  const unsigned plane = (unsigned)J * (unsigned)I, vplane = (unsigned)(J - 1) * (unsigned)I;
  const unsigned r2 = (unsigned)j * (unsigned)I;

  // Staged rows of a level: 3 f + r, field f = U, Phi, V, yU, yPhi, yV, row r =
  // j-1, j, j+1; then 18, 19 psi, 20, 21 Dbar, 22, 23 W at j, j+1, 24 the
  // adjoint of Phi, 25..27 the stage sum's U, Phi, V of the level above.  A
  // quarter of the threads each: a thread four columns of seven rows, next to
  // each other, or tr apart where rows are not aligned.  Rows outside the grid
  // are zeros.
  const bool al = VEC < 0 ? a.vec != 0 : VEC != 0;
  const int tr = NTW >> 2, cr = t / tr, cc = (al ? 4 : 1) * (t - cr * tr);
  int c4 = cstart + cc;
  while (c4 >= I) c4 -= I;
  const unsigned turns = own_columns(cc, al ? 1 : tr, H, own) | (al ? 0u : row_turns(c4, tr, I));
  const int jr = cr < 3 ? j + cr - 1 : j;
  const bool in = cc < NT, ok3 = in && jr >= 0 && jr < J, okv = in && jr >= 0 && jr < J - 1;
  const bool oks = in && hasS;
  const unsigned so = (unsigned)(ok3 ? jr : j) * (unsigned)I + (unsigned)c4, ro = r2 + (unsigned)c4;
  const unsigned ring_s = smem_addr(ring);
  auto chunk = [&](auto vec, int row, int s, const T* src, bool ok, bool inplace = false) __attribute__((always_inline)) {
    const unsigned d = ring_s + (unsigned)(((s * kAdjRaw + row) * NTP + cc) * (int)sizeof(T));
    if constexpr (decltype(vec)::value) {
#pragma unroll
      for (int e = 0; e < 4; e += 16 / (int)sizeof(T)) copy16_g2s(d + e * sizeof(T), src + e, true, ok && (!inplace || turns & 128u));
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        copy_elem_g2s<sizeof(T)>(d + (unsigned)(e * tr * (int)sizeof(T)), src + (e * tr - (int)(turns >> 8 * e & 127u) * I),
                                 true, ok && (!inplace || turns >> 8 * e & 128u));
    }
  };
  auto issue_form = [&](auto vec, int k, int s) __attribute__((always_inline)) {
    const unsigned p3 = (unsigned)k * plane, pv = (unsigned)k * vplane;
    if (cr < 3) {
      const unsigned ov = pv + (okv ? so : 0u);
      chunk(vec, cr, s, a.U + (p3 + so), ok3);
      chunk(vec, 3 + cr, s, a.Phi + (p3 + so), ok3);
      chunk(vec, 6 + cr, s, a.V + ov, okv);
      chunk(vec, 9 + cr, s, a.yU + (p3 + so), ok3);
      chunk(vec, 12 + cr, s, a.yPhi + (p3 + so), ok3);
      chunk(vec, 15 + cr, s, a.yV + ov, okv);
      if (a.rU && k > 0) {  // quarter cr: field U, Phi, V
        const T* const r = cr == 0 ? a.rU : (cr == 1 ? a.rPhi : a.rV);
        const unsigned q = cr == 2 ? (hasS ? pv - vplane + ro : 0u) : p3 - plane + ro;
        chunk(vec, 25 + cr, s, r + q, in && (cr < 2 || hasS), true);
      }
    } else {
      const unsigned q = p3 + ro, qs = oks ? q + I : q;
      chunk(vec, 18, s, a.psi + q, in);
      chunk(vec, 19, s, a.psi + qs, oks);
      chunk(vec, 20, s, a.Db + q, in);
      chunk(vec, 21, s, a.Db + qs, oks);
      chunk(vec, 22, s, a.W + q, in && k > 0);  // W_0 = 0 is not stored
      chunk(vec, 23, s, a.W + qs, oks && k > 0);
      chunk(vec, 24, s, a.aPhi + q, in);
    }
  };
  auto issue_level = [&](int k, int s) __attribute__((always_inline)) {
    if (al)
      issue_form(std::true_type{}, k, s);
    else
      issue_form(std::false_type{}, k, s);
  };
  pdl_wait();  // the column pass is done
  for (int s = 0; s < R; ++s) {
    if (s < K) issue_level(s, s);
    copy_commit();
  }

  // ---- the factors of the own column, rows j-1, j, j+1 (index r)
  T rP[3], rPu[3], rPv[3], kP[3], kU[3], kV[3], b[3], aF[2];
  T Pu0 = 0, Pv0 = 0;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int jj = j - 1 + r;
    const bool ok = jj >= 0 && jj < J, kv = jj >= 0 && jj < J - 1;
    const unsigned n = ok ? (unsigned)jj * (unsigned)I + (unsigned)c : r2 + (unsigned)c;
    rP[r] = ok ? cs.rP[n] : T(0);
    rPu[r] = ok ? cs.rPu[n] : T(0);
    kP[r] = ok ? -ldg(g.r2A + jj) * rP[r] : T(0);
    kU[r] = ok ? T(-0.5) * ldg(g.r2A + jj) * rPu[r] : T(0);
    const T Pu = ok && r > 0 ? cs.Pu[n] : T(0);
    if (r == 1) Pu0 = Pu;
    // row j+1's flux carries V row j's face length
    if (r > 0) aF[r - 1] = r == 1 ? ldg(g.zf + j) * Pu : (hasS ? ldg(g.zfv + j) * Pu : T(0));
    rPv[r] = kv ? cs.rPv[n] : T(0);
    kV[r] = kv ? T(-0.5) * ldg(g.r2Av + jj) * rPv[r] : T(0);
    const T Pv = kv ? cs.Pv[n] : T(0);
    if (r == 1) Pv0 = Pv;
    b[r] = kv ? ldg(g.yv + jj) * Pv : T(0);
  }
  // ---- row scalars
  const T zf = g.zf[j], rdx = g.rdx[j], f0 = g.f0[j], cota = g.cota[j], rady = g.rady;
  const T zS = hasS ? g.zfv[j] : T(0), zN = hasN ? g.zfv[j - 1] : T(0), rm = M1 ? T(1) : zS / zf;
  const T f1 = hasS ? g.f0[j + 1] : T(0), cota1 = hasS ? g.cota[j + 1] : T(0);
  const T cn = hasS ? g.cn[j] : T(0), csn = hasN ? g.cs[j - 1] : T(0), yvS = hasS ? g.yv[j] : T(0);
  const T nr2A = -g.r2A[j], nr2Av = hasS ? -g.r2Av[j] : T(0);
  const T s0 = hasS ? g.sv[j] * g.rdy[j] : T(0), s1 = hasS ? g.sv[j] * g.rdy[j + 1] : T(0);
  const T A = T(0.5) / g.r2A[j], Av = hasS ? T(0.5) / g.r2Av[j] : T(0);
  // ---- offsets of the stencil from the own column.  A halo thread's partner
  // may lie outside the segment: such reads land in the neighbouring arrays
  // and feed only results that nobody writes.
  const int oa0 = -(M - 1) / 2, ob0 = (M + 1) / 2, oa1 = -(M + 1) / 2, ob1 = (M - 1) / 2;
  const int ocS = -(Mv - 1) / 2, odS = (Mv + 1) / 2, ofE = (Mv - 1) / 2, ofW = -(Mv + 1) / 2;
  const int ocN = -(Mvm - 1) / 2, odN = (Mvm + 1) / 2;

  // ---- carries: sums over the levels, and of the level above: h / dsigma and
  // G, the adjoints so far, x and -ybar / (2 A) / dsigma (late terms)
  T aPu = 0, arPu = 0, aPv = 0, arPv = 0, arP = owner ? a.arPcol[r2 + c] : T(0);
  T hvU = 0, hvP = 0, hvV = 0, GuP = 0, GsP = 0, GvP = 0;
  T bU = 0, bP = 0, bV = 0, xU = 0, xP = 0, xV = 0, yrU = 0, yrP = 0, yrV = 0;
  const bool rmw = a.rU != nullptr;
  unsigned q3 = r2 + (unsigned)c, qv = q3;  // the own column at the level being written
  auto write = [&](T accU, T accP, T accV) __attribute__((always_inline)) {
    const T vU = o.scale * bU, vP = o.scale * bP, vV = o.scale * bV;
    if (owner) {
      if (o.sU) {
        o.oU[q3] = vU;
        o.oPhi[q3] = vP;
        o.sU[q3] = accU + vU;
        o.sPhi[q3] = accP + vP;
        if (hasS) {
          o.oV[qv] = vV;
          o.sV[qv] = accV + vV;
        }
      } else {
        o.oU[q3] = accU + vU;  // accU = 0 unless accumulating
        o.oPhi[q3] = accP + vP;
        if (hasS) o.oV[qv] = accV + vV;
      }
    }
    q3 += plane;
    qv += vplane;
  };

  copy_wait<R - 1>();
  row_sync(NTW);  // the level table and the first level are staged
  int sl0 = 0;
  auto level = [&](const int k, auto SL) __attribute__((always_inline)) {
    constexpr int sl = decltype(SL)::value;
    const int slot = sl0 + sl;
    const T* const raw = ring + (size_t)slot * (kAdjRaw * NTP) + t;
    T* const P = pub + (size_t)sl * kAdjPub * NTP + t;
    auto X = [&](int row) { return raw[row * NTP]; };
    const T rds = s_rds[k], rA = rds * A, rAv = rds * Av;
    T U[3], Ph[3], V[3], yU[3], yP[3], yV[3], hP[3], hU[3], hV[3], Gs[3], Gu[3], Gv[3], FT[3], FL[2];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      U[r] = X(r);
      Ph[r] = X(3 + r);
      V[r] = X(6 + r);
      yU[r] = X(9 + r);
      yP[r] = X(12 + r);
      yV[r] = X(15 + r);
      hP[r] = yP[r] * kP[r];
      Gs[r] = Ph[r] * rP[r];
      hU[r] = yU[r] * kU[r];
      Gu[r] = U[r] * rPu[r];
      hV[r] = yV[r] * kV[r];
      Gv[r] = V[r] * rPv[r];
      FT[r] = b[r] * V[r];
      if (r > 0) FL[r - 1] = aF[r - 1] * U[r];
    }
    const T fs = f0 + cota * Gu[1];
    const T cU = yU[1] * fs + yU[2] * (f1 + cota1 * Gu[2]);
    const T yC = cn * yV[1] + csn * yV[0], vs = V[0] + V[1];
    const T eU = hU[1] * Gu[2] - hU[2] * Gu[1];
    P[kpHP * NTP] = hP[1];
    P[kpGs * NTP] = Gs[1];
    P[kpHU * NTP] = hU[1];
    P[kpGu * NTP] = Gu[1];
    P[kpFL * NTP] = FL[0];
    P[kpHV * NTP] = hV[1];
    P[kpGv * NTP] = Gv[1];
    P[kpFT * NTP] = FT[1];
    P[kpFLs * NTP] = FL[1];
    P[kpHVm * NTP] = hV[0];
    P[kpGvm * NTP] = Gv[0];
    P[kpFTm * NTP] = FT[0];
    P[kpYC * NTP] = yC;
    P[kpVs * NTP] = vs;
    P[kpCU * NTP] = cU;
    P[kpEU * NTP] = eU;
    // the staged rows read as they are
    const T dpsi = raw[18 * NTP + ob0] - raw[18 * NTP + oa0], dpsv = X(19) - X(18);
    const T dDb = raw[20 * NTP + oa0] - raw[20 * NTP + ob0], dDv = s0 * X(20) - s1 * X(21);
    const T W0 = X(22), WU = W0 + raw[22 * NTP + 1], WV = W0 + X(23), aPh = X(24);
    // ---- the level above: its bottom face is this level's top face
    const T hU0 = hU[1] * rA, hP0 = hP[1] * rA, hV0 = hV[1] * rAv;
    if (k > 0) {
      const T dU = -hU0 * WU, dP = -hP0 * W0, dV = -hV0 * WV;
      bU += dU * rPu[1];
      bP += dP * rP[1];
      bV += dV * rPv[1];
      arPu += dU * xU + yrU * (WU * Gu[1]);
      arP += dP * xP + yrP * (W0 * Gs[1]);
      arPv += dV * xV + yrV * (WV * Gv[1]);
      write(rmw ? X(25) : T(0), rmw ? X(26) : T(0), rmw ? X(27) : T(0));
    }
    // ---- what needs no neighbour column
    const T hyU = T(0.5) * nr2A * yU[1], hyP = nr2A * yP[1], hyV = T(0.5) * nr2Av * yV[1];
    T agU = hvU * WU, agP = hvP * W0, agV = hvV * WV;
    agP += hP[0] * FT[0];
    agP -= hP[2] * FT[1];
    yrU = hyU * rA;
    yrP = hyP * rA;
    yrV = hyV * rAv;
    arPu -= yrU * (WU * GuP);
    arP -= yrP * (W0 * GsP);
    arPv -= yrV * (WV * GvP);
    T horP = FT[1] * Gs[2] - FT[0] * Gs[0];
    T eV = eU + hP[1] * Gs[2];
    eV -= hP[2] * Gs[1];
    eV += hV[1] * (Gv[2] - Gv[0]);
    eV += (hV[0] - hV[2]) * Gv[1];
    const T YSv = FT[1] + FT[2], YNv = FT[0] + FT[1];
    agV += hV[0] * YNv;
    agV -= hV[2] * YSv;
    T horV = YSv * Gv[2] - YNv * Gv[0];
    hvU = hU0;
    hvP = hP0;
    hvV = hV0;
    GuP = Gu[1];
    GsP = Gs[1];
    GvP = Gv[1];
    copy_wait<R - 2>();
    row_sync(NTW);
    // every thread is past its reads of this ring slot: fetch level k + R into it
    if (k + R < K) issue_level(k + R, slot);
    copy_commit();
    auto N = [&](int arr, int off) { return P[arr * NTP + off]; };
    // ---- partners at +-M, +-Mv
    const T hPE = N(kpHP, M), hPW = N(kpHP, -M), GsE = N(kpGs, M), GsW = N(kpGs, -M);
    const T hUE = N(kpHU, M), hUW = N(kpHU, -M), GuE = N(kpGu, M), GuW = N(kpGu, -M);
    const T hVE = N(kpHV, Mv), hVW = N(kpHV, -Mv), GvE = N(kpGv, Mv), GvW = N(kpGv, -Mv);
    const T Fb0 = N(kpFL, ob0), Fa1 = N(kpFL, oa1);
    const T Fa0 = M1 ? FL[0] : N(kpFL, oa0), Fb1 = M1 ? FL[0] : N(kpFL, ob1);
    const T FTp = N(kpFT, 1), FTmp = N(kpFTm, 1);
    // ---------------- U point and F^u
    T e, aFl;
    if (M1) {
      e = hP[1] * GsE;
      e -= hPE * Gs[1];
      e += hU[1] * (GuE - GuW);
      e += (hUW - hUE) * Gu[1];
      e += hV[1] * GvE;
      e -= hVE * Gv[1];
      e += hV[0] * N(kpGvm, 1);
      e -= N(kpHVm, 1) * Gv[0];
      aFl = zf * e + rdx * dDb;
    } else {
      e = (N(kpHP, oa0) * N(kpGs, ob0) - N(kpHP, ob0) * N(kpGs, oa0)) +
          (N(kpHU, oa0) * N(kpGu, ob0) - N(kpHU, ob0) * N(kpGu, oa0)) +
          (N(kpHU, oa1) * N(kpGu, ob1) - N(kpHU, ob1) * N(kpGu, oa1));
      aFl = zf * e + zS * (N(kpHV, ocS) * N(kpGv, odS) - N(kpHV, odS) * N(kpGv, ocS)) +
            zN * (N(kpHVm, ocN) * N(kpGvm, odN) - N(kpHVm, odN) * N(kpGvm, ocN)) + rdx * dDb;
    }
    {
      const T ZE = Fb1 + Fb0, ZW = Fa1 + Fa0, YS = FT[1] + FTp, YN = FT[0] + FTmp;
      const T Cu = yC + N(kpYC, 1), v = vs + N(kpVs, 1);
      agU += hUW * ZW;
      agU -= hUE * ZE;
      agU += hU[0] * YN;
      agU -= hU[2] * YS;
      agU += cota * (Cu * U[1] - T(0.25) * yU[1] * v);
      T hor = ZE * GuE;
      hor -= ZW * GuW;
      hor += YS * Gu[2];
      hor -= YN * Gu[0];
      bU = Cu * fs + aFl * Pu0 + agU * rPu[1];
      aPu += aFl * U[1] - yU[1] * (dpsi * rdx);
      arPu += agU * U[1] + hyU * hor;
    }
    // ---------------- Phi point
    agP += hPW * Fa1;
    agP -= hPE * Fb1;
    horP += Fb1 * GsE;
    horP -= Fa1 * GsW;
    bP = aPh + agP * rP[1];
    arP += agP * Ph[1] + hyP * horP;
    // ---------------- V point
    if (hasS) {
      const T ZE = M1 ? FL[0] + FL[1] : rm * N(kpFL, ofE) + N(kpFLs, ofE);
      const T ZW = (M1 ? Fa1 : rm * N(kpFL, ofW)) + N(kpFLs, ofW);
      const T aFt = yvS * (eV + N(kpEU, -1)) + dDv;
      agV += hVW * ZW;
      agV -= hVE * ZE;
      horV += ZE * GvE;
      horV -= ZW * GvW;
      bV = T(-0.25) * (cU + N(kpCU, -1)) + aFt * Pv0 + agV * rPv[1];
      aPv += aFt * V[1] - yV[1] * (dpsv * rady);
      arPv += agV * V[1] + hyV * horV;
    }
    xU = U[1];
    xP = Ph[1];
    xV = V[1];
  };
  int k = 0;
  for (; k + 1 < K; k += 2) {
    level(k, std::integral_constant<int, 0>{});
    level(k + 1, std::integral_constant<int, 1>{});
    if (R == 4) sl0 ^= 2;
  }
  if (k < K) level(k, std::integral_constant<int, 0>{});
  {  // the last level has no level below
    T accU = 0, accP = 0, accV = 0;
    if (rmw && owner) {
      accU = a.rU[q3];
      accP = a.rPhi[q3];
      if (hasS) accV = a.rV[qv];
    }
    write(accU, accP, accV);
  }
  if (owner) {
    const unsigned n = r2 + (unsigned)c;
    m.mub[n] = aPu * T(0.5) * rPu[1] - arPu * T(0.5) * rPu[1] * rPu[1] * rPu[1];
    m.mvb[n] = hasS ? aPv * T(0.5) * rPv[1] - arPv * T(0.5) * rPv[1] * rPv[1] * rPv[1] : T(0);
    m.mcb[n] = -arP * T(0.5) * rP[1] * rP[1] * rP[1];
  }
}

template <class T, int VEC = -1>
__global__ void __launch_bounds__(kRowB, sizeof(T) == 4 ? AGCM_ROW_MINB : AGCM_ROW_MINB64)
    k_adj_rows(const __grid_constant__ Geom<T> g, const __grid_constant__ ColState<T> cs,
               const __grid_constant__ AdjRowArgs<T> a, const __grid_constant__ AdjM<T> m,
               const __grid_constant__ AdjOut<T> o, const int nany) {
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_launch();
  const int4 item = a.items[blockIdx.x];
  if ((int)blockIdx.x >= nany)
    adj_row<T, true, VEC>(g, cs, a, m, o, item, smem);
  else
    adj_row<T, false, VEC>(g, cs, a, m, o, item, smem);
}

// The same in CTAs of 192 threads, two an SM (12 warps, as above): FP32 rows of
// halo 33 to 48, of which a CTA of kRowB threads would own under half, where
// they make one and a half CTAs an SM.  Reverse step's gather with strides of 35
// (45) in every row, 720x360x30: 1008 (1165) us, 2685 in k_adj_gather; in a
// tenth of the rows 659 (681) against 787; with fewer the one wave's latency
// counts (256x128x30, a third of the rows: 230 against 198).  256 threads and
// 128 registers: 1166 (1263), 84 B of spills.
constexpr int kAdjWide = 192;
template <class T>
__global__ void __launch_bounds__(kAdjWide, 2)
    k_adj_rows_wide(const __grid_constant__ Geom<T> g, const __grid_constant__ ColState<T> cs,
                    const __grid_constant__ AdjRowArgs<T> a, const __grid_constant__ AdjM<T> m,
                    const __grid_constant__ AdjOut<T> o) {
  extern __shared__ __align__(128) unsigned char smem[];
  adj_row<T, false, -1, kAdjWide>(g, cs, a, m, o, a.items[blockIdx.x], smem);
}

// pi-bar = direct psi part + m-bar, with m^u_i = (m_i + m_{i+1})/2 and
// m^v_j = (m_j + m_{j+1})/2 transposed as gathers.
template <class T>
__global__ void __launch_bounds__(256) k_adj_colstate(Geom<T> g, AdjM<T> m, const T* aPiD,
                                                      AdjOut<T> o) {
  const int I = g.I, J = g.J;
  pdl_launch();
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= I * J) return;
  pdl_wait();
  const int j = n / I, i = n - j * I;
  T mb = m.mcb[n] + T(0.5) * (m.mub[n] + m.mub[j * I + wrapi(i - 1, I)]);
  if (j < J - 1) mb += T(0.5) * m.mvb[n];
  if (j > 0) mb += T(0.5) * m.mvb[n - I];
  const T v = o.scale * (aPiD[n] + mb);
  o.opi[n] = (o.accumulate ? o.opi[n] : T(0)) + v;
  if (o.spi) o.spi[n] = o.rpi[n] + v;
}

}  // namespace agcm
