// Three-dimensional solver of liblbm.so (lbm3d_*): the D3Q19 lattice with
// the same multiple-relaxation-time collision, Guo forcing and curved slip
// boundary scheme (Eq. EqNewBDSC) per link as the two-dimensional solver --
// the extension the paper names as future work (Sec. 5).
//
// The paper's parameters (Sec. 3.B: tau_s from Kn, per-link l and r, the
// uniform tau_q) come from a two-dimensional analysis.  Carried out for
// D3Q19 (a flow u_x(z) between walls normal to z), that analysis involves
// the x-odd moments j_x, q_x, p_xz and the third-order m_x, and reaches
// exactly the wall relation of Eq. u1u0Coeff when m relaxes with tau_q; so
// m takes tau_q here, and the two-dimensional closed forms hold for the 3-D
// flat channel (tested against the oracle).
//
// Layout: a dense lattice (every node has slots; solid ones are never
// touched), populations stored as deviations d_q = f_q - w_q in FP64 or
// FP32, plane q of N elements (N = nodes rounded up to 32), then a link
// tail.  Pull scheme as in 2-D: step t stores f'_q(x, t) in x's own slot
// q N + x and step t+1 gathers f_q(x, t+1) = f'_q(x - c_q, t) from the slot
// of x - c_q, or, where x - c_q is solid (a boundary link), from the link's
// tail element 19 N + k, which Eq. EqNewBDSC (local to x) filled during
// step t.  Per node: a flag word (bit q: x - c_q solid; kSolid3 for solid
// nodes) and the index of its first link (links sorted by node, then
// direction); the step runs one thread per fluid node from a list of the
// fluid nodes (index, flag word and the node's first link).  The collision
// works in moment space with the D3Q19 basis built here from its defining
// polynomials (d'Humieres et al. 2002): m - m_eq = M (d - d_eq), M Fbar,
// then f' - f = M^T diag(1/|M_k|^2) (m' - m) (the basis is orthogonal), and
// the rest population closes the mass.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <string>
#include <type_traits>
#include <vector>

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm3 {

constexpr int Q = 19;
constexpr uint32_t kSolid3 = 0xFFFFFFFFu;
// an entry of the fluid-node list: the node's index, and its flag word (bits
// 1..18) with the node's first link, counted from its group of 32 entries'
// first, in the bits above
constexpr uint32_t kFlags3 = (1u << 19) - 1u;
constexpr int kRank3 = 19;
constexpr int kThreads3 = 128;
constexpr int kResBlocks3 = 2048;
constexpr int kResThreads3 = 256;

// velocities: rest, the six axes (+x, -x, +y, -y, +z, -z), then the
// diagonals of the xy, xz and yz planes, each (+, +), (+, -), (-, +), (-, -)
#define LBM3_CX {0, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1, 1, 1, -1, -1, 0, 0, 0, 0}
#define LBM3_CY {0, 0, 0, 1, -1, 0, 0, 1, -1, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1}
#define LBM3_CZ {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1}
#define LBM3_OPP {0, 2, 1, 4, 3, 6, 5, 10, 9, 8, 7, 14, 13, 12, 11, 18, 17, 16, 15}

// component a (0 x, 1 y, 2 z) of c_q, and the opposite direction
__host__ __device__ constexpr int cvel3(int q, int a) {
  const int cx[Q] = LBM3_CX, cy[Q] = LBM3_CY, cz[Q] = LBM3_CZ;
  return a == 0 ? cx[q] : (a == 1 ? cy[q] : cz[q]);
}
__host__ __device__ constexpr int opp3(int q) {
  const int o[Q] = LBM3_OPP;
  return o[q];
}

// Moment basis of d'Humieres et al. (2002): row r evaluated at c_q.  Rows:
// rho, e, eps, j_x, q_x, j_y, q_y, j_z, q_z, 3p_xx, 3pi_xx, p_ww, pi_ww,
// p_xy, p_yz, p_xz, m_x, m_y, m_z.  Every entry is an integer.
__host__ __device__ constexpr int m3(int r, int q) {
  const int x = cvel3(q, 0), y = cvel3(q, 1), z = cvel3(q, 2), c2 = x * x + y * y + z * z;
  switch (r) {
    case 0: return 1;
    case 1: return 19 * c2 - 30;
    case 2: return (21 * c2 * c2 - 53 * c2 + 24) / 2;
    case 3: return x;
    case 4: return (5 * c2 - 9) * x;
    case 5: return y;
    case 6: return (5 * c2 - 9) * y;
    case 7: return z;
    case 8: return (5 * c2 - 9) * z;
    case 9: return 3 * x * x - c2;
    case 10: return (3 * c2 - 5) * (3 * x * x - c2);
    case 11: return y * y - z * z;
    case 12: return (3 * c2 - 5) * (y * y - z * z);
    case 13: return x * y;
    case 14: return y * z;
    case 15: return x * z;
    case 16: return (y * y - z * z) * x;
    case 17: return (z * z - x * x) * y;
    default: return (x * x - y * y) * z;
  }
}

// the rows odd in c (j, q and the third-order m): m3(r, opp q) = -m3(r, q);
// the others are even
__host__ __device__ constexpr bool odd_row3(int r) { return (r >= 3 && r <= 8) || r >= 16; }

// one direction of each pair (q, opp q)
constexpr int kPairs3 = 9;
__host__ __device__ constexpr int rep3(int p) {
  const int t[kPairs3] = {1, 3, 5, 7, 8, 11, 12, 15, 16};
  return t[p];
}

__host__ __device__ constexpr int norm3(int r) {
  int s = 0;
  for (int q = 0; q < Q; q++) s += m3(r, q) * m3(r, q);
  return s;
}

// The basis is orthogonal, each row even or odd as odd_row3 says, and the
// representatives with their opposites cover directions 1..18 once.
constexpr bool basis3_ok() {
  for (int r = 0; r < Q; r++) {
    for (int s = 0; s < Q; s++) {
      int dot = 0;
      for (int q = 0; q < Q; q++) dot += m3(r, q) * m3(s, q);
      if (r != s && dot != 0) return false;
    }
    for (int q = 0; q < Q; q++)
      if (m3(r, opp3(q)) != (odd_row3(r) ? -m3(r, q) : m3(r, q))) return false;
  }
  int seen = 0;
  for (int p = 0; p < kPairs3; p++) seen |= (1 << rep3(p)) | (1 << opp3(rep3(p)));
  return seen == ((1 << Q) - 2);
}
static_assert(basis3_ok(), "D3Q19 moment basis");
static_assert(norm3(0) == 19 && norm3(1) == 2394 && norm3(2) == 252 && norm3(3) == 10 &&
                  norm3(4) == 40 && norm3(13) == 4 && norm3(16) == 8,
              "D3Q19 moment norms");

struct Lattice {
  int c[Q][3];
  int opp[Q];
  double w[Q];
  double M[Q][Q];  // moment basis, rows = moments
  double norm[Q];  // |M_k|^2
  Lattice() {
    for (int q = 0; q < Q; q++) {
      for (int a = 0; a < 3; a++) c[q][a] = cvel3(q, a);
      opp[q] = opp3(q);
      const int c2 = c[q][0] * c[q][0] + c[q][1] * c[q][1] + c[q][2] * c[q][2];
      w[q] = c2 == 0 ? 1.0 / 3.0 : (c2 == 1 ? 1.0 / 18.0 : 1.0 / 36.0);
    }
    for (int r = 0; r < Q; r++) {
      norm[r] = norm3(r);
      for (int q = 0; q < Q; q++) M[r][q] = m3(r, q);
    }
  }
};

const Lattice &lattice() {
  static const Lattice L;
  return L;
}

// p / d for 0 <= p < 2^31 by a multiplication (Granlund and Montgomery
// 1994): m = ceil(2^(31 + l) / d) with 2^l >= d, the quotient the product's
// bits from 31 + l up; m = 0 stands for d = 1.
struct DivBy3 {
  uint32_t m = 0, shift = 0;
  DivBy3() = default;
  explicit DivBy3(uint32_t d) {
    uint32_t l = 0;
    while ((uint64_t(1) << l) < d) l++;
    if (l == 0) return;
    m = static_cast<uint32_t>(((uint64_t(1) << (31 + l)) + d - 1) / d);
    shift = l - 1;
  }
  __device__ __forceinline__ uint32_t operator()(uint32_t p) const {
    return m ? __umulhi(p, m) >> shift : p;
  }
};

// Kernel constants of one case (passed by value): the relaxation rates
// s_k and forcing weights 1 - s_k/2 of the 19 moments, each divided by
// |M_k|^2 (the scale of M^-1 = M^T diag(1/|M_k|^2)).
template <typename C>
struct Const3 {
  C s_scaled[Q], f_scaled[Q];
  C ax, ay, az;
  int32_t nx, ny, nz, px, py, pz;
  DivBy3 by_nx, by_ny;
  int32_t diffuse_mode;
  int64_t plane;    // N
  int64_t n_links;  // the exact-mass variant: where the per-node carries start
  uint32_t sr_seed; // the exact-mass variant: random-bit seed of the step
};

// per link: k1, k2, k3, alpha of the folded form of Eq. EqNewBDSC (LinkCoef)
template <typename C>
struct Link3 {
  C k1, k2, k3, alpha;
};

// lattice weight of direction q
template <typename C>
__host__ __device__ constexpr C w3(int q) {
  return q == 0 ? C(1) / C(3) : (q < 7 ? C(1) / C(18) : C(1) / C(36));
}

// Coordinates of lattice node p (row-major x fastest; p < 2^31).
struct Coord3 {
  int x, y, z;
};
template <typename C>
__device__ __forceinline__ Coord3 coord3(const Const3<C> &k, int64_t p) {
  const unsigned u = static_cast<unsigned>(p), row = k.by_nx(u), z = k.by_ny(row);
  return Coord3{static_cast<int>(u - row * static_cast<unsigned>(k.nx)),
                static_cast<int>(row - z * static_cast<unsigned>(k.ny)), static_cast<int>(z)};
}

// Slot of f_q(x, t) for node p (pull layout): the neighbour x - c_q's own
// slot, or the node's tail element when x - c_q is solid.  A coordinate
// that leaves the lattice wraps (periodic axis); on a walled axis the link
// flag is set there, so the wrapped value is never used.
template <typename C>
__device__ __forceinline__ int64_t pull_slot3(const Const3<C> &k, int q, Coord3 c, uint32_t fl,
                                              uint32_t lbase, int64_t N) {
  if (fl & (1u << q)) return 19 * N + lbase + __popc(fl & ((1u << q) - 1u));
  int xs = c.x - cvel3(q, 0), ys = c.y - cvel3(q, 1), zs = c.z - cvel3(q, 2);
  xs += xs < 0 ? k.nx : (xs >= k.nx ? -k.nx : 0);
  ys += ys < 0 ? k.ny : (ys >= k.ny ? -k.ny : 0);
  zs += zs < 0 ? k.nz : (zs >= k.nz ? -k.nz : 0);
  return static_cast<int64_t>(q) * N + (static_cast<int64_t>(zs) * k.ny + ys) * k.nx + xs;
}

// acc + m x for a compile-time integer m (zero terms vanish, +-1 add)
template <typename C>
__device__ __forceinline__ C mac3(C acc, int m, C x) {
  return m == 0 ? acc : (m == 1 ? acc + x : (m == -1 ? acc - x : fma(C(m), x, acc)));
}

// Runtime forms of the velocity components and of the opposite direction
// (the link epilogue meets each direction as a value): two bits per
// direction hold c + 1.
constexpr uint64_t pack_c3(int a) {
  uint64_t t = 0;
  for (int q = 0; q < Q; q++) t |= static_cast<uint64_t>(cvel3(q, a) + 1) << (2 * q);
  return t;
}
constexpr uint64_t kPackX3 = pack_c3(0), kPackY3 = pack_c3(1), kPackZ3 = pack_c3(2);
__device__ __forceinline__ int cvel3_rt(int q, int a) {
  const uint64_t t = a == 0 ? kPackX3 : (a == 1 ? kPackY3 : kPackZ3);
  return static_cast<int>((t >> (2 * q)) & 3u) - 1;
}
__host__ __device__ constexpr int opp3_rt(int j) {
  return j <= 6 ? ((j - 1) ^ 1) + 1 : j + 3 - 2 * ((j - 7) & 3);
}
constexpr bool opp3_rt_ok() {
  for (int q = 1; q < Q; q++)
    if (opp3_rt(q) != opp3(q)) return false;
  return true;
}
static_assert(opp3_rt_ok(), "opposite directions");

// What the links of a boundary node read of it, one column per lane of a
// warp: f'_q (rows 0..17, q = 1..18), f_q (rows 18..35), drho, rho, u_x,
// u_y, u_z (rows 36..40); 33 columns so that a lane's rows fall in
// different banks.
constexpr int kLinkVals3 = 2 * (Q - 1) + 5;
template <typename C>
struct Warp3 {
  C v[kLinkVals3][33];
};

// lattice weight of direction q in the arithmetic type A
template <typename A>
__device__ __forceinline__ A wq3(int q) {
  return w3<A>(q);
}

// The second half of the collision: from d - d_eq as pair sums (NS) and
// differences (NA) plus the rest direction's (n0), rho, u and the body force
// a, the change ch[q] = f'_q - f_q (ch[0] = 0):
// m' - m = -s (m - m_eq) + (1 - s/2) M Fbar, scaled by 1/|M_k|^2.  M Fbar
// has a closed form (F = rho a; the moments of Eq. LBEforce): e 38 u.F, eps
// -11 u.F, j F, q -2/3 F, 3p_xx 2 (3 u_x F_x - u.F), p_ww 2 (u_y F_y -
// u_z F_z), the fourth-order ones -1/2 of these, p_ab u_a F_b + u_b F_a, m 0.
// rho does not change and j changes by F exactly, for any s_j, since rho u =
// j + F/2: taken as such.  (Formed from d - d_eq like the other rows, j came
// out as F plus rho u times the rounding of the equilibrium's weights, 1e-8
// every step.)
template <typename A>
__device__ __forceinline__ void transform3(const A n0, const A (&NS)[kPairs3],
                                           const A (&NA)[kPairs3], const A rho, const A (&u)[3],
                                           const Const3<A> &k, A (&ch)[Q]) {
  const A F[3] = {rho * k.ax, rho * k.ay, rho * k.az};
  const A uF[3] = {u[0] * F[0], u[1] * F[1], u[2] * F[2]};
  const A uf = uF[0] + uF[1] + uF[2];
  const A pxx = A(2) * (A(3) * uF[0] - uf), pww = A(2) * (uF[1] - uF[2]);
  const A b[Q] = {A(0), A(38) * uf, A(-11) * uf,
                  A(0), A(-2.0 / 3.0) * F[0], A(0), A(-2.0 / 3.0) * F[1],
                  A(0), A(-2.0 / 3.0) * F[2],
                  pxx, A(-0.5) * pxx, pww, A(-0.5) * pww,
                  u[0] * F[1] + u[1] * F[0], u[1] * F[2] + u[2] * F[1], u[0] * F[2] + u[2] * F[0],
                  A(0), A(0), A(0)};
  A dm[Q];
#pragma unroll
  for (int r = 1; r < Q; r++) {
    if (r == 3 || r == 5 || r == 7) {
      dm[r] = A(1.0 / norm3(3)) * F[(r - 3) / 2];
      continue;
    }
    A a = A(0);
    if (!odd_row3(r)) a = mac3(a, m3(r, 0), n0);
#pragma unroll
    for (int pp = 0; pp < kPairs3; pp++) a = mac3(a, m3(r, rep3(pp)), odd_row3(r) ? NA[pp] : NS[pp]);
    dm[r] = r >= 16 ? -k.s_scaled[r] * a : k.f_scaled[r] * b[r] - k.s_scaled[r] * a;
  }
  // f' - f = M^T dm: even rows give the same change to q and opp q, odd
  // rows opposite ones
  ch[0] = A(0);
#pragma unroll
  for (int pp = 0; pp < kPairs3; pp++) {
    const int q = rep3(pp), qb = opp3(q);
    A ev = A(0), od = A(0);
#pragma unroll
    for (int r = 1; r < Q; r++) {
      if (odd_row3(r)) od = mac3(od, m3(r, q), dm[r]);
      else ev = mac3(ev, m3(r, q), dm[r]);
    }
    ch[q] = ev + od;
    ch[qb] = ev - od;
  }
}

__device__ __forceinline__ float recip3(float r) { return __frcp_rn(r); }
__device__ __forceinline__ double recip3(double r) { return 1.0 / r; }

// The collision change f' - f of one node from its deviations d (Eq.
// FluidMacr, Eq. LBEequi, Eq. LBEforce, Eq. MomentPost through M^-1), in
// the arithmetic type A: ch[1..18] (f'_0 closes the mass instead), and the
// node's rho - 1, rho and u.  It runs on the pairs (q, opp q): d_q + d_opp
// carries the even moments and d_q - d_opp the odd ones, so each row of M
// touches at most ten values and, M being integer and known here at compile
// time, only its non-zero entries cost an instruction.
template <typename A>
__device__ __forceinline__ void collide3(const A (&d)[Q], const Const3<A> &k, A &drho, A &rho,
                                         A (&u)[3], A (&ch)[Q]) {
  // Eq. FluidMacr on the pair sums and differences
  A S[kPairs3], D[kPairs3];
  drho = d[0];
#pragma unroll
  for (int pp = 0; pp < kPairs3; pp++) {
    S[pp] = d[rep3(pp)] + d[opp3(rep3(pp))];
    D[pp] = d[rep3(pp)] - d[opp3(rep3(pp))];
    drho += S[pp];
  }
  A j[3] = {A(0), A(0), A(0)};
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int pp = 0; pp < kPairs3; pp++) j[a] = mac3(j[a], cvel3(rep3(pp), a), D[pp]);
  rho = A(1) + drho;
  const A inv = recip3(rho), half = A(0.5) * rho;
  u[0] = lbm::dev::quotient(fma(half, k.ax, j[0]), rho, inv);
  u[1] = lbm::dev::quotient(fma(half, k.ay, j[1]), rho, inv);
  u[2] = lbm::dev::quotient(fma(half, k.az, j[2]), rho, inv);
  const A ux = u[0], uy = u[1], uz = u[2];
  const A uu = ux * ux + uy * uy + uz * uz;
  // d - d_eq (Eq. LBEequi), as pair sums and differences; the rest
  // direction alone.  Per pair of weight w: the sum's 2 w (rho - 1 + rho (9/2
  // (c.u)^2 - 3/2 u.u)), the difference's 6 w rho c.u.  (The sum's terms
  // common to all pairs are not formed once and shared: their one rounding
  // would lean the same way in every pair, and the velocity error of the
  // sphere pack tripled.)
  A NS[kPairs3], NA[kPairs3];
  const A uu15 = A(-1.5) * uu;
  const A n0 = d[0] - wq3<A>(0) * fma(rho, uu15, drho);
  const A ga = A(1.0 / 3) * rho, gd = A(0.5) * ga;     // 6 w rho
#pragma unroll
  for (int pp = 0; pp < kPairs3; pp++) {
    const int q = rep3(pp);
    const A cu = mac3(mac3(mac3(A(0), cvel3(q, 0), ux), cvel3(q, 1), uy), cvel3(q, 2), uz);
    NS[pp] = fma(A(-2) * wq3<A>(q), fma(rho, fma(A(4.5) * cu, cu, uu15), drho), S[pp]);
    NA[pp] = fma(-(q < 7 ? ga : gd), cu, D[pp]);
  }
  transform3<A>(n0, NS, NA, rho, u, k, ch);
}

// The exact-mass variant's first half of the collision (FP32 storage).  The
// pair sums and d_eq are ~100 times their difference d - d_eq, so the FP32
// rounding errors of the former become relative errors of ~1e-5 of the
// latter, and in a steady flow they repeat every step; so rho - 1, j, rho,
// u and d - d_eq are formed in double-FP32 (the pair sums exactly, by
// TwoSum) and d - d_eq is rounded once to FP32 for the transform.  rho - 1,
// rho, u and -3/2 |u|^2 are returned in double-FP32 for the links.
// Sums of several terms run in twice the working precision without
// normalising in between (Sum), products by lattice weights are formed once
// per node for the axes and halved (exactly) for the diagonals, and rho's
// reciprocal serves the three quotients: about 950 operations, straight-line
// (the form before, one general double-FP32 operation per term, took 3 to 4
// times as many).
using lbm::dev::DF;
using lbm::dev::Sum;
struct Force3 {
  DF a[3];  // the body acceleration as double-FP32 pairs
};
inline DF df_of(double x) {
  const float h = static_cast<float>(x);
  return DF{h, static_cast<float>(x - static_cast<double>(h))};
}
__device__ __forceinline__ DF df_third() {
  constexpr float h = static_cast<float>(1.0 / 3.0);
  return DF{h, static_cast<float>(1.0 / 3.0 - static_cast<double>(h))};
}
__device__ __forceinline__ DF df_ninth() {
  constexpr float h = static_cast<float>(1.0 / 9.0);
  return DF{h, static_cast<float>(1.0 / 9.0 - static_cast<double>(h))};
}
__device__ __forceinline__ void exact_moments3(const float (&d)[Q], const Force3 &force, DF &drho,
                                               DF &rho, DF (&u)[3], DF &uu15, float &n0,
                                               float (&NS)[kPairs3], float (&NA)[kPairs3]) {
  using namespace lbm::dev;
  DF S[kPairs3], D[kPairs3];
  Sum sr(DF{d[0], 0.0f});
#pragma unroll
  for (int pp = 0; pp < kPairs3; pp++) {
    const int q = rep3(pp), qb = opp3(q);
    two_sum(d[q], d[qb], S[pp].h, S[pp].l);
    two_sum(d[q], -d[qb], D[pp].h, D[pp].l);
    sr.add(S[pp]);
  }
  drho = sr.value();
  rho = df_add(DF{1.0f, 0.0f}, drho);
  const float inv = __frcp_rn(rho.h);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    Sum sj(D[a]);  // pair a is the axis a
#pragma unroll
    for (int pp = 3; pp < kPairs3; pp++) {
      const int c = cvel3(rep3(pp), a);
      if (c != 0) sj.add(c > 0 ? D[pp] : df_neg(D[pp]));
    }
    DF j = sj.value();
    if (force.a[a].h != 0.0f) j = df_add(j, df_mul(df_scale(0.5f, rho), force.a[a]));
    u[a] = df_div_inv(j, rho, inv);
  }
  const DF uu = df_add(df_add(df_mul(u[0], u[0]), df_mul(u[1], u[1])), df_mul(u[2], u[2]));
  uu15 = df_mul_f(uu, -1.5f);
  const DF e0 = df_add(drho, df_mul(rho, uu15));
  n0 = df_sub_f(DF{d[0], 0.0f}, df_mul(e0, df_third()));
  const DF ea = df_mul(e0, df_ninth()), ed = df_scale(0.5f, ea);
  const DF ra = df_scale(0.5f, rho), rd = df_scale(0.25f, rho);
  const DF ga = df_mul(rho, df_third()), gd = df_scale(0.5f, ga);
#pragma unroll
  for (int pp = 0; pp < kPairs3; pp++) {
    const int q = rep3(pp);
    DF cu{0.0f, 0.0f};
    bool first = true;
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const int c = cvel3(q, a);
      if (c == 0) continue;
      const DF t = c > 0 ? u[a] : df_neg(u[a]);
      cu = first ? t : df_add(cu, t);
      first = false;
    }
    const DF eq = df_add(df_mul(df_mul(cu, cu), q < 7 ? ra : rd), q < 7 ? ea : ed);
    NS[pp] = df_sub_f(S[pp], eq);
    NA[pp] = df_sub_f(D[pp], df_mul(q < 7 ? ga : gd, cu));
  }
}

// The exact-mass variant's extra record per warp: rho - 1, rho, u_x, u_y,
// u_z, -3/2 |u|^2 of each boundary node in double-FP32 (pairs of rows).
struct Warp3X {
  float v[12][33];
};

// Gather, collide and store one fluid node (pull layout); a boundary node
// leaves what its links need in the warp's shared record.
//
// kExact (FP32 storage): the stored mass must follow the FP64 trajectory to
// ~1e-10 over thousands of steps where walls move, and a moving wall
// exchanges mass at a rate set by the populations next to it.  Any rounding
// that leans the same way step after step shifts that rate: the storage
// rounding of f' (round to nearest), and equally the FP32 arithmetic of the
// collision, whose rounding errors repeat every step once the flow is
// steady.  So d - d_eq is formed in double-FP32 (exact_moments3; kd: the
// body force as double-FP32 pairs) before the FP32 transform to f' - f,
// f'_1..f'_18 are rounded to FP32 stochastically, and f'_0 closes the
// node's mass in double-FP32 plus the node's carry c0 (what FP32 storage
// dropped from its earlier values); stored rounded to nearest, the new
// remainder is kept in c0.
//
// I indexes the lattice's elements: 32 bits where all of them, link tail
// included, fit (half the address arithmetic), else 64.
template <typename C, bool kExact, typename I>
__device__ __forceinline__ void node3(const C *src, C *dst, const Const3<C> &k, const uint32_t p,
                                      const uint32_t fl, const uint32_t lb, Warp3<C> &sh,
                                      const int lane, float *c0 = nullptr, const uint32_t rs = 0u,
                                      Warp3X *shx = nullptr, const Force3 *force = nullptr) {
  const I N = static_cast<I>(k.plane);
  const Coord3 c = coord3(k, p);
  C d[Q];
  {
    // x - c_q from the wrapped coordinates, or the node's next tail element
    // where x - c_q is solid (a select, so interior and boundary nodes run
    // the same instructions; on a walled axis the wrapped value is unused)
    const int xw[3] = {c.x + 1 < k.nx ? c.x + 1 : 0, c.x, c.x > 0 ? c.x - 1 : k.nx - 1};
    const int yw[3] = {c.y + 1 < k.ny ? c.y + 1 : 0, c.y, c.y > 0 ? c.y - 1 : k.ny - 1};
    const int zw[3] = {c.z + 1 < k.nz ? c.z + 1 : 0, c.z, c.z > 0 ? c.z - 1 : k.nz - 1};
    uint32_t row[3][3];  // lattice nodes are below 2^31
#pragma unroll
    for (int z = 0; z < 3; z++)
#pragma unroll
      for (int y = 0; y < 3; y++)
        row[z][y] = static_cast<uint32_t>((zw[z] * k.ny + yw[y]) * k.nx);
    I t = 19 * N + lb;
    lbm::dev::chain_wait();
    d[0] = src[p];
#pragma unroll
    for (int q = 1; q < Q; q++) {
      const I nb = static_cast<I>(q) * N +
                   (row[cvel3(q, 2) + 1][cvel3(q, 1) + 1] + static_cast<uint32_t>(xw[cvel3(q, 0) + 1]));
      const bool link = (fl & (1u << q)) != 0u;
      d[q] = src[link ? t : nb];
      t += link ? 1 : 0;
    }
  }
  C o[Q];
  if constexpr (kExact) {
    static_assert(std::is_same<C, float>::value, "the exact-mass variant is FP32 storage");
    DF drx, rhx, ux3[3], uu15;
    float n0, NS[kPairs3], NA[kPairs3], ch[Q];
    exact_moments3(d, *force, drx, rhx, ux3, uu15, n0, NS, NA);
    const float uf[3] = {ux3[0].h, ux3[1].h, ux3[2].h};
    transform3<float>(n0, NS, NA, rhx.h, uf, k, ch);
    // f'_q = f_q + ch_q rounded to FP32 stochastically (16 random bits
    // each: the halves of the node's nine random words)
    uint32_t rw[kPairs3];
    rw[0] = lbm::dev::fmix32(rs);
#pragma unroll
    for (int pp = 1; pp < kPairs3; pp++) rw[pp] = lbm::dev::fmix32(rw[0] + 0x9E3779B9u * pp);
#pragma unroll
    for (int pp = 0; pp < kPairs3; pp++) {
      const int q = rep3(pp), qb = opp3(q);
      o[q] = lbm::dev::add_stochastic(d[q], ch[q], rw[pp] & 0xFFFFu);
      o[qb] = lbm::dev::add_stochastic(d[qb], ch[qb], rw[(pp + 4) % kPairs3] >> 16);
    }
    // f'_0 = f_0 - sum (f'_q - f_q) plus the carry, in double-FP32 (each
    // change is the exact difference of two FP32 values); stored rounded to
    // nearest, the remainder kept
    Sum sum(DF{d[0], 0.0f});
#pragma unroll
    for (int q = 1; q < Q; q++) {
      DF dd;
      lbm::dev::two_sum(d[q], -o[q], dd.h, dd.l);
      sum.add(dd);
    }
    sum.add(DF{*c0, 0.0f});
    float e0;
    lbm::dev::two_sum(sum.s, sum.e, o[0], e0);
    *c0 = e0;
#pragma unroll
    for (int q = 0; q < Q; q++) dst[static_cast<I>(q) * N + p] = o[q];
    if (fl) {
#pragma unroll
      for (int q = 1; q < Q; q++) {
        sh.v[q - 1][lane] = o[q];
        sh.v[Q - 2 + q][lane] = d[q];
      }
      // rho - 1, rho, u and -3/2 |u|^2 as pairs of FP32 values for the links
      const DF nv[6] = {drx, rhx, ux3[0], ux3[1], ux3[2], uu15};
#pragma unroll
      for (int i = 0; i < 6; i++) {
        shx->v[2 * i][lane] = nv[i].h;
        shx->v[2 * i + 1][lane] = nv[i].l;
      }
    }
  } else {
    C drho, rho, u[3], ch[Q];
    collide3<C>(d, k, drho, rho, u, ch);
    // f'_0 closes the mass from the stored changes
    C sum = C(0);
#pragma unroll
    for (int pp = 0; pp < kPairs3; pp++) {
      const int q = rep3(pp), qb = opp3(q);
      o[q] = d[q] + ch[q];
      o[qb] = d[qb] + ch[qb];
      sum += (o[q] - d[q]) + (o[qb] - d[qb]);
    }
    o[0] = d[0] - sum;
#pragma unroll
    for (int q = 0; q < Q; q++) dst[static_cast<I>(q) * N + p] = o[q];
    if (fl) {
#pragma unroll
      for (int q = 1; q < Q; q++) {
        sh.v[q - 1][lane] = o[q];
        sh.v[Q - 2 + q][lane] = d[q];
      }
      sh.v[36][lane] = drho;
      sh.v[37][lane] = rho;
      sh.v[38][lane] = u[0];
      sh.v[39][lane] = u[1];
      sh.v[40][lane] = u[2];
    }
  }
}

// One lattice step of every fluid node, then Eq. EqNewBDSC for every
// boundary link of the step's nodes into the lattice's tail.  The links of
// a warp's 32 nodes are consecutive in the link table (sorted by node); the
// warp spreads them over its lanes, one link per lane, each reading its
// node's values from the warp's shared record -- the links of a node
// cluster would otherwise run direction by direction on few lanes.
// Each lane finds its link's node (lane of the warp) and direction in the
// link's entry of ldesc.
// kExact: 96 registers and 5 CTAs per SM.
template <typename C, bool kExact, typename I>
__global__ void __launch_bounds__(kThreads3, kExact ? 5 : (sizeof(C) == 4 ? 8 : 2))
step3_kernel(const C *src, C *dst, const uint32_t *__restrict__ gbase,
             const uint16_t *__restrict__ ldesc, const Link3<C> *__restrict__ links,
             const uint2 *__restrict__ fluid, const __grid_constant__ Const3<C> k, int64_t n_fluid,
             const lbm::LinkCoefDF *__restrict__ links_df, float *carry,
             const __grid_constant__ Force3 force) {
  constexpr int kW = kThreads3 / 32;
  __shared__ Warp3<C> sh[kW];
  __shared__ Warp3X shx[kExact ? kW : 1];
  // thread t of the launch runs the t-th fluid node (node order), so no
  // lane idles on a solid node
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int lane = static_cast<int>(threadIdx.x & 31u), w = static_cast<int>(threadIdx.x >> 5);
  const bool live = t0 < n_fluid;
  // the fluid-node list holds each node's index and flag word together, the
  // flag word the node's first link within its group of 32 (a warp)
  const uint2 pf = live ? fluid[t0] : make_uint2(0u, 0u);
  const uint32_t fl = pf.y & kFlags3;
  const uint32_t base = t0 - lane < n_fluid ? gbase[t0 / 32] : 0u;  // the warp's first link
  // the exact-mass variant's carries: one per link, then one per fluid node
  if (live) {
    if constexpr (kExact)
      node3<C, true, I>(src, dst, k, pf.x, fl, base + (pf.y >> kRank3), sh[w], lane,
                        carry + k.n_links + t0, static_cast<uint32_t>(t0) ^ k.sr_seed, &shx[w],
                        &force);
    else
      node3<C, false, I>(src, dst, k, pf.x, fl, base + (pf.y >> kRank3), sh[w], lane);
  }
  const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, static_cast<uint32_t>(__popc(fl)));
  if (total == 0u) return;
  __syncwarp();
  const Warp3<C> &ws = sh[w];
  C *tail = dst + 19 * k.plane;
  for (uint32_t t = static_cast<uint32_t>(lane); t < total; t += 32u) {
    const uint32_t lj = base + t, dsc = ldesc[lj];
    const int s = static_cast<int>(dsc >> 5), j = static_cast<int>(dsc & 31u), jb = opp3_rt(j);
    const C oj = ws.v[j - 1][s], ojb = ws.v[jb - 1][s], djb = ws.v[Q - 2 + jb][s];
    if constexpr (kExact) {
      // Eq. EqNewBDSC in double-FP32 with the link's carry
      using namespace lbm::dev;
      const Warp3X &wx = shx[w];
      const DF drho{wx.v[0][s], wx.v[1][s]}, rho{wx.v[2][s], wx.v[3][s]};
      DF cu{0.0f, 0.0f};
#pragma unroll
      for (int a = 0; a < 3; a++) {
        const DF t1 = df_scale(static_cast<float>(cvel3_rt(j, a)),
                               DF{wx.v[4 + 2 * a][s], wx.v[5 + 2 * a][s]});
        cu = a == 0 ? t1 : df_add(cu, t1);
      }
      tail[lj] = link_value_exact(links_df[lj], k.diffuse_mode, djb, oj, ojb, drho, rho, cu,
                                  DF{wx.v[10][s], wx.v[11][s]}, carry + lj);
    } else {
      const Link3<C> cl = links[lj];
      const C drho = ws.v[36][s], rho = ws.v[37][s], ux = ws.v[38][s], uy = ws.v[39][s],
              uz = ws.v[40][s];
      const C uu = ux * ux + uy * uy + uz * uz;
      const C wj = j < 7 ? C(1) / C(18) : C(1) / C(36);
      const C r = cl.k1 + cl.k2 + cl.k3;
      C c0, c2;
      if (k.diffuse_mode == 0) {
        c0 = cl.alpha;
        c2 = (C(1) - r) * wj;
      } else {
        c0 = cl.alpha + (r - C(1)) * wj;
        c2 = C(0);
      }
      const C cu = C(cvel3_rt(j, 0)) * ux + C(cvel3_rt(j, 1)) * uy + C(cvel3_rt(j, 2)) * uz;
      const C pj = C(3) * cu + C(4.5) * cu * cu - C(1.5) * uu;
      tail[lj] = cl.k1 * djb + cl.k2 * oj + cl.k3 * ojb + c0 + cl.alpha * drho +
                 c2 * (drho + rho * pj);
    }
  }
}

// Residual pass (FP64 sums, fixed grid and order): num, den, mass
// deviation, non-finite count of the states in cur and prev.
template <typename C>
__global__ void __launch_bounds__(kResThreads3)
residual3_kernel(const C *__restrict__ cur, const C *__restrict__ prev,
                 const uint32_t *__restrict__ gbase, const uint2 *__restrict__ fluid,
                 const Const3<C> k, int64_t n_fluid, double *__restrict__ partials) {
  // per node: rho and j of both states in the storage's arithmetic type,
  // the node's mass deviation summed in FP64; sums over nodes in FP64
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const int64_t G = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < n_fluid;
       t += G) {
    const uint2 pf = fluid[t];
    const int64_t p = pf.x;
    const uint32_t fl = pf.y & kFlags3;
    const Coord3 c = coord3(k, p);
    C r1 = C(0), r0 = C(0), j1[3] = {C(0), C(0), C(0)}, j0[3] = {C(0), C(0), C(0)};
    double dm = 0.0;
    const uint32_t lb = gbase[t / 32] + (pf.y >> kRank3);
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const int64_t s = pull_slot3(k, q, c, fl, lb, k.plane);
      const C a = cur[s], b = prev[s];
      r1 += a;
      r0 += b;
      dm += static_cast<double>(a);
#pragma unroll
      for (int e = 0; e < 3; e++) {
        j1[e] = mac3(j1[e], cvel3(q, e), a);
        j0[e] = mac3(j0[e], cvel3(q, e), b);
      }
    }
    r1 += C(1);
    r0 += C(1);
    const C acc3[3] = {k.ax, k.ay, k.az};
    double num = 0.0, den = 0.0;
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const C u1 = (j1[e] + C(0.5) * r1 * acc3[e]) / r1, u0 = (j0[e] + C(0.5) * r0 * acc3[e]) / r0;
      const double du = static_cast<double>(u1) - static_cast<double>(u0);
      num += du * du;
      den += static_cast<double>(u1) * static_cast<double>(u1);
    }
    if (!(isfinite(num) && isfinite(den) && isfinite(dm))) {
      acc[3] += 1.0;
      continue;
    }
    acc[0] += num;
    acc[1] += den;
    acc[2] += dm;
  }
  __shared__ double sh[kResThreads3 / 32][4];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int cc = 0; cc < 4; cc++) {
    const double v = lbm::dev::warp_sum(acc[cc]);
    if (lane == 0) sh[w][cc] = v;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int i = 0; i < kResThreads3 / 32; i++) t += sh[i][threadIdx.x];
    partials[blockIdx.x * 4 + threadIdx.x] = t;
  }
}

__global__ void __launch_bounds__(1024) residual3_final(const double *partials, double *out) {
  __shared__ double sh[32][4];
  double v[4];
  for (int c = 0; c < 4; c++) {
    double t = 0.0;
    for (int b = threadIdx.x; b < kResBlocks3; b += 1024) t += partials[b * 4 + c];
    v[c] = lbm::dev::warp_sum(t);
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0)
    for (int c = 0; c < 4; c++) sh[w][c] = v[c];
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int i = 0; i < 32; i++) s += sh[i][threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// Conversions between the lattice and caller arrays of full populations
// f[19][nz][ny][nx] (export: solid nodes as the rest state w_q; import:
// solid entries ignored).
template <typename C>
__global__ void export3_kernel(const C *__restrict__ f, const uint32_t *__restrict__ flags,
                               const uint32_t *__restrict__ lbase, const Const3<C> k,
                               int64_t n_nodes, double *out) {
  for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < n_nodes;
       p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const uint32_t fl = flags[p];
    const Coord3 c = coord3(k, p);
    const uint32_t lb = fl != kSolid3 && fl ? lbase[p] : 0u;
#pragma unroll
    for (int q = 0; q < Q; q++) {
      double v = w3<double>(q);
      if (fl != kSolid3) v += static_cast<double>(f[pull_slot3(k, q, c, fl, lb, k.plane)]);
      out[q * n_nodes + p] = v;
    }
  }
}

// Eq. FluidMacr at every node (solid nodes 0): rho, ux, uy, uz arrays of
// nx*ny*nz doubles.
struct HalfAccel3 {
  double a[3];
};
template <typename C>
__global__ void fields3_kernel(const C *__restrict__ f, const uint32_t *__restrict__ flags,
                               const uint32_t *__restrict__ lbase, const Const3<C> k,
                               const HalfAccel3 half, int64_t n_nodes, double *__restrict__ out) {
  for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < n_nodes;
       p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const uint32_t fl = flags[p];
    double r = 0.0, u[3] = {0.0, 0.0, 0.0};
    if (fl != kSolid3) {
      const Coord3 c = coord3(k, p);
      const uint32_t lb = fl ? lbase[p] : 0u;
      C d[Q];
#pragma unroll
      for (int q = 0; q < Q; q++) d[q] = f[pull_slot3(k, q, c, fl, lb, k.plane)];
      C j[3][10];
#pragma unroll
      for (int e = 0; e < 3; e++) {
        int at = 0;
#pragma unroll
        for (int q = 1; q < Q; q++)
          if (cvel3(q, e) != 0) j[e][at++] = cvel3(q, e) > 0 ? d[q] : -d[q];
      }
      lbm::dev::node_fields(d, j, half.a, r, u);
    }
    out[p] = r;
    out[n_nodes + p] = u[0];
    out[2 * n_nodes + p] = u[1];
    out[3 * n_nodes + p] = u[2];
  }
}

template <typename C>
__global__ void import3_kernel(const double *__restrict__ in, const uint32_t *__restrict__ flags,
                               const uint32_t *__restrict__ lbase, const Const3<C> k,
                               int64_t n_nodes, C *f) {
  for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < n_nodes;
       p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const uint32_t fl = flags[p];
    if (fl == kSolid3) continue;
    const Coord3 c = coord3(k, p);
    const uint32_t lb = fl ? lbase[p] : 0u;
#pragma unroll
    for (int q = 0; q < Q; q++)
      f[pull_slot3(k, q, c, fl, lb, k.plane)] = static_cast<C>(in[q * n_nodes + p] - w3<double>(q));
  }
}

// a case's constants in both arithmetic types (the one of its precision is set)
struct Const3Both {
  Const3<double> d;
  Const3<float> f;
  Const3<double> &get(double *) { return d; }
  Const3<float> &get(float *) { return f; }
  const Const3<double> &get(double *) const { return d; }
  const Const3<float> &get(float *) const { return f; }
};

int grid_for3(int64_t n, int threads) {
  const int64_t b = (n + threads - 1) / threads;
  return static_cast<int>(b < 1 ? 1 : (b > 65536 ? 65536 : b));
}

}  // namespace lbm3

using lbm3::Const3Both;
struct lbm3d {
  int precision = LBM_FP32;
  cudaStream_t stream = nullptr;
  int32_t nx = 0, ny = 0, nz = 0;
  int64_t n_nodes = 0, plane = 0, n_fluid = 0, n_links = 0, steps = 0;
  double ax = 0.0, ay = 0.0, az = 0.0;
  lbm::CaseParams cp{};
  void *f[2] = {nullptr, nullptr};
  int cur = 0;
  uint32_t *flags = nullptr;
  uint32_t *lbase = nullptr;
  uint2 *fluid = nullptr;  // the fluid nodes in node order: index, flag word (kFlags3)
  uint32_t *gbase = nullptr;   // per 32 of them: the first link of the first
  uint16_t *ldesc = nullptr;   // per link: its node's place among the 32 << 5 | direction
  // the exact-mass variant (FP32): link coefficients as FP32 pairs and the
  // carries (one per link, then one per fluid node)
  int exact = 0;
  int64_t dev_bytes = 0;  // device memory the handle holds
  lbm::LinkCoefDF *links_df = nullptr;
  float *carry = nullptr;
  void *links = nullptr;
  Const3Both kc;
  lbm3::Force3 force{};  // the exact-mass variant's body force
  double *partials = nullptr, *result = nullptr;
  std::vector<double> link_r, link_l;
  std::string err;
};

namespace {

thread_local std::string g_err3;

int fail3(lbm3d_t *h, int code, const std::string &m) {
  if (h) h->err = m;
  else g_err3 = m;
  return code;
}

void release3(lbm3d_t *h) {
  if (!h) return;
  cudaStreamSynchronize(h->stream);
  for (void *p : {h->f[0], h->f[1], static_cast<void *>(h->flags), static_cast<void *>(h->lbase),
                  static_cast<void *>(h->fluid), static_cast<void *>(h->gbase),
                  static_cast<void *>(h->ldesc), static_cast<void *>(h->links_df),
                  static_cast<void *>(h->carry),
                  h->links, static_cast<void *>(h->partials),
                  static_cast<void *>(h->result)})
    if (p) cudaFree(p);
  delete h;
}

template <typename F>
cudaError_t dispatch3(int precision, F &&fn) {
  if (precision == LBM_FP64) return fn(static_cast<double *>(nullptr));
  return fn(static_cast<float *>(nullptr));
}

}  // namespace

extern "C" {

int lbm3d_create(const lbm3d_domain_t *dom, const uint8_t *solid, size_t n_links,
                 const int32_t *link_x, const int32_t *link_y, const int32_t *link_z,
                 const int32_t *link_dir, const double *link_q, const double *link_ub, double Kn,
                 const lbm_params_t *params, lbm3d_t **out) {
  using namespace lbm3;
  g_err3.clear();
  if (!out) return fail3(nullptr, LBM_EINVAL, "null output");
  *out = nullptr;
  if (!dom || !solid || !params) return fail3(nullptr, LBM_EINVAL, "null argument");
  if (n_links && (!link_x || !link_y || !link_z || !link_dir || !link_q || !link_ub))
    return fail3(nullptr, LBM_EINVAL, "null link array");
  const lbm_params_t &p = *params;
  if (p.precision != LBM_FP64 && p.precision != LBM_FP32)
    return fail3(nullptr, LBM_EINVAL, "the 3-D solver stores LBM_FP64 or LBM_FP32");
  if (p.diffuse_mode != 0 && p.diffuse_mode != 1)
    return fail3(nullptr, LBM_EINVAL, "diffuse_mode must be 0 or 1");
  if (p.collision != 0) return fail3(nullptr, LBM_EINVAL, "the 3-D solver is MRT only");
  if (p.mass_mode < -1 || p.mass_mode > 1)
    return fail3(nullptr, LBM_EINVAL, "mass_mode must be -1, 0 or 1");
  const int32_t nx = dom->nx, ny = dom->ny, nz = dom->nz;
  if (nx < 1 || ny < 1 || nz < 1) return fail3(nullptr, LBM_EINVAL, "nx, ny, nz must be >= 1");
  const int64_t n = static_cast<int64_t>(nx) * ny * nz;
  if (n >= (int64_t(1) << 31)) return fail3(nullptr, LBM_EINVAL, "lattice too large");
  if (!std::isfinite(dom->ax) || !std::isfinite(dom->ay) || !std::isfinite(dom->az))
    return fail3(nullptr, LBM_EINVAL, "non-finite force");
  const int per[3] = {dom->periodic_x ? 1 : 0, dom->periodic_y ? 1 : 0, dom->periodic_z ? 1 : 0};
  const Lattice &L = lattice();
  auto node = [&](int64_t x, int64_t y, int64_t z) { return (z * ny + y) * nx + x; };
  // neighbour x + s c_q, or -1 outside a non-periodic axis
  auto nbr = [&](int x, int y, int z, int q, int s) -> int64_t {
    int a[3] = {x + s * L.c[q][0], y + s * L.c[q][1], z + s * L.c[q][2]};
    const int d[3] = {nx, ny, nz};
    for (int e = 0; e < 3; e++) {
      if (a[e] < 0 || a[e] >= d[e]) {
        if (!per[e]) return -1;
        a[e] = (a[e] + d[e]) % d[e];
      }
    }
    return node(a[0], a[1], a[2]);
  };
  // flags: unknown directions of fluid nodes
  std::vector<uint32_t> flags(static_cast<size_t>(n), kSolid3);
  int64_t n_fluid = 0;
  for (int z = 0; z < nz; z++)
    for (int y = 0; y < ny; y++)
      for (int x = 0; x < nx; x++) {
        const int64_t pn = node(x, y, z);
        if (solid[pn]) continue;
        n_fluid++;
        uint32_t fl = 0;
        for (int q = 1; q < Q; q++) {
          const int64_t r = nbr(x, y, z, q, -1);
          if (r < 0 || solid[r]) fl |= 1u << q;
        }
        flags[pn] = fl;
      }
  // links: validate, one per unknown (node, direction), sorted by node then direction
  std::vector<uint32_t> lbase(static_cast<size_t>(n), 0);
  int64_t total = 0;
  for (int64_t pn = 0; pn < n; pn++) {
    lbase[pn] = static_cast<uint32_t>(total);
    if (flags[pn] != kSolid3) total += __builtin_popcount(flags[pn]);
  }
  if (total > static_cast<int64_t>(UINT32_MAX))
    return fail3(nullptr, LBM_EINVAL, "more than 2^32 - 1 boundary links");
  if (static_cast<int64_t>(n_links) != total)
    return fail3(nullptr, LBM_EINVAL,
                 "links must cover every unknown (node, direction) once: " +
                     std::to_string(total) + " unknown, " + std::to_string(n_links) + " given");
  std::vector<int64_t> slot(n_links);
  std::vector<uint8_t> seen(static_cast<size_t>(total), 0);
  std::vector<double> cub(n_links), wq(n_links), uu(n_links);
  for (size_t k = 0; k < n_links; k++) {
    const int x = link_x[k], y = link_y[k], z = link_z[k], q = link_dir[k];
    if (x < 0 || x >= nx || y < 0 || y >= ny || z < 0 || z >= nz || q < 1 || q >= Q)
      return fail3(nullptr, LBM_EINVAL, "link " + std::to_string(k) + ": out of range");
    if (!(link_q[k] > 0.0 && link_q[k] <= 1.0))
      return fail3(nullptr, LBM_EINVAL, "link " + std::to_string(k) + ": gamma outside (0, 1]");
    const int64_t pn = node(x, y, z);
    const uint32_t fl = flags[pn];
    if (fl == kSolid3 || !(fl & (1u << q)))
      return fail3(nullptr, LBM_EINVAL,
                   "link " + std::to_string(k) + ": node must be fluid and x - c_i solid");
    const int64_t s = lbase[pn] + __builtin_popcount(fl & ((1u << q) - 1u));
    if (seen[s]) return fail3(nullptr, LBM_EINVAL, "link " + std::to_string(k) + ": duplicate");
    seen[s] = 1;
    slot[k] = s;
    const double *ub = link_ub + 3 * k;
    cub[k] = L.c[q][0] * ub[0] + L.c[q][1] * ub[1] + L.c[q][2] * ub[2];
    wq[k] = L.w[q];
    uu[k] = ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2];
  }
  // Sec. 3.B parameters (the two-dimensional closed forms) and the folded
  // per-link coefficients
  lbm::CaseParams cp;
  std::string msg = lbm::compute_case_params(Kn, dom->H, p, &cp);
  if (!msg.empty()) return fail3(nullptr, LBM_EINVAL, msg);
  std::vector<double> r(n_links), l(n_links), coef(8 * n_links);
  msg = lbm::compute_link_coefs_general(cp, p, n_links, link_q, cub.data(), wq.data(), uu.data(),
                                        r.data(), l.data(), coef.data(), &cp.n_clamped);
  if (!msg.empty()) return fail3(nullptr, LBM_EINVAL, msg);

  lbm3d_t *h = new (std::nothrow) lbm3d_t();
  if (!h) return fail3(nullptr, LBM_ENOMEM, "host allocation failed");
  h->precision = p.precision;
  h->stream = static_cast<cudaStream_t>(p.stream);
  h->nx = nx;
  h->ny = ny;
  h->nz = nz;
  h->n_nodes = n;
  h->plane = (n + 31) / 32 * 32;
  h->n_fluid = n_fluid;
  h->n_links = static_cast<int64_t>(n_links);
  h->ax = dom->ax;
  h->ay = dom->ay;
  h->az = dom->az;
  h->cp = cp;
  h->link_r = r;
  h->link_l = l;
  // relaxation times of the 19 moments: rho, e, eps, j_x, q_x, j_y, q_y,
  // j_z, q_z, 3p_xx, 3pi_xx, p_ww, pi_ww, p_xy, p_yz, p_xz, m_x, m_y, m_z
  const double tau[Q] = {cp.tau_rho, cp.tau_e, cp.tau_eps, cp.tau_j, cp.tau_q, cp.tau_j,
                         cp.tau_q,   cp.tau_j, cp.tau_q,   cp.tau_s, cp.tau_eps, cp.tau_s,
                         cp.tau_eps, cp.tau_s, cp.tau_s,   cp.tau_s, cp.tau_q,   cp.tau_q,
                         cp.tau_q};
  cudaError_t e = cudaSuccess;
  const size_t es = p.precision == LBM_FP64 ? 8 : 4;
  const size_t fbytes = (19 * static_cast<size_t>(h->plane) + (n_links + 63) / 64 * 64) * es;
  auto alloc = [&](void **ptr, size_t bytes) {
    h->dev_bytes += static_cast<int64_t>(std::max<size_t>(bytes, 16));
    return cudaMalloc(ptr, std::max<size_t>(bytes, 16));
  };
  if (e == cudaSuccess) e = alloc(&h->f[0], fbytes);
  if (e == cudaSuccess) e = alloc(&h->f[1], fbytes);
  if (e == cudaSuccess) e = alloc(reinterpret_cast<void **>(&h->flags), n * 4);
  if (e == cudaSuccess) e = alloc(reinterpret_cast<void **>(&h->lbase), n * 4);
  if (e == cudaSuccess) e = alloc(&h->links, std::max<size_t>(1, n_links) * 4 * es);
  if (e == cudaSuccess)
    e = alloc(reinterpret_cast<void **>(&h->partials), kResBlocks3 * 4 * sizeof(double));
  if (e == cudaSuccess) e = alloc(reinterpret_cast<void **>(&h->result), 4 * sizeof(double));
  if (e == cudaSuccess) e = cudaMemset(h->f[0], 0, fbytes);
  if (e == cudaSuccess) e = cudaMemset(h->f[1], 0, fbytes);
  if (e == cudaSuccess) e = cudaMemcpy(h->flags, flags.data(), n * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(h->lbase, lbase.data(), n * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    std::vector<uint2> fluid(static_cast<size_t>(n_fluid));
    std::vector<uint32_t> gbase(static_cast<size_t>((n_fluid + 31) / 32));
    std::vector<uint16_t> ldesc(std::max<size_t>(1, n_links));
    uint32_t i = 0, l = 0;  // fluid nodes and links so far
    for (int64_t pn = 0; pn < n; pn++) {
      const uint32_t fl = flags[pn];
      if (fl == kSolid3) continue;
      const uint32_t at = i % 32;
      if (at == 0) gbase[i / 32] = l;
      // (at most 31 x 18 links precede it in its group)
      fluid[i] = make_uint2(static_cast<uint32_t>(pn), fl | (l - gbase[i / 32]) << kRank3);
      i++;
      for (uint32_t m = fl; m; m &= m - 1u)
        ldesc[l++] = static_cast<uint16_t>(at << 5 | static_cast<uint32_t>(__builtin_ctz(m)));
    }
    e = alloc(reinterpret_cast<void **>(&h->fluid), std::max<size_t>(1, fluid.size()) * 8);
    if (e == cudaSuccess)
      e = alloc(reinterpret_cast<void **>(&h->gbase), std::max<size_t>(1, gbase.size()) * 4);
    if (e == cudaSuccess) e = alloc(reinterpret_cast<void **>(&h->ldesc), ldesc.size() * 2);
    if (e == cudaSuccess && !fluid.empty())
      e = cudaMemcpy(h->fluid, fluid.data(), fluid.size() * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !gbase.empty())
      e = cudaMemcpy(h->gbase, gbase.data(), gbase.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = cudaMemcpy(h->ldesc, ldesc.data(), ldesc.size() * 2, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess)
    e = dispatch3(h->precision, [&](auto tag) {
      using C = std::remove_pointer_t<decltype(tag)>;
      std::vector<Link3<C>> lk(std::max<size_t>(1, n_links));
      for (size_t k = 0; k < n_links; k++) {
        const double *cf = &coef[8 * k];
        lk[slot[k]] = Link3<C>{static_cast<C>(cf[0]), static_cast<C>(cf[1]), static_cast<C>(cf[2]),
                               static_cast<C>(cf[3])};
      }
      // the case's constants in each arithmetic type
      auto fill = [&](auto &kc) {
        using A = std::remove_reference_t<decltype(kc.ax)>;
        for (int a = 0; a < Q; a++) {
          const double s = 1.0 / tau[a];
          kc.s_scaled[a] = static_cast<A>(s / L.norm[a]);
          kc.f_scaled[a] = static_cast<A>((1.0 - 0.5 * s) / L.norm[a]);
        }
        kc.ax = static_cast<A>(dom->ax);
        kc.ay = static_cast<A>(dom->ay);
        kc.az = static_cast<A>(dom->az);
        kc.nx = nx;
        kc.ny = ny;
        kc.nz = nz;
        kc.px = per[0];
        kc.py = per[1];
        kc.pz = per[2];
        kc.by_nx = DivBy3(static_cast<uint32_t>(nx));
        kc.by_ny = DivBy3(static_cast<uint32_t>(ny));
        kc.diffuse_mode = p.diffuse_mode;
        kc.plane = h->plane;
        kc.n_links = h->n_links;
        kc.sr_seed = 0u;
      };
      fill(h->kc.f);
      fill(h->kc.d);
      return cudaMemcpy(h->links, lk.data(), lk.size() * sizeof(Link3<C>), cudaMemcpyHostToDevice);
    });
  // the exact-mass variant (FP32): where mass_mode asks for it, or by
  // default where a wall moves or the lattice has no boundary links
  bool moving = false;
  for (size_t k = 0; k < 3 * n_links && !moving; k++) moving = link_ub[k] != 0.0;
  h->exact = p.precision == LBM_FP32 && p.mass_mode >= 0 &&
             (p.mass_mode > 0 || moving || n_links == 0);
  if (e == cudaSuccess && h->exact) {
    const double acc[3] = {dom->ax, dom->ay, dom->az};
    for (int a = 0; a < 3; a++) h->force.a[a] = df_of(acc[a]);
    std::vector<lbm::LinkCoefDF> ldf(std::max<size_t>(1, n_links));
    for (size_t k = 0; k < n_links; k++) ldf[slot[k]] = lbm::link_coef_df(&coef[8 * k], wq[k], p.diffuse_mode);
    e = alloc(reinterpret_cast<void **>(&h->links_df), ldf.size() * sizeof(lbm::LinkCoefDF));
    if (e == cudaSuccess)
      e = cudaMemcpy(h->links_df, ldf.data(), ldf.size() * sizeof(lbm::LinkCoefDF),
                     cudaMemcpyHostToDevice);
    const size_t nc = std::max<size_t>(1, n_links) + static_cast<size_t>(n_fluid);
    if (e == cudaSuccess) e = alloc(reinterpret_cast<void **>(&h->carry), nc * 4);
    if (e == cudaSuccess) e = cudaMemset(h->carry, 0, nc * 4);
  }
  if (e != cudaSuccess) {
    const int code = e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
    g_err3 = std::string("device setup: ") + cudaGetErrorString(e);
    release3(h);
    return code;
  }
  *out = h;
  return LBM_OK;
}

int lbm3d_step(lbm3d_t *h, int64_t n) {
  using namespace lbm3;
  if (!h) return LBM_EINVAL;
  if (n < 0) return fail3(h, LBM_EINVAL, "negative step count");
  for (int64_t s = 0; s < n; s++) {
    const int src = h->cur, dst = 1 - h->cur;
    cudaError_t e = dispatch3(h->precision, [&](auto tag) {
      using C = std::remove_pointer_t<decltype(tag)>;
      if (h->n_fluid == 0) return cudaSuccess;
      const dim3 blocks(static_cast<unsigned>((h->n_fluid + kThreads3 - 1) / kThreads3));
      Const3<C> kc = h->kc.get(tag);
      kc.sr_seed = lbm::dev::step_seed(h->steps);
      auto go = [&](auto *kernel) {
        return lbm::launch_chained(kernel, blocks, kThreads3, 0, h->stream,
                                   static_cast<const C *>(h->f[src]), static_cast<C *>(h->f[dst]),
                                   h->gbase, h->ldesc, static_cast<const Link3<C> *>(h->links),
                                   h->fluid, kc, h->n_fluid, h->links_df, h->carry, h->force);
      };
      const bool small = 19 * h->plane + h->n_links < (int64_t(1) << 32);
      if constexpr (std::is_same<C, float>::value) {
        if (h->exact)
          return small ? go(step3_kernel<C, true, uint32_t>) : go(step3_kernel<C, true, int64_t>);
      }
      return small ? go(step3_kernel<C, false, uint32_t>) : go(step3_kernel<C, false, int64_t>);
    });
    if (e != cudaSuccess) return fail3(h, LBM_ECUDA, std::string("step: ") + cudaGetErrorString(e));
    h->cur = dst;
    h->steps++;
  }
  return LBM_OK;
}

int lbm3d_residual(lbm3d_t *h, double *residual, double *mass) {
  using namespace lbm3;
  if (!h) return LBM_EINVAL;
  double tot[4];
  cudaError_t e = dispatch3(h->precision, [&](auto tag) {
    using C = std::remove_pointer_t<decltype(tag)>;
    residual3_kernel<C><<<kResBlocks3, kResThreads3, 0, h->stream>>>(
        static_cast<const C *>(h->f[h->cur]), static_cast<const C *>(h->f[1 - h->cur]), h->gbase,
        h->fluid, h->kc.get(tag), h->n_fluid, h->partials);
    residual3_final<<<1, 1024, 0, h->stream>>>(h->partials, h->result);
    return cudaGetLastError();
  });
  if (e == cudaSuccess) e = cudaMemcpyAsync(tot, h->result, sizeof tot, cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return fail3(h, LBM_ECUDA, std::string("residual: ") + cudaGetErrorString(e));
  double res;
  if (std::isnan(tot[0]) || std::isnan(tot[1])) res = std::numeric_limits<double>::quiet_NaN();
  else res = tot[1] > 0.0 ? std::sqrt(tot[0] / tot[1]) : (tot[0] > 0.0 ? INFINITY : 0.0);
  if (residual) *residual = res;
  if (mass) *mass = static_cast<double>(h->n_fluid) + tot[2];
  if (tot[3] > 0.0) return fail3(h, LBM_EUNSTABLE, "fluid nodes with non-finite density or velocity");
  return LBM_OK;
}

int lbm3d_get_f(lbm3d_t *h, double *f) {
  using namespace lbm3;
  if (!h || !f) return h ? fail3(h, LBM_EINVAL, "null output") : LBM_EINVAL;
  double *d = nullptr;
  const size_t bytes = static_cast<size_t>(Q) * h->n_nodes * sizeof(double);
  cudaError_t e = cudaMalloc(&d, bytes);
  if (e == cudaSuccess)
    e = dispatch3(h->precision, [&](auto tag) {
      using C = std::remove_pointer_t<decltype(tag)>;
      export3_kernel<C><<<grid_for3(h->n_nodes, 256), 256, 0, h->stream>>>(
          static_cast<const C *>(h->f[h->cur]), h->flags, h->lbase, h->kc.get(tag), h->n_nodes, d);
      return cudaGetLastError();
    });
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e == cudaSuccess) e = cudaMemcpy(f, d, bytes, cudaMemcpyDeviceToHost);
  if (d) cudaFree(d);
  if (e != cudaSuccess) return fail3(h, LBM_ECUDA, std::string("get_f: ") + cudaGetErrorString(e));
  return LBM_OK;
}

int lbm3d_set_f(lbm3d_t *h, const double *f) {
  using namespace lbm3;
  if (!h || !f) return h ? fail3(h, LBM_EINVAL, "null input") : LBM_EINVAL;
  double *d = nullptr;
  const size_t bytes = static_cast<size_t>(Q) * h->n_nodes * sizeof(double);
  cudaError_t e = cudaMalloc(&d, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(d, f, bytes, cudaMemcpyHostToDevice);
  for (int b = 0; b < 2 && e == cudaSuccess; b++)
    e = dispatch3(h->precision, [&](auto tag) {
      using C = std::remove_pointer_t<decltype(tag)>;
      import3_kernel<C><<<grid_for3(h->n_nodes, 256), 256, 0, h->stream>>>(
          d, h->flags, h->lbase, h->kc.get(tag), h->n_nodes, static_cast<C *>(h->f[b]));
      return cudaGetLastError();
    });
  if (e == cudaSuccess && h->carry)  // a new state owes no carries
    e = cudaMemsetAsync(h->carry, 0, (std::max<int64_t>(1, h->n_links) + h->n_fluid) * 4,
                        h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (d) cudaFree(d);
  if (e != cudaSuccess) return fail3(h, LBM_ECUDA, std::string("set_f: ") + cudaGetErrorString(e));
  h->steps = 0;
  return LBM_OK;
}

int lbm3d_fields(lbm3d_t *h, double *rho, double *ux, double *uy, double *uz) {
  using namespace lbm3;
  if (!h) return LBM_EINVAL;
  double *d = nullptr;
  const size_t n = static_cast<size_t>(h->n_nodes);
  cudaError_t e = cudaMalloc(&d, 4 * n * sizeof(double));
  if (e == cudaSuccess)
    e = dispatch3(h->precision, [&](auto tag) {
      using C = std::remove_pointer_t<decltype(tag)>;
      fields3_kernel<C><<<grid_for3(h->n_nodes, 256), 256, 0, h->stream>>>(
          static_cast<const C *>(h->f[h->cur]), h->flags, h->lbase, h->kc.get(tag),
          HalfAccel3{{0.5 * h->ax, 0.5 * h->ay, 0.5 * h->az}}, h->n_nodes, d);
      return cudaGetLastError();
    });
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  double *outs[4] = {rho, ux, uy, uz};
  for (int a = 0; a < 4 && e == cudaSuccess; a++)
    if (outs[a]) e = cudaMemcpy(outs[a], d + a * n, n * sizeof(double), cudaMemcpyDeviceToHost);
  if (d) cudaFree(d);
  if (e != cudaSuccess) return fail3(h, LBM_ECUDA, std::string("fields: ") + cudaGetErrorString(e));
  return LBM_OK;
}

int lbm3d_link_params(const lbm3d_t *h, double *r, double *l) {
  if (!h) return LBM_EINVAL;
  if (r) std::copy(h->link_r.begin(), h->link_r.end(), r);
  if (l) std::copy(h->link_l.begin(), h->link_l.end(), l);
  return LBM_OK;
}

int lbm3d_get_info(const lbm3d_t *h, lbm_info_t *info) {
  if (!h || !info) return LBM_EINVAL;
  *info = lbm_info_t{};
  info->n_nodes = h->n_nodes;
  info->n_fluid = h->n_fluid;
  info->n_links = h->n_links;
  info->steps = h->steps;
  info->tau_s = h->cp.tau_s;
  info->tau_q = h->cp.tau_q;
  info->E = h->cp.E;
  info->E_max = h->cp.E_max;
  info->L1 = h->cp.L1;
  info->L2 = h->cp.L2;
  info->n_clamped = h->cp.n_clamped;
  info->device_bytes = h->dev_bytes;
  info->precision = h->precision;
  info->pitch = h->nx;
  info->exact_mass = h->exact;
  return LBM_OK;
}

void lbm3d_destroy(lbm3d_t *h) { release3(h); }

const char *lbm3d_last_error(const lbm3d_t *h) { return h ? h->err.c_str() : g_err3.c_str(); }

}  // extern "C"
