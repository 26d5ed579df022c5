// Setup kernel: FP64 corrections C_ts = N_ts - Q_ts for near element pairs.
//
// N_ts (near rule) = (1/4pi) int_t psi_s(x) dx with psi_s the closed-form
// potential of the uniform source element, integrated over the target by a
// composite collapsed Gauss-Legendre rule (target refined k times: a tet
// into 8 children with the inner octahedron cut along the x02-x13 diagonal,
// a triangle into its 4 midpoint children).  Q_ts is the product rule the
// point passes apply to the same pair (self point r = 0 skipped).  This is
// the library's own evaluation of the near field of Sec. 3.3; the paper's
// singularity-removing transforms are replaced by the closed-form inner
// integral.
#include <cmath>
#include <cstring>

#include "kernels.cuh"

namespace bcfmm {

constexpr double kInv4PiN = 0.079577471545947667884441881686257;

struct V3 { double x, y, z; };
__device__ __forceinline__ V3 vsub(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double vdot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 vcross(V3 a, V3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }
__device__ __forceinline__ V3 vscale(V3 a, double s) { return {a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ V3 vmid(V3 a, V3 b) { return {0.5 * (a.x + b.x), 0.5 * (a.y + b.y), 0.5 * (a.z + b.z)}; }

// int_T ds_y / |x - y| over the flat triangle (A, B, C): edge terms
// d_e ln((t2 + R2)/(t1 + R1)) from the in-plane divergence theorem, minus
// |w| times the solid angle (Van Oosterom-Strackee) for the height w.
__device__ double tri_pot(V3 x, const V3* P) {
  V3 n = vcross(vsub(P[1], P[0]), vsub(P[2], P[0]));
  const double nn = sqrt(vdot(n, n));
  n = vscale(n, 1.0 / nn);
  const double w = vdot(vsub(x, P[0]), n);
  const V3 rho = vsub(x, vscale(n, w));
  const double scale = sqrt(nn);
  double acc = 0.0;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const V3 A = P[e], B = P[(e + 1) % 3];
    V3 t = vsub(B, A);
    const double Lt = sqrt(vdot(t, t));
    t = vscale(t, 1.0 / Lt);
    const V3 m = vcross(t, n);
    const double d = vdot(vsub(A, rho), m);
    if (fabs(d) <= 1e-14 * scale) continue;
    const V3 ax = vsub(A, x), bx = vsub(B, x);
    const double t1 = vdot(ax, t), t2 = vdot(bx, t);
    const double R1 = sqrt(vdot(ax, ax)), R2 = sqrt(vdot(bx, bx));
    const double lg = (t1 + t2 >= 0.0) ? log((R2 + t2) / (R1 + t1)) : log((R1 - t1) / (R2 - t2));
    acc += d * lg;
  }
  const V3 r1 = vsub(P[0], x), r2 = vsub(P[1], x), r3 = vsub(P[2], x);
  const double l1 = sqrt(vdot(r1, r1)), l2 = sqrt(vdot(r2, r2)), l3 = sqrt(vdot(r3, r3));
  const double num = vdot(r1, vcross(r2, r3));
  const double den = l1 * l2 * l3 + vdot(r1, r2) * l3 + vdot(r1, r3) * l2 + vdot(r2, r3) * l1;
  const double omega = 2.0 * atan2(num, den);
  return acc - fabs(w) * fabs(omega);
}

// int_T n.(x-y)/|x-y|^3 ds_y over the flat triangle with normal
// n = (P1-P0) x (P2-P0) / |.|: the solid angle T subtends at x, signed
// positive on the side n points to (for y in the plane n.(x-y) is the
// height of x).  Van Oosterom-Strackee: tan(Omega/2) = r1.(r2 x r3) /
// (l1 l2 l3 + (r1.r2) l3 + (r1.r3) l2 + (r2.r3) l1), r_i = P_i - x; the
// triple product is negative for x on the + side, hence the minus sign.
__device__ double tri_solid(V3 x, const V3* P) {
  const V3 r1 = vsub(P[0], x), r2 = vsub(P[1], x), r3 = vsub(P[2], x);
  const double l1 = sqrt(vdot(r1, r1)), l2 = sqrt(vdot(r2, r2)), l3 = sqrt(vdot(r3, r3));
  const double num = vdot(r1, vcross(r2, r3));
  const double den = l1 * l2 * l3 + vdot(r1, r2) * l3 + vdot(r1, r3) * l2 + vdot(r2, r3) * l1;
  return -2.0 * atan2(num, den);
}

// int_tet dy/|x-y| = 1/2 sum_F h_F(x) I_F(x), h_F = n_F.(y_F - x), n_F
// outward, with I_F the flat-triangle integral above.  Everything that does
// not depend on x (edge lengths, face normals, in-plane edge normals) is
// prepared once per pair by the warp, and the quantities faces share (vertex
// distances and their products, the log term of each of the 6 edges) are
// computed once per point.
//
// FP64 instructions are what this costs (two lanes a cycle and SM), so the
// two transcendental functions are tabulated with one short division each:
//  - edge term: ln((R_a + t_a) / (R_b + t_b)) along the edge equals
//    ln((S + l) / (S - l)), S = R_a + R_b, l the edge length (both numerators
//    are squares' differences over the same (S - l)); ln(a / b) = ln c + 2
//    artanh((a - c b) / (a + c b)) with c the nearest of 33 table points in
//    [1, 2] to the ratio of the mantissas, artanh by its Taylor series
//    (|z| <= 1/127: terms to z^7, the next, z^8 / 9 of z, is below 2^-59);
//  - solid angle: tan(Omega / 2) = |h| 2A / den; atan(y / x) = atan c +
//    atan((y - c x) / (x + c y)), c the nearest of 65 points in [0, 1],
//    again by Taylor's series to z^7 (|z| <= 1/127).
// This is the table-driven scheme of P. T. P. Tang (ACM Trans. Math. Softw. 16,
// 1990) with the functions' addition theorems in place of his products.  Errors:
// the difference a - c b is one FMA, so z is off by at most three roundings
// (sum, quotient, difference), and the result by at most four of 2^-52: for c = 1
// (0) the result is the series itself, else the table's value is at least as
// large as the series' part of it.  The table entries (ln c, atan c) come from
// the host's libm.
__device__ constexpr int kTetEdge[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
__device__ constexpr int kTetFace[4][3] = {{1, 2, 3}, {0, 3, 2}, {0, 1, 3}, {0, 2, 1}};
__device__ constexpr int kFaceEdge[4][3] = {{3, 5, 4}, {2, 5, 1}, {0, 4, 2}, {1, 3, 0}};   // edge of (F[j], F[j+1])
__constant__ int c_tet_edge[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
__constant__ int c_tet_face[4][3] = {{1, 2, 3}, {0, 3, 2}, {0, 1, 3}, {0, 2, 1}};

constexpr int kLogTab = 33, kAtanTab = 65;
struct NearTabs {
  double2 lg[kLogTab];     // (c, ln c), c = 1 + i / 32
  double at[kAtanTab];     // atan(i / 64)
};

struct SrcTet {
  V3 v[4];
  double len[6];       // length of edge k
  V3 nout[4];          // outward unit normal of face f
  V3 nf[4];            // unit normal of the face's vertex order
  double nn[4];        // twice the face's area
  V3 m[4][3];          // in-plane outward normal of the face's edge j (vertex order of the face)
  double thr[4];       // |d| below this: x on the edge's line within the face plane
};

// the warp prepares S from the vertices v (12 doubles)
__device__ __forceinline__ void src_tet_prepare(const double* __restrict__ v, SrcTet& S, int lane) {
  if (lane < 12) (&S.v[0].x)[lane] = v[lane];
  __syncwarp();
  if (lane < 6) {
    const V3 t = vsub(S.v[c_tet_edge[lane][1]], S.v[c_tet_edge[lane][0]]);
    const double l = sqrt(vdot(t, t));
    S.len[lane] = l;
  } else if (lane >= 8 && lane < 12) {
    const int f = lane - 8;
    V3 cen = {0, 0, 0};
    for (int i = 0; i < 4; ++i) { cen.x += 0.25 * S.v[i].x; cen.y += 0.25 * S.v[i].y; cen.z += 0.25 * S.v[i].z; }
    const V3 T0 = S.v[c_tet_face[f][0]], T1 = S.v[c_tet_face[f][1]], T2 = S.v[c_tet_face[f][2]];
    V3 n = vcross(vsub(T1, T0), vsub(T2, T0));
    const double nn = sqrt(vdot(n, n));
    n = vscale(n, 1.0 / nn);             // normal of the face's vertex order
    S.nn[f] = nn;
    S.thr[f] = 1e-14 * sqrt(nn);
    S.nf[f] = n;
    S.nout[f] = vdot(vsub(T0, cen), n) < 0 ? vscale(n, -1.0) : n;
  }
  __syncwarp();
  if (lane < 12) {
    const int f = lane / 3, j = lane - 3 * f;
    V3 t = vsub(S.v[c_tet_face[f][j == 2 ? 0 : j + 1]], S.v[c_tet_face[f][j]]);
    t = vscale(t, 1.0 / sqrt(vdot(t, t)));
    S.m[f][j] = vcross(t, S.nf[f]);
  }
  __syncwarp();
}

// n / d, both normal and the quotient far from the ends of the range: one step r <-
// r + r (1 - d r) of Newton's iteration for 1 / d from the hardware's approximation
// (twenty bits: e0 about 2^-19, so e0^2 = 2^-38 after it), then Markstein's
// correction of the quotient z = n r by its residual, z + r (n - d z) (IBM J. Res.
// Dev. 34, 1990): the residual is one FMA, so its own error is 2^-53 of 2^-38, and
// the quotient is within one unit of 2^-52.
__device__ __forceinline__ double div_nr(double n, double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  r = fma(r, fma(-d, r, 1.0), r);
  const double z = n * r;
  return fma(fma(-d, z, n), r, z);
}

// mantissa in [1, 2) of a positive double, to 20 bits
__device__ __forceinline__ float mant_f(int hi) { return __int_as_float(0x3f800000 | ((hi & 0xfffff) << 3)); }

// ln(a / b), a >= b > 0
__device__ __forceinline__ double log_ratio(double a, double b, const NearTabs& T) {
  const int ha = __double2hiint(a), hb = __double2hiint(b);
  int k = (ha >> 20) - (hb >> 20);
  float rm = __fdividef(mant_f(ha), mant_f(hb));          // in (1/2, 2)
  int up = 0;
  // (k = 0: the mantissas' ratio is at least 1, whatever their leading bits give;
  // ln 2 would cancel against the table's)
  if (rm < 1.f && k > 0) { rm *= 2.f; k -= 1; up = 1 << 20; }
  const int i = min(kLogTab - 1, (int)fmaf(rm - 1.f, 32.f, 0.5f));
  const double2 c = T.lg[i];
  const double am = __hiloint2double(((ha & 0xfffff) | 0x3ff00000) + up, __double2loint(a));
  const double bm = __hiloint2double((hb & 0xfffff) | 0x3ff00000, __double2loint(b));
  const double z = div_nr(fma(-c.x, bm, am), fma(c.x, bm, am));
  const double z2 = z * z, t = z + z;
  double s = fma(t * z2, fma(z2, fma(z2, 1.0 / 7, 1.0 / 5), 1.0 / 3), t);
  s += c.y;
  // k as a double by its bits (2^52 + 2^31 + k)
  const double kd = __hiloint2double(0x43300000, (int)(0x80000000u + (unsigned)k)) - 4503601774854144.0;
  return k ? fma(kd, 0.69314718055994530942, s) : s;
}

// atan2(y, x) for y > 0
__device__ __forceinline__ double atan_pos(double y, double x, const NearTabs& T) {
  const double ax = fabs(x);
  const int hy = __double2hiint(y), hx = __double2hiint(ax);
  const bool sw = hy > hx;
  const double num = sw ? ax : y, den = sw ? y : ax;
  const int hn = sw ? hx : hy, hd = sw ? hy : hx;
  const int diff = (hn >> 20) - (hd >> 20);               // <= 0
  const float t = diff < -20 ? 0.f : __fdividef(mant_f(hn), mant_f(hd)) * __int_as_float((127 + diff) << 23);
  const int i = min(kAtanTab - 1, (int)fmaf(t, 64.f, 0.5f));
  const double c = (double)((float)i * (1.f / 64));
  const double z = div_nr(fma(-c, den, num), fma(c, num, den));
  const double z2 = z * z;
  double r = fma(z * z2, fma(z2, fma(z2, -1.0 / 7, 1.0 / 5), -1.0 / 3), z) + T.at[i];
  if (sw) r = 1.57079632679489661923 - r;
  return x < 0 ? 3.14159265358979323846 - r : r;
}

__device__ __forceinline__ double tet_pot(V3 x, const SrcTet& S, const NearTabs& T) {
  V3 r[4];
  double R[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { r[i] = vsub(S.v[i], x); R[i] = sqrt(vdot(r[i], r[i])); }
  double L[6], rr[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int a = kTetEdge[k][0], b = kTetEdge[k][1];
    const double s = R[a] + R[b], l = S.len[k];
    // (s - l = 0: x on the edge, whose distance d is below the threshold)
    L[k] = log_ratio(s + l, fmax(s - l, 0x1p-60 * s), T);
    rr[k] = vdot(r[a], r[b]);
  }
  double acc = 0.0;
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int i0 = kTetFace[f][0], i1 = kTetFace[f][1], i2 = kTetFace[f][2];
    const double h = vdot(S.nout[f], r[i0]);
    double e = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double d = vdot(r[kTetFace[f][j]], S.m[f][j]);
      if (fabs(d) > S.thr[f]) e = fma(d, L[kFaceEdge[f][j]], e);
    }
    // edges (i0, i1), (i1, i2), (i2, i0) of the face
    const double den = fma(R[i0] * R[i1], R[i2],
                           fma(rr[kFaceEdge[f][0]], R[i2], fma(rr[kFaceEdge[f][2]], R[i1], rr[kFaceEdge[f][1]] * R[i0])));
    const double ah = fabs(h);
    if (h != 0.0) acc = fma(0.5 * h, e - ah * (2.0 * atan_pos(ah * S.nn[f], den, T)), acc);
  }
  return acc;
}

__device__ double tet_vol6(const V3* v) {
  return fabs(vdot(vcross(vsub(v[1], v[0]), vsub(v[2], v[0])), vsub(v[3], v[0])));
}
__device__ double tri_area2(const V3* v) {
  const V3 n = vcross(vsub(v[1], v[0]), vsub(v[2], v[0]));
  return sqrt(vdot(n, n));
}

// children as pairs of parent vertices (i == j: the vertex, else the midpoint)
__constant__ int c_tet_child[8][4][2] = {
    {{0, 0}, {0, 1}, {0, 2}, {0, 3}}, {{0, 1}, {1, 1}, {1, 2}, {1, 3}},
    {{0, 2}, {1, 2}, {2, 2}, {2, 3}}, {{0, 3}, {1, 3}, {2, 3}, {3, 3}},
    {{0, 1}, {0, 2}, {0, 3}, {1, 3}}, {{0, 1}, {0, 2}, {1, 2}, {1, 3}},
    {{0, 2}, {0, 3}, {1, 3}, {2, 3}}, {{0, 2}, {1, 2}, {1, 3}, {2, 3}}};
__constant__ int c_tri_child[4][3][2] = {
    {{0, 0}, {0, 1}, {2, 0}}, {{0, 1}, {1, 1}, {1, 2}}, {{2, 0}, {1, 2}, {2, 2}}, {{0, 1}, {1, 2}, {2, 0}}};

constexpr int kMaxGL = 8;
constexpr int kNearPairs = 64;       // pairs per CTA
constexpr int kNearPts = 256;        // outer points staged per round

struct NearRuleArgs {
  const int64_t* sel;
  const int *row, *col;
  const double *tgt_v, *src_v, *tgt_qp, *tgt_qw, *src_qp, *src_qw, *glx, *glw;
  double* cor_val;
  const NearTabs* tabs;
  int64_t nnz;
  int n, k, compact;
};

// outer point idx of target element v (nvt vertices) and its weight
template <bool TGT_TET>
__device__ __forceinline__ void outer_point(const V3* tv, const double* gx, const double* gw, int n, int k, int npc,
                                            int npieces, int idx, V3& x, double& wt) {
  constexpr int nvt = TGT_TET ? 4 : 3, nch = TGT_TET ? 8 : 4;
  const int piece = idx / npc, q = idx % npc;
  // descend k levels (most significant digit = first refinement)
  V3 v[4] = {tv[0], tv[1], tv[2], tv[TGT_TET ? 3 : 0]};
  int div = npieces;
  for (int lev = 0; lev < k; ++lev) {
    div /= nch;
    const int c = (piece / div) % nch;
    V3 w[4];
    for (int i = 0; i < nvt; ++i) {
      const int a = TGT_TET ? c_tet_child[c][i][0] : c_tri_child[c][i][0];
      const int b = TGT_TET ? c_tet_child[c][i][1] : c_tri_child[c][i][1];
      w[i] = (a == b) ? v[a] : vmid(v[a], v[b]);
    }
    for (int i = 0; i < nvt; ++i) v[i] = w[i];
  }
  if (TGT_TET) {
    const int ia = q / (n * n), ib = (q / n) % n, ic = q % n;
    const double u = gx[ia], vv = gx[ib], ww = gx[ic];
    const double x1 = u, x2 = (1 - u) * vv, x3 = (1 - u) * (1 - vv) * ww;
    const double jac = (1 - u) * (1 - u) * (1 - vv);
    x.x = v[0].x + x1 * (v[1].x - v[0].x) + x2 * (v[2].x - v[0].x) + x3 * (v[3].x - v[0].x);
    x.y = v[0].y + x1 * (v[1].y - v[0].y) + x2 * (v[2].y - v[0].y) + x3 * (v[3].y - v[0].y);
    x.z = v[0].z + x1 * (v[1].z - v[0].z) + x2 * (v[2].z - v[0].z) + x3 * (v[3].z - v[0].z);
    wt = gw[ia] * gw[ib] * gw[ic] * jac * tet_vol6(v);
  } else {
    const int ia = q / n, ib = q % n;
    const double u = gx[ia], vv = gx[ib];
    const double x1 = u, x2 = (1 - u) * vv, jac = 1 - u;
    x.x = v[0].x + x1 * (v[1].x - v[0].x) + x2 * (v[2].x - v[0].x);
    x.y = v[0].y + x1 * (v[1].y - v[0].y) + x2 * (v[2].y - v[0].y);
    x.z = v[0].z + x1 * (v[1].z - v[0].z) + x2 * (v[2].z - v[0].z);
    wt = gw[ia] * gw[ib] * jac * tri_area2(v);
  }
}

// this lane's part of the product rule of the point passes for the pair (t, s):
// target point lane / nvs, source point lane % nvs (lanes beyond nvt nvs: zero)
template <bool TGT_TET, int SRC>
__device__ __forceinline__ double product_term(const NearRuleArgs& A, int t, int s, int lane) {
  constexpr int nvt = TGT_TET ? 4 : 3, nvs = SRC == 0 ? 4 : 3;
  if (lane >= nvt * nvs) return 0.0;
  const int ti = lane / nvs, sj = lane % nvs;
  const double* xp = A.tgt_qp + 3 * ((int64_t)t * nvt + ti);
  const double* yp = A.src_qp + 3 * ((int64_t)s * nvs + sj);
  const double dx = xp[0] - yp[0], dy = xp[1] - yp[1], dz = xp[2] - yp[2];
  const double r = sqrt(dx * dx + dy * dy + dz * dz);
  if (r == 0.0) return 0.0;
  double q = A.tgt_qw[(int64_t)t * nvt + ti] * A.src_qw[(int64_t)s * nvs + sj] * kInv4PiN / r;
  if constexpr (SRC == 2) {
    const double* svp = A.src_v + (int64_t)s * 3 * nvs;
    const V3 e0 = {svp[3] - svp[0], svp[4] - svp[1], svp[5] - svp[2]}, e1 = {svp[6] - svp[0], svp[7] - svp[1], svp[8] - svp[2]};
    V3 ns = vcross(e0, e1);
    ns = vscale(ns, 1.0 / sqrt(vdot(ns, ns)));
    q *= (ns.x * dx + ns.y * dy + ns.z * dz) / (r * r);
  }
  return q;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 64 consecutive pairs of the CSR (or of the selection list) per CTA.  The
// pairs of one target share its outer points, staged in shared memory; a warp
// takes one pair at a time, its lanes the outer points.  SRC: 0 tets, 1
// triangles (single layer), 2 triangles (double layer, kernel dG/dn_y).  The
// result of pair ii (CSR position k = sel[ii], or ii without a selection)
// goes to cor_val[k].
// Bound by the FP64 pipe: 216 points x about 400 FP64 instructions a pair of
// tets (about 750 with libm's functions, the outer points computed anew for
// every pair and the source tet prepared by one lane).  Build of a 3,072-tet
// cube, default rule, 467,000 pairs: 184 -> 102 ms.  Against extended
// precision the potential's error is as before (rms 9e-15 around the tet,
// 6e-16 inside, both forms).
template <bool TGT_TET, int SRC>
__global__ void __launch_bounds__(128) k_near_rule(NearRuleArgs A) {
  constexpr int nvt = TGT_TET ? 4 : 3, nvs = SRC == 0 ? 4 : 3, nch = TGT_TET ? 8 : 4;
  __shared__ double4_32a pts[kNearPts];        // outer points x, y, z, weight
  __shared__ double part[kNearPairs];           // sums of the rounds so far
  __shared__ SrcTet sS[SRC == 0 ? 4 : 1];
  __shared__ NearTabs tabs;
  __shared__ double gx[kMaxGL], gw[kMaxGL];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t p0 = (int64_t)blockIdx.x * kNearPairs;
  const int np = (int)min((int64_t)kNearPairs, A.nnz - p0);
  if (SRC == 0) {
    const double* src = reinterpret_cast<const double*>(A.tabs);
    for (int i = threadIdx.x; i < (int)(sizeof(NearTabs) / sizeof(double)); i += 128) reinterpret_cast<double*>(&tabs)[i] = src[i];
  }
  if (threadIdx.x < A.n) { gx[threadIdx.x] = A.glx[threadIdx.x]; gw[threadIdx.x] = A.glw[threadIdx.x]; }
  int npc = TGT_TET ? A.n * A.n * A.n : A.n * A.n, npieces = 1;
  for (int i = 0; i < A.k; ++i) npieces *= nch;
  const int total = npieces * npc;
  auto pos = [&](int i) { return A.sel ? A.sel[p0 + i] : p0 + i; };
  for (int a = 0; a < np;) {
    const int t = A.row[pos(a)];
    int b = a + 1;
    while (b < np && A.row[pos(b)] == t) ++b;            // (the same for every thread)
    V3 tv[4];
    for (int i = 0; i < nvt; ++i) {
      const double* q = A.tgt_v + ((int64_t)t * nvt + i) * 3;
      tv[i] = {q[0], q[1], q[2]};
    }
    for (int c0 = 0; c0 < total; c0 += kNearPts) {
      const int m = min(kNearPts, total - c0);
      __syncthreads();
      for (int i = threadIdx.x; i < m; i += 128) {
        V3 x;
        double wt;
        outer_point<TGT_TET>(tv, gx, gw, A.n, A.k, npc, npieces, c0 + i, x, wt);
        pts[i] = make_double4_32a(x.x, x.y, x.z, wt);
      }
      __syncthreads();
      for (int i = a + warp; i < b; i += 4) {
        const int64_t kk = pos(i);
        const int s = A.col[kk];
        const double* svp = A.src_v + (int64_t)s * 3 * nvs;
        double sum = 0.0;
        if constexpr (SRC == 0) {
          SrcTet& S = sS[warp];
          __syncwarp();
          src_tet_prepare(svp, S, lane);
          for (int j = lane; j < m; j += 32) {
            const double4_32a q = pts[j];
            sum = fma(q.w, tet_pot({q.x, q.y, q.z}, S, tabs), sum);
          }
        } else {
          V3 sv[3];
          for (int v = 0; v < 3; ++v) sv[v] = {svp[3 * v], svp[3 * v + 1], svp[3 * v + 2]};
          for (int j = lane; j < m; j += 32) {
            const double4_32a q = pts[j];
            const V3 x = {q.x, q.y, q.z};
            sum += q.w * (SRC == 2 ? tri_solid(x, sv) : tri_pot(x, sv));
          }
        }
        sum *= kInv4PiN;
        if (c0 + kNearPts >= total) sum -= product_term<TGT_TET, SRC>(A, t, s, lane);
        sum = warp_sum(sum);
        if (lane == 0) {
          if (c0 > 0) sum += part[i];
          part[i] = sum;
          if (c0 + kNearPts >= total) A.cor_val[kk] = sum;
        }
      }
    }
    a = b;
  }
}

// The same for selections whose neighbouring pairs have different targets (the
// strided samples of a training set): one warp per pair, its lanes compute the
// outer points themselves.  The kernel above would find one pair per target, so
// one warp in four at work, with two barriers a pair.  Cube of 3,072 tets, 2,000
// of its near-singular VtV pairs with features and labels: 7.2 -> 0.76 ms, BtV
// 6.6 -> 0.68 ms; 50,000: 11.5 -> 10.2 and 5.0 -> 3.9 ms.
template <bool TGT_TET, int SRC>
__global__ void __launch_bounds__(128) k_near_rule_each(NearRuleArgs A) {
  constexpr int nvt = TGT_TET ? 4 : 3, nvs = SRC == 0 ? 4 : 3, nch = TGT_TET ? 8 : 4;
  __shared__ SrcTet sS[SRC == 0 ? 4 : 1];
  __shared__ NearTabs tabs;
  __shared__ double gx[kMaxGL], gw[kMaxGL];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (SRC == 0) {
    const double* src = reinterpret_cast<const double*>(A.tabs);
    for (int i = threadIdx.x; i < (int)(sizeof(NearTabs) / sizeof(double)); i += 128) reinterpret_cast<double*>(&tabs)[i] = src[i];
  }
  if (threadIdx.x < A.n) { gx[threadIdx.x] = A.glx[threadIdx.x]; gw[threadIdx.x] = A.glw[threadIdx.x]; }
  __syncthreads();
  const int64_t ii = blockIdx.x * (int64_t)4 + warp;
  if (ii >= A.nnz) return;
  int npc = TGT_TET ? A.n * A.n * A.n : A.n * A.n, npieces = 1;
  for (int i = 0; i < A.k; ++i) npieces *= nch;
  const int total = npieces * npc;
  const int64_t kk = A.sel ? A.sel[ii] : ii;
  const int t = A.row[kk], s = A.col[kk];
  V3 tv[4];
  for (int i = 0; i < nvt; ++i) {
    const double* q = A.tgt_v + ((int64_t)t * nvt + i) * 3;
    tv[i] = {q[0], q[1], q[2]};
  }
  const double* svp = A.src_v + (int64_t)s * 3 * nvs;
  V3 sv[3];
  if constexpr (SRC == 0) src_tet_prepare(svp, sS[warp], lane);
  else
    for (int v = 0; v < 3; ++v) sv[v] = {svp[3 * v], svp[3 * v + 1], svp[3 * v + 2]};
  double sum = 0.0;
  for (int j = lane; j < total; j += 32) {
    V3 x;
    double wt;
    outer_point<TGT_TET>(tv, gx, gw, A.n, A.k, npc, npieces, j, x, wt);
    if constexpr (SRC == 0) sum = fma(wt, tet_pot(x, sS[warp], tabs), sum);
    else sum += wt * (SRC == 2 ? tri_solid(x, sv) : tri_pot(x, sv));
  }
  sum = warp_sum(sum * kInv4PiN - product_term<TGT_TET, SRC>(A, t, s, lane));
  if (lane == 0) A.cor_val[A.compact ? ii : kk] = sum;
}

static NearTabs make_tabs() {
  NearTabs T;
  for (int i = 0; i < kLogTab; ++i) T.lg[i] = make_double2(1.0 + i / 32.0, std::log(1.0 + i / 32.0));
  for (int i = 0; i < kAtanTab; ++i) T.at[i] = std::atan(i / 64.0);
  return T;
}

size_t near_rule_tabs_bytes() { return sizeof(NearTabs); }
void near_rule_tabs_fill(void* host) {
  const NearTabs T = make_tabs();
  std::memcpy(host, &T, sizeof T);
}

// out[i] = a[i] / b[i] (kind 0), ln(a / b) (1), atan2(a, b) (2) by the functions above
__global__ void k_debug_near_math(int kind, int64_t n, const double* __restrict__ a, const double* __restrict__ b,
                                  const NearTabs* __restrict__ tabs, double* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = kind == 0 ? div_nr(a[i], b[i]) : kind == 1 ? log_ratio(a[i], b[i], *tabs) : atan_pos(a[i], b[i], *tabs);
}
cudaError_t launch_debug_near_math(int kind, int64_t n, const double* a, const double* b, const void* tabs, double* out,
                                   cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_debug_near_math<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(kind, n, a, b, static_cast<const NearTabs*>(tabs), out);
  return cudaGetLastError();
}

cudaError_t launch_near_rule(int task, int64_t nnz, const int64_t* sel, const int* row, const int* col,
                             const double* tgt_v, const double* src_v,
                             const double* tgt_qp, const double* tgt_qw,
                             const double* src_qp, const double* src_qw,
                             const double* glx, const double* glw, int n, int k,
                             int compact, const void* tabs, double* cor_val, cudaStream_t st) {
  if (nnz == 0) return cudaSuccess;
  if (n > kMaxGL) return cudaErrorInvalidValue;
  const NearRuleArgs A{sel, row, col, tgt_v, src_v, tgt_qp, tgt_qw, src_qp, src_qw, glx, glw, cor_val,
                       static_cast<const NearTabs*>(tabs), nnz, n, k, compact};
  // compact: the results of a training set's sample (see k_near_rule_each)
  if (compact) {
    const unsigned grid = (unsigned)((nnz + 3) / 4);
    switch (task) {
      case 0: k_near_rule_each<true, 0><<<grid, 128, 0, st>>>(A); break;
      case 1: k_near_rule_each<false, 0><<<grid, 128, 0, st>>>(A); break;
      case 2: k_near_rule_each<true, 1><<<grid, 128, 0, st>>>(A); break;
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  const unsigned grid = (unsigned)((nnz + kNearPairs - 1) / kNearPairs);
  switch (task) {
    case 0: k_near_rule<true, 0><<<grid, 128, 0, st>>>(A); break;
    case 1: k_near_rule<false, 0><<<grid, 128, 0, st>>>(A); break;
    case 2: k_near_rule<true, 1><<<grid, 128, 0, st>>>(A); break;
    case 3: k_near_rule<true, 2><<<grid, 128, 0, st>>>(A); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace bcfmm
