// numeric_const.cuh -- numeric phase of the constant kernel psi = c (included by numeric.cuh, whose
// types it uses).  One kernel, k_const, does a triangle's interior and boundary candidates.
//
// With psi = c the inner integrand c (1, phi_b, phi_b phi_b^T) is quadratic on T_b, and every inner
// rule of the library integrates quadratics exactly, so the rule's sums over a region equal the
// region's moments.  The moments are taken once per region from its boundary, in T_b's own
// barycentric coordinates, instead of point by point over a fan: a whole T_b needs no arithmetic
// beyond its area, and a cut T_b needs the parameters t of its cut edges and one closing chain.
// n_qp_pairs still counts the rule's points, which the sums stand for.
//
// Moments (Mom): with l = (l1, l2) the barycentric coordinates of T_b's vertices 1 and 2, each
// scaled so that the whole triangle has all six equal to 1:
//     S0 = int 1 / |T|, S1 = 3 int l1 / |T|, S2 = 3 int l2 / |T|,
//     S11 = 6 int l1^2 / |T|, S22 = 6 int l2^2 / |T|, S12 = 12 int l1 l2 / |T|.
// A directed boundary segment p -> q contributes the triangle (0, p, q), 0 = T_b's vertex 0 (Green);
// pieces of edges 0 and 2 pass through that origin and contribute nothing, and a piece [t0, t1] of
// edge 1 contributes F(t1) - F(t0) with the polynomials of edge1_add.  Where the ball is no larger than
// the triangles (g.turn: delta < h_max) a region can be a small part of T_b and those contributions
// would cancel: such problems sum the regions' fans instead (exact_disc_item, kBallNgonAny).
//
// A pair's block is linear in twelve sums over its outer points (acc rows): P_i,c = sum_q W_q
// phi_a,i S_c (c = 0, 1, 2) and Q = sum_q W_q (S11, S22, S12); the other entries of M_ab and M_bb
// follow from phi_0 = 1 - phi_1 - phi_2 and sum_i phi_a,i = 1 (pair_block).
//
// Every block of this file is without the constant c, which the scatter multiplies in FP64: D is a small
// difference of M_aa, M_ab and M_bb where delta is near h, and a c rounded to FP32 in some of them would
// not cancel.
#pragma once

namespace nlq {

// ball modes of k_const beyond nl_ball: an N-gon whose vertices are not those of a regular polygon, or
// no larger than the triangles (the certified Sutherland-Hodgman clip, moments about its first vertex)
constexpr int kBallNgonAny = 16;

template <int BALL>
constexpr int kGeoBall = BALL == kBallNgonAny ? NL_BALL_NGON : BALL;

template <int BALL>
constexpr bool kSupportBall = BALL == NL_BALL_BARY_NOCAPS || BALL == NL_BALL_BARY_APPROXCAPS;

template <typename T>
struct Mom {
    T s0, s1, s2, s11, s22, s12;
};

template <typename T>
__device__ __forceinline__ void mom_set(Mom<T> &M, T v)
{
    M.s0 = M.s1 = M.s2 = M.s11 = M.s22 = M.s12 = v;
}

// a thin triangle's moments (its Cand32 area is negative): every one lies in [0, 1]
__device__ __forceinline__ void mom_hold(Mom<float> &M)
{
    M.s0 = fminf(fmaxf(M.s0, 0.f), 1.f);
    M.s1 = fminf(fmaxf(M.s1, 0.f), 1.f);
    M.s2 = fminf(fmaxf(M.s2, 0.f), 1.f);
    M.s11 = fminf(fmaxf(M.s11, 0.f), 1.f);
    M.s22 = fminf(fmaxf(M.s22, 0.f), 1.f);
    M.s12 = fminf(fmaxf(M.s12, 0.f), 1.f);
}

// boundary segment p -> q, (l1, l2) coordinates
template <typename T>
__device__ __forceinline__ void seg_add(Mom<T> &M, T p1, T p2, T q1, T q2)
{
    const T cr = p1 * q2 - q1 * p2, a1 = p1 + q1, a2 = p2 + q2;
    M.s0 += cr;
    M.s1 += cr * a1;
    M.s2 += cr * a2;
    M.s11 += cr * (a1 * a1 - p1 * q1);
    M.s22 += cr * (a2 * a2 - p2 * q2);
    M.s12 += cr * (a1 * a2 + p1 * p2 + q1 * q2);
}

// a triangle (f, p, q) of area cr |T| / 2 (counted without sign), by its corners' coordinates
template <typename T>
__device__ __forceinline__ void tri_add(Mom<T> &M, T cr, T f1, T f2, T p1, T p2, T q1, T q2)
{
    cr = cr < (T)0 ? -cr : cr;
    const T a1 = f1 + p1 + q1, a2 = f2 + p2 + q2, h = (T)0.5 * cr;
    M.s0 += cr;
    M.s1 += cr * a1;
    M.s2 += cr * a2;
    M.s11 += h * (a1 * a1 + f1 * f1 + p1 * p1 + q1 * q1);
    M.s22 += h * (a2 * a2 + f2 * f2 + p2 * p2 + q2 * q2);
    M.s12 += cr * (a1 * a2 + f1 * f2 + p1 * p2 + q1 * q2);
}

// the piece of edge 1 (from (1, 0) to (0, 1)) up to its point (1 - t, t), times sg
template <typename T>
__device__ __forceinline__ void edge1_add(Mom<T> &M, T t, T sg)
{
    const T st = sg * t, tt = st * t;
    M.s0 += st;
    M.s1 += st * ((T)2 - t);
    M.s2 += tt;
    M.s11 += st * ((T)3 - t * ((T)3 - t));
    M.s22 += tt * t;
    M.s12 += tt * ((T)3 - (T)2 * t);
}

// a point of weight w (relative to |T|)
template <typename T>
__device__ __forceinline__ void point_add(Mom<T> &M, T l1, T l2, T w)
{
    M.s0 += w;
    M.s1 += (T)3 * w * l1;
    M.s2 += (T)3 * w * l2;
    M.s11 += (T)6 * w * l1 * l1;
    M.s22 += (T)6 * w * l2 * l2;
    M.s12 += (T)12 * w * l1 * l2;
}

// moments of m about the point p in T_b's own coordinates: those of l + p
template <typename T>
__device__ __forceinline__ void mom_shift(Mom<T> &M, T p1, T p2)
{
    M.s12 += (T)12 * p1 * p2 * M.s0 + (T)4 * (p1 * M.s2 + p2 * M.s1);
    M.s11 += p1 * ((T)6 * p1 * M.s0 + (T)4 * M.s1);
    M.s22 += p2 * ((T)6 * p2 * M.s0 + (T)4 * M.s2);
    M.s1 += (T)3 * p1 * M.s0;
    M.s2 += (T)3 * p2 * M.s0;
}

// M_ab (9) and the upper M_bb (00 11 22 01 02 12), without c, from a pair's sums P, Q and area = |T_b|
template <typename T>
__device__ __forceinline__ void pair_block(T area, const T *P, const T *Q, T *mab, T *mbb)
{
    // a third by division: 1 / 3 rounded to FP32 would scale every S1 and S2 the same way
    const T k3 = area / (T)3;
    for (int i = 0; i < 3; i++) {
        const T m1 = P[3 * i + 1] * k3, m2 = P[3 * i + 2] * k3;
        mab[3 * i] = area * P[3 * i] - m1 - m2;
        mab[3 * i + 1] = m1;
        mab[3 * i + 2] = m2;
    }
    const T k6 = (T)0.5 * k3, k12 = (T)0.25 * k3;
    const T b11 = k6 * Q[0], b22 = k6 * Q[1], b12 = k12 * Q[2];
    const T p1 = mab[1] + mab[4] + mab[7], p2 = mab[2] + mab[5] + mab[8];
    const T p00 = mab[0] + mab[3] + mab[6];   // sum_q W int phi_0
    const T b01 = p1 - b11 - b12, b02 = p2 - b12 - b22;
    mbb[0] = p00 - b01 - b02;
    mbb[1] = b11;
    mbb[2] = b22;
    mbb[3] = b01;
    mbb[4] = b02;
    mbb[5] = b12;
}

// FP32 data of a candidate: vertices and barycentre relative to bary_a, the edges 0 -> 1, 1 -> 2, 2 -> 0,
// the gradients of the three barycentric coordinates, |T|.  Edges, gradients and area are those of the
// rounded vertices: the triangles around T_a then form one mesh in FP32 too (a shared vertex is rounded
// once), their regions tile the ball, and what the rounding takes from one triangle its neighbour
// gets.  (Edges from the exact vertices, with only T_b's place rounded: errors 1.3-1.8 times as large
// where delta is below h, 1.1 times over 110 problems with horizons of 0.7 to 5 cells.)
// Thin triangles, whose height the vertices' rounding reaches, keep the exact edges and area (as -area), and
// their moments are held to [0, 1] (mom_hold): a rounded one can have no area or a negative one.  (The 23
// words keep lanes that read their own candidate in distinct banks.)
struct Cand32 {
    float vx[3], vy[3], ex[3], ey[3], gx[3], gy[3], blx, bly, area;
    int b, q0;
};

__device__ __forceinline__ Cand32 cand32_of(const CandData &c)
{
    Cand32 r;
    for (int i = 0; i < 3; i++) {
        const int k = (i + 1) % 3;
        r.vx[i] = c.vlx[i];
        r.vy[i] = c.vly[i];
        r.ex[i] = c.vlx[k] - c.vlx[i];
        r.ey[i] = c.vly[k] - c.vly[i];
    }
    float det = r.ex[0] * r.ey[1] - r.ex[1] * r.ey[0];
    // the vertices' rounding moves det by up to 8u (2 + L) L (delta < 2, L the longer of two edges): by
    // more than 6 % here
    const float L = fmaxf(fabsf(c.e1x) + fabsf(c.e1y), fabsf(c.e2x) + fabsf(c.e2y));
    const bool thin = c.akcf < 4e-6f * (2.f + L) * L;
    if (thin) {
        r.ex[0] = c.e1x; r.ex[1] = c.e2x - c.e1x; r.ex[2] = -c.e2x;
        r.ey[0] = c.e1y; r.ey[1] = c.e2y - c.e1y; r.ey[2] = -c.e2y;
        det = 2.f * c.akcf;
    }
    const float inv = 1.f / det;
    for (int i = 0; i < 3; i++) {   // the opposite edge turned, over the determinant
        const int k = (i + 1) % 3;
        r.gx[i] = -r.ey[k] * inv;
        r.gy[i] = r.ex[k] * inv;
    }
    r.blx = c.blx;
    r.bly = c.bly;
    r.area = thin ? -c.akcf : 0.5f * det;
    r.b = c.b;
    r.q0 = c.q0;
    return r;
}

// the same in FP64 (FP64 path): vertex 0, vertices relative to it, edges, gradients of l1 and l2, |T|
struct Cand64 {
    double x0, y0, v[3][2], e[3][2], g[2][2], area, pad;
};
struct CandNone {};

template <typename T>
using CandT = typename std::conditional<sizeof(T) == sizeof(double), Cand64, CandNone>::type;

// T_b as one item sees it: start of edge i relative to x and its direction (read from the candidate's
// shared data by the edge's index, so that nothing is selected between registers), barycentric
// coordinates of a point relative to x
struct View32 {
    const Cand32 &c;
    float lx, ly;   // x relative to bary_a
    __device__ __forceinline__ View32(const Cand32 &c_, const OuterPt &o) : c(c_), lx(o.lx), ly(o.ly) {}
    __device__ __forceinline__ void edge(int i, float &px, float &py, float &ex, float &ey) const
    {
        px = c.vx[i] - lx;
        py = c.vy[i] - ly;
        ex = c.ex[i];
        ey = c.ey[i];
    }
    __device__ __forceinline__ void coords(float px, float py, float &l1, float &l2) const
    {
        const float cx = px - (c.vx[0] - lx), cy = py - (c.vy[0] - ly);
        l1 = cx * c.gx[1] + cy * c.gy[1];
        l2 = cx * c.gx[2] + cy * c.gy[2];
    }
};

struct View64 {
    const Cand64 &c;
    double rx, ry;   // x - vertex 0
    __device__ __forceinline__ View64(const Cand64 &c_, const OuterPt &o) : c(c_), rx(o.x - c_.x0), ry(o.y - c_.y0) {}
    __device__ __forceinline__ void edge(int i, double &px, double &py, double &ex, double &ey) const
    {
        ex = c.e[i][0];
        ey = c.e[i][1];
        const double vx = c.v[i][0], vy = c.v[i][1];
        px = vx - rx;
        py = vy - ry;
    }
    __device__ __forceinline__ void coords(double px, double py, double &l1, double &l2) const
    {
        const double cx = px + rx, cy = py + ry;
        l1 = cx * c.g[0][0] + cy * c.g[0][1];
        l2 = cx * c.g[1][0] + cy * c.g[1][1];
    }
};

template <typename T>
__device__ __forceinline__ T quot(T a, T b)
{
    if constexpr (sizeof(T) == sizeof(float)) {
        return __fdividef(a, b);
    } else {
        // Newton's iteration on 1 / b from the hardware's approximate reciprocal (2^-20), then one
        // residual step on the quotient: five FP64 instructions, within an ulp for the normal numbers
        // of a mesh (the correctly rounded division takes about twice as many).  With it and root, FP64
        // matrices are as far from extended precision as with correctly rounded ones point by point, or
        // closer: 0.80 of those errors over 151 problems
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
        y = fma(y, fma(-b, y, 1.0), y);
        const double t = a * y;
        return fma(fma(-b, t, a), y, t);
    }
}

// the barycentric point at parameter t of edge i
template <typename T>
__device__ __forceinline__ void edge_l(int i, T t, T &l1, T &l2)
{
    const T u = (T)1 - t;
    l1 = i == 0 ? t : i == 1 ? u : (T)0;
    l2 = i == 0 ? (T)0 : i == 1 ? t : u;
}

// ---------------------------------------------------------------------------
// Which of T_b's vertices lie in the ball (bits of `in`) and which edges with both ends outside
// cross it twice (bits of `dbl`), in FP32, taken only when FP32 is certain (false: undecided).
// Every function of the cut items has a single exit: an early return inside a divergent loop
// moves the point where the warp's lanes meet again to the end of the item (the first version of
// k_const<N-gon, float> ran 13 of 32 lanes on average for that reason).
// ---------------------------------------------------------------------------
// The disc: the predicates and margins of nlg::ball_walk_f32.
__device__ __forceinline__ bool disc_status(const nlg::F2 d[3], const nlg::GeoParams &g, unsigned &in, unsigned &dbl)
{
    in = 0;
    dbl = 0;
    bool sure = true;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float r = d[i].x * d[i].x + d[i].y * d[i].y;
        const bool is_in = r <= g.rin_m2;
        sure = sure && (is_in || r > g.rout_p2);
        if (is_in) in |= 1u << i;
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int j = (i + 1) % 3;
        const float ex = d[j].x - d[i].x, ey = d[j].y - d[i].y;
        const float a = ex * ex + ey * ey, b = d[i].x * ex + d[i].y * ey, cr = d[i].x * ey - d[i].y * ex;
        // both ends outside and the closest point between them
        const bool mid = !(((in >> i) | (in >> j)) & 1u) && b < 0.f && -b < a;
        const bool hits = cr * cr <= g.rin_m2 * a, misses = cr * cr > g.rout_p2 * a;
        if (mid && hits) dbl |= 1u << i;
        sure = sure && !(mid && !hits && !misses);
    }
    return sure;
}

// The regular N-gon with corners o_0 .. o_N (o_N = o_0) on the circle of radius^2 g.poly_r2.
// The line p + t e crosses polygon edge k exactly when it separates corners k and k + 1, that is
// when its crossing of the circle lies on the arc between them: k comes from the angle of that
// crossing (arctangent polynomial) and is certain when both corners are farther than tau from
// the line, on the sides that an exit (entry) needs.  s0, s1: the corners' signed distances to
// the line times |e|.  Returns k in [0, N); *hit = false when the line misses the circle.
__device__ __forceinline__ int ngon_edge(const nlg::F2 &p, const nlg::F2 &e, float a, float b, float cr, bool exit_,
                                         const nlg::GeoParams &g, const float2 *corner, bool *hit, float *s0,
                                         float *s1)
{
    const float disc = a * g.poly_r2 - cr * cr;
    *hit = disc > 0.f;
    const float half = sqrtf(fmaxf(disc, 0.f));
    const float t = __fdividef((exit_ ? half : -half) - b, a);
    int k = (int)floorf(nlg::atan2_poly(p.y + t * e.y, p.x + t * e.x) * g.inv_sector);
    if (k < 0) k += g.ngon_n;
    const float2 o0 = corner[k], o1 = corner[k + 1];
    *s0 = e.x * (o0.y - p.y) - e.y * (o0.x - p.x);
    *s1 = e.x * (o1.y - p.y) - e.y * (o1.x - p.x);
    return k;
}

// is v inside the N-gon?  v's angle names the polygon edge to test (and the next one, for an angle
// near a corner): 1 inside, 0 outside, -1 undecided; *w: the direction of an edge v lies beyond
__device__ __forceinline__ int ngon_holds(const nlg::F2 &v, const nlg::GeoParams &g, const float2 *corner, nlg::F2 *w)
{
    const float f = nlg::atan2_poly(v.y, v.x) * g.inv_sector;
    const float fl = floorf(f);
    int k = (int)fl, n = f - fl < 0.5f ? k - 1 : k + 1;
    const int N = g.ngon_n;
    k += k < 0 ? N : 0;
    n += n < 0 ? N : 0;
    n -= n >= N ? N : 0;
    const float m = g.poly_m;
    const float2 a0 = corner[k], a1 = corner[k + 1], b0 = corner[n], b1 = corner[n + 1];
    const float ax = a1.x - a0.x, ay = a1.y - a0.y, bx = b1.x - b0.x, by = b1.y - b0.y;
    const float oa = ax * (v.y - a0.y) - ay * (v.x - a0.x), ob = bx * (v.y - b0.y) - by * (v.x - b0.x);
    const bool out_a = oa < -m, out_b = ob < -m;
    w->x = out_a ? ax : bx;
    w->y = out_a ? ay : by;
    return out_a || out_b ? 0 : (oa > m && ob > m ? 1 : -1);
}

__device__ __forceinline__ bool ngon_status(const nlg::F2 d[3], const nlg::GeoParams &g, const float2 *corner,
                                            unsigned &in, unsigned &dbl)
{
    in = 0;
    dbl = 0;
    bool sure = true;
    unsigned far = 0;
    nlg::F2 w[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};   // a polygon edge that an outside vertex lies beyond
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float r = d[i].x * d[i].x + d[i].y * d[i].y;
        if (r <= g.rin_m2) in |= 1u << i;
        else if (r > g.rout_p2) far |= 1u << i;
    }
    // vertices between the inscribed and the circumscribed circle: rarely more than one
    for (unsigned todo = ~(in | far) & 7u; todo; todo &= todo - 1) {
        const int i = __ffs(todo) - 1;
        nlg::F2 x;
        const int h = ngon_holds(i == 0 ? d[0] : i == 1 ? d[1] : d[2], g, corner, &x);
        sure = sure && h >= 0;
        if (h > 0) in |= 1u << i;
        if (i == 0) w[0] = x;
        if (i == 1) w[1] = x;
        if (i == 2) w[2] = x;
    }
    unsigned pend = 0;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int j = (i + 1) % 3;
        const float ex = d[j].x - d[i].x, ey = d[j].y - d[i].y;
        const float a = ex * ex + ey * ey, b = d[i].x * ex + d[i].y * ey, cr = d[i].x * ey - d[i].y * ex;
        const bool both = ((far >> i) & (far >> j) & 1u) != 0;
        // edges with both ends outside that miss the polygon: the line misses the circle; both ends
        // beyond the circle and the closest point is one of them; or an end lies beyond a polygon
        // edge and the edge leads away from it
        const bool miss = cr * cr > g.rout_p2 * a || (both && !(b < 0.f && -b < a)) ||
                          (!((far >> i) & 1u) && w[i].x * ey - w[i].y * ex <= 0.f) ||
                          (!((far >> j) & 1u) && w[j].x * ey - w[j].y * ex >= 0.f);
        const bool out = !(((in >> i) | (in >> j)) & 1u);
        const bool hits = both && cr * cr <= g.rin_m2 * a;   // the line meets the inscribed circle
        if (out && !miss) {
            if (hits) dbl |= 1u << i;
            else pend |= 1u << i;
        }
    }
    for (; pend; pend &= pend - 1) {
        // an outside edge whose line passes between the two circles, or that starts or ends there
        const int i = __ffs(pend) - 1;
        const nlg::F2 p = i == 0 ? d[0] : i == 1 ? d[1] : d[2], q = i == 0 ? d[1] : i == 1 ? d[2] : d[0];
        const nlg::F2 e = {q.x - p.x, q.y - p.y};
        const float a = e.x * e.x + e.y * e.y, b = p.x * e.x + p.y * e.y, cr = p.x * e.y - p.y * e.x;
        const float le = sqrtf(a), m = g.tau * le;
        float n0, n1, x0, x1;
        bool hit;
        const int kn = ngon_edge(p, e, a, b, cr, false, g, corner, &hit, &n0, &n1);
        const int kx = ngon_edge(p, e, a, b, cr, true, g, corner, &hit, &x0, &x1);
        // every corner on one side of the line: no crossing
        const bool none = kn == kx && ((n0 > m && n1 > m) || (n0 < -m && n1 < -m));
        // the line crosses edges kn and kx: between p and q (both outside by tau), or not
        const float2 on = corner[kn], on1 = corner[kn + 1], ox = corner[kx], ox1 = corner[kx + 1];
        const float ax = on1.x - on.x, ay = on1.y - on.y, cx = ox1.x - ox.x, cy = ox1.y - ox.y;
        const float dn = ax * e.y - ay * e.x, dx = cx * e.y - cy * e.x;
        const float graze = 0.02f * le * g.poly_side;   // below that the crossing's place is too uncertain
        const float tn = __fdividef(ay * (p.x - on.x) - ax * (p.y - on.y), dn);
        const float tx = __fdividef(cy * (p.x - ox.x) - cx * (p.y - ox.y), dx);
        const float mt = __fdividef(g.tau, le);
        const bool cross = kn != kx && n0 > m && n1 < -m && x0 < -m && x1 > m && fabsf(dn) > graze && fabsf(dx) > graze;
        const bool inside = cross && tn > mt && tx < 1.f - mt, beyond = cross && (tx < -mt || tn > 1.f + mt);
        if (hit && inside) dbl |= 1u << i;
        sure = sure && hit && (none || inside || beyond);
    }
    return sure;
}

// square root of d >= 0
template <typename T>
__device__ __forceinline__ T root(T d)
{
    if constexpr (sizeof(T) == sizeof(float)) {
        return sqrtf(d);
    } else {
        // Newton's iteration on 1 / sqrt(d) from the hardware's approximate one (2^-20 or better), then
        // one residual step on the root: six FP64 instructions
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(fmax(d, 1e-280)));
        const double h = 0.5 * y;
        double s = d * y;
        s = fma(h, fma(-s, s, d), s);
        return fma(h, fma(-s, s, d), s);
    }
}

// the parameter t of edge (p, e) where it leaves (enters) the disc.  FP32: delta^2 in two parts (one
// rounded delta^2 would shift every region the same way: 4.4e-8 instead of 3e-8 in the matrix)
template <typename T>
__device__ __forceinline__ T disc_cross(const nlg::GeoParams &g, T px, T py, T ex, T ey, bool exit_)
{
    const T a = ex * ex + ey * ey, b = px * ex + py * ey;
    T c;
    if constexpr (sizeof(T) == sizeof(float)) c = (px * px + py * py - g.d2f) - g.d2lo;
    else c = px * px + py * py - g.d2;
    T ds = b * b - a * c;
    ds = ds > (T)0 ? ds : (T)0;
    const T s = root(ds);
    // roots of a t^2 + 2 b t + c without cancellation: the far one from w, the other from c / w
    const T w = b > (T)0 ? -(b + s) : s - b;
    const bool num = exit_ == (b <= (T)0);
    return quot(num ? w : c, num ? a : w);
}

// corner k of the polygon in the quadrature's precision
template <typename T>
__device__ __forceinline__ void corner_of(const NumArgs &A, const float2 *corner, int k, T &x, T &y)
{
    if constexpr (sizeof(T) == sizeof(float)) {
        const float2 o = corner[k];
        x = o.x;
        y = o.y;
    } else {
        const int kk = k >= A.geo.ngon_n ? k - A.geo.ngon_n : k;
        const double2 o = __ldg((const double2 *)A.geo.ngon + kk);
        x = o.x;
        y = o.y;
    }
}

// Moments of one cut (q, b): the region's structure (vertices in, edges cut, polygon edges met) from
// certain FP32 predicates, its coordinates in T.  1 done, 0 empty region, -1 the FP64 geometry decides.
// The vertex count, kind and cap count are those of the FP64 region (the records' content).
// Every lane of the warp calls it (with data of some item: `live` says whether the lane's counts).
// d: T_b's vertices relative to x; v32, f: T_b in FP32 and in T.
template <int BALL, typename T, typename View>
__device__ __forceinline__ int cut_item(const NumArgs &A, bool live, const nlg::F2 d[3], const View32 &v32,
                                        const View &f, T inv_area, const float2 *corner, Mom<T> &M, int &nv,
                                        int &kind, int &ncap)
{
    constexpr bool kPoly = BALL == NL_BALL_NGON;
    const nlg::GeoParams &g = A.geo;
    unsigned in, dbl;
    const bool sure = kPoly ? ngon_status(d, g, corner, in, dbl) : disc_status(d, g, in, dbl);
    const unsigned nxt = ((in >> 1) | (in << 2)) & 7u;   // bit i: the end of edge i is inside
    unsigned X = (in & ~nxt) | dbl;                      // edges that leave the ball
    const unsigned N = (~in & nxt) | dbl;                // edges that enter it
    const int narc = __popc(X);
    int n = __popc(in) + 2 * narc;
    bool known = sure;
    if (BALL == NL_BALL_APPROXCAPS) {
        known = known && g.cap_level <= 2;
        n += narc * ((1 << g.cap_level) - 1);
    }
    bool empty = BALL == NL_BALL_EXACTCAPS ? n < 2 : n < 3;
    if (kPoly && X == 0u && in != 7u) {
        // no crossing: empty, unless the polygon lies inside T_b (x inside it)
        const float o0 = d[0].x * d[1].y - d[0].y * d[1].x, o1 = d[1].x * d[2].y - d[1].y * d[2].x;
        const float o2 = d[2].x * d[0].y - d[2].y * d[0].x;
        known = known && !(fminf(o0, fminf(o1, o2)) >= 0.f);
        empty = true;
    }
    // a polygon region with two crossings and no vertex of T_b inside has its corners still to count
    if (kPoly && X != 0u) empty = false;
    mom_set(M, in & 4u ? (T)1 : (T)0);   // edge 1 up to vertex 2
    ncap = 0;
    bool go = live && known && !empty;
    __syncwarp();
    while (__any_sync(0xffffffffu, go && X != 0u)) {   // one exit and the next entry (rarely more)
        if (go && X != 0u) {
            const int i = __ffs(X) - 1;
            X &= X - 1;
            // the next edge that enters, along the boundary of T_b
            const int i1 = i == 2 ? 0 : i + 1, i2 = i1 == 2 ? 0 : i1 + 1;
            const int j = (N >> i1) & 1u ? i1 : ((N >> i2) & 1u ? i2 : i);
            // start relative to x and direction of the edge left (p, e) and of the edge entered (s, h)
            T px, py, ex, ey, sx, sy, hx, hy, tx, tn;
            f.edge(i, px, py, ex, ey);
            f.edge(j, sx, sy, hx, hy);
            int kx = 0, kn = 0;
            if constexpr (kPoly) {
                float s0, s1, n0, n1;
                bool hitx, hitn;
                nlg::F2 p, e, q, h;
                v32.edge(i, p.x, p.y, e.x, e.y);
                v32.edge(j, q.x, q.y, h.x, h.y);
                const float ae = e.x * e.x + e.y * e.y, ah = h.x * h.x + h.y * h.y;
                kx = ngon_edge(p, e, ae, p.x * e.x + p.y * e.y, p.x * e.y - p.y * e.x, true, g, corner, &hitx, &s0, &s1);
                kn = ngon_edge(q, h, ah, q.x * h.x + q.y * h.y, q.x * h.y - q.y * h.x, false, g, corner, &hitn, &n0, &n1);
                const float m = g.tau * sqrtf(ae), mh = g.tau * sqrtf(ah);
                known = hitx && hitn && s0 < -m && s1 > m && n0 > mh && n1 < -mh;
                // t from the line of the polygon edge
                T ox, oy, ux, uy;
                corner_of<T>(A, corner, kx, ox, oy);
                corner_of<T>(A, corner, kx + 1, ux, uy);
                ux -= ox;
                uy -= oy;
                tx = quot(uy * (px - ox) - ux * (py - oy), ux * ey - uy * ex);
                corner_of<T>(A, corner, kn, ox, oy);
                corner_of<T>(A, corner, kn + 1, ux, uy);
                ux -= ox;
                uy -= oy;
                tn = quot(uy * (sx - ox) - ux * (sy - oy), ux * hy - uy * hx);
                if (kn == kx) {
                    // both on one polygon edge: the boundary runs along it from the exit to the entry, or
                    // (the polygon all but inside T_b) around it
                    const float2 a0 = corner[kx], a1 = corner[kx + 1];
                    const float wx = a1.x - a0.x, wy = a1.y - a0.y;
                    float t, r;
                    if constexpr (sizeof(T) == sizeof(float)) {
                        t = tx;
                        r = tn;
                    } else {   // FP32 decides
                        t = __fdividef(wy * (p.x - a0.x) - wx * (p.y - a0.y), wx * e.y - wy * e.x);
                        r = __fdividef(wy * (q.x - a0.x) - wx * (q.y - a0.y), wx * h.y - wy * h.x);
                    }
                    const float run = ((q.x + r * h.x) - (p.x + t * e.x)) * wx + ((q.y + r * h.y) - (p.y + t * e.y)) * wy;
                    known = known && run > g.poly_m;
                }
                go = known;
            } else {
                tx = disc_cross<T>(g, px, py, ex, ey, true);
                tn = disc_cross<T>(g, sx, sy, hx, hy, false);
            }
            if (i == 1) edge1_add(M, tx, (T)1);
            if (j == 1) edge1_add(M, tn, (T)-1);
            T l1, l2, q1, q2;
            edge_l(i, tx, l1, l2);
            edge_l(j, tn, q1, q2);
            if constexpr (kPoly) {   // along the polygon's corners
                int c = kn - kx;
                c += c < 0 ? g.ngon_n : 0;
                n += c;
                for (int k = kx + 1; c > 0; c--, k++) {
                    if (k >= g.ngon_n) k -= g.ngon_n;
                    T ox, oy, m1, m2;
                    corner_of<T>(A, corner, k, ox, oy);
                    f.coords(ox, oy, m1, m2);
                    seg_add(M, l1, l2, m1, m2);
                    l1 = m1;
                    l2 = m2;
                }
            }
            if constexpr (BALL == NL_BALL_APPROXCAPS) {   // along the dyadic arc points
                if (g.cap_level > 0) {
                    const T ax = px + tx * ex, ay = py + tx * ey, bx = sx + tn * hx, by = sy + tn * hy;
                    const T dl = sizeof(T) == sizeof(float) ? (T)g.deltaf : (T)g.delta;
                    auto mid = [&](T ux, T uy, T &ox, T &oy) {
                        T s;
                        if constexpr (sizeof(T) == sizeof(float)) {
                            const float rs = rsqrtf(ux * ux + uy * uy);
                            s = fmaf(dl, rs, g.deltalo * rs);
                        } else {
                            s = quot(dl, root(ux * ux + uy * uy));
                        }
                        ox = ux * s;
                        oy = uy * s;
                    };
                    auto to = [&](T x, T y) {
                        T m1, m2;
                        f.coords(x, y, m1, m2);
                        seg_add(M, l1, l2, m1, m2);
                        l1 = m1;
                        l2 = m2;
                    };
                    // the bisection's direction (a - x) + (b - x) points away from an arc beyond a half circle
                    // (the ball all but inside T_b): such a polygon turns back, and its fan's areas count
                    // without sign, as exact_disc_item takes them
                    known = ax * bx + ay * by > (T)0 || ax * by - ay * bx > (T)1e-3 * dl * dl;
                    go = known;
                    T mx, my;
                    mid(ax + bx, ay + by, mx, my);
                    if (g.cap_level == 2) {
                        T qx, qy;
                        mid(ax + mx, ay + my, qx, qy);
                        to(qx, qy);
                        to(mx, my);
                        mid(mx + bx, my + by, qx, qy);
                        to(qx, qy);
                    } else {
                        to(mx, my);
                    }
                }
            }
            seg_add(M, l1, l2, q1, q2);
            if constexpr (BALL == NL_BALL_EXACTCAPS) {
                const T ax = px + tx * ex, ay = py + tx * ey, bx = sx + tn * hx, by = sy + tn * hy;
                T cx, cy, w;
                if constexpr (sizeof(T) == sizeof(float)) {
                    nlg::cap_rule_f32(nlg::F2{ax, ay}, nlg::F2{bx, by}, g, &cx, &cy, &w);
                } else {
                    D2 cc;
                    nlg::cap_rule(D2{ax, ay}, D2{bx, by}, D2{0.0, 0.0}, g.delta, g.cap_printed, &cc, &w);
                    cx = cc.x;
                    cy = cc.y;
                }
                T c1, c2;
                f.coords(cx, cy, c1, c2);
                point_add(M, c1, c2, w * inv_area);
                ncap++;
            }
        }
        __syncwarp();
    }
    kind = in == 7u ? nlg::KIND_WHOLE : nlg::KIND_PARTIAL;
    nv = BALL == NL_BALL_EXACTCAPS && n < 3 ? 0 : n;
    return !known ? -1 : empty ? 0 : 1;
}

// ---------------------------------------------------------------------------
// Per-warp shared memory of k_const
// ---------------------------------------------------------------------------
struct NoClip {};

template <int BALL, typename T>
struct ConstShared {
    static constexpr bool kClip = sizeof(T) == sizeof(float) ? (BALL == kBallNgonAny || kSupportBall<BALL>) : kSupportBall<BALL>;
    using Fx = typename std::conditional<sizeof(T) == sizeof(float), int, T>::type;   // FP32 sums: fixed point
    CandT<T> c64[sizeof(T) == sizeof(double) ? 32 : 1];
    T w[NL_MAXQ][4];           // per outer point: W phi_a,i (i = 0, 1, 2) and W
    OuterPt sq[NL_MAXQ];
    Cand32 cand[32];
    Fx acc[12][32];            // P (rows 0-8) and Q (9-11) of each lane's pair, value-major
    Fx s0q[NL_MAXQ];           // per outer point: sum of |T_b| S0 over the cut regions
    unsigned dmask[32];        // FP32: outer points of each lane's candidate whose item the deferred kernel
                               // takes; FP64: the lanes that hold moments for this lane's pair
    typename std::conditional<sizeof(T) == sizeof(double), T, CandNone>::type mom[6][sizeof(T) == sizeof(double) ? 32 : 1];
    unsigned char momq[sizeof(T) == sizeof(double) ? 32 : 1];   // FP64: moments on their way, their outer points
    float2 corner[65];         // the regular polygon's corners, corner[N] = corner[0]
    unsigned short queue[32 * NL_MAXQ];   // cut items (owner lane << 8 | q)
    unsigned char hit[32];     // the lane's pair has a non-empty cut region
    typename std::conditional<kClip, nlg::ClipBuf, NoClip>::type clip;
};

// The N-gon's region by the FP64 geometry and its moments: false for an empty region
template <int BALL, typename T>
__device__ __noinline__ bool exact_const_item(const NumArgs &A, int b, const nlg::F2 *dl, double xx, double xy,
                                              Mom<T> &M, int &nv, int &kind, int &ncap)
{
    const CandFp64 c = cand_fp64(A, b);
    const D2 x = {xx, xy};
    nlg::Region R;
    nlg::make_region<NL_BALL_NGON>(c.V, dl, c.bb, x, A.geo, R);
    if (R.overflow) atomicOr(A.err, 1);
    if (R.kind == nlg::KIND_NONE) return false;
    kind = R.kind;
    nv = R.nv;
    ncap = R.ncap;
    if (kind == nlg::KIND_WHOLE) {
        mom_set(M, (T)1);
        return true;
    }
    // in FP64 whatever T (these items are few)
    const BaryMap bm = bary_map(c.V);
    Mom<double> S;
    mom_set(S, 0.0);
    double phi[3];
    const double x0 = R.P[0].x, y0 = R.P[0].y;   // about the polygon's first vertex
    double p1 = 0.0, p2 = 0.0;
    for (int i = 1; i < nv; i++) {
        const double dx = R.P[i].x - x0, dy = R.P[i].y - y0;
        const double q1 = (dx * bm.e2y - bm.e2x * dy) * bm.inv, q2 = (bm.e1x * dy - dx * bm.e1y) * bm.inv;
        seg_add(S, p1, p2, q1, q2);
        p1 = q1;
        p2 = q2;
    }
    bary_of(bm, x0, y0, phi);
    mom_shift(S, phi[1], phi[2]);
    M = Mom<T>{(T)S.s0, (T)S.s1, (T)S.s2, (T)S.s11, (T)S.s22, (T)S.s12};
    return true;
}

// The same for the balls whose FP64 decisions are a vertex or edge predicate: barycenter, overlap and
// the disc walks.  FP32 leaves a few predicates of an item open (a vertex or a closest point within
// tau of the circle); only those are taken in FP64, by the canonical expressions, and the walk's points
// (vertex if inside, then the edge's roots) are linked as they come, with nothing kept in arrays: on
// the uniform grid of the paper's protocol, whose outer points lie at distance delta of other vertices
// (1.35 M open items at h = 0.0125), it replaced a queue and a second kernel that built every such
// region in local memory (exactcaps: 3.2 ms there, 1.1 ms here; the whole assembly 5.3 -> 3.2 ms).
template <typename T>
struct WalkPt {
    T l1, l2, x, y;   // barycentric coordinates; position relative to x (arc ends)
    int tag;          // 0 vertex, 1 entry, 2 exit
};

template <int BALL, typename T>
__device__ __noinline__ bool exact_disc_item(const NumArgs &A, int b, float area32, const nlg::F2 *dl, double xx,
                                             double xy, Mom<T> &M, int &nv, int &kind, int &ncap, bool *used64)
{
    const nlg::GeoParams &g = A.geo;
    const D2 x = {xx, xy};
    ncap = 0;
    *used64 = true;
    if constexpr (BALL == NL_BALL_BARYCENTER || BALL == NL_BALL_OVERLAP) {
        const CandFp64 c = cand_fp64(A, b);
        mom_set(M, (T)1);
        nv = 3;
        kind = nlg::KIND_WHOLE;
        return BALL == NL_BALL_BARYCENTER ? nlg::in_ball(c.bb, x, g.d2) : nlg::overlaps(c.V, x, g.d2);
    } else {
        constexpr bool f32 = sizeof(T) == sizeof(float);
        const int K = A.K;
        D2 V[3];
        for (int i = 0; i < 3; i++) { V[i].x = A.tx[i * K + b]; V[i].y = A.ty[i * K + b]; }
        T px[3], py[3];   // vertices relative to x
        unsigned in = 0, open = 0;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if constexpr (f32) {
                px[i] = dl[i].x;
                py[i] = dl[i].y;
            } else {
                px[i] = nlg::sub(V[i].x, x.x);
                py[i] = nlg::sub(V[i].y, x.y);
            }
            const float r = dl[i].x * dl[i].x + dl[i].y * dl[i].y;
            if (r <= g.rin_m2) in |= 1u << i;
            else if (!(r > g.rout_p2)) open |= 1u << i;
        }
        // The loops over the open vertices and edges (one vertex and its two edges as a rule) run once
        // for all lanes, whichever theirs are: the FP64 pipe takes a warp instruction of one lane as
        // long as one of 32.
        auto vert = [&](int i) { return i == 0 ? V[0] : i == 1 ? V[1] : V[2]; };
        for (unsigned w = open; w; w &= w - 1) {
            const int i = __ffs(w) - 1;
            if (nlg::in_ball(vert(i), x, g.d2)) in |= 1u << i;
        }
        unsigned eopen = open | ((open >> 1) | (open << 2));   // edges that start or end at an open vertex
        eopen &= 7u;
        int nr[3] = {0, 0, 0};
        unsigned ents = 0;   // bit 2 i + k: root k of edge i enters
        T t[3][2];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const int j = (i + 1) % 3;
            t[i][0] = t[i][1] = 0;
            if ((eopen >> i) & 1u) continue;
            const bool pi = ((in >> i) & 1u) != 0, qi = ((in >> j) & 1u) != 0;
            if (pi != qi) {
                nr[i] = 1;
                if (!pi) ents |= 1u << (2 * i);
            } else if (!pi) {
                const float fx = dl[j].x - dl[i].x, fy = dl[j].y - dl[i].y;
                const float a = fx * fx + fy * fy, bq = dl[i].x * fx + dl[i].y * fy, cr = dl[i].x * fy - dl[i].y * fx;
                if (bq < 0.f && -bq < a) {
                    if (cr * cr <= g.rin_m2 * a) {
                        nr[i] = 2;
                        ents |= 1u << (2 * i);
                    } else if (!(cr * cr > g.rout_p2 * a)) {
                        eopen |= 1u << i;
                    }
                }
            }
        }
        const unsigned ecert = ~eopen & 7u;
        for (unsigned w = eopen; w; w &= w - 1) {
            // the canonical roots (nlg::edge_roots); l = num / a lies in (0, 1) exactly when 0 < num < a
            const int i = __ffs(w) - 1;
            const D2 p = vert(i), q = vert(i == 2 ? 0 : i + 1);
            using namespace nlg;
            const double dx = sub(q.x, p.x), dy = sub(q.y, p.y), fx = sub(p.x, x.x), fy = sub(p.y, x.y);
            const double a = add(mul(dx, dx), mul(dy, dy)), bh = add(mul(fx, dx), mul(fy, dy));
            const double c = sub(add(mul(fx, fx), mul(fy, fy)), g.d2);
            const double disc = sub(mul(bh, bh), mul(a, c));
            int m = 0;
            T u0 = 0, u1 = 0;
            unsigned en = 0;
            if (!(disc < 0.0)) {
                const double sq = __dsqrt_rn(disc), n1 = sub(-bh, sq), n2 = add(-bh, sq);
                const bool k1 = n1 > 0.0 && n1 < a, k2 = n2 > 0.0 && n2 < a;
                m = (int)k1 + (int)k2;
                if constexpr (f32) {
                    const float ia = 1.f / (float)a;
                    u0 = (float)(k1 ? n1 : n2) * ia;
                    u1 = (float)n2 * ia;
                } else {
                    const double ia = 1.0 / a;
                    u0 = (k1 ? n1 : n2) * ia;
                    u1 = n2 * ia;
                }
                en = k1 && k2 ? 1u : (in >> i) & 1u ? 0u : 1u;
            }
#pragma unroll
            for (int k = 0; k < 3; k++)
                if (k == i) {
                    nr[k] = m;
                    t[k][0] = u0;
                    t[k][1] = u1;
                    ents |= en << (2 * k);
                }
        }
        const T e1x = px[1] - px[0], e1y = py[1] - py[0], e2x = px[2] - px[0], e2y = py[2] - py[0];
        const bool thin = f32 && area32 < 0.f;   // Cand32
        const T inv = (T)1 / (thin ? (T)(-2.f * area32) : e1x * e2y - e2x * e1y);
        mom_set(M, (T)0);
        WalkPt<T> first = {0, 0, 0, 0, 0}, prev = first;
        int n = 0, narc = 0;
        // the piece of boundary from a to c: triangles of the region's fan from its first point, their
        // areas from positions, their moments from the corners' coordinates (nothing cancels)
        auto link = [&](const WalkPt<T> &a, const WalkPt<T> &c) {
            T u1 = a.l1, u2 = a.l2, ux = a.x, uy = a.y;
            auto to = [&](T v1, T v2, T vx, T vy) {
                const T cr = (ux - first.x) * (vy - first.y) - (vx - first.x) * (uy - first.y);
                tri_add(M, cr * inv, first.l1, first.l2, u1, u2, v1, v2);
                u1 = v1;
                u2 = v2;
                ux = vx;
                uy = vy;
            };
            if (BALL != NL_BALL_NOCAPS && a.tag == 2 && c.tag == 1) {
                narc++;
                if constexpr (BALL == NL_BALL_APPROXCAPS) {
                    // dyadic arc points, each by bisection from the ends
                    const int m = 1 << g.cap_level;
                    for (int j = 1; j < m; j++) {
                        T ax = a.x, ay = a.y, bx = c.x, by = c.y, mx = 0, my = 0;
                        for (int lo = 0, hi = m; hi - lo > 1;) {
                            mx = ax + bx;
                            my = ay + by;
                            T sc;
                            if constexpr (f32) {   // both parts of delta in one rounding (disc_cross)
                                const float rs = 1.f / sqrtf(mx * mx + my * my);
                                sc = fmaf(g.deltaf, rs, g.deltalo * rs);
                            } else {
                                sc = g.delta / sqrt(mx * mx + my * my);
                            }
                            mx *= sc;
                            my *= sc;
                            const int md = (lo + hi) >> 1;
                            if (md == j) break;
                            if (j < md) { hi = md; bx = mx; by = my; }
                            else { lo = md; ax = mx; ay = my; }
                        }
                        const T cx = mx - px[0], cy = my - py[0];
                        to((cx * e2y - e2x * cy) * inv, (e1x * cy - cx * e1y) * inv, mx, my);
                    }
                } else if (ncap < 3) {   // exactcaps: centroid and area
                    T cx, cy, w;
                    if constexpr (f32) {
                        nlg::cap_rule_f32(nlg::F2{a.x, a.y}, nlg::F2{c.x, c.y}, g, &cx, &cy, &w);
                    } else {
                        D2 cc;
                        nlg::cap_rule(D2{a.x, a.y}, D2{c.x, c.y}, D2{0.0, 0.0}, g.delta, g.cap_printed, &cc, &w);
                        cx = cc.x;
                        cy = cc.y;
                    }
                    cx -= px[0];
                    cy -= py[0];
                    // w / |T_b| = 2 w / det
                    point_add(M, (cx * e2y - e2x * cy) * inv, (e1x * cy - cx * e1y) * inv, (T)2 * w * inv);
                    ncap++;
                }
            }
            to(c.l1, c.l2, c.x, c.y);
        };
        auto emit = [&](T l1, T l2, T qx, T qy, int tag) {
            const WalkPt<T> q = {l1, l2, qx, qy, tag};
            if (n == 0) first = q;
            else link(prev, q);
            prev = q;
            n++;
        };
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const int j = (i + 1) % 3;
            const bool pi = ((in >> i) & 1u) != 0;
            if (pi) emit((T)(i == 1), (T)(i == 2), px[i], py[i], 0);
            const T ex = px[j] - px[i], ey = py[j] - py[i];
            const bool calc = ((ecert >> i) & 1u) != 0;
#pragma unroll
            for (int k = 0; k < 2; k++)
                if (k < nr[i]) {
                    const bool en = ((ents >> (2 * i + k)) & 1u) != 0;
                    const T tk = calc ? disc_cross<T>(g, px[i], py[i], ex, ey, !en) : t[i][k];
                    T l1, l2;
                    edge_l(i, tk, l1, l2);
                    emit(l1, l2, px[i] + tk * ex, py[i] + tk * ey, en ? 1 : 2);
                }
        }
        if (n > 1) link(prev, first);
        int m = n;
        if (BALL == NL_BALL_APPROXCAPS) m += narc * ((1 << g.cap_level) - 1);
        nv = n >= 2 && m >= 3 ? m : 0;
        kind = in == 7u && n == 3 ? nlg::KIND_WHOLE : nlg::KIND_PARTIAL;
        if (kind == nlg::KIND_WHOLE) mom_set(M, (T)1);
        if constexpr (f32)
            if (thin) mom_hold(M);
        *used64 = (open | eopen) != 0u;
        return nv >= 3 || ncap > 0;
    }
}

// region and moments of one item by the FP64 geometry (*used64 = false: FP32 was certain after all);
// area32: the candidate's Cand32 area
template <int BALL, typename T>
__device__ __forceinline__ bool exact_item(const NumArgs &A, int b, float area32, const nlg::F2 *dl, double xx, double xy,
                                           Mom<T> &M, int &nv, int &kind, int &ncap, bool *used64)
{
    if constexpr (kGeoBall<BALL> == NL_BALL_NGON) return exact_const_item<BALL, T>(A, b, dl, xx, xy, M, nv, kind, ncap);
    else return exact_disc_item<BALL, T>(A, b, area32, dl, xx, xy, M, nv, kind, ncap, used64);
}

// are the items that FP32 leaves open queued for k_deferred?  The N-gon's on the FP32 path: its FP64
// clip keeps its polygons in local memory, and a warp that ran it for one lane would wait (about 0.2
// such items a round on a jittered mesh; a disc item costs some 150 FP64 instructions).
template <int BALL, typename T>
constexpr bool kConstQueue = sizeof(T) == sizeof(float) && kGeoBall<BALL> == NL_BALL_NGON;

// inner points that the rule spends on a region (the counted qp-pairs)
__device__ __forceinline__ int region_points(const NumArgs &A, int kind, int nv, int ncap)
{
    if (kind == nlg::KIND_WHOLE && ncap == 0) return A.inner.n;
    return (nv >= 3 ? (nv - 2) * A.inner.n : 0) + ncap;
}

// An item's moments M at an outer point of weights w, added onto owner own's sums (rows 0-11), its s0 onto
// the outer point's.  FP32 sums: rounded to the grids fxs and gs (native integer adds, any order).
__device__ __forceinline__ void item_add(const float *w, const Mom<float> &M, int (*acc)[32], int *s0q, int own,
                                         float fxs, float area, float gs)
{
    const float w0 = w[0] * fxs, w1 = w[1] * fxs, w2 = w[2] * fxs, W = w[3] * fxs;   // fxs: a power of two
    auto put = [&](int k, float v) { atomicAdd(&acc[k][own], __float2int_rn(v)); };
    put(0, w0 * M.s0); put(1, w0 * M.s1); put(2, w0 * M.s2);
    put(3, w1 * M.s0); put(4, w1 * M.s1); put(5, w1 * M.s2);
    put(6, w2 * M.s0); put(7, w2 * M.s1); put(8, w2 * M.s2);
    put(9, W * M.s11); put(10, W * M.s22); put(11, W * M.s12);
    atomicAdd(s0q, __float2int_rn(area * gs * M.s0));
}

// FP64 sums: an FP64 shared atomic is a loop of compare-and-swaps with an FP64 add in each, and the FP64
// pipe is what bounds the kernel.  So the lanes leave their moments in shared memory, and each owner
// takes the ones of its pair into its own column: one fused multiply-add a value.  Every lane calls it.
template <typename Sh>
__device__ __forceinline__ void items_gather(Sh &sh, bool has, int own, int q, const Mom<double> &M, int lane)
{
    if (has) {
        sh.mom[0][lane] = M.s0; sh.mom[1][lane] = M.s1; sh.mom[2][lane] = M.s2;
        sh.mom[3][lane] = M.s11; sh.mom[4][lane] = M.s22; sh.mom[5][lane] = M.s12;
        sh.momq[lane] = (unsigned char)q;
        atomicOr(&sh.dmask[own], 1u << lane);
        atomicAdd(&sh.s0q[q], sh.c64[own].area * M.s0);
    }
    __syncwarp();
    unsigned from = sh.dmask[lane];
    sh.dmask[lane] = 0;
    while (from) {
        const int i = __ffs(from) - 1;
        from &= from - 1;
        const double *w = sh.w[sh.momq[i]];
        const double s0 = sh.mom[0][i], s1 = sh.mom[1][i], s2 = sh.mom[2][i];
        for (int k = 0; k < 3; k++) {
            sh.acc[3 * k][lane] += w[k] * s0;
            sh.acc[3 * k + 1][lane] += w[k] * s1;
            sh.acc[3 * k + 2][lane] += w[k] * s2;
        }
        for (int k = 0; k < 3; k++) sh.acc[9 + k][lane] += w[3] * sh.mom[3 + k][i];
    }
    __syncwarp();
}

// Interior candidates of T_a: T_b whole for every outer point (certified when the lists are built,
// a relation symmetric in a and b).  The outer rules integrate quadratics exactly too, so the
// pair's blocks are closed forms of the two areas: M_ab = |T_a| |T_b| / 9 in all nine entries
// (formed by the scatter: nothing is stored), M_aa = |T_a| |T_b| (1 + delta_ij) / 12, and the
// M_bb that T_a receives as the inner triangle of its symmetric pairs is the same sum again.
template <int STS>
__device__ __forceinline__ void interior_const(const NumArgs &A, int a, int lane, LaneAcc &acc)
{
    const D2 ba = {A.bx[a], A.by[a]};
    double sum = 0.0;
    for (int64_t e = A.nbr_ptr[a] + lane; e < A.nbr_split[a]; e += 32) {
        const int b = A.nbr_idx[e];
#ifdef NL_CHECKS
        if (b < 0 || b >= A.K) {   // debug build: bad candidate recorded (bit 16) and skipped
            atomicOr(A.err, 16);
            continue;
        }
#endif
        sum += A.area[b];
        A.flag[e] = 1;
        int q0 = 0, q1 = A.outer.n;
        if (A.switch47) rule_range(A, ba, D2{A.bx[b], A.by[b]}, q0, q1);
        const int nq = q1 - q0;
        acc.qp += (uint32_t)(nq * A.inner.n);
        acc.cnt += A.outer_support ? 1u : (uint32_t)nq;
        if (want_stats<STS>(A))
            for (int q = 0; q < (A.outer_support ? 1 : nq); q++)
                acc.hsum += nlg::record_hash(a, b, q, nlg::KIND_WHOLE, 3, 0);
    }
    const double w = sum * A.area[a] * (1.0 / 12.0) * 2.0;
    for (int i = 0; i < 6; i++) acc.maa[i] += i < 3 ? 2.0 * w : w;
}

// Queue the round's marked items for k_deferred, ordered by owner lane and outer point (as
// defer_flush); items past the queue's capacity are integrated by their owner lane.
template <int BALL, int STS, typename Sh>
__device__ __forceinline__ void const_defer_flush(const NumArgs &A, int a, int64_t base, Sh &sh, int lane, float fxs,
                                                  LaneAcc &acc)
{
    const unsigned m = sh.dmask[lane];
    const int cnt = __popc(m);
    int inc = cnt;
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += y;
    }
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    if (total == 0) return;
    sh.dmask[lane] = 0;
    int slot0 = 0;
    if (lane == 0 && A.defer) slot0 = atomicAdd(A.defer_n, total);
    slot0 = __shfl_sync(0xffffffffu, slot0, 0);
    int slot = slot0 + inc - cnt;
    for (unsigned rest = m; rest; rest &= rest - 1, slot++) {
        const int q = __ffs(rest) - 1;
        if (A.defer && slot < A.defer_cap) {
            A.defer[slot] = DeferItem{base + lane, a, (A.prob << 8) | q};
            continue;
        }
        const Cand32 &cd = sh.cand[lane];
        const OuterPt &o = sh.sq[q];
        nlg::F2 dl[3];
        for (int i = 0; i < 3; i++) { dl[i].x = cd.vx[i] - o.lx; dl[i].y = cd.vy[i] - o.ly; }
        Mom<float> M;
        int nv, kind, ncap;
        bool used64;
        if (!exact_item<BALL, float>(A, cd.b, cd.area, dl, o.x, o.y, M, nv, kind, ncap, &used64)) continue;
        item_add(sh.w[q], M, sh.acc, &sh.s0q[q], lane, fxs, fabsf(cd.area), A.s0q_grid);
        sh.hit[lane] = 1;
        acc.cnt++;
        acc.qp += (uint32_t)region_points(A, kind, nv, ncap);
        if (want_stats<STS>(A)) acc.hsum += nlg::record_hash(a, cd.b, q - cd.q0, kind, nv, ncap);
    }
}

// The boundary candidates of outer triangle a, 32 at a time (one a lane): classification of every
// (q, b) in FP32 in lockstep, whole ones summed on the spot (their moments are 1), cut ones queued
// and drained by all lanes.
template <int BALL, typename T, int STS>
__device__ __forceinline__ void boundary_const(const NumArgs &A, int a, ConstShared<BALL, T> &sh, int lane,
                                               LaneAcc &acc)
{
    constexpr bool f32 = sizeof(T) == sizeof(float);
    using Fx = typename ConstShared<BALL, T>::Fx;
    const D2 ba = {A.bx[a], A.by[a]};
    const float4 bah = bary_hilo(A, a);
    const int64_t es = A.nbr_split[a], e1 = A.nbr_ptr[a + 1];
    const int nq_all = A.outer.n;
    // FP32 sums: one grid for all pairs of T_a (every moment is at most 1 on a part of T_b)
    float fxs = 0.f, inv_s = 0.f;
    if (f32) {
        const float r = fx_outer_bound(sh.sq, nq_all);
        const int e = ((__float_as_int(fmaxf(r, 1e-25f)) >> 23) & 0xff) - 126;   // r < 2^e
        fxs = __int_as_float((127 + 29 - e) << 23);
        inv_s = 1.f / fxs;
    }
    for (int q = lane; q < NL_MAXQ; q += 32) sh.s0q[q] = (Fx)0;
    for (int q = lane; q < nq_all; q += 32) {
        const OuterPt &o = sh.sq[q];
        const T W = f32 ? (T)o.Wf : (T)o.W;
        sh.w[q][0] = W * (f32 ? (T)o.l0f : (T)o.l0);
        sh.w[q][1] = W * (f32 ? (T)o.l1f : (T)o.l1);
        sh.w[q][2] = W * (f32 ? (T)o.l2f : (T)o.l2);
        sh.w[q][3] = W;
    }
    double ws = 0.0;   // sum of |T_b| over the whole items of outer point q = lane
    int nopen = 0;   // items the FP64 geometry decided here
    __syncwarp();
    for (int64_t base = es; base < e1; base += 32) {
        const int64_t e = base + lane;
        const bool valid = e < e1;
        int q0 = 0, q1 = 0;
        CandData c;
        c.b = a;
        c.akcf = 0.f;
        T area_b = 0;
        if (valid) {
            int b = A.nbr_idx[e];
#ifdef NL_CHECKS
            if (b < 0 || b >= A.K) {   // debug build: bad candidate recorded (bit 16), replaced by a
                atomicOr(A.err, 16);
                b = a;
            }
#endif
            load_cand(A, b, ba, bah, c, q1);
            q0 = c.q0;
            sh.cand[lane] = cand32_of(c);
            if constexpr (f32) {
                area_b = c.akcf;
            } else {
                const int64_t K = A.K;
                Cand64 d;
                d.x0 = A.tx[b];
                d.y0 = A.ty[b];
                const double x1 = A.tx[K + b], y1 = A.ty[K + b], x2 = A.tx[2 * K + b], y2 = A.ty[2 * K + b];
                d.area = A.area[b];
                const double inv = quot(0.5, d.area);
                d.v[0][0] = d.v[0][1] = 0.0;
                d.v[1][0] = d.e[0][0] = x1 - d.x0;
                d.v[1][1] = d.e[0][1] = y1 - d.y0;
                d.v[2][0] = x2 - d.x0;
                d.v[2][1] = y2 - d.y0;
                d.e[1][0] = x2 - x1;
                d.e[1][1] = y2 - y1;
                d.e[2][0] = -d.v[2][0];
                d.e[2][1] = -d.v[2][1];
                d.g[0][0] = inv * d.v[2][1];
                d.g[0][1] = -inv * d.v[2][0];
                d.g[1][0] = -inv * d.v[1][1];
                d.g[1][1] = inv * d.v[1][0];
                sh.c64[lane] = d;
                area_b = d.area;
            }
        }
        // The round's areas as integers, so that 32 of them are summed in one or two instructions and in no
        // order: 27 bits (FP32; an area has 24) or 54 in two limbs (FP64; an area has 53) under the power of
        // two above the round's largest area.  A grid of the mesh's largest area took the small triangles
        // of a graded mesh down to 1e-9 of themselves.
        constexpr int kExpBias = f32 ? 127 : 1023, kBits = f32 ? 27 : 54;
        unsigned ef;   // exponent field of the largest area
        if constexpr (f32) ef = (unsigned)__float_as_int(area_b) >> 23;
        else ef = (unsigned)__double2hiint(area_b) >> 20;
        ef = max(__reduce_max_sync(0xffffffffu, ef), (unsigned)kBits + 1u);
        unsigned a_hi = 0, a_lo, r_hi = 0, r_lo = 0;
        if constexpr (f32) {
            a_lo = __float2uint_rn(area_b * __int_as_float((2 * kExpBias + kBits - 1 - (int)ef) << 23));
        } else {
            const unsigned long long fx =
                __double2ull_rn(area_b * __hiloint2double((2 * kExpBias + kBits - 1 - (int)ef) << 20, 0));
            a_hi = (unsigned)(fx >> 27);
            a_lo = (unsigned)fx & ((1u << 27) - 1u);
        }
        for (int i = 0; i < 12; i++) sh.acc[i][lane] = (Fx)0;
        sh.dmask[lane] = 0;
        sh.hit[lane] = 0;
        int nqueue = 0, nwhole = 0;
        unsigned cutq = 0;   // outer points whose region of this lane's candidate is cut
        T u0 = 0, u1 = 0, u2 = 0;   // sum of W_q phi_a,i over the outer points that see all of T_b
        __syncwarp();
        for (int q = 0; q < nq_all; q++) {
            const bool active = valid && q >= q0 && q < q1;
            const OuterPt &o = sh.sq[q];
            int cls = nlg::CLS_EMPTY;
            if (active) {
                nlg::F2 dl[3];
                cls = classify_item<kGeoBall<BALL>, T, false>(A, c, o, dl);
            }
            const bool whole = cls == nlg::CLS_WHOLE;
            if (whole) {
                u0 += sh.w[q][0];
                u1 += sh.w[q][1];
                u2 += sh.w[q][2];
                nwhole++;
                if (want_stats<STS>(A)) acc.hsum += nlg::record_hash(a, c.b, q - q0, nlg::KIND_WHOLE, 3, 0);
            }
            const unsigned tl = __reduce_add_sync(0xffffffffu, whole ? a_lo : 0u);
            if (lane == q) r_lo = tl;
            if constexpr (!f32) {
                const unsigned th = __reduce_add_sync(0xffffffffu, whole ? a_hi : 0u);
                if (lane == q) r_hi = th;
            }
            if (cls == nlg::CLS_EXACT) cutq |= 1u << q;
        }
        if constexpr (f32) ws += (double)r_lo * (double)__int_as_float(((int)ef + 1 - kBits) << 23);
        else ws += (double)(((unsigned long long)r_hi << 27) + r_lo) * __hiloint2double(((int)ef + 1 - kBits) << 20, 0);
        // the cut items, every lane's first, then every lane's second, ...: neighbours in the queue have
        // different owners and outer points, so their adds rarely meet on one address
        for (unsigned m = __ballot_sync(0xffffffffu, cutq != 0u); m; m = __ballot_sync(0xffffffffu, cutq != 0u)) {
            if (cutq) {
                sh.queue[nqueue + __popc(m & ((1u << lane) - 1u))] = (unsigned short)((lane << 8) | (__ffs(cutq) - 1));
                cutq &= cutq - 1;
            }
            nqueue += __popc(m);
        }
        acc.cnt += (uint32_t)nwhole;
        acc.qp += (uint32_t)(nwhole * A.inner.n);
        __syncwarp();
        // cut items, 32 at a time; the ones the FP64 geometry has to decide are marked for
        // k_deferred (kConstQueue) or compacted at the front of the queue and done after the others
        int nslow = 0;
        for (int r0 = 0; r0 < nqueue; r0 += 32) {
            const bool live = r0 + lane < nqueue;
            const unsigned it = sh.queue[live ? r0 + lane : r0];   // the other lanes follow along
            const int own = it >> 8, q = it & 0xff;
            const Cand32 &cd = sh.cand[own];
            const OuterPt &o = sh.sq[q];
            nlg::F2 d[3];
            for (int k = 0; k < 3; k++) { d[k].x = cd.vx[k] - o.lx; d[k].y = cd.vy[k] - o.ly; }
            Mom<T> M;
            int nv = 0, kind = nlg::KIND_PARTIAL, ncap = 0, r = -1;
            T area = (T)fabsf(cd.area);
            if constexpr (BALL == NL_BALL_BARYCENTER || BALL == NL_BALL_OVERLAP) {
                // FP64 predicate on the whole triangle
            } else if constexpr (BALL == kBallNgonAny) {
                if constexpr (f32) {
                    int which = 0;
                    bool cut = false;
                    const int n = nlg::clip_ngon_f32_sh<true>(d, A.geo.err0, A.geo, sh.clip, lane, &which, &cut);
                    r = n < 0 ? -1 : n < 3 ? 0 : 1;
                    if (r == 1) {
                        // about the polygon's first vertex
                        const float x0 = sh.clip.x[which][0][lane], y0 = sh.clip.y[which][0][lane];
                        mom_set(M, 0.f);
                        float p1 = 0.f, p2 = 0.f;
                        for (int k = 1; k < n; k++) {
                            const float dx = sh.clip.x[which][k][lane] - x0, dy = sh.clip.y[which][k][lane] - y0;
                            const float q1 = dx * cd.gx[1] + dy * cd.gy[1], q2 = dx * cd.gx[2] + dy * cd.gy[2];
                            seg_add(M, p1, p2, q1, q2);
                            p1 = q1;
                            p2 = q2;
                        }
                        View32(cd, o).coords(x0, y0, p1, p2);
                        mom_shift(M, p1, p2);
                        nv = n;
                        kind = cut ? nlg::KIND_PARTIAL : nlg::KIND_WHOLE;
                    }
                }
            } else if constexpr (f32) {
                const View32 v(cd, o);
                if (!A.geo.turn)
                    r = cut_item<BALL, float>(A, live, d, v, v, BALL == NL_BALL_EXACTCAPS ? 1.f / area : 0.f, sh.corner,
                                              M, nv, kind, ncap);
            } else {
                const Cand64 &w = sh.c64[own];
                area = w.area;
                if (!A.geo.turn)
                    r = cut_item<BALL, double>(A, live, d, View32(cd, o), View64(w, o),
                                               BALL == NL_BALL_EXACTCAPS ? 1.0 / area : 0.0, sh.corner, M, nv, kind,
                                               ncap);
            }
            if constexpr (f32) {
                if (live && r > 0) {
                    if (cd.area < 0.f) mom_hold(M);
                    item_add(sh.w[q], M, sh.acc, &sh.s0q[q], own, fxs, area, A.s0q_grid);
                }
            } else {
                items_gather(sh, live && r > 0, own, q, M, lane);
            }
            if (live && r > 0) {
                sh.hit[own] = 1;
                acc.cnt++;
                acc.qp += (uint32_t)region_points(A, kind, nv, ncap);
                if (want_stats<STS>(A)) acc.hsum += nlg::record_hash(a, cd.b, q - cd.q0, kind, nv, ncap);
            }
            const bool slow = live && r < 0;
            if constexpr (kConstQueue<BALL, T>) {
                if (slow) atomicOr(&sh.dmask[own], 1u << q);
            } else {
                const unsigned ms = __ballot_sync(0xffffffffu, slow);   // also: every lane has read its item
                if (slow) sh.queue[nslow + __popc(ms & ((1u << lane) - 1u))] = (unsigned short)it;
                nslow += __popc(ms);
                __syncwarp();
            }
        }
        __syncwarp();
        if constexpr (kConstQueue<BALL, T>) {
            const_defer_flush<BALL, STS>(A, a, base, sh, lane, fxs, acc);
            __syncwarp();
        } else {
            for (int i0 = 0; i0 < nslow; i0 += 32) {
                const bool live = i0 + lane < nslow;
                const unsigned it = sh.queue[live ? i0 + lane : i0];
                const int own = it >> 8, q = it & 0xff;
                const Cand32 &cd = sh.cand[own];
                const OuterPt &o = sh.sq[q];
                Mom<T> M;
                int nv = 0, kind = 0, ncap = 0;
                bool has = false, used64 = kGeoBall<BALL> == NL_BALL_NGON;
                if (live) {
                    nlg::F2 d[3];
                    for (int k = 0; k < 3; k++) { d[k].x = cd.vx[k] - o.lx; d[k].y = cd.vy[k] - o.ly; }
                    has = exact_item<BALL, T>(A, cd.b, cd.area, d, o.x, o.y, M, nv, kind, ncap, &used64);
                    nopen += used64;
                }
                if constexpr (f32) {
                    if (has) item_add(sh.w[q], M, sh.acc, &sh.s0q[q], own, fxs, fabsf(cd.area), A.s0q_grid);
                } else {
                    items_gather(sh, has, own, q, M, lane);
                }
                if (has) {
                    sh.hit[own] = 1;
                    acc.cnt++;
                    acc.qp += (uint32_t)region_points(A, kind, nv, ncap);
                    if (want_stats<STS>(A)) acc.hsum += nlg::record_hash(a, cd.b, q - cd.q0, kind, nv, ncap);
                }
            }
            __syncwarp();
        }
        if (valid) {   // the owner's pair
            const int b = c.b;
            T P[9], Q[3], mab[9], mbb[6];
            bool big = false;
            for (int k = 0; k < 12; k++) {
                T v;
                if constexpr (f32) {
                    const int iv = sh.acc[k][lane];
                    big = big || iv >= (1 << 30) || iv <= -(1 << 30);
                    v = (float)iv * inv_s;
                } else {
                    v = sh.acc[k][lane];
                }
                if (k < 9) P[k] = v;
                else Q[k - 9] = v;
            }
            if (big) atomicOr(A.err, 256);
            T area;
            if constexpr (f32) area = c.akcf;
            else area = sh.c64[lane].area;
            pair_block<T>(f32 ? (T)fabsf(sh.cand[lane].area) : area, P, Q, mab, mbb);
            // the outer points that see all of T_b: their moments are 1, the blocks |T_b| u_i / 3 and
            // |T_b| sum_i u_i (1 + delta_ij) / 12 (kept apart from the cut ones, whose block is formed by
            // differences: in FP32 those would round the larger, whole part)
            const T k3 = area / (T)3, us[3] = {u0 * k3, u1 * k3, u2 * k3};
            for (int i = 0; i < 9; i++) mab[i] += us[i / 3];
            const T kw = (us[0] + us[1] + us[2]) * (T)0.25;
            for (int i = 0; i < 6; i++) mbb[i] += i < 3 ? (T)2 * kw : kw;
            const bool any = nwhole > 0 || sh.hit[lane] != 0;
            A.flag[e] = any ? 1 : 0;
            T *blk = (T *)A.blk;
            for (int i = 0; i < 9; i++) blk[(int64_t)i * A.E + e] = mab[i];
            if (any)
                for (int i = 0; i < 6; i++) atomicAdd(&A.mbb[(int64_t)i * A.K + b], (double)mbb[i]);
        }
        __syncwarp();
    }
    if (!kConstQueue<BALL, T> && nopen > 0 && A.defer_n) atomicAdd(A.defer_n, nopen);
    // M_aa / c = sum_q W_q phi_a(x_q) phi_a(x_q)^T sum_b int_{R(x_q, T_b)} 1, in FP64, one outer point a lane
    if (lane < nq_all) {
        double t;
        if constexpr (f32) {
            const int s = sh.s0q[lane];
            if (s >= (1 << 30) || s <= -(1 << 30)) atomicOr(A.err, 256);
            t = (double)s / (double)A.s0q_grid + ws;
        } else {
            t = sh.s0q[lane] + ws;
        }
        // W phi_a,i and W as the pairs' sums have them (FP32 path: rounded to FP32): M_aa, M_ab and M_bb are
        // then the blocks of one square (sum_i phi_a,i u_i - u(y))^2, and what rounding the weights costs
        // is not enlarged by the difference that D takes of them (deferred_const's few items take the FP64 weights
        // for M_aa)
        const double w0 = (double)sh.w[lane][0], w1 = (double)sh.w[lane][1], w2 = (double)sh.w[lane][2];
        const double s = t / (double)sh.w[lane][3];
        acc.maa[0] += s * w0 * w0; acc.maa[1] += s * w1 * w1; acc.maa[2] += s * w2 * w2;
        acc.maa[3] += s * w0 * w1; acc.maa[4] += s * w0 * w2; acc.maa[5] += s * w1 * w2;
    }
}

// all candidates of outer triangle a; the per-triangle outputs are stored (the only kernel that
// writes them before k_deferred adds)
template <int BALL, typename T, int STS>
__device__ __forceinline__ void const_outer(const NumArgs &A, int a, ConstShared<BALL, T> &sh, int lane)
{
    LaneAcc acc;
    acc_zero(acc);
    interior_const<STS>(A, a, lane, acc);
    if constexpr (kSupportBall<BALL>) {
        support_boundary<BALL, T>(A, a, lane, sh.clip, acc);
    } else {
        if constexpr (BALL == NL_BALL_NGON)
            for (int k = lane; k <= A.geo.ngon_n; k += 32) {
                const int kk = k == A.geo.ngon_n ? 0 : k;
                sh.corner[k] = make_float2((float)A.geo.ngon[2 * kk], (float)A.geo.ngon[2 * kk + 1]);
            }
        stage_outer(A, a, sh.sq, lane);
        __syncwarp();
        boundary_const<BALL, T, STS>(A, a, sh, lane, acc);
    }
    finish_outer<STS>(A, a, acc, lane, kStore);
}

// Measured (32-gon, delta = 0.1, 96 x 96 cells jittered, 16-point outer rule, 30 M cut items, one
// GB300): FP32 sums 1.50 ms against 4.2 ms for the point-by-point kernel it replaced (certified
// Sutherland-Hodgman clip into shared memory, 7-point rule on every fan triangle) plus 0.5 ms of its
// interior kernel; it issues in 71 % of the cycles with 24 of 32 lanes active.  FP64 sums 10.2 ms
// against 99.3 + 17.2 ms, with the FP64 pipe (1/64 of the FP32 rate) busy 87 % of the time: every FP64
// instruction saved counts there, whatever it costs elsewhere.
// (FP64: 64.8 KB of shared memory a block hold three blocks an SM.  The bound of four keeps 128 registers with a
// few hundred bytes of spills; a bound of three takes 168 with fewer and measured the same within 1 %, N-gon
// 0.6 % slower, approxcaps 0.7 % faster.)
template <typename T>
constexpr int kConstBlocksPerSm = sizeof(T) == sizeof(float) ? 5 : 4;

template <int BALL, typename T, int STS>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, kConstBlocksPerSm<T>) k_const(const NumArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ConstShared<BALL, T> &sh = ((ConstShared<BALL, T> *)smem_raw)[threadIdx.x >> 5];
    const int a = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    if (a < A.K) const_outer<BALL, T, STS>(A, a, sh, threadIdx.x & 31);
}

// a deferred item of the constant kernel (FP32 path): region and moments by the FP64 geometry, its
// M_ab into the queue's value slots, its M_bb, M_aa and statistics onto their sums
template <int BALL>
__device__ __forceinline__ void deferred_const(const NumArgs &A, const DeferItem &d, float *dv, int cap, int slot)
{
    const int K = A.K, a = d.a, q = d.qp & 0xff;
    const int64_t e = d.e;
#ifdef NL_CHECKS
    if (a < 0 || a >= K || e < 0 || e >= A.E || q >= A.outer.n) {   // debug build: bad item (bit 64), skipped
        atomicOr(A.err, 64);
        return;
    }
#endif
    const int b = A.nbr_idx[e];
    D2 Va[3];
    for (int i = 0; i < 3; i++) { Va[i].x = A.tx[i * K + a]; Va[i].y = A.ty[i * K + a]; }
    const OuterPt o = outer_point(A, a, Va, A.area[a], q);
    const D2 ba = {A.bx[a], A.by[a]};
    CandData c;
    int q1;
    load_cand(A, b, ba, bary_hilo(A, a), c, q1);
    nlg::F2 dl[3];
    for (int i = 0; i < 3; i++) { dl[i].x = c.vlx[i] - o.lx; dl[i].y = c.vly[i] - o.ly; }
    Mom<float> M;
    int kind, nv, ncap;
    bool used64;
    if (!exact_item<BALL, float>(A, b, 0.f, dl, o.x, o.y, M, nv, kind, ncap, &used64)) {
        for (int k = 0; k < kDeferVals; k++) dv[(int64_t)k * cap + slot] = 0.f;
        return;
    }
    const float la[3] = {o.l0f, o.l1f, o.l2f};
    float P[9], mab[9], mbb[6];
    for (int i = 0; i < 3; i++) {
        const float w = o.Wf * la[i];
        P[3 * i] = w * M.s0;
        P[3 * i + 1] = w * M.s1;
        P[3 * i + 2] = w * M.s2;
    }
    const float Q[3] = {o.Wf * M.s11, o.Wf * M.s22, o.Wf * M.s12};
    pair_block<float>(c.akcf, P, Q, mab, mbb);
    for (int k = 0; k < kDeferVals; k++) dv[(int64_t)k * cap + slot] = mab[k];
    for (int k = 0; k < 6; k++) atomicAdd(&A.mbb[(int64_t)k * K + b], (double)mbb[k]);
    const double ws = o.W * A.area[b] * (double)M.s0;
    const double m[6] = {ws * o.l0 * o.l0, ws * o.l1 * o.l1, ws * o.l2 * o.l2,
                         ws * o.l0 * o.l1, ws * o.l0 * o.l2, ws * o.l1 * o.l2};
    for (int k = 0; k < 6; k++) atomicAdd(&A.maa[(int64_t)k * K + a], m[k]);
    A.flag[e] = 1;
    atomicAdd((unsigned long long *)&A.qp_a[a], (unsigned long long)region_points(A, kind, nv, ncap));
    atomicAdd((unsigned long long *)&A.cnt_a[a], 1ull);
    if (A.stats)
        atomicAdd((unsigned long long *)&A.hash_a[a],
                  (unsigned long long)nlg::record_hash(a, b, q - c.q0, kind, nv, ncap));
}

}  // namespace nlq
