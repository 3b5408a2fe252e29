// Link-based lubrication of Ding and Aidun, as summarised in Sec. II
// (Eq. methods:dlub), for comparison with the contact-based corrections: for
// every D3Q19 link c_r that ends on a lattice site of particle i and stems
// from a site of particle j, or from a fluid site midway along 2 c_r from a
// site of j, a partial force
//   df = -3 qbar mu / (2 c_r^2 lambda*) c^ (c^ . (v_bi - v_bj)) (1/h*^2 - 1/c_r^2)
// on i where 0 < h* < c_r, and -df on j; h* is the distance along the link
// (or pair of links) between where it leaves j's surface and where it enters
// i's, v_b the rigid-body velocities there, lambda* the mean of the two
// surfaces' mean curvatures there.  Lattice sites are the integer points of
// the box coordinates (spacing 1); a site belongs to a particle when it lies
// in or on its spheroid, and a site in both is no stem; particle j is taken
// at its minimum image from i; a fluid site is in neither particle; the forces
// act at the two intersection points, torques about the centres; walls give
// nothing.
//
// A warp takes up to 8 pairs at a time (as few as give every resident warp some:
// below some 24,000 pairs the list does not fill the GPU and a warp's own chain
// is what counts).  What bounds the work is the FP64 pipe (two
// lanes per clock and SM: one warp instruction costs as much as some 70 on
// the other pipes), so every FP64 operation runs with all lanes busy, and
// what need not be FP64 is not:
//   set-up    the 16 bodies of the 8 pairs, one per lane, into shared memory;
//   sites     the integer points of the box where i's extent meets j's extent
//             widened by 2 on every axis (a link, or two, moves a site by at
//             most 2 per axis), one per lane, as integer offsets from each
//             centre's integer part: membership is decided in FP32 from
//             (float) offset - fraction (exact to about 1e-7) with a margin,
//             and again in FP64 inside the margin, so every decision is the
//             FP64 one; sites too deep in i or too far from j for any link
//             are dropped by the norms sqrt(quad) (a step of length s changes
//             one by at most s / R_min), the rest are gathered;
//   links     the (site, direction) pairs of the gathered sites, one per lane;
//             the links that qualify queue up, over all 8 pairs;
//   measure   32 queued links at a time, one per lane, in FP64, and their
//             sums per pair, nine components x three thirds of the links, one
//             per lane, in a fixed order.
// Measuring across pairs fills the lanes (a pair has some 35 links, so one
// batch of 32 per pair would be followed by a nearly empty one), and the
// set-up of one body per lane replaces one by all lanes for every pair.
// Measured: 65k pairs of a mixed suspension 1.175 ms (FP64 pipe 81 % busy),
// against 4.03 ms for one pair per warp with the set-up by all lanes and a
// measure per pair, and 1.335 with the measure on the box's own axes; 103 pairs
// 49 us (103 and, with batches of 8 whatever the list's length, 201).
#include "lub_internal.cuh"

namespace {

constexpr int LB = 8;             // most pairs per warp and batch (two bodies each: one per lane)
constexpr int LBLOCKS = 5;        // resident blocks (of four warps) per SM
constexpr int LQ = 64;            // queued links and gathered sites per warp: at most 31 waiting plus 32 new

// A particle at its (image) centre r: what the tests and the measure need.
struct Body {
    double r[3], o[3];
    double ia2, dc;     // 1 / R_perp^2, 1 / R_par^2 - 1 / R_perp^2
    double c2, kk;      // R_par^2, (R_perp^2 - R_par^2) / R_par^2 (curvature)
    double rr, rq;      // R_par R_perp, R_par / R_perp
    double v[3], w[3];
    int nint[3];        // floor of the centre (the anchor of the site offsets)
    float f[3];         // centre - floor, in float
    float of[3], ia2f, dcf;  // axis, 1 / R_perp^2 and dc in float
    float half[3];      // half extents along the axes
    float irmin;        // 1 / the smaller semi-axis
    float margin;       // of the FP32 membership test (decide)
};

// one queued link: the site of i (offset from i's anchor) and direction |
// (links from j's site: 1 or 2) << 8 | pair of the batch << 16
struct LinkEntry {
    int m[3];
    int tag;
};

struct LinkWarp {
    Body body[2 * LB];        // pair q: i at 2 q, j at 2 q + 1
    double res[9][33];        // the measured links' force on i and torques on i and j (rows padded)
    double acc[3][9][LB];     // their sums per pair, by thirds of the batches
    LinkEntry queue[LQ];
    int site[LQ][3];
    int nl[LB];
};

__device__ __forceinline__ void body_at(Body &b, const PView &P, int k, const V3<double> &r)
{
    const V3<double> o = quat_axis<double>(__ldg(P.qw + k), __ldg(P.qx + k), __ldg(P.qy + k), __ldg(P.qz + k));
    const float rpar = __ldg(P.rpar + k), rperp = __ldg(P.rperp + k);
    const double Rpar = widen_bits(rpar), Rperp = widen_bits(rperp);
    const double ia2 = 1.0 / (Rperp * Rperp), ic2 = 1.0 / (Rpar * Rpar);
    const double rv[3] = {r.x, r.y, r.z}, ov[3] = {o.x, o.y, o.z};
    b.ia2 = ia2;
    b.dc = ic2 - ia2;
    b.c2 = Rpar * Rpar;
    b.kk = (Rperp * Rperp - Rpar * Rpar) * ic2;
    b.rr = Rpar * Rperp;
    b.rq = Rpar * rcp64(Rperp);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double fl = floor(rv[a]);
        b.r[a] = rv[a];
        b.o[a] = ov[a];
        b.nint[a] = (int)fl;
        b.f[a] = (float)(rv[a] - fl);
        b.of[a] = (float)ov[a];
    }
    // the half extent sqrt(R_perp^2 (1 - o_a^2) + R_par^2 o_a^2) as a sum of
    // positive terms (1 - o_a^2 from the other two components, |o| = 1 to
    // 2^-23), which is good to some 2^-22 of itself for any shape: as
    // R_perp^2 + (R_par^2 - R_perp^2) o_a^2 it cancels for a disc whose axis is
    // close to a, and a site just inside a thin one (R_perp / R_par above some
    // 200 at R_perp = 100) would be missed; 1e-6 outward for the rounding
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float u = b.of[a], v = b.of[a == 2 ? 0 : a + 1], w = b.of[a == 0 ? 2 : a - 1];
        b.half[a] = 1.000001f * sqrtf(rperp * rperp * (v * v + w * w) + rpar * rpar * (u * u));
    }
    b.ia2f = (float)ia2;
    b.dcf = (float)(ic2 - ia2);
    b.irmin = 1.0f / fminf(rpar, rperp);
    const float ratio = fmaxf(rpar, rperp) * b.irmin;
    b.margin = 8e-6f * (1.0f + ratio * ratio) + 1e-6f * ratio * b.irmin;
    b.v[0] = widen_bits(__ldg(P.vx + k));
    b.v[1] = widen_bits(__ldg(P.vy + k));
    b.v[2] = widen_bits(__ldg(P.vz + k));
    b.w[0] = widen_bits(__ldg(P.wx + k));
    b.w[1] = widen_bits(__ldg(P.wy + k));
    b.w[2] = widen_bits(__ldg(P.wz + k));
}

// (x - r)^T M^-1 (x - r) for the site x = floor(r) + m (m: integer offset
// from the body's anchor), in FP32 from (float) m - frac r, and in FP64
__device__ __forceinline__ float quad_f(const Body &b, int m0, int m1, int m2)
{
    const float u0 = (float)m0 - b.f[0], u1 = (float)m1 - b.f[1], u2 = (float)m2 - b.f[2];
    const float ou = b.of[0] * u0 + b.of[1] * u1 + b.of[2] * u2;
    return (u0 * u0 + u1 * u1 + u2 * u2) * b.ia2f + ou * ou * b.dcf;
}

__device__ __noinline__ bool inside_d(const Body &b, int m0, int m1, int m2)
{
    const int m[3] = {m0, m1, m2};
    double u[3];
    for (int a = 0; a < 3; ++a) u[a] = (double)(b.nint[a] + m[a]) - b.r[a];
    const double ou = b.o[0] * u[0] + b.o[1] * u[1] + b.o[2] * u[2];
    return (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) * b.ia2 + ou * ou * b.dc <= 1.0;
}

// membership from the FP32 value q, decided in FP64 inside the margin: the
// terms of quad_f are of order ratio^2 (|u|^2 / R_perp^2 against a negative
// (o.u)^2 dc for a prolate), each within a few 2^-24 of its value, so q is
// within some 20 2^-24 (1 + ratio^2) of the exact one, and the fraction's
// rounding adds 2^-23 ratio / R_min; the margin is six to eight times that
__device__ __forceinline__ bool decide(const Body &b, float q, int m0, int m1, int m2)
{
    if (q < 1.0f - b.margin) return true;
    if (q > 1.0f + b.margin) return false;
    return inside_d(b, m0, m1, m2);
}

__device__ __forceinline__ bool inside(const Body &b, int m0, int m1, int m2)
{
    return decide(b, quad_f(b, m0, m1, m2), m0, m1, m2);
}

// the 18 nonzero D3Q19 lattice vectors, two bits per component and vector
// (component + 1): (+-1,0,0), (0,+-1,0), (0,0,+-1), then the face diagonals
// (+-1,+-1,0), (+-1,0,+-1), (0,+-1,+-1)
constexpr int kD3Q19[18][3] = {{1, 0, 0},  {-1, 0, 0}, {0, 1, 0},  {0, -1, 0},  {0, 0, 1},  {0, 0, -1},
                               {1, 1, 0},  {-1, -1, 0}, {1, -1, 0}, {-1, 1, 0},  {1, 0, 1},  {-1, 0, -1},
                               {1, 0, -1}, {-1, 0, 1},  {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
constexpr unsigned long long d3q19_bits(int a)
{
    unsigned long long v = 0;
    for (int r = 0; r < 18; ++r) v |= (unsigned long long)(kD3Q19[r][a] + 1) << (2 * r);
    return v;
}
__device__ __forceinline__ int d3q19(int r, int a)
{
    constexpr unsigned long long bits[3] = {d3q19_bits(0), d3q19_bits(1), d3q19_bits(2)};
    return (int)((a == 0 ? bits[0] : a == 1 ? bits[1] : bits[2]) >> (2 * r) & 3) - 1;
}

// the double of an integer below 2^24 in magnitude, off the FP64 pipe
__device__ __forceinline__ double small_int(int m)
{
    return abs(m) < (1 << 24) ? widen_bits((float)m) : (double)m;
}

// c x for c = -1 or 1, and for c = -1, 0 or 1, on the integer pipe
__device__ __forceinline__ double with_sign(int c, double x)
{
    return __hiloint2double(__double2hiint(x) ^ (c & 0x80000000), __double2loint(x));
}
__device__ __forceinline__ double times_sign(int c, double x) { return c ? with_sign(c, x) : 0.0; }

// The measure works on axes turned cyclically, (p, q, k), so that the lattice
// vector is (cp, cq, 0) with cp = -1 or 1: its products with vectors are then
// one addition each instead of two, and its cross products one instead of
// three.  The bodies' components come from shared memory at the turned
// indices, so the turn costs address arithmetic only.
struct LinkAxes {
    int p, q, k, cp, cq;
};
__device__ __forceinline__ LinkAxes link_axes(int r)
{
    LinkAxes x;
    x.p = r < 6 ? r >> 1 : r < 10 ? 0 : r < 14 ? 2 : 1;
    x.q = x.p == 2 ? 0 : x.p + 1;
    x.k = x.p == 0 ? 2 : x.p - 1;
    x.cp = d3q19(r, x.p);
    x.cq = d3q19(r, x.q);
    return x;
}

// The line x0 + t c (c: a lattice vector in turned axes) and body b: t of the
// smaller or larger crossing of its surface, from x0 - r = u; false where it
// misses.  uxc: the third component of u x c (the others are -cq u_k and
// cp u_k).  H: twice the mean curvature at the crossing (radii of
// curvature of Eq. lub:curvature-radii): with z the crossing's height along
// the axis and sin^2 p = z^2 / R_par^2, cos^2 p = 1 - sin^2 p on the surface,
// s1^2 = R_perp^2 sin^2 p + R_par^2 cos^2 p, 1/S1 = R_par R_perp / s1^3 and
// 1/S2 = R_par / (R_perp s1).  (Signs and zeros are tested on the integer
// pipe: a comparison costs as much as a multiply-add.)
template <bool LARGER>
__device__ __forceinline__ bool cross_surface(const Body &b, const double u[3], const LinkAxes &c, double &t, double &H,
                                              double &uxc)
{
    const double op = b.o[c.p], oq = b.o[c.q], ok = b.o[c.k];
    const double ou = op * u[0] + oq * u[1] + ok * u[2];
    const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const double oc = with_sign(c.cp, op) + times_sign(c.cq, oq);
    const double uc = with_sign(c.cp, u[0]) + times_sign(c.cq, u[1]);
    const int diag = c.cq != 0;
    const double ia2 = b.ia2, dc = b.dc;
    // |c|^2 / R_perp^2 by the exponent
    const double ccia2 = __hiloint2double(__double2hiint(ia2) + (diag << 20), __double2loint(ia2));
    const double dou = dc * ou;
    const double A = fma(oc * oc, dc, ccia2);
    const double B = fma(dou, oc, uc * ia2);  // half the linear coefficient
    const double C = fma(dou, ou, fma(uu, ia2, -1.0));
    const double disc = fma(B, B, -A * C);
    if ((unsigned)__double2hiint(disc) >= 0x7ff00000u) return false;  // negative (never -0) or not finite
    const double sq = __double2hiint(disc) | __double2loint(disc) ? disc * rsqrt64(disc) : 0.0;
    t = ((LARGER ? sq : -sq) - B) * rcp64(A);
    const double z = fma(t, oc, ou);
    const double is1 = rsqrt64(fma(b.kk * z, z, b.c2));
    H = is1 * fma(b.rr * is1, is1, b.rq);
    uxc = times_sign(c.cq, u[0]) - with_sign(c.cp, u[1]);
    return true;
}

// Measures the first min(32, queued) entries of the queue, adds their forces
// and torques to the pairs' sums and moves the rest of the queue to the front;
// returns what is left.  Out of line: called from two places, and the scan's
// loops then stay small (inlined, the warps waited for instructions).
__device__ __noinline__ int measure_links(LinkWarp &W, int queued, double2 pre)
{
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    __syncwarp();
    const int n = queued < 32 ? queued : 32;
    // (an entry past the queue's end is read but not used)
    const int tag = W.queue[lane].tag;
    const LinkAxes c = link_axes(lane < n ? tag & 255 : 0);
    const int m[3] = {W.queue[lane].m[c.p], W.queue[lane].m[c.q], W.queue[lane].m[c.k]};
    const LinkEntry nx = W.queue[32 + lane];
    __syncwarp();
    if (lane < queued - 32) W.queue[lane] = nx;
    double Fp = 0.0, Fq = 0.0, Ti[3] = {0, 0, 0}, Tj[3] = {0, 0, 0};  // in turned axes (F has no third)
    const int pr = lane < n ? tag >> 16 : 0;
    if (lane < n) {
        const Body &bi = W.body[2 * pr], &bj = W.body[2 * pr + 1];
        const int r = tag & 255, kind = (tag >> 8) & 255;
        const int ax[3] = {c.p, c.q, c.k}, cs[3] = {c.cp, c.cq, 0};
        double ui[3], uj[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double x0 = small_int(bi.nint[ax[a]] + m[a] - kind * cs[a]);
            ui[a] = x0 - bi.r[ax[a]];
            uj[a] = x0 - bj.r[ax[a]];
        }
        double ti, tj, Hi, Hj, xi, xj;
        const bool mi = cross_surface<false>(bi, ui, c, ti, Hi, xi);
        const bool mj = cross_surface<true>(bj, uj, c, tj, Hj, xj);
        const double tau = ti - tj;  // h* / c_r; 0 < tau < 1:
        const int th = __double2hiint(tau);
        if (mi && mj && (unsigned)th < 0x3ff00000u && (th | __double2loint(tau))) {
            // c.(v_i + w_i x a_i - v_j - w_j x a_j), with c.(w x a) = w.(a x c) = w.(u x c)
            const double cv = with_sign(c.cp, bi.v[c.p] - bj.v[c.p]) + times_sign(c.cq, bi.v[c.q] - bj.v[c.q]) +
                              ui[2] * (with_sign(c.cp, bi.w[c.q]) - times_sign(c.cq, bi.w[c.p])) + bi.w[c.k] * xi -
                              uj[2] * (with_sign(c.cp, bj.w[c.q]) - times_sign(c.cq, bj.w[c.p])) - bj.w[c.k] * xj;
            // df = -3 qbar mu / (2 c_r^2 lambda) (c/c_r) (c/c_r . dv) (1/h*^2 - 1/c_r^2),
            // lambda = (H_i + H_j) / 4, h* = tau c_r, c_r^6 = 8 on the diagonals
            const double t2 = tau * tau;
            const double s = (r >= 6 ? pre.y : pre.x) * cv * (1.0 - t2) * rcp64((Hi + Hj) * t2);
            Fp = with_sign(c.cp, s);
            Fq = times_sign(c.cq, s);
            const double sui = s * ui[2], suj = s * uj[2];
            Ti[0] = -times_sign(c.cq, sui);
            Ti[1] = with_sign(c.cp, sui);
            Ti[2] = s * xi;
            Tj[0] = times_sign(c.cq, suj);
            Tj[1] = -with_sign(c.cp, suj);
            Tj[2] = -s * xj;
            atomicAdd(&W.nl[pr], 1);
        }
    }
    {
        const double F[3] = {Fp, Fq, 0.0};
        const int ax[3] = {c.p, c.q, c.k};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            W.res[ax[a]][lane] = F[a];
            W.res[3 + ax[a]][lane] = Ti[a];
            W.res[6 + ax[a]][lane] = Tj[a];
        }
    }
    __syncwarp();
    const int part = lane / 9, comp = lane - 9 * part;
    const int e0 = part * 11, e1 = part < 2 ? e0 + 11 : 32;
    int cur = -1;
    double run = 0.0;
    for (int e = 0; e < 11; ++e) {
        const int at = e0 + e < e1 ? e0 + e : 31;
        const int p = __shfl_sync(FULL, pr, at);
        if (part < 3 && e0 + e < e1 && e0 + e < n) {
            if (p != cur) {
                if (cur >= 0) W.acc[part][comp][cur] += run;
                cur = p;
                run = 0.0;
            }
            run += W.res[comp][at];
        }
    }
    if (cur >= 0) W.acc[part][comp][cur] += run;
    __syncwarp();
    return queued - n;
}

template <bool ENS>
__global__ void __launch_bounds__(128, LBLOCKS) k_links(PView P, const __grid_constant__ DView D0, Ens E,
                                               const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                                               const int32_t *__restrict__ d_count, int32_t cap, double mu,
                                               double qbar, double *__restrict__ force, double *__restrict__ torque,
                                               int32_t *__restrict__ nlinks, int resident)
{
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char links_raw[];
    LinkWarp &W = reinterpret_cast<LinkWarp *>(links_raw)[threadIdx.x >> 5];
    const int count = pair_count(d_count, cap);
    const size_t C = (size_t)cap;
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu, below = (1u << lane) - 1u;
    const int nwarp = (gridDim.x * blockDim.x) >> 5;
    // pairs per batch: enough that every resident warp has one.  Measured with
    // 1, 2, 4 and 8 (us): 100 pairs 57, 75, 108, 195; 2,000 92, 90, 131, 221;
    // 6,000 161, 156, 181, 255; 20,000 474, 417, 408, 416; 60,000 1321, 1107,
    // 1003, 1047
    const int per = min(LB, max(1, (count + resident - 1) / resident));
    // factors of a link along an axis, and of a diagonal (c_r^6 = 8)
    const double2 pre = make_double2(-6.0 * qbar * mu, -6.0 * qbar * mu * 0.125);
    for (int64_t k0 = (int64_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per; k0 < count;
         k0 += (int64_t)nwarp * per) {
        const int np = (int)(count - k0 < per ? count - k0 : per);
        // the bodies: lane 2 q takes i of pair q, lane 2 q + 1 takes j
        unsigned valid;
        {
            const int q = lane >> 1;
            bool ok = false;
            if (q < np) {
                const int i = __ldg(pi + k0 + q), j = __ldg(pj + k0 + q);
                bool alien = false;
                const DView &D = pair_domain<ENS>(D0, E, i, j, &alien);
                ok = !alien && i >= 0 && i < P.n && j >= 0 && j < P.n && i != j &&
                     shape_ok(__ldg(P.rpar + i), __ldg(P.rperp + i)) && shape_ok(__ldg(P.rpar + j), __ldg(P.rperp + j));
                if (ok) {
                    V3<double> r = load_pos(P, i);
                    if (lane & 1) r = add(r, min_image(D, sub(load_pos(P, j), r)));
                    body_at(W.body[lane], P, lane & 1 ? j : i, r);
                }
            }
            valid = __ballot_sync(FULL, ok);
            for (int e = lane; e < 3 * 9 * LB; e += 32) (&W.acc[0][0][0])[e] = 0.0;
            if (lane < LB) W.nl[lane] = 0;
        }
        __syncwarp();
        int queued = 0;  // links waiting (warp-uniform)
        for (int q = 0; q < np; ++q) {
            if (!((valid >> (2 * q)) & 1u)) continue;
            const Body &bi = W.body[2 * q], &bj = W.body[2 * q + 1];
            // the box of sites as offsets m from i's anchor (the same site is
            // m + dij from j's); 1e-3 outward for the FP32 sums
            int lo[3], nn[3], dij[3];
            int nsites = 1;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                dij[a] = bi.nint[a] - bj.nint[a];
                const int l = max((int)ceilf(bi.f[a] - bi.half[a] - 1e-3f),
                                  (int)ceilf(bj.f[a] - bj.half[a] - 2.001f) - dij[a]);
                const int h = min((int)floorf(bi.f[a] + bi.half[a] + 1e-3f),
                                  (int)floorf(bj.f[a] + bj.half[a] + 2.001f) - dij[a]);
                lo[a] = l;
                nn[a] = max(h - l + 1, 0);
                nsites *= nn[a];
            }
            if (nsites <= 0) continue;
            // a site that ends a link is in i within sqrt(2) of a site outside
            // i, and within 2 sqrt(2) of a site of j
            const float deep = fmaxf(1.0f - 1.4143f * bi.irmin, 0.f), far = 1.0f + 2.8286f * bj.irmin;
            const float qi_min = deep * deep - 2.0f * bi.margin, qj_max = far * far * (1.0f + 2.0f * bj.margin);
            const int n0 = nn[0], n01 = nn[0] * nn[1];
            const float in0 = 1.0f / (float)n0, in01 = 1.0f / (float)n01;
            int ns = 0;  // gathered sites (warp-uniform)
            for (int q0 = 0;; q0 += 32) {
                const bool last = q0 + 32 >= nsites;
                const int e = q0 + lane;
                int m0 = 0, m1 = 0, m2 = 0;
                bool site = false;
                if (e < nsites) {
                    // e = (z n1 + y) n0 + x by FP32 quotients, corrected to the exact ones
                    int z = (int)((float)e * in01);
                    int rem = e - z * n01;
                    if (rem < 0) { --z; rem += n01; }
                    if (rem >= n01) { ++z; rem -= n01; }
                    int y = (int)((float)rem * in0);
                    int x = rem - y * n0;
                    if (x < 0) { --y; x += n0; }
                    if (x >= n0) { ++y; x -= n0; }
                    m0 = lo[0] + x;
                    m1 = lo[1] + y;
                    m2 = lo[2] + z;
                    const float qi = quad_f(bi, m0, m1, m2);
                    site = qi >= qi_min && qi <= 1.0f + bi.margin &&
                           quad_f(bj, m0 + dij[0], m1 + dij[1], m2 + dij[2]) <= qj_max && decide(bi, qi, m0, m1, m2);
                }
                const unsigned hit = __ballot_sync(FULL, site);
                if (site) {
                    int *s = W.site[ns + __popc(hit & below)];
                    s[0] = m0;
                    s[1] = m1;
                    s[2] = m2;
                }
                ns += __popc(hit);
                // the links of the gathered sites, 32 sites at a time
                while (ns >= 32 || (last && ns > 0)) {
                    __syncwarp();
                    const int n = ns < 32 ? ns : 32;
                    const int total = 18 * n;
                    for (int e0 = 0; e0 < total; e0 += 32) {
                        const int e = e0 + lane;
                        int kind = 0, m0 = 0, m1 = 0, m2 = 0, r = 0;
                        if (e < total) {
                            const int sidx = (e * 3641) >> 16;  // e / 18 for e < 576
                            r = e - 18 * sidx;
                            m0 = W.site[sidx][0];
                            m1 = W.site[sidx][1];
                            m2 = W.site[sidx][2];
                            const int c0 = d3q19(r, 0), c1 = d3q19(r, 1), c2 = d3q19(r, 2);
                            const int a0 = m0 - c0, a1 = m1 - c1, a2 = m2 - c2;
                            if (!inside(bi, a0, a1, a2)) {
                                if (inside(bj, a0 + dij[0], a1 + dij[1], a2 + dij[2])) {
                                    kind = 1;
                                } else {
                                    const int b0 = a0 - c0, b1 = a1 - c1, b2 = a2 - c2;
                                    if (inside(bj, b0 + dij[0], b1 + dij[1], b2 + dij[2]) && !inside(bi, b0, b1, b2))
                                        kind = 2;
                                }
                            }
                        }
                        const unsigned hit = __ballot_sync(FULL, kind != 0);
                        if (!hit) continue;
                        if (kind) {
                            LinkEntry &en = W.queue[queued + __popc(hit & below)];
                            en.m[0] = m0;
                            en.m[1] = m1;
                            en.m[2] = m2;
                            en.tag = r | kind << 8 | q << 16;
                        }
                        queued += __popc(hit);
                        if (queued >= 32) queued = measure_links(W, queued, pre);
                    }
                    // the rest to the front
                    __syncwarp();
                    int s0 = 0, s1 = 0, s2 = 0;
                    const bool mv = lane < ns - 32;
                    if (mv) {
                        s0 = W.site[32 + lane][0];
                        s1 = W.site[32 + lane][1];
                        s2 = W.site[32 + lane][2];
                    }
                    __syncwarp();
                    if (mv) {
                        W.site[lane][0] = s0;
                        W.site[lane][1] = s1;
                        W.site[lane][2] = s2;
                    }
                    ns -= n;
                }
                if (last) break;
            }
        }
        while (queued > 0) queued = measure_links(W, queued, pre);
        __syncwarp();
        // rows of consecutive pairs: lane = pair (half warps take alternate rows)
        const int q = lane & (LB - 1), row0 = lane / LB;
        if (q < np) {
            for (int row = row0; row < 9; row += 32 / LB) {
                const double v = W.acc[0][row][q] + W.acc[1][row][q] + W.acc[2][row][q];
                double *dst = row < 3 ? force + row * C : torque + (row - 3) * C;
                dst[k0 + q] = v;
            }
            if (nlinks && row0 == 0) nlinks[k0 + q] = W.nl[q];
        }
        __syncwarp();  // the batch's shared memory is reused
    }
}

}  // namespace

int launch_links(lub_ctx *ctx, const PView &P, const DView &D, const Ens &E, const int32_t *pi, const int32_t *pj,
                 const int32_t *d_count, int32_t cap, double mu, double qbar, double *force, double *torque,
                 int32_t *nlinks, cudaStream_t st)
{
    if (cap == 0) return LUB_OK;
    const int block = 128;
    const size_t smem = (block / 32) * sizeof(LinkWarp);
    static_assert(LBLOCKS * (4 * sizeof(LinkWarp) + 1024) <= 228 * 1024, "the resident blocks fit an SM's shared memory");
    const int warps = block / 32;
    // a warp per batch of LB pairs, or (short lists, in batches of fewer) one wave of blocks
    int64_t grid = ((int64_t)cap + LB * warps - 1) / (LB * warps);
    const int64_t wave = (int64_t)LBLOCKS * ctx->num_sms, each = ((int64_t)cap + warps - 1) / warps;
    if (grid < wave) grid = each < wave ? each : wave;
    if (grid > 64 * (int64_t)ctx->num_sms) grid = 64 * (int64_t)ctx->num_sms;
    const int resident = (int)wave * warps;
    int rc = lub_check_cuda(ctx,
                            cudaFuncSetAttribute(E.nb ? k_links<true> : k_links<false>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                            "shared memory attribute");
    if (rc) return rc;
    const auto kernel = E.nb ? k_links<true> : k_links<false>;
    cudaError_t e;
    if (grid <= wave) {
        // (a plain launch: its blocks are spread over all SMs, not packed on those
        // that the kernel before leaves first)
        kernel<<<(int)grid, block, smem, st>>>(P, D, E, pi, pj, d_count, cap, mu, qbar, force, torque, nlinks, resident);
        e = cudaGetLastError();
    } else {
        e = launch_pdl(kernel, (int)grid, block, smem, st, P, D, E, pi, pj, d_count, cap, mu, qbar, force, torque,
                       nlinks, resident);
    }
    return lub_check_cuda(ctx, e, "k_links launch");
}
