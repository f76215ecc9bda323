// K1: per-primitive projection for every registered view -- the range key, the sign that turns
// the normal towards the sensor, and the conservative spherical bounding box of the region of the
// 3-sigma box where the primitive can reach alpha_min, with its tile rectangle (Sec. 3.2.1 tiles
// and range sort; Sec. 3.2.3 bounding box computation; Supp. B).
//
// Everything in this file takes integer decisions (which tiles, which order, which sign), so it
// follows a fixed binary32 contract: every value is produced by the same sequence of correctly
// rounded IEEE operations on every machine.  The file is compiled with -fmad=false so that no
// a*b+c is fused; fused multiply-adds appear only where written as fmaf.  The arctangent and
// exponential and logarithm used by the contract are evaluated from their series (see
// contract_atan2, contract_exp, contract_log), never through a math library.
//
// A CTA takes a block of primitives, kProjectThreads at a time; a thread reads its primitive's 40
// bytes once (coalesced float4/float2 loads) and, view by view, forms the pair's centre and bounds
// the box with approximate arithmetic (quick_box).  The contract's box costs about
// 1,400 instructions, most of them correctly rounded roots and quotients; what it decides is four
// integers, and wherever the approximate bounds of all four lie clear of the next pixel by more
// than both computations' errors the integers are already known.  The few pairs left (a bound
// within a few thousandths of a pixel of a boundary, near or steep primitives: 1 % of the
// pairs along a long street, 3-4 % in a street or block) are queued per warp and boxed by the
// contract 32 at a time.  Projection of 12 x 500 k pairs: 0.214 -> 0.19 ms, in a refinement with
// the gradient accumulators zeroed on the way; of 8 x 1 M pairs along a 600 m street: 0.278
// -> 0.188 ms.  Bound by instruction issue: in that refinement 67 % of the slots, 700 instructions
// per warp and view.
//
// A pair leaves its pixel rectangle with the normal-flip bit (8 bytes, zero when it touches no
// tile).  A pair that touches a tile also appends its tile rectangle and range key (12 bytes) to
// the segment of its view and block, from which the lists are built; the pairs of a view that was
// not drawn for this step leave nothing.  Each primitive also gets the
// 64 bytes the compositing kernels stage for it -- its scaled tangent axes, normal, opacity and
// centre, in the world frame -- so that they need not redo the quaternion and exponentials for
// every (block, list entry), and read them as two whole sectors.

#include <cmath>

#include "splat_internal.cuh"

namespace splat {
namespace {

constexpr float kPi = 3.14159274f;      // nearest binary32 values
constexpr float kHalfPi = 1.57079637f;
constexpr float kTwoPi = 6.28318548f;
constexpr float kQuarterPi = 0.785398163f;
constexpr float kTanPi8 = 0.414213562f;
constexpr float kPixelMargin = 0.01f;   // pixel units, both axes

// atan2 from the arctangent series: reduce to t = min/max in [0, 1], fold t > tan(pi/8) with
// atan t = pi/4 + atan((t - 1)/(t + 1)), then z - z^3/3 + ... + z^17/17 on |z| <= tan(pi/8).
__device__ float contract_atan2(float y, float x)
{
    const float ax = fabsf(x), ay = fabsf(y);
    const float hi = ax > ay ? ax : ay;
    const float lo = ax > ay ? ay : ax;
    if (hi == 0.0f) return 0.0f;
    const float t = lo / hi;
    float z, base;
    if (t > kTanPi8) {
        z = (t - 1.0f) / (t + 1.0f);
        base = kQuarterPi;
    } else {
        z = t;
        base = 0.0f;
    }
    const float z2 = z * z;
    float p = 0.0588235294f;
    p = fmaf(p, z2, -0.0666666667f);
    p = fmaf(p, z2, 0.0769230769f);
    p = fmaf(p, z2, -0.0909090909f);
    p = fmaf(p, z2, 0.111111111f);
    p = fmaf(p, z2, -0.142857143f);
    p = fmaf(p, z2, 0.2f);
    p = fmaf(p, z2, -0.333333333f);
    p = fmaf(p, z2, 1.0f);
    float a = fmaf(z, p, base);
    if (ay > ax) a = kHalfPi - a;
    if (x < 0.0f) a = kPi - a;
    if (y < 0.0f) a = -a;
    return a;
}

// exp from a Cody-Waite split of ln 2 (2839/4096 plus its binary32 remainder) and the
// exponential series through r^7/7!; 2^k is assembled in the exponent field.
__device__ float contract_exp(float x)
{
    x = x > 80.0f ? 80.0f : x;
    x = x < -80.0f ? -80.0f : x;
    const float k = rintf(x * 1.44269504f);
    const float r = (x - k * 0.693115234375f) - k * 3.19461849e-05f;
    float p = 1.98412698e-04f;
    p = fmaf(p, r, 1.38888889e-03f);
    p = fmaf(p, r, 8.33333333e-03f);
    p = fmaf(p, r, 4.16666667e-02f);
    p = fmaf(p, r, 0.166666667f);
    p = fmaf(p, r, 0.5f);
    p = fmaf(p, r, 1.0f);
    p = fmaf(p, r, 1.0f);
    const int ki = static_cast<int>(k);
    return p * __uint_as_float(static_cast<uint32_t>(ki + 127) << 23);
}

// ln for the contract, x >= 1: x = 2^e m with m folded into [1/sqrt2, sqrt2), then
// ln m = 2 atanh z, z = (m - 1)/(m + 1), from the series 2(z + z^3/3 + ... + z^9/9).
__device__ float contract_log(float x)
{
    const uint32_t u = __float_as_uint(x);
    int e = static_cast<int>((u >> 23) & 0xFFu) - 127;
    float m = __uint_as_float((u & 0x7FFFFFu) | 0x3F800000u);
    if (m > 1.41421354f) {
        m = m * 0.5f;
        e = e + 1;
    }
    const float z = (m - 1.0f) / (m + 1.0f);
    const float z2 = z * z;
    float p = 0.111111111f;
    p = fmaf(p, z2, 0.142857143f);
    p = fmaf(p, z2, 0.2f);
    p = fmaf(p, z2, 0.333333333f);
    p = fmaf(p, z2, 1.0f);
    return fmaf(static_cast<float>(e), 0.693147182f, 2.0f * z * p);
}

struct v3 {
    float x, y, z;
};

// R v with R row-major, each row summed as ((a + b) + c)
__device__ __forceinline__ v3 rot(const float *R, v3 v)
{
    return v3{(R[0] * v.x + R[1] * v.y) + R[2] * v.z, (R[3] * v.x + R[4] * v.y) + R[5] * v.z,
              (R[6] * v.x + R[7] * v.y) + R[8] * v.z};
}

// keep the higher and the lower of the points seen so far, by elevation atan2(z, r), r >= 0:
// z r' > z' r says that (z, r) lies above (z', r'); the first of equal points stays
__device__ __forceinline__ void elev_candidate(float z, float r, float &zh, float &rh, float &zl,
                                               float &rl, bool &have)
{
    if (!have) {
        zh = z; rh = r; zl = z; rl = r;
        have = true;
        return;
    }
    if (z * rh > zh * r) { zh = z; rh = r; }
    if (z * rl < zl * r) { zl = z; rl = r; }
}

// The view-independent part: the reach radius r_o, the half-side a and the octagon's cut c (in
// units of a) of a primitive with opacity o; false when o stays below alpha_min everywhere.
struct Octagon {
    float a, k, c;
};

__device__ bool contract_octagon(float o, float alpha_min, float sigma, Octagon &oct)
{
    float x = o / alpha_min;
    if (x < 0.999f) return false;
    if (x < 1.0f) x = 1.0f;
    const float ro = sqrtf(2.0f * contract_log(x)) * 1.001f + 0.002f;
    const float a = ro < sigma ? ro : sigma;
    const float k = (1.41421356f * ro) / a;
    // the octagon (|u|, |w| <= 1, |u| + |w| <= k in units of a); when the diamond misses the
    // square's corners (k >= 2) the cut c = 1 repeats each corner, and the repeated vertices give
    // zero-length edges that add nothing
    oct.a = a;
    oct.k = k;
    oct.c = k < 2.0f ? k - 1.0f : 1.0f;
    return true;
}

// Spherical bounding box of the splat-space region where the primitive can contribute: the
// 3-sigma box |s|_inf <= sigma intersected with the disk where o G(s) >= alpha_min, i.e.
// |s| <= r_o = sqrt(2 ln(o / alpha_min)), bounded by |s|_inf <= a = min(sigma, r_o) and the
// diamond |s_a| + |s_b| <= sqrt2 r_o (an octagon when it cuts the corners), r_o widened by
// 0.1 % + 0.002.  The polygon maps to P = b_c + s_a b_alpha + s_b b_beta.  Azimuth: every column
// when the z axis pierces the polygon's xy-shadow, else the extreme vertex azimuths relative to
// the centre direction.  Elevation: the extreme of the vertices and each edge's interior extremum
// (where z / |xy| is stationary along the edge), and the pole the z axis reaches.  Returns the tile count and
// fills the record's pixel rectangle.
__device__ uint32_t contract_bbox(v3 ba, v3 bb, v3 bc, const Octagon &oct, const ViewDesc &vd,
                                  int th_shift, int tw_shift, PairRec &rec)
{
    const float a = oct.a, k = oct.k, c = oct.c;
    const v3 A{a * ba.x, a * ba.y, a * ba.z};
    const v3 B{a * bb.x, a * bb.y, a * bb.z};
    const v3 C = bc;
    const float u[8] = {1.0f, 1.0f, c, -c, -1.0f, -1.0f, -c, c};
    const float w[8] = {-c, c, 1.0f, 1.0f, c, -c, -1.0f, -1.0f};
    v3 P[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        P[i] = v3{(C.x + u[i] * A.x) + w[i] * B.x, (C.y + u[i] * A.y) + w[i] * B.y,
                  (C.z + u[i] * A.z) + w[i] * B.z};

    // does the z axis cross the polygon's xy-shadow?  c + u A + w B = 0 with |u|, |w| <= 1 and
    // |u| + |w| <= k
    const float det = A.x * B.y - A.y * B.x;
    const float cxb = C.x * B.y - C.y * B.x;
    const float axc = A.x * C.y - A.y * C.x;
    const float la = fabsf(A.x) + fabsf(A.y), lb = fabsf(B.x) + fabsf(B.y);
    const float lc = fabsf(C.x) + fabsf(C.y);
    const float tol = 1e-5f * ((la + lb) * ((lc + la) + lb));
    const float adet = fabsf(det);
    const bool axis_in = (fabsf(cxb) <= adet + tol) && (fabsf(axc) <= adet + tol) &&
                         (fabsf(cxb) + fabsf(axc) <= k * adet + 2.0f * tol);
    bool north = false, south = false;
    if (axis_in) {
        if (adet > tol) {
            const float uu = -cxb / det, ww = -axc / det;
            const float zh = (C.z + uu * A.z) + ww * B.z;
            const float tz = 1e-5f * ((fabsf(C.z) + fabsf(A.z)) + fabsf(B.z));
            north = zh > -tz;
            south = zh < tz;
        } else {
            north = south = true;
        }
    }

    // elevation: the highest and the lowest of the vertices and of the edges' interior extrema,
    // ordered by z / |xy| without a division (z_i r_j against z_j r_i); one arctangent each
    float zh = 0.0f, rh = 0.0f, zl = 0.0f, rl = 0.0f;
    bool have = false;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const v3 p = P[i], q = P[(i + 1) & 7];
        elev_candidate(p.z, sqrtf(p.x * p.x + p.y * p.y), zh, rh, zl, rl, have);
        const v3 d{q.x - p.x, q.y - p.y, q.z - p.z};
        const float pd = p.x * d.x + p.y * d.y;
        const float pp = p.x * p.x + p.y * p.y;
        const float dd = d.x * d.x + d.y * d.y;
        const float num = p.z * pd - d.z * pp;
        const float den = d.z * pd - p.z * dd;
        // the quotient can round into (0, 1) only when num and den are non-zero with one sign
        // and |num| < |den| (a quotient >= 1 rounds to >= 1): testing that first skips the
        // division for most edges and changes no result
        if (den != 0.0f && num != 0.0f && (num > 0.0f) == (den > 0.0f) &&
            fabsf(num) < fabsf(den)) {
            const float lam = num / den;
            if (lam > 0.0f && lam < 1.0f) {
                const v3 X{p.x + lam * d.x, p.y + lam * d.y, p.z + lam * d.z};
                elev_candidate(X.z, sqrtf(X.x * X.x + X.y * X.y), zh, rh, zl, rl, have);
            }
        }
    }
    float el_hi = contract_atan2(zh, rh), el_lo = contract_atan2(zl, rl);
    if (north) el_hi = kHalfPi;
    if (south) el_lo = -kHalfPi;

    const int H = vd.rows, W = vd.cols;
    const float vhi = (vd.elev_max - el_hi) * vd.kr - kPixelMargin;
    const float vlo = (vd.elev_max - el_lo) * vd.kr + kPixelMargin;
    int r0 = static_cast<int>(ceilf(vhi));
    int r1 = static_cast<int>(floorf(vlo));
    r0 = r0 < 0 ? 0 : r0;
    r1 = r1 > H - 1 ? H - 1 : r1;
    if (r0 > r1) return 0u;

    int c0, nc;
    if (axis_in) {
        c0 = 0;
        nc = W;
    } else {
        // the polygon's xy-shadow misses the origin, so it spans less than pi in azimuth: the
        // extreme vertices follow from the signs of cross products, one arctangent each,
        // relative to the centre direction
        const float gc = contract_atan2(C.y, C.x);
        float xmin = P[0].x, ymin = P[0].y, xmax = P[0].x, ymax = P[0].y;
#pragma unroll
        for (int i = 1; i < 8; ++i) {
            if (xmax * P[i].y - ymax * P[i].x > 0.0f) { xmax = P[i].x; ymax = P[i].y; }
            if (xmin * P[i].y - ymin * P[i].x < 0.0f) { xmin = P[i].x; ymin = P[i].y; }
        }
        const float dmax = contract_atan2(C.x * ymax - C.y * xmax, C.x * xmax + C.y * ymax);
        const float dmin = contract_atan2(C.x * ymin - C.y * xmin, C.x * xmin + C.y * ymin);
        const float glo = gc + dmin, ghi = gc + dmax;
        const float kc = static_cast<float>(W) / kTwoPi;
        const float uf = ((kPi - ghi) * kc - 0.5f) - kPixelMargin;
        const float ul = ((kPi - glo) * kc - 0.5f) + kPixelMargin;
        const int cf = static_cast<int>(ceilf(uf));
        const int cl = static_cast<int>(floorf(ul));
        if (cf > cl) return 0u;
        nc = cl - cf + 1;
        if (nc >= W) {
            c0 = 0;
            nc = W;
        } else {
            const int rem = cf % W;   // in (-W, W)
            c0 = rem < 0 ? rem + W : rem;
        }
    }
    rec.r0 = static_cast<int16_t>(r0);
    rec.r1 = static_cast<int16_t>(r1);
    rec.c0 = static_cast<int16_t>(c0);
    rec.nc = static_cast<int16_t>(nc);
    const TileRect tr = tile_rect(rec, W, vd.tiles_c, th_shift, tw_shift);
    return static_cast<uint32_t>(tr.nr * tr.nc);
}

// C3 of the contract for one pair: the sensor-frame centre, the range key and whether the normal
// is turned (binary32 T^c_w)
struct SensorCentre {
    v3 bc;
    float kappa;
    bool flip;
};

__device__ __forceinline__ SensorCentre contract_centre(const float *R, const float *t, v3 mu,
                                                        v3 tn, int flip_normals)
{
    const v3 rm = rot(R, mu);
    SensorCentre s;
    s.bc = v3{rm.x + t[0], rm.y + t[1], rm.z + t[2]};
    const v3 nr = rot(R, tn);
    const float dot = (nr.x * s.bc.x + nr.y * s.bc.y) + nr.z * s.bc.z;
    s.flip = flip_normals && dot > 0.0f;
    s.kappa = sqrtf((s.bc.x * s.bc.x + s.bc.y * s.bc.y) + s.bc.z * s.bc.z);
    return s;
}

__device__ __forceinline__ float approx_rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float approx_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// atan z for |z| <= tan(pi/8) (the next term of the series is below 1.3e-7) and for |z| <= 0.27
// (8.5e-7; 5.2e-7 at the 0.2555 that an azimuth reaches)
__device__ __forceinline__ float approx_atan_mid(float z)
{
    const float z2 = z * z;
    float p = fmaf(0.0769230769f, z2, -0.0909090909f);
    p = fmaf(p, z2, 0.111111111f);
    p = fmaf(p, z2, -0.142857143f);
    p = fmaf(p, z2, 0.2f);
    p = fmaf(p, z2, -0.333333333f);
    return fmaf(z * z2, p, z);
}

__device__ __forceinline__ float approx_atan_small(float z)
{
    const float z2 = z * z;
    float p = fmaf(-0.142857143f, z2, 0.2f);
    p = fmaf(p, z2, -0.333333333f);
    return fmaf(z * z2, p, z);
}

// atan(y / x) for x > 0, |y| <= 8 x
__device__ __forceinline__ float approx_atan(float y, float x)
{
    const float ay = fabsf(y);
    const float hi = fmaxf(ay, x), lo = fminf(ay, x);
    const bool fold = lo > kTanPi8 * hi;
    const float z = (fold ? lo - hi : lo) * approx_rcp(fold ? lo + hi : hi);
    float a = approx_atan_mid(z) + (fold ? kQuarterPi : 0.0f);
    a = ay > x ? kHalfPi - a : a;
    return copysignf(a, y);
}

// What contract_bbox will decide for a polygon well away from the z axis, from approximate
// arithmetic: kQuickEmpty (it meets no pixel centre), kQuickBox (rec holds its rectangle) or
// kQuickUnsure.
//
// The extreme elevations and azimuths are taken over the vertices.  Against the contract's values
// these are off by the rounding of both computations, below 3e-6 rad (positions to a few units in
// 2^24 of the range, angles to 2^-22, series to 1e-6, approximate reciprocals and roots to 2.4e-7),
// for which kQuickAngle stands at twice that, plus the final product's rounding of up to a few
// 2^-24 of the image size in pixels; and the contract also takes the interior extrema of the
// edges.  Where a great-circle arc of length phi reaches its highest elevation theta_m inside, its
// nearer end is at most tan(theta_m) phi^2 / 8 lower: `bulge` bounds that for the longest edge, and
// only widens the box.  So the contract's row bounds lie in [vhi - eps - bulge, vhi + eps] and
// [vlo - eps, vlo + eps + bulge], its column bounds within eps; an integer is taken only when both
// ends of its interval round to it.
enum { kQuickUnsure = 0, kQuickEmpty, kQuickBox };
constexpr float kQuickAngle = 6e-6f;

// what a pair needs of its view, in five 16-byte words of shared memory
struct __align__(16) QuickView {
    float R[9], t[3];
    float kr, elev_max, er;   // rows a radian, top elevation, row bounds' error in pixels
    float kc, ec;             // columns a radian, column bounds' error in pixels
    int rows, cols, tiles_c;
};

__device__ __forceinline__ QuickView quick_view(const ViewDesc &vd)
{
    QuickView q;
#pragma unroll
    for (int k = 0; k < 9; ++k) q.R[k] = vd.R_hi[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) q.t[k] = vd.t_hi[k];
    q.kr = vd.kr;
    q.elev_max = vd.elev_max;
    q.rows = vd.rows;
    q.cols = vd.cols;
    q.tiles_c = vd.tiles_c;
    q.er = fmaf(q.kr, kQuickAngle, fmaf(3e-7f, static_cast<float>(q.rows), 1e-5f));
    q.kc = static_cast<float>(q.cols) / kTwoPi;
    q.ec = fmaf(q.kc, kQuickAngle, fmaf(6e-7f, static_cast<float>(q.cols), 1e-5f));
    return q;
}

__device__ __forceinline__ int quick_box(v3 ba, v3 bb, v3 C, float sa, float sb, float sigma,
                                         const Octagon &oct, const QuickView &vd, PairRec &rec)
{
    const float F0 = fmaf(C.x, C.x, C.y * C.y);
    const float rxy = F0 * approx_rsqrt(F0);
    const float reach = sigma * (sa + sb) * 1.01f;   // the polygon lies in this ball about C
    if (!(reach <= 0.25f * rxy) || !(fabsf(C.z) <= 4.0f * rxy) || !(rxy > 1e-6f) ||
        !(rxy < 1e12f))
        return kQuickUnsure;
    const float a = oct.a, k = oct.k, c = oct.c;
    const v3 A{a * ba.x, a * ba.y, a * ba.z};
    const v3 B{a * bb.x, a * bb.y, a * bb.z};
    // the contract's own axis test, operation by operation: an edge-on shadow can pass it at any
    // distance
    const float det = A.x * B.y - A.y * B.x;
    const float cxb = C.x * B.y - C.y * B.x;
    const float axc = A.x * C.y - A.y * C.x;
    const float la = fabsf(A.x) + fabsf(A.y), lb = fabsf(B.x) + fabsf(B.y);
    const float lc = fabsf(C.x) + fabsf(C.y);
    const float tol = 1e-5f * ((la + lb) * ((lc + la) + lb));
    const float adet = fabsf(det);
    if ((fabsf(cxb) <= adet + tol) && (fabsf(axc) <= adet + tol) &&
        (fabsf(cxb) + fabsf(axc) <= k * adet + 2.0f * tol))
        return kQuickUnsure;
    // half the vertices relative to the centre; the others are their opposites.  With L = C x d
    // and f = C . d in the xy plane, vertex C +- d has squared distance F0 + |d|^2 +- 2 f from the
    // axis and azimuth tangent +- L / (F0 +- f) from the centre
    const v3 D[4] = {v3{fmaf(-c, B.x, A.x), fmaf(-c, B.y, A.y), fmaf(-c, B.z, A.z)},
                     v3{fmaf(c, B.x, A.x), fmaf(c, B.y, A.y), fmaf(c, B.z, A.z)},
                     v3{fmaf(c, A.x, B.x), fmaf(c, A.y, B.y), fmaf(c, A.z, B.z)},
                     v3{fmaf(-c, A.x, B.x), fmaf(-c, A.y, B.y), fmaf(-c, A.z, B.z)}};
    float t_hi = -INFINITY, t_lo = INFINITY, q_hi = -INFINITY, q_lo = INFINITY;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const v3 d = D[i];
        const float L = fmaf(C.x, d.y, -(C.y * d.x)), f = fmaf(C.x, d.x, C.y * d.y);
        const float G = fmaf(d.x, d.x, fmaf(d.y, d.y, F0));
        const float tp = (C.z + d.z) * approx_rsqrt(fmaf(2.0f, f, G));   // tan of the elevation
        const float tq = (C.z - d.z) * approx_rsqrt(fmaf(-2.0f, f, G));
        const float qp = L * approx_rcp(F0 + f), qm = -L * approx_rcp(F0 - f);
        t_hi = fmaxf(t_hi, fmaxf(tp, tq));
        t_lo = fminf(t_lo, fminf(tp, tq));
        q_hi = fmaxf(q_hi, fmaxf(qp, qm));
        q_lo = fminf(q_lo, fminf(qp, qm));
    }
    const float phi = 2.1f * a * fmaxf(sa, sb) * approx_rcp(rxy - reach);
    const float tm = fmaxf(fabsf(t_hi), fabsf(t_lo));
    const float bulge = 0.15f * (phi * phi) * fmaf(1.3f * phi, fmaf(tm, tm, 1.0f), tm) * vd.kr;
    // the higher elevation as the lower one plus the small angle between them
    const float el_lo = approx_atan(t_lo, 1.0f);
    const float dt = (t_hi - t_lo) * approx_rcp(fmaf(t_hi, t_lo, 1.0f));
    const float el_hi = el_lo + (fabsf(dt) <= 0.27f ? approx_atan_small(dt)
                                                    : approx_atan(t_hi, 1.0f) - el_lo);
    const int H = vd.rows, W = vd.cols;
    const float vhi = (vd.elev_max - el_hi) * vd.kr - kPixelMargin;
    const float vlo = (vd.elev_max - el_lo) * vd.kr + kPixelMargin;
    const int r0 = max(static_cast<int>(ceilf(vhi - vd.er - bulge)), 0);
    const int r1 = min(static_cast<int>(floorf(vlo + vd.er + bulge)), H - 1);
    if (r0 > r1) return kQuickEmpty;
    const bool rows = r0 == max(static_cast<int>(ceilf(vhi + vd.er)), 0) &&
                      r1 == min(static_cast<int>(floorf(vlo - vd.er)), H - 1);
    const float ax = fabsf(C.x), ay = fabsf(C.y);
    float gc = approx_atan(fminf(ax, ay), fmaxf(ax, ay));
    gc = ay > ax ? kHalfPi - gc : gc;
    gc = C.x < 0.0f ? kPi - gc : gc;
    gc = copysignf(gc, C.y);
    const float uf = (kPi - (gc + approx_atan_small(q_hi))) * vd.kc - 0.5f - kPixelMargin;
    const float ul = (kPi - (gc + approx_atan_small(q_lo))) * vd.kc - 0.5f + kPixelMargin;
    const int cf = static_cast<int>(ceilf(uf - vd.ec)), cl = static_cast<int>(floorf(ul + vd.ec));
    if (cf > cl) return kQuickEmpty;
    const int nc = cl - cf + 1;
    // cf and the columns lie within one turn of [0, W): less than a quarter turn from the centre
    const int c0 = cf < 0 ? cf + W : (cf >= W ? cf - W : cf);
    if (!rows || cf != static_cast<int>(ceilf(uf + vd.ec)) ||
        cl != static_cast<int>(floorf(ul - vd.ec)) || nc >= W || c0 < 0 || c0 >= W)
        return kQuickUnsure;
    rec.r0 = static_cast<int16_t>(r0);
    rec.r1 = static_cast<int16_t>(r1);
    rec.c0 = static_cast<int16_t>(c0);
    rec.nc = static_cast<int16_t>(nc);
    return kQuickBox;
}

// Pairs waiting for the contract's box, kQueueSlots per warp (structure of arrays)
constexpr int kProjectThreads = 256, kProjectWarps = kProjectThreads / 32;
constexpr int kQueueSlots = 64;
struct BoxQueue {
    float f[14][kProjectWarps * kQueueSlots];   // b_a, b_b, b_c, octagon (a, k, c), key, s_a + s_b
    uint32_t pair[kProjectWarps * kQueueSlots]; // view << 13 | normal flipped << 12 | local place
};

struct ProjectShared {
    QuickView view[kMaxViews];
    BoxQueue q;
    uint32_t count[kMaxViews];        // pairs of the block that touch a tile, per view
    uint32_t left[kProjectWarps];     // pairs left in each warp's queue at the end
    unsigned long long rows;
};

__global__ void __launch_bounds__(kProjectThreads, 3) k_project(const ProjectArgs A)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char s_raw[];
    ProjectShared &sh = *reinterpret_cast<ProjectShared *>(s_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t block0 = static_cast<int64_t>(blockIdx.x) * A.block_prims;
    const int th_shift = __ffs(A.tile_h) - 1, tw_shift = __ffs(A.tile_w) - 1;   // powers of two
    for (int v = threadIdx.x; v < A.n_views; v += kProjectThreads) {
        sh.count[v] = 0u;
        sh.view[v] = quick_view(A.views[v]);
    }
    if (threadIdx.x == 0) sh.rows = 0ull;
    __syncthreads();
    float rows8 = 0.0f;   // rows of 8-pixel columns that this thread's touching pairs meet

    // append a touching pair (its primitive's place in the block is `local`) to the block's
    // segment of the view, with one counter update for the lanes `peers` of that view (the whole
    // warp takes part)
    auto append = [&](bool touch, uint32_t peers, int v, uint32_t local, const PairRec &rec) {
        const int lead = __ffs(peers) - 1;
        uint32_t at = 0;
        if (touch && lane == lead) at = atomicAdd(&sh.count[v], __popc(peers));
        at = __shfl_sync(0xFFFFFFFFu, at, lead) + __popc(peers & ((1u << lane) - 1u));
        if (touch) {
            const int64_t o = static_cast<int64_t>(v) * A.n + block0 + at;
            A.touch[o] = pack_touch(tile_rect(rec, sh.view[v].cols, sh.view[v].tiles_c, th_shift,
                                              tw_shift), local);
            A.kappa[o] = rec.kappa;
            // (a wrapping rectangle meets one column of 8 more at the seam)
            rows8 += static_cast<float>((rec.r1 - rec.r0 + 1) *
                                        (((rec.c0 + rec.nc - 1) >> 3) - (rec.c0 >> 3) + 2));
        }
    };

    // box the queued pair of slot s, one per lane with `has`
    auto box = [&](bool has, int s) {
        const uint32_t e = has ? sh.q.pair[s] : 0u;
        const uint32_t local = e & 0xFFFu;
        const int v = static_cast<int>(e >> 13);
        const ViewDesc &vd = A.views[v];
        PairRec rec;
        rec.r0 = rec.r1 = rec.c0 = rec.nc = 0;
        rec.kappa = 0.0f;
        rec.cf = (e & 0x1000u) ? kPairFlip : 0u;
        uint32_t count = 0;
        if (has) {
            const float(*f)[kProjectWarps * kQueueSlots] = sh.q.f;
            rec.kappa = f[12][s];
            const v3 bc{f[6][s], f[7][s], f[8][s]};
            // A pair whose whole 3-sigma box lies beyond the view's culling cones (two rows past
            // the top or bottom row) and away from the z axis reaches no row: every point of the
            // box is within R = sigma (s_a + s_b) of b_c, and z - t |xy| changes by at most l R
            // over that ball.
            const float rxy = sqrtf(bc.x * bc.x + bc.y * bc.y);
            const float reach = A.sigma * f[13][s] * 1.01f;
            const bool clear = rxy * 0.99f - reach > 1e-3f;
            const bool above = bc.z - vd.cull_t_top * rxy > reach * vd.cull_l_top;
            const bool below = vd.cull_t_bot * rxy - bc.z > reach * vd.cull_l_bot;
            // C4: bounding box
            if (!(clear && (above || below)))
                count = contract_bbox(v3{f[0][s], f[1][s], f[2][s]},
                                      v3{f[3][s], f[4][s], f[5][s]}, bc,
                                      Octagon{f[9][s], f[10][s], f[11][s]}, vd, th_shift, tw_shift,
                                      rec);
            A.prect[static_cast<int64_t>(v) * A.n + block0 + local] =
                count ? pack_pixel_rect(rec) : 0ull;
        }
        append(count != 0u, __match_any_sync(0xFFFFFFFFu, count ? v : -1), v, local, rec);
    };

    const int q0 = warp * kQueueSlots;
    int qn = 0;
    for (int base = 0; base < A.block_prims; base += kProjectThreads) {
        const uint32_t local = static_cast<uint32_t>(base) + threadIdx.x;
        const int64_t i = block0 + local;
        const bool in = i < A.n;
        if (block0 + base + 32 * warp >= A.n) break;   // the whole warp
        float4 pl = make_float4(0.0f, 0.0f, 0.0f, 0.0f), q4 = pl;
        float2 ls = make_float2(0.0f, 0.0f);
        if (in) {
            pl = A.pos_logit[i];
            q4 = A.quat[i];
            ls = A.log_scale[i];
        }
        bool ok = isfinite(pl.x) && isfinite(pl.y) && isfinite(pl.z) && isfinite(pl.w) &&
                  isfinite(q4.x) && isfinite(q4.y) && isfinite(q4.z) && isfinite(q4.w) &&
                  isfinite(ls.x) && isfinite(ls.y);
        // C1: normalised quaternion and scales
        float w = q4.x, x = q4.y, y = q4.z, z = q4.w;
        const float qq = ((w * w + x * x) + y * y) + z * z;
        ok = ok && qq > 0.0f && isfinite(qq);
        v3 ta{}, tb{}, tn{};
        float sa = 0.0f, sb = 0.0f, oc = 0.0f;
        Octagon oct{};
        bool opaque = false;   // the opacity reaches alpha_min somewhere
        if (ok) {
            const float r = sqrtf(qq);
            w = w / r;
            x = x / r;
            y = y / r;
            z = z / r;
            // C2: rotation columns
            ta = v3{1.0f - 2.0f * (y * y + z * z), 2.0f * (x * y + w * z),
                    2.0f * (x * z - w * y)};
            tb = v3{2.0f * (x * y - w * z), 1.0f - 2.0f * (x * x + z * z),
                    2.0f * (y * z + w * x)};
            tn = v3{2.0f * (x * z + w * y), 2.0f * (y * z - w * x),
                    1.0f - 2.0f * (x * x + y * y)};
            sa = contract_exp(ls.x);
            sb = contract_exp(ls.y);
            oc = 1.0f / (1.0f + contract_exp(-pl.w));
            opaque = contract_octagon(oc, A.alpha_min, A.sigma, oct);
        } else if (in) {
            atomicOr(A.status, SPLAT_STATUS_NONFINITE);
        }
        const v3 mu{pl.x, pl.y, pl.z};
        if (in) {   // what the compositing kernels stage for every (block, list entry)
            float4 *e = A.prim + kPrimRow * i;
            e[0] = make_float4(sa * ta.x, sa * ta.y, sa * ta.z, oc);
            e[1] = make_float4(sb * tb.x, sb * tb.y, sb * tb.z, ok ? 1.0f : 0.0f);
            e[2] = make_float4(tn.x, tn.y, tn.z, 0.0f);
            e[3] = make_float4(mu.x, mu.y, mu.z, 0.0f);
            if (A.wgrad) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    A.wgrad[4 * i + k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
        }

        for (int v = 0; v < A.n_views; ++v) {
            if (A.active && !A.active[v]) continue;   // views not drawn take no pairs
            const QuickView &vd = sh.view[v];
            int state = kQuickEmpty;
            SensorCentre sc{};
            v3 ba{}, bb{};
            PairRec rec;
            rec.r0 = rec.r1 = rec.c0 = rec.nc = 0;
            if (ok && in && opaque) {
                // C3
                sc = contract_centre(vd.R, vd.t, mu, tn, A.flip_normals);
                const v3 ra = rot(vd.R, ta), rb = rot(vd.R, tb);
                ba = v3{sa * ra.x, sa * ra.y, sa * ra.z};
                bb = v3{sb * rb.x, sb * rb.y, sb * rb.z};
                state = quick_box(ba, bb, sc.bc, sa, sb, A.sigma, oct, vd, rec);
            }
            const bool unsure = state == kQuickUnsure;
            rec.kappa = sc.kappa;
            rec.cf = sc.flip ? kPairFlip : 0u;
            if (in && !unsure)
                A.prect[static_cast<int64_t>(v) * A.n + i] =
                    state == kQuickBox ? pack_pixel_rect(rec) : 0ull;
            append(state == kQuickBox, __ballot_sync(0xFFFFFFFFu, state == kQuickBox), v, local,
                   rec);
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, unsure);
            if (m == 0u) continue;
            if (unsure) {
                const int s = q0 + qn + __popc(m & ((1u << lane) - 1u));
                const float f[14] = {ba.x, ba.y, ba.z, bb.x, bb.y, bb.z, sc.bc.x, sc.bc.y, sc.bc.z,
                                     oct.a, oct.k, oct.c, sc.kappa, sa + sb};
#pragma unroll
                for (int k = 0; k < 14; ++k) sh.q.f[k][s] = f[k];
                sh.q.pair[s] = static_cast<uint32_t>(v) << 13 | (sc.flip ? 0x1000u : 0u) | local;
            }
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32) {   // the newest 32, so that nothing moves
                qn -= 32;
                box(true, q0 + qn + lane);
                __syncwarp();
            }
        }
    }
    // what is left in the warps' queues (fewer than 32 each), 32 at a time over the CTA
    if (lane == 0) sh.left[warp] = static_cast<uint32_t>(qn);
    __syncthreads();
    uint32_t total = 0;
    for (int w = 0; w < kProjectWarps; ++w) total += sh.left[w];
    for (uint32_t e0 = 32u * warp; e0 < total; e0 += 32u * kProjectWarps) {
        uint32_t e = e0 + lane;
        const bool has = e < total;
        int w = 0;
        while (has && e >= sh.left[w]) e -= sh.left[w++];
        box(has, w * kQueueSlots + static_cast<int>(e));
    }
    unsigned long long r64 = static_cast<unsigned long long>(rows8 * 1.001f) + 1ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r64 += __shfl_xor_sync(0xFFFFFFFFu, r64, o);
    if (lane == 0 && r64) atomicAdd(&sh.rows, r64);
    __syncthreads();
    if (threadIdx.x == 0 && sh.rows) atomicAdd(A.n_rows, sh.rows);
    // the segments' lengths, and the pairs that touch a tile
    uint32_t nv = 0;
    for (int v = threadIdx.x; v < A.n_views; v += kProjectThreads) {
        A.touch_count[static_cast<int64_t>(v) * gridDim.x + blockIdx.x] = sh.count[v];
        nv += sh.count[v];
    }
    if (warp < (kMaxViews + 31) / 32) {
        nv = __reduce_add_sync(0xFFFFFFFFu, nv);
        if (lane == 0 && nv) atomicAdd(A.n_valid, nv);
    }
}

// The records of the last render as the debugging interface gives them, from what the
// projection kept: rectangles of the pairs, and the primitives' own centre and normal for the
// range key and the flip (the contract's operations again, so the same bits).
__global__ void __launch_bounds__(256) k_records(int64_t n, const ViewDesc *__restrict__ views,
                                                 int flip_normals, int tile_h, int tile_w,
                                                 const float4 *__restrict__ prim,
                                                 const uint64_t *__restrict__ prect,
                                                 const uint8_t *__restrict__ active,
                                                 PairRec *__restrict__ recs)
{
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int v = blockIdx.y;
    if (i >= n) return;
    const int64_t p = static_cast<int64_t>(v) * n + i;
    const uint64_t word = !active || active[v] ? prect[p] : 0ull;
    PairRec rec = unpack_pixel_rect(word);
    rec.cf = 0u;
    if (prim[kPrimRow * i + 1].w == 0.0f) {
        rec.cf = kPairInvalid;
    } else {
        const float4 t = prim[kPrimRow * i + 2], m = prim[kPrimRow * i + 3];
        const SensorCentre sc = contract_centre(views[v].R_hi, views[v].t_hi, v3{m.x, m.y, m.z},
                                                v3{t.x, t.y, t.z}, flip_normals);
        rec.kappa = sc.kappa;
        if (sc.flip) rec.cf |= kPairFlip;
    }
    if (word) {
        const TileRect tr = tile_rect(rec, views[v].cols, views[v].tiles_c, __ffs(tile_h) - 1,
                                      __ffs(tile_w) - 1);
        rec.cf |= static_cast<uint32_t>(tr.nr * tr.nc);
    }
    recs[p] = rec;
}

}  // namespace

cudaError_t launch_project(const ProjectArgs &a, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    ProjectArgs b = a;
    b.block_prims = block_prims(a.n);
    return launch_chained(chained_size(a.n * a.n_views), k_project,
                          dim3(static_cast<unsigned>(project_blocks(a.n))),
                          kProjectThreads, sizeof(ProjectShared), st, b);
}

cudaError_t launch_records(int64_t n, int n_views, const ViewDesc *views, int flip_normals,
                           int tile_h, int tile_w, const float4 *prim, const uint64_t *prect,
                           const uint8_t *active, PairRec *recs, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const dim3 grid(static_cast<unsigned>((n + 255) / 256), static_cast<unsigned>(n_views));
    k_records<<<grid, 256, 0, st>>>(n, views, flip_normals, tile_h, tile_w, prim, prect, active,
                                    recs);
    return cudaGetLastError();
}

}  // namespace splat
