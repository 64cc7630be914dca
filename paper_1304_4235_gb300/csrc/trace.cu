// Column tracing (Sec. 3.2 and Eq. colden): for each (origin particle,
// HEALPix direction) the segment r_i + t n_k, t in [0, l_ray], is walked
// through the LBVH and every smoothing sphere it crosses adds
//   A_j x_j * int W(q) du      (A_j = sigma_th m_j/m_p (8/pi) / h_j^2)
// with the line integral in closed form: the M4 spline of Eq. spline via
// antiderivatives of q, q^2, q^3 along the chord, or the truncated Gaussian
// of Eq. Gt via the erf form I(h,b,z1,z2).
//
// Work distribution: a persistent grid; each warp takes tasks of 32
// neighbouring origins in one direction from an atomic queue, so the 32 rays
// of a warp are parallel and start close together (a beam).  The beam walks
// the 32-ary box tree as one packet, each lane testing one child of the
// current entry against the beam; at a block of 32 each lane tests one sphere
// against the beam, and the spheres that pass are staged in shared memory.
// Every 32 staged spheres, each lane tests them against its own ray in the
// beam's frame (a handful of packed FP32 operations per sphere, conservative)
// and keeps the ones it may cross as a bit mask.  The (ray, sphere) pairs of
// the masks are listed ray by ray, and the exact hit test and the chord
// integral run over the list 32 pairs at a time, whichever rays they belong
// to; each lane then adds its own ray's values in list order, so that the
// expensive part works on full warps while every ray still sums its hits in
// the tree's fixed order.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"

namespace urchin {

namespace {

struct TraceParams {
    const float2* ktab;           // [kKTab + 1] full-chord M4 table (value, slope x dt)
    const float4* boxes;          // 32-ary tree (urchin_bvh::boxes)
    int n_lev;
    int lev_off[kMaxLevels], lev_cnt[kMaxLevels];
    int n;
    const float4* xyzh;
    const float* w32;
    const double* w64;
    const double* dirs;
    int R;
    double l_ray;
    float l_beam;                 // length of the filters' segments (beam_length)
    const int32_t* items;
    int64_t n_items;
    int64_t row_stride, k_stride;
    const int32_t* out_row;
    void* out;
    unsigned* counter;
    unsigned* status;
    unsigned long long* hits;
    int periodic;
    double Lbox;
    int nimg;
    float root_lo[3], root_hi[3];
    double gt_t2, gt_t, gt_pref;
    int64_t n_chunks;             // packets per direction
    int packet;                   // origins per packet (32, or fewer where 32 leave warps idle)
    // stored-segment modes
    uint32_t* counts;             // MODE_COUNT: hits per ray, index k * n_items + item
    const uint64_t* row_ptr;      // MODE_FILL: first segment of each ray (same index), size + 1
    int32_t* seg_col;             // MODE_FILL: Morton index of the particle, or NULL:
    uint16_t* seg_lo;             //   its low 16 bits
    uint8_t* seg_hi;              //   and high 8 bits (indices below 2^24; NULL: below 2^16)
    void* seg_val;                // MODE_FILL: A_j * chord integral (float or double)
    const float* A32;
    const double* A64;
    // transpose mode
    const void* coef;             // MODE_SCATTER: coefficient of each ray, indexed like out
    double* xbar;                 // MODE_SCATTER: xbar[j] += coef * A_j * chord integral (Morton)
    const int32_t* order;         // [R * n_items] per-direction item order, or NULL
    // near/far split
    void* out_near;               // [slot + k * near_k_stride] near column (x = 1)
    const float* w32_2;           // kThree: the other tracers' weights (as w32)
    const float* w32_3;
    float* out_2;                 //   and columns (indexed like out)
    float* out_3;
    int64_t near_k_stride;
    // MODE_CHUNK: segment lists in chunks of kChunk entries taken while tracing
    uint32_t* chunk_head;         // [R * n] first chunk of each ray (rays with hits)
    uint32_t* chunk_next;         // [cap] the chunk after each chunk of a ray
    unsigned long long* chunk_counter;   // chunks handed out (may exceed cap: then the lists are incomplete)
    unsigned long long chunk_cap;
    int2* chunk_seg;              // [cap * kChunk] (particle, value bits): one 8-byte store per full chord
};

constexpr int MODE_TAU = 0, MODE_COUNT = 1, MODE_FILL = 2, MODE_SCATTER = 3, MODE_CHUNK = 4;
// MODE_CHUNK: the columns as in MODE_TAU, the hit counts as in MODE_COUNT, and
// every ray's segments stored while tracing, in chunks of kChunk entries that
// the warp takes from a global counter kStash at a time (the counts are not
// known before the traversal); the chunks of a ray are linked through
// chunk_next.  Used by the solver's first sweep, so that a solve of two sweeps
// traces once.
// Flag beside MODE_TAU or MODE_CHUNK (FP32): columns of two more tracers in the
// same traversal (helium), each summed as a traversal of its own would.
constexpr int kThree = 8;
// Flag beside MODE_TAU: the form for many rays (k_trace's comment).
constexpr int kWide = 16;
constexpr int kChunk = kChunkEntries;   // entries per chunk (a multiple of kSegPad)
constexpr int kStash = 64;        // chunks a warp takes from the counter at a time

// Where a ray's hits go: the running column sum, and in MODE_FILL the
// cursor into the ray's stored segment list.
template <typename Real>
struct Sink {
    Real sum, comp;               // full chords, in traversal order
    Real psum, pcomp;             // partial chords (FP32 queue), in the ray's queue order
    unsigned nhit, ntest;
    int64_t pos, end;
    Real coef;                    // MODE_SCATTER
    Real near, near_c;            // near/far: near column and its compensation
    Real sum2, comp2, psum2, pcomp2, sum3, comp3, psum3, pcomp3;   // kThree: the other tracers' sums
    int64_t ray;                  // MODE_CHUNK: row k n + origin slot
    int coff;                     // MODE_CHUNK: entries used in it (kChunk: none or full; kChunk + 1: pool exhausted)
    uint32_t cur;                 // MODE_CHUNK: its index (kNoChunk before the first)
};
constexpr uint32_t kNoChunk = 0xffffffffu;

// Near/far split (Sec. 3.3.3): particle j is near the ray's origin when the
// origin lies inside j's smoothing sphere.  For a crossed sphere that is the
// case exactly when its chord starts before the origin, tc - ch < 0 (the
// origin at distance^2 = tc^2 + b^2 < h^2); that test decides unless the
// origin sits within rounding of the sphere's surface, where the distance is
// compared in double from the float positions (the differences are exact),
// like the reference definition, so both sides classify every pair alike.
template <typename Real>
__device__ __forceinline__ bool is_near(const double* o, float4 q, Real tc, Real ch)
{
    const Real gap = tc - ch;
    if (fabs((double)gap) > 1e-4 * (double)q.w) return gap < Real(0);
    const double ex = (double)q.x - o[0], ey = (double)q.y - o[1], ez = (double)q.z - o[2];
    const double hh = (double)q.w;
    return fma(ez, ez, fma(ey, ey, __dmul_rn(ex, ex))) < __dmul_rn(hh, hh);
}

// Rounded arithmetic the compiler may not contract into multiply-adds.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }

template <typename Real> struct RealOps;
template <> struct RealOps<float> {
    static __device__ __forceinline__ float exp_(float x) { return expf(x); }
    static __device__ __forceinline__ float erf_(float x) { return erff(x); }
};
template <> struct RealOps<double> {
    static __device__ __forceinline__ double exp_(double x) { return exp(x); }
    static __device__ __forceinline__ double erf_(double x) { return erf(x); }
};

// ---- M4 chord integrals in units of h -------------------------------------
// With q = sqrt(beta^2 + a^2) and L(a) = asinh(a/beta) = ln(a + q) - ln(beta):
//   inner piece (q <= 1/2), integrand 1 - 6q^2 + 6q^3:
//     Fi(a) = a(1 - 6b2 - 2a^2) + 3/2 a q^3 + 9/4 b2 a q + 9/4 b2^2 L
//   outer piece (1/2 < q <= 1), integrand 2(1-q)^3:
//     Fo(a) = a(2 + 6b2 + 2a^2) - 3 a q - 1/2 a q^3 - 3/4 b2 a q - (3 b2 + 3/4 b2^2) L
// and the odd antiderivative from 0 is H(a) = Fi(a) for a <= s, else
// Fo(a) + Fi(s) - Fo(s) with s = sqrt(1/4 - b2) (b2 < 1/4), where
//   Fi(s) - Fo(s) = -s(1/4 + 13/2 b2) + (3 b2 + 3 b2^2) L(s).
// At the chord end a = c = sqrt(1 - b2) (q = 1):
//   Fo(c) = c(1/2 + 13/4 b2) - (3 b2 + 3/4 b2^2) L(c).
// In double (the FP32 chords are below).  The FP64 pipe bounds this path (2
// results per clock and SM), so a chord takes as few FP64 operations as it can:
// one ln b and one join for both ends, the two pieces' polynomials as one with
// selected coefficients, and logarithms from a table (after Tang, 1990):
// x = 2^e m, c about 1 / m from the top 7 bits of m, r = m c - 1 rounded once,
// ln x = e ln 2 - ln c + log1p(r), |r| < 0.004, the series to r^7; absolute
// error about 1e-16, 11 operations where log() takes some 27.
constexpr int kLogTab = 128;

__device__ __forceinline__ void log_table(double2* tab)
{
    for (int i = threadIdx.x; i < kLogTab; i += blockDim.x) {
        const double c = (double)(float)(1.0 / (1.0 + (i + 0.5) / kLogTab));
        tab[i] = make_double2(c, -log(c));
    }
}

__device__ __forceinline__ double log_tab(const double2* tab, double x)
{
    const int hi = __double2hiint(x);
    if (hi < 0x00100000 || hi >= 0x7ff00000) return log(x);        // zero, denormal, negative, infinite, NaN
    const double2 T = tab[(hi >> 13) & (kLogTab - 1)];
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    const double r = fma(m, T.x, -1.0);
    double p = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    p = fma(r, p, 0.2);
    p = fma(r, p, -0.25);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -0.5);
    return fma((double)((hi >> 20) - 1023), 0.6931471805599453, T.y) + fma(r * r, p, r);
}

// ln b of b^2, and Fi(s) - Fo(s) with s = sqrt(1/4 - b^2) (b^2 < 1/4)
__device__ __forceinline__ double m4_join(const double2* lt, double b2, double lb, double& s)
{
    s = sqrt(0.25 - b2);
    const double Ls = b2 > 0.0 ? log_tab(lt, s + 0.5) - lb : 0.0;
    return fma(fma(3.0 * b2, b2, 3.0 * b2), Ls, -s * fma(6.5, b2, 0.25));
}

__device__ __forceinline__ double m4_full(const double2* lt, double b2, double c)
{
    const double lb = b2 > 0.0 ? 0.5 * log_tab(lt, b2) : 0.0;
    const double Lc = b2 > 0.0 ? log_tab(lt, c + 1.0) - lb : 0.0;
    double H = c * fma(3.25, b2, 0.5) - fma(0.75 * b2, b2, 3.0 * b2) * Lc;
    if (b2 < 0.25) {
        double s;
        H += m4_join(lt, b2, lb, s);
    }
    return 2.0 * H;
}

__device__ __forceinline__ double m4_part(const double2* lt, double b2, double u1, double u2)
{
    const double lb = b2 > 0.0 ? 0.5 * log_tab(lt, b2) : 0.0;
    double s = -1.0, join = 0.0;
    if (b2 < 0.25) join = m4_join(lt, b2, lb, s);
    const double kLo = fma(0.75 * b2, b2, 3.0 * b2), kLi = 2.25 * b2 * b2, kqo = -fma(0.75, b2, 3.0), kqi = 2.25 * b2;
    double H[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const double a = fabs(e == 0 ? u1 : u2), q2 = fma(a, a, b2), q = sqrt(q2);
        const double L = b2 > 0.0 ? log_tab(lt, a + q) - lb : 0.0;
        const bool in = a <= s;
        // a (k0 + k1 (6 b2 + 2 a^2) + q (kq + k3 q^2)) + kL L
        const double g = fma(4.0, b2, 2.0 * q2);
        const double P = (in ? 1.0 - g : 2.0 + g) + q * fma(in ? 1.5 : -0.5, q2, in ? kqi : kqo);
        const double v = fma(a, P, (in ? kLi : -kLo) * L) + (in ? 0.0 : join);
        H[e] = (e == 0 ? u1 : u2) >= 0.0 ? v : -v;
    }
    return H[1] - H[0];
}

// ---- truncated Gaussian (Eq. Gt, I(h,b,z1,z2)) ----------------------------
template <typename Real>
__device__ __forceinline__ Real gt_chord(const TraceParams& P, Real b2, Real u1, Real u2)
{
    using O = RealOps<Real>;
    Real t = Real(P.gt_t);
    return Real(P.gt_pref) * O::exp_(-Real(P.gt_t2) * b2) * (O::erf_(t * u2) - O::erf_(t * u1));
}

// ---- FP32 chord evaluation ------------------------------------------------
// The antiderivatives above lose about two digits in FP32 over the outer
// spline piece (terms of order 4 cancel to the small value of 2(1-q)^3), so
// the FP32 path evaluates
//   * full chords from a table of K(t) = int W du over the whole chord,
//     t = b^2/h^2, with cubic Hermite interpolation (values and slopes at
//     kKTab + 1 nodes, built on the host in double and staged in shared
//     memory), and
//   * partial chords piece by piece: the inner piece (q <= 1/2) by the
//     antiderivative Fi (well conditioned), the outer piece by 8-point
//     Gauss-Legendre quadrature of 2(1-q)^3, a smooth non-negative
//     integrand on [s, c].
__device__ __forceinline__ float m4_full_tab(const float2* tab, float t)
{
    float x = fminf(t, 1.0f) * (float)kKTab;
    int i = min((int)x, kKTab - 1);
    float f = x - (float)i;
    float2 a = tab[i], b = tab[i + 1];
    float f2 = f * f, f3 = f2 * f;
    return (2.f * f3 - 3.f * f2 + 1.f) * a.x + (f3 - 2.f * f2 + f) * a.y + (3.f * f2 - 2.f * f3) * b.x +
           (f3 - f2) * b.y;
}

// int_{a1}^{a2} M4shape(sqrt(b2 + u^2)) du for 0 <= a1 <= a2 <= sqrt(1 - b2):
// the inner piece (q <= 1/2) by its antiderivative Fi (Fi(0) = 0), the
// outer piece by 6-point Gauss-Legendre quadrature of 2(1 - q)^3 (within
// 6e-8 of the integral for every b2 and interval; K(0) = 0.75).  Integrating
// over the interval itself keeps a short piece's relative accuracy (as a
// difference of antiderivatives from 0 it would lose it).
__constant__ float kGL6x[6] = {-0.9324695142031521f, -0.6612093864662645f, -0.2386191860831969f,
                               0.2386191860831969f,  0.6612093864662645f,  0.9324695142031521f};
__constant__ float kGL6w[6] = {0.1713244923791704f, 0.3607615730481386f, 0.4679139345726910f,
                               0.4679139345726910f, 0.3607615730481386f, 0.1713244923791704f};

__device__ __forceinline__ float m4_inner_fi(float b2, float rb, float a)
{
    const float q = sqrtf(fmaf(a, a, b2));
    const float L = b2 > 0.f ? logf((a + q) * rb) : 0.f;
    return a * (1.f - 6.f * b2 - 2.f * a * a) + 1.5f * a * q * q * q + 2.25f * b2 * a * q + 2.25f * b2 * b2 * L;
}

__device__ __forceinline__ float m4_seg_f(float b2, float a1, float a2)
{
    const float s = b2 < 0.25f ? sqrtf(0.25f - b2) : 0.f;
    const float rb = b2 > 0.f ? rsqrtf(b2) : 0.f;
    float r = 0.f;
    if (a1 < s) {
        // one copy of the code for both ends: the traversal's loop has to stay
        // in the instruction cache
        const int ends = a1 > 0.f ? 2 : 1;
#pragma unroll 1
        for (int e = 0; e < ends; ++e) {
            const float fi = m4_inner_fi(b2, rb, e == 0 ? fminf(a2, s) : a1);
            r = e == 0 ? fi : r - fi;
        }
    }
    const float lo = fmaxf(a1, s);
    if (a2 > lo) {
        const float m = 0.5f * (lo + a2), h = 0.5f * (a2 - lo);
        float acc = 0.f;
#pragma unroll
        for (int g = 0; g < 6; ++g) {
            const float u = fmaf(h, kGL6x[g], m);
            const float v = 1.f - sqrtf(fmaf(u, u, b2));
            acc = fmaf(kGL6w[g], v * v * v, acc);
        }
        r += 2.f * h * acc;
    }
    return r;
}

// Partial M4 chord over [u1, u2] (units of h, -c <= u1 < u2 <= c).  A chord
// that straddles the closest approach (u1 < 0 < u2) is the sum of its two
// halves, and a half that the segment does not clip is K(b2)/2 from the
// full-chord table, so a chord clipped at one end costs one piece; a chord
// on one side (the segment starts past the closest approach, or ends
// before it) is integrated over its own interval.
__device__ __forceinline__ float m4_part_q(const float2* tab, float b2, float u1, float u2, bool clip_lo,
                                           bool clip_hi)
{
    const bool straddle = u1 < 0.f && u2 > 0.f;
    // the first piece: the clipped half of a straddling chord, or the chord
    float a1 = straddle ? 0.f : fminf(fabsf(u1), fabsf(u2));
    float a2 = straddle ? (clip_hi ? u2 : -u1) : fmaxf(fabsf(u1), fabsf(u2));
    const bool both = straddle && clip_hi && clip_lo;
    float F = 0.f;
#pragma unroll 1
    for (int e = 0;; ++e) {
        const float r = m4_seg_f(b2, a1, a2);
        F = e == 0 ? r : F + r;
        if (e == 1 || !both) break;
        a1 = 0.f;
        a2 = -u1;
    }
    if (straddle && !both) F += 0.5f * m4_full_tab(tab, b2);
    return F;
}

// a*b - c*d with one rounding (Kahan's difference of products via FMA)
__device__ __forceinline__ float dop(float a, float b, float c, float d)
{
    float w = __fmul_rn(c, d);
    float e = fmaf(-c, d, w);
    float f = fmaf(a, b, -w);
    return f + e;
}

struct Kahan {
    __device__ __forceinline__ static void add(float& s, float& c, float v)
    {
        float y = v - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    // s += a b, the product not rounded
    __device__ __forceinline__ static void add_product(float& s, float& c, float a, float b)
    {
        float y = fmaf(a, b, -c);
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ static void add(double& s, double& c, double v)
    {
        double y = v - c;
        double t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

// ---- the packet's beam ------------------------------------------------------
// The 32 rays of a packet are parallel (one direction d).  In the frame
// (e1, e2, d) anchored at C, a lane's segment is the point (u_i, v_i) across
// the direction and the depths [t_i, t_i + l_ray]; the beam is the box
// |u| <= hu, |v| <= hv, |t| <= ht that holds the live lanes' segments.
// Everything decided in this frame (child boxes, spheres against the beam,
// spheres against a lane's ray) is a conservative filter in front of the exact
// hit test: distances carry a margin of several times the roundings of the
// projections (each coordinate difference is rounded once and projected with
// a frame orthonormal to ~3e-7, together below 2e-6 of the distances
// involved; the margin is 4e-6 of them, plus 3e-7 of the coordinates for an
// origin held in double), so no crossing is dropped and the hits are those of
// testing every sphere.
struct Beam {
    float4 c;                     // C, ht
    float4 e1;                    // e1, hu
    float4 e2;                    // e2, hv
    float4 d;                     // d, margin
    float4 o;                     // half extents of the beam's axis-aligned bounds, margin included; 0
    float4 r;                     // its radii along d x (x, y, z), margin included; 0
};

// Smallest and largest of the warp's values (one reduction instruction each).
__device__ __forceinline__ float wmin(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float wmax(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Called by all 32 lanes with the same direction d and length L; (sx, sy, sz)
// is the lane's (shifted) origin.  Writes the warp's beam to shared memory and
// returns the lane's point and depth (u, v, t); at least one lane is live.
// A called function: it runs once per image, and the traversal's loop has to
// stay in the instruction cache.
template <typename Real>
__device__ __noinline__ float3 make_beam(Beam* out, unsigned lv, bool live, Real sx, Real sy, Real sz, float dx,
                                         float dy, float dz, float L)
{
    float u, v, t;
    const int a = __ffs(lv) - 1;
    const Real bx = __shfl_sync(0xffffffffu, sx, a), by = __shfl_sync(0xffffffffu, sy, a),
               bz = __shfl_sync(0xffffffffu, sz, a);
    // e1 perpendicular to d, from the coordinate axis least aligned with it
    float ax = 0.f, ay = 0.f, az = 0.f;
    if (fabsf(dx) <= fabsf(dy) && fabsf(dx) <= fabsf(dz)) ax = 1.f;
    else if (fabsf(dy) <= fabsf(dz)) ay = 1.f;
    else az = 1.f;
    float e1x = dy * az - dz * ay, e1y = dz * ax - dx * az, e1z = dx * ay - dy * ax;
    const float inv = rsqrtf(e1x * e1x + e1y * e1y + e1z * e1z);
    e1x *= inv;
    e1y *= inv;
    e1z *= inv;
    const float e2x = dy * e1z - dz * e1y, e2y = dz * e1x - dx * e1z, e2z = dx * e1y - dy * e1x;
    // the live lanes' bounds relative to lane a's origin give the centre
    float rx = (float)(sx - bx), ry = (float)(sy - by), rz = (float)(sz - bz);
    u = rx * e1x + ry * e1y + rz * e1z;
    v = rx * e2x + ry * e2y + rz * e2z;
    t = rx * dx + ry * dy + rz * dz;
    const float um = 0.5f * (wmin(live ? u : INFINITY) + wmax(live ? u : -INFINITY));
    const float vm = 0.5f * (wmin(live ? v : INFINITY) + wmax(live ? v : -INFINITY));
    const float tm = 0.5f * (wmin(live ? t : INFINITY) + wmax(live ? t : -INFINITY) + L);
    const float cx = (float)bx + (um * e1x + vm * e2x + tm * dx);
    const float cy = (float)by + (um * e1y + vm * e2y + tm * dy);
    const float cz = (float)bz + (um * e1z + vm * e2z + tm * dz);
    rx = (float)(sx - Real(cx));
    ry = (float)(sy - Real(cy));
    rz = (float)(sz - Real(cz));
    u = rx * e1x + ry * e1y + rz * e1z;
    v = rx * e2x + ry * e2y + rz * e2z;
    t = rx * dx + ry * dy + rz * dz;
    float hu = wmax(live ? fabsf(u) : 0.f), hv = wmax(live ? fabsf(v) : 0.f);
    float ht = wmax(live ? fmaxf(fabsf(t), fabsf(t + L)) : 0.f);
    const float eps = 4e-6f * (hu + hv + ht) + 3e-7f * (fabsf(cx) + fabsf(cy) + fabsf(cz));
    hu += eps;
    hv += eps;
    ht += eps;
    __syncwarp();                    // the previous beam's readers are done
    if ((threadIdx.x & 31) == 0) {
        out->c = make_float4(cx, cy, cz, ht);
        out->e1 = make_float4(e1x, e1y, e1z, hu);
        out->e2 = make_float4(e2x, e2y, e2z, hv);
        out->d = make_float4(dx, dy, dz, eps);
        out->o = make_float4(hu * fabsf(e1x) + hv * fabsf(e2x) + ht * fabsf(dx) + eps,
                             hu * fabsf(e1y) + hv * fabsf(e2y) + ht * fabsf(dy) + eps,
                             hu * fabsf(e1z) + hv * fabsf(e2z) + ht * fabsf(dz) + eps, 0.f);
        // d x axis lies in the (e1, e2) plane: its components are those of the axis on e2 and e1
        out->r = make_float4(hu * fabsf(e2x) + hv * fabsf(e1x) + eps, hu * fabsf(e2y) + hv * fabsf(e1y) + eps,
                             hu * fabsf(e2z) + hv * fabsf(e1z) + eps, 0.f);
    }
    __syncwarp();
    return make_float3(u, v, t);
}

// Whether the beam may reach the box [lo, hi]: separating axes x, y, z (on
// the differences to C, so that near-touching faces are exact), e1, e2, d and
// d x (x, y, z).  Comparisons are written so that a NaN passes.
__device__ __forceinline__ bool beam_box(const Beam& B, float4 lo, float4 hi)
{
    const float4 c4 = B.c, o4 = B.o;
    const float lx = lo.x - c4.x, ly = lo.y - c4.y, lz = lo.z - c4.z;
    const float hx = hi.x - c4.x, hy = hi.y - c4.y, hz = hi.z - c4.z;
    if (lx > o4.x || ly > o4.y || lz > o4.z || hx < -o4.x || hy < -o4.y || hz < -o4.z) return false;
    const float4 d4 = B.d, a4 = B.e1, b4 = B.e2, r4 = B.r;
    const float cx = 0.5f * (lx + hx), cy = 0.5f * (ly + hy), cz = 0.5f * (lz + hz);
    const float ex = 0.5f * (hx - lx), ey = 0.5f * (hy - ly), ez = 0.5f * (hz - lz);
    const float m = 2e-6f * (ex + ey + ez + fabsf(cx) + fabsf(cy) + fabsf(cz));
    const float adx = fabsf(d4.x), ady = fabsf(d4.y), adz = fabsf(d4.z);
    bool out = fabsf(cx * a4.x + cy * a4.y + cz * a4.z) > ex * fabsf(a4.x) + ey * fabsf(a4.y) + ez * fabsf(a4.z) + a4.w + m;
    out = out || fabsf(cx * b4.x + cy * b4.y + cz * b4.z) > ex * fabsf(b4.x) + ey * fabsf(b4.y) + ez * fabsf(b4.z) + b4.w + m;
    out = out || fabsf(cx * d4.x + cy * d4.y + cz * d4.z) > ex * adx + ey * ady + ez * adz + c4.w + m;
    out = out || fabsf(cy * d4.z - cz * d4.y) > ey * adz + ez * ady + r4.x + m;
    out = out || fabsf(cz * d4.x - cx * d4.z) > ez * adx + ex * adz + r4.y + m;
    out = out || fabsf(cx * d4.y - cy * d4.x) > ex * ady + ey * adx + r4.z + m;
    return !out;
}

// ---- staged spheres and pairs ---------------------------------------------------
// A warp's work space: a block of up to 32 spheres that the beam may reach and
// the list of (ray, sphere) pairs that the lanes' masks give for it, at most
// kPairs at a time (4 spheres never give more than 128).  The sizes keep three
// blocks of 8 warps on an SM (TraceLayout asserts it).
template <typename Real>
struct alignas(4 * sizeof(Real)) Origin {
    Real x, y, z;                 // a lane's (image-shifted) origin
    Real coef;                    // MODE_SCATTER: its ray's coefficient
};
template <typename Real, int XMODE, bool NF>
struct Staged {
    static constexpr int MODE = XMODE & 7;
    static constexpr bool k3 = (XMODE & kThree) != 0;
    static constexpr bool kF32 = sizeof(Real) == 4;
    static constexpr bool kStored = MODE == 2 || MODE == 4;   // MODE_FILL, MODE_CHUNK
    static constexpr int kPairs = kF32 && kStored ? (NF ? 128 : 192) : 256;
    float4 q[32];                 // x, y, z, h
    Origin<Real> org[32];
    union {
        struct {
            float u[32], v[32], t[32], hh[32];        // in the beam's frame; hh = (h + margin)^2
        };
        Real tc[kF32 || kStored ? kPairs : 1];        // once the masks are made: depths of the closest approach,
    };                                                //   where they are kept; then (FP32) a pair's weight
    Real val[kF32 || kStored ? kPairs : 1];   // b^2, where it is kept; then (FP32) a pair's chord integral
    int64_t base0[MODE == 2 ? 32 : 1];        // MODE_FILL, per lane: where its next hits are stored
    uint32_t chunk0[MODE == 4 ? 32 : 1], chunk1[MODE == 4 ? 32 : 1];   // MODE_CHUNK, per lane: its chunk and the next
    int room[kStored ? 32 : 1];               // per lane: hits that fit (there)
    unsigned lane_hits[kStored ? 32 : 1];     // per lane: which of its pairs are hits
    int lane_off[kStored ? 32 : 1];           // per lane: its first pair
    double ih[kF32 ? 1 : 32];     // FP64: 1/h
    double near_o[NF ? 32 : 1][3];            // near/far: shifted origin in double (the near test)
    float2 aw[kF32 ? 32 : 1];     // A_j and the tracer weight A_j x_j
    float2 g[kF32 ? 32 : 1];      // 1/h and h^2
    float2 w23[k3 ? 32 : 1];      // the other tracers' weights
    int j[32];                    // Morton slot
    int img_lo[3], img_n[2], img_batches;     // image_range, and the images' number / 32
    unsigned hit[kPairs / 32 + 1], full[kPairs / 32 + 1], any[kPairs / 32 + 1];   // bit per pair; any: near ones too
    uint16_t pair[kPairs];        // sphere << 5 | lane
};

// The lanes' candidates among the block's first m spheres (bit e: sphere e):
// the lane's segment comes within h + margin of the sphere's centre,
//   (u_e - u)^2 + (v_e - v)^2 + dt^2 < hh,  dt the distance of t_e to [t, t + L].
// Two spheres per packed FP32 operation.
template <typename St>
__device__ __forceinline__ unsigned candidates(const St& S, int m, float u, float v, float t, float L)
{
    const float2 nu = make_float2(-u, -u), nv = make_float2(-v, -v), nt = make_float2(-t, -t), nL = make_float2(-L, -L);
    unsigned mask = 0u;
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        if (e >= m) break;
        const float4 u4 = *reinterpret_cast<const float4*>(S.u + e), v4 = *reinterpret_cast<const float4*>(S.v + e);
        const float4 t4 = *reinterpret_cast<const float4*>(S.t + e), h4 = *reinterpret_cast<const float4*>(S.hh + e);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float2 du = __fadd2_rn(p ? make_float2(u4.z, u4.w) : make_float2(u4.x, u4.y), nu);
            const float2 dv = __fadd2_rn(p ? make_float2(v4.z, v4.w) : make_float2(v4.x, v4.y), nv);
            const float2 a = __fadd2_rn(p ? make_float2(t4.z, t4.w) : make_float2(t4.x, t4.y), nt);
            const float2 b = __fadd2_rn(a, nL);
            const float2 w = make_float2(fmaxf(fmaxf(-a.x, b.x), 0.f), fmaxf(fmaxf(-a.y, b.y), 0.f));
            float2 r = __fmul2_rn(dv, dv);
            r = __ffma2_rn(du, du, r);
            r = __ffma2_rn(w, w, r);
            if (!(r.x >= (p ? h4.z : h4.x))) mask |= 1u << (e + 2 * p);
            if (!(r.y >= (p ? h4.w : h4.y))) mask |= 2u << (e + 2 * p);
        }
    }
    return m < 32 ? mask & ((1u << m) - 1u) : mask;
}

// Particle index of stored segment pos: an int32, or split into 16 + 8 bits
// (neighbouring lanes store neighbouring positions of one ray's list).
__device__ __forceinline__ void store_index(const TraceParams& P, int64_t pos, int j)
{
    if (P.seg_col) {
        P.seg_col[pos] = j;
        return;
    }
    P.seg_lo[pos] = (uint16_t)((uint32_t)j & 0xffffu);
    if (P.seg_hi) P.seg_hi[pos] = (uint8_t)(((uint32_t)j >> 16) & 0xffu);
}

// ---- deferred partial chords ------------------------------------------------
// A partial chord (a sphere cut by the segment's start or end) takes the
// piecewise evaluation of m4_part_f, an order of magnitude more arithmetic
// than a full chord's table lookup, and with rays of a few smoothing lengths
// most hits are partial (every sphere holding the origin or the end point).
// Evaluated where it is met, a warp would run that code for the few lanes
// whose ray met one.  Instead the warp appends its partial chords to a queue
// in shared memory and evaluates them 32 at a time, one per lane; every ray
// then adds its own results in queue order (the lanes of one ray's items
// found by a bit mask per ray), so the sums stay deterministic.
constexpr int kPQ = 64;           // queue capacity per warp; a round takes 32
constexpr int kPQNear = 32;       // owner flag: a near particle (near/far split)
constexpr int kPQClipLo = 64;     // owner flag: the segment's start cuts the chord
constexpr int kPQClipHi = 128;    // owner flag: the segment's end cuts the chord
template <int XMODE, bool NF>
struct PartQueue {
    static constexpr int MODE = XMODE & 7;
    static constexpr bool k3 = (XMODE & kThree) != 0;
    static constexpr bool kAux = MODE != 0;   // every mode but MODE_TAU, of whose items the near ones need A_j
    float4 item[kPQ];             // b^2/h^2 and [u1, u2] in units of h; the tracer weight A_j x_j (MODE_SCATTER: the ray's coefficient)
    int4 aux[kAux ? kPQ : 1];     // particle (Morton slot), low half of the segment's position, bits of A_j; 0
    float A[NF && !kAux ? kPQ : 1];
    float2 w23[k3 ? kPQ : 1];     // the other tracers' weights
    float val2[k3 ? 32 : 1], val3[k3 ? 32 : 1];
    int owner[kPQ];               // lane of the ray | kPQNear | kPQClipLo | kPQClipHi | high half of the position << 16
    float val[32];                // results of the round being flushed
    unsigned own[NF ? 64 : 32];   // per owner (lane, lane + kPQNear): items of the round
};

// Items waiting in a ring of kPQ and where it begins (full: FP64 only).
struct Queued {
    int part, full, part_head, full_head;
};

// Position of a stored segment in a queue item: 47 bits and "nowhere" (-1).
__device__ __forceinline__ int pos_hi(int64_t pos) { return pos < 0 ? (int)0xffff0000 : (int)(pos >> 32) << 16; }
__device__ __forceinline__ int64_t pos_of(int owner, int lo)
{
    const int hi = (owner >> 16) & 0xffff;
    return hi == 0xffff ? -1 : ((int64_t)hi << 32) | (uint32_t)lo;
}

// Evaluate the first n (<= 32) queued chords, one per lane.  Every lane of the
// warp calls it.  Inlined: as a called function its reference arguments kept
// the ray's running state (sums, cursor, queue length) in local memory for the
// whole traversal, which cost 7 % of the traversal's time.
template <int KERNEL, int XMODE, bool NF, typename Queue>
__device__ __forceinline__ void flush_partials(const TraceParams& P, const float2* tab, Queue* pq, Queued& qn, int n,
                                               Sink<float>& k)
{
    constexpr int MODE = XMODE & 7;
    constexpr bool k3 = (XMODE & kThree) != 0;
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const int at = (qn.part_head + lane) & (kPQ - 1);
        const int ow = pq->owner[at];
        const float4 q = pq->item[at];
        const float F = KERNEL == URCHIN_KERNEL_M4 ? m4_part_q(tab, q.x, q.y, q.z, (ow & kPQClipLo) != 0, (ow & kPQClipHi) != 0)
                                                   : gt_chord<float>(P, q.x, q.y, q.z);
        int4 x = make_int4(0, 0, 0, 0);
        if (Queue::kAux) x = pq->aux[at];
        const float A = NF && !Queue::kAux ? pq->A[at] : __int_as_float(x.z);
        if (MODE == MODE_SCATTER) {
            atomicAdd(P.xbar + x.x, (double)(q.w * (A * F)));
        } else {
            pq->val[lane] = NF && (ow & kPQNear) ? A * F : q.w * F;
            if constexpr (k3) {
                const float2 w = pq->w23[at];
                pq->val2[lane] = w.x * F;
                pq->val3[lane] = w.y * F;
            }
            if (MODE == MODE_FILL || MODE == MODE_CHUNK) {
                const int64_t pos = pos_of(ow, x.y);
                if (MODE == MODE_FILL && pos >= 0) static_cast<float*>(P.seg_val)[pos] = A * F;
                if (MODE == MODE_CHUNK && pos >= 0) P.chunk_seg[pos] = make_int2(x.x, __float_as_int(A * F));
            }
            atomicOr(&pq->own[ow & (NF ? 31 | kPQNear : 31)], 1u << lane);
        }
    }
    __syncwarp();
    if (MODE != MODE_SCATTER) {
        for (unsigned m = pq->own[lane]; m; m &= m - 1) {
            Kahan::add(k.psum, k.pcomp, pq->val[__ffs(m) - 1]);
            if constexpr (k3) {
                Kahan::add(k.psum2, k.pcomp2, pq->val2[__ffs(m) - 1]);
                Kahan::add(k.psum3, k.pcomp3, pq->val3[__ffs(m) - 1]);
            }
        }
        if (NF)
            for (unsigned m = pq->own[lane + kPQNear]; m; m &= m - 1)
                Kahan::add(k.near, k.near_c, pq->val[__ffs(m) - 1]);
        __syncwarp();
        pq->own[lane] = 0u;
        if (NF) pq->own[lane + kPQNear] = 0u;
        __syncwarp();
    }
    qn.part_head = (qn.part_head + n) & (kPQ - 1);
    qn.part -= n;
}

// FP64: hits wait in two queues, full chords and partial ones (which cost
// twice as much), and either is evaluated 32 at a time.  Each ray's values are
// added in its queues' orders, full and partial chords apart, as in FP32.
template <bool kStored, bool NF>
struct HitQueue {
    double b2[2][kPQ];            // [0] full, [1] partial chords: b^2
    double tc[kPQ];               // partial: depth of the closest approach
    int64_t pos[2][kStored ? kPQ : 1];    // MODE_FILL: the segment's position
    double val[32];
    double ih[2][kPQ];            // 1/h
    float h[2][kPQ];
    int j[2][kPQ];                // particle (Morton slot)
    int owner[2][kPQ];            // lane of the ray | kPQNear
    unsigned own[NF ? 64 : 32];   // as PartQueue::own
};

template <int KERNEL, int MODE, bool NF, int KIND, typename Queue, typename St>
__device__ __forceinline__ void flush_hits(const TraceParams& P, const double2* lt, Queue* hq, const St& S,
                                           int& count, int& head, int n, double L, Sink<double>& k)
{
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const int at = (head + lane) & (kPQ - 1);
        const int j = hq->j[KIND][at], ow = hq->owner[KIND][at];
        const double b2 = hq->b2[KIND][at], h = (double)hq->h[KIND][at], ih = hq->ih[KIND][at];
        const double ch = sqrt(__fma_rn(h, h, -b2));
        const double beta2 = b2 * ih * ih;
        double F;
        if (KIND == 0) {
            const double c = ch * ih;
            // erf is odd: both ends of a full chord from one
            F = KERNEL == URCHIN_KERNEL_M4 ? m4_full(lt, beta2, c)
                                           : P.gt_pref * exp(-P.gt_t2 * beta2) * (2.0 * erf(P.gt_t * c));
        } else {
            const double tc = hq->tc[at];
            const double u1 = (fmax(0.0, tc - ch) - tc) * ih, u2 = (fmin(L, tc + ch) - tc) * ih;
            F = KERNEL == URCHIN_KERNEL_M4 ? m4_part(lt, beta2, u1, u2) : gt_chord(P, beta2, u1, u2);
        }
        if (MODE == MODE_SCATTER) {
            atomicAdd(P.xbar + j, S.org[ow].coef * (__ldg(P.A64 + j) * F));
        } else {
            const bool near = NF && (ow & kPQNear);
            hq->val[lane] = near ? __ldg(P.A64 + j) * F : __ldg(P.w64 + j) * F;
            if (MODE == MODE_FILL && hq->pos[KIND][at] >= 0)
                static_cast<double*>(P.seg_val)[hq->pos[KIND][at]] = __ldg(P.A64 + j) * F;
            atomicOr(&hq->own[ow & (31 | kPQNear)], 1u << lane);
        }
    }
    __syncwarp();
    if (MODE != MODE_SCATTER) {
        for (unsigned m = hq->own[lane]; m; m &= m - 1) {
            if (KIND == 0) Kahan::add(k.sum, k.comp, hq->val[__ffs(m) - 1]);
            else Kahan::add(k.psum, k.pcomp, hq->val[__ffs(m) - 1]);
        }
        if (NF)
            for (unsigned m = hq->own[lane + kPQNear]; m; m &= m - 1)
                Kahan::add(k.near, k.near_c, hq->val[__ffs(m) - 1]);
        __syncwarp();
        hq->own[lane] = 0u;
        if (NF) hq->own[lane + kPQNear] = 0u;
    }
    __syncwarp();
    head = (head + n) & (kPQ - 1);
    count -= n;
}

// MODE_CHUNK: `want` consecutive chunks from the warp's block of chunks in
// shared memory, a new block of kStash (or more) from the global counter when
// it runs out.  Called by lane 0 with the warp converged.
__device__ __forceinline__ unsigned long long chunk_block(const TraceParams& P, unsigned long long* stash, int want)
{
    unsigned long long b = stash[0];
    if (b + (unsigned long long)want > stash[1]) {
        const unsigned long long take = want > kStash ? (unsigned long long)want : (unsigned long long)kStash;
        b = atomicAdd(P.chunk_counter, take);
        stash[1] = b + take;
    }
    stash[0] = b + (unsigned long long)want;
    return b;
}

// Where a lane's next h hits go (MODE_FILL, MODE_CHUNK; called with the warp
// converged): consecutive positions of its ray's segment list, in MODE_CHUNK
// the rest of its chunk and then a new one (h <= 32 = kChunk, so one is enough).
template <int MODE, typename Real, typename St>
__device__ __forceinline__ void assign_positions(const TraceParams& P, unsigned long long* stash, St& S, int h,
                                                 Sink<Real>& k, unsigned& err)
{
    const int lane = threadIdx.x & 31;
    if constexpr (MODE == MODE_FILL) {
        int r = h;
        if ((int64_t)h > k.end - k.pos) {              // more hits than were counted
            r = (int)(k.end - k.pos);
            err |= kStSegment;
        }
        S.base0[lane] = k.pos;
        S.room[lane] = r;
        k.pos += r;
    } else {
        // coff: entries used of the current chunk (kChunk: none left, or no
        // chunk yet; kChunk + 1: the pool is exhausted, nothing more is stored)
        const int r = k.coff <= kChunk ? kChunk - k.coff : 0;
        const bool need = k.coff <= kChunk && h > r;
        S.chunk0[lane] = k.cur;
        S.room[lane] = r;
        uint32_t next = kNoChunk;
        const unsigned nm = __ballot_sync(0xffffffffu, need);
        if (nm) {
            unsigned long long base = 0;
            if (lane == 0) base = chunk_block(P, stash, __popc(nm));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (need) {
                const unsigned long long c = base + (unsigned long long)__popc(nm & ((1u << lane) - 1u));
                if (c < P.chunk_cap) {
                    if (k.cur == kNoChunk) P.chunk_head[k.ray] = (uint32_t)c;
                    else P.chunk_next[k.cur] = (uint32_t)c;
                    next = (uint32_t)c;
                    k.cur = next;
                    k.coff = h - r;
                } else {
                    k.coff = kChunk + 1;
                }
            }
        }
        if (!need && k.coff <= kChunk) k.coff += h;
        S.chunk1[lane] = next;
    }
}

// Position of pair p, a hit of lane o (-1: not stored).
template <int MODE, typename St>
__device__ __forceinline__ int64_t hit_position(const St& S, int p, int o)
{
    const int i = __popc(S.lane_hits[o] & ((1u << (p - S.lane_off[o])) - 1u)), r = S.room[o];
    if constexpr (MODE == MODE_FILL) return i < r ? S.base0[o] + i : -1;
    const uint32_t c = i < r ? S.chunk0[o] : S.chunk1[o];
    // the first chunk's free entries are its last r
    return c == kNoChunk ? -1 : (int64_t)c * kChunk + (i < r ? kChunk - r + i : i - r);
}

// Bits [off, off + c) of a list of flag words, c <= 32.
__device__ __forceinline__ unsigned flag_bits(const unsigned* w, int off, int c)
{
    const unsigned b = __funnelshift_r(w[off >> 5], w[(off >> 5) + 1], off & 31);
    return c < 32 ? b & ((1u << c) - 1u) : b;
}

// Hit decision of pair (sphere e, lane o).  Written with explicit roundings
// (no multiply-add contraction left to the compiler), so that the counting and
// the filling traversal, separate instantiations, find exactly the same hits.
// FP32: the impact parameter from an error-free cross product.
template <typename St>
__device__ __forceinline__ bool decide(const St& S, int e, int o, float dx, float dy, float dz, float L, float& b2,
                                       float& tc, float& ch)
{
    const float4 q = S.q[e];
    const Origin<float> s = S.org[o];
    const float ex = q.x - s.x, ey = q.y - s.y, ez = q.z - s.z;
    const float cx = dop(ey, dz, ez, dy);
    const float cy = dop(ez, dx, ex, dz);
    const float cz = dop(ex, dy, ey, dx);
    const float h2 = S.g[e].y;
    b2 = fmaf(cz, cz, fmaf(cy, cy, __fmul_rn(cx, cx)));
    if (!(b2 < h2)) return false;
    tc = fmaf(ez, dz, fmaf(ey, dy, __fmul_rn(ex, dx)));
    ch = sqrtf(__fsub_rn(h2, b2));
    return __fadd_rn(tc, ch) > 0.f && __fsub_rn(tc, ch) < L;
}

// In double the half chord ch stays squared, w = h^2 - b^2 = ch^2: tc + ch > 0,
// tc - ch < L, and (full) tc - ch >= 0, tc + ch <= L by comparing squares.
template <typename St>
__device__ __forceinline__ bool decide(const St& S, int e, int o, double dx, double dy, double dz, double L,
                                       double& b2, double& tc, bool& full)
{
    const float4 q = S.q[e];
    const Origin<double> s = S.org[o];
    const double ex = (double)q.x - s.x, ey = (double)q.y - s.y, ez = (double)q.z - s.z;
    const double cx = __fma_rn(ey, dz, -mul_rn(ez, dy));
    const double cy = __fma_rn(ez, dx, -mul_rn(ex, dz));
    const double cz = __fma_rn(ex, dy, -mul_rn(ey, dx));
    b2 = __fma_rn(cz, cz, __fma_rn(cy, cy, mul_rn(cx, cx)));
    const double w = __fma_rn((double)q.w, (double)q.w, -b2);
    if (!(w > 0.0)) return false;
    tc = __fma_rn(ez, dz, __fma_rn(ey, dy, mul_rn(ex, dx)));
    const double d = sub_rn(L, tc), t2 = mul_rn(tc, tc), d2 = mul_rn(d, d);
    full = tc >= 0.0 && d >= 0.0 && w <= t2 && w <= d2;
    return (tc > 0.0 || w > t2) && (d > 0.0 || w > d2);
}

// The pairs of the lanes' masks mm (at most kPairs in all): listed, decided,
// evaluated and added up (file comment).  FP32: full chords from the table at
// once, partial chords queued for flush_partials.  Where hits are stored
// (MODE_FILL, MODE_CHUNK) all pairs are decided first, which gives every hit
// its position.
template <int KERNEL, int XMODE, bool NF, typename Queue, typename St>
__device__ __forceinline__ void pairs_f32(const TraceParams& P, const float2* tab, Queue* pq, Queued& qn,
                                          unsigned long long* stash, St& S, unsigned mm, bool drain, float dx, float dy,
                                          float dz, float L, Sink<float>& k, unsigned& err)
{
    constexpr int MODE = XMODE & 7;
    constexpr bool k3 = (XMODE & kThree) != 0;
    constexpr bool kStored = MODE == MODE_FILL || MODE == MODE_CHUNK;
    const int lane = threadIdx.x & 31;
    const int c = __popc(mm);
    int off = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, off, d);
        if (lane >= d) off += y;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= c;
    {
        int i = off;
        for (unsigned m = mm; m; m &= m - 1u) S.pair[i++] = (uint16_t)(((__ffs(m) - 1) << 5) | lane);
    }
    __syncwarp();
    if constexpr (kStored) {
        for (int p0 = 0; p0 < total; p0 += 32) {
            const int p = p0 + lane;
            bool hit = false, near = false;
            if (p < total) {
                const int pr = S.pair[p], e = pr >> 5, o = pr & 31;
                float b2, tc = 0.f, ch = 0.f;
                hit = decide(S, e, o, dx, dy, dz, L, b2, tc, ch);
                if (hit) {
                    near = NF && is_near(S.near_o[o], S.q[e], tc, ch);
                    S.val[p] = b2;
                    S.tc[p] = tc;
                }
            }
            const unsigned ha = __ballot_sync(0xffffffffu, hit), hw = __ballot_sync(0xffffffffu, hit && !near);
            if (lane == 0) {
                S.any[p0 >> 5] = ha;
                S.hit[p0 >> 5] = hw;
            }
        }
        __syncwarp();
        const unsigned hm = c ? flag_bits(S.hit, off, c) : 0u;
        k.nhit += (unsigned)__popc(hm);
        S.lane_hits[lane] = hm;
        S.lane_off[lane] = off;
        assign_positions<MODE>(P, stash, S, __popc(hm), k, err);
        __syncwarp();
    }
    for (int p0 = 0; p0 < total || drain; p0 += 32) {
        const int p = p0 + lane;
        bool hit = false, near = false, full = false, part = false;
        int clip = 0, e = 0, o = 0;
        float beta2 = 0.f, u1 = 0.f, u2 = 0.f;
        float2 aw = make_float2(0.f, 0.f);
        int64_t pos = -1;
        if (p < total) {
            const int pr = S.pair[p];
            e = pr >> 5;
            o = pr & 31;
            float b2, tc = 0.f, ch = 0.f;
            if constexpr (kStored) {
                hit = (S.any[p0 >> 5] >> lane) & 1u;
                if (hit) {
                    b2 = S.val[p];
                    tc = S.tc[p];
                    ch = sqrtf(__fsub_rn(S.g[e].y, b2));
                    near = NF && !((S.hit[p0 >> 5] >> lane) & 1u);
                    if (!near) {
                        pos = hit_position<MODE>(S, p, o);
                        if (MODE == MODE_FILL && pos >= 0) store_index(P, pos, S.j[e]);
                    }
                }
            } else {
                hit = decide(S, e, o, dx, dy, dz, L, b2, tc, ch);
                if (hit) near = NF && is_near(S.near_o[o], S.q[e], tc, ch);
            }
            if (hit && MODE != MODE_COUNT) {
                const float ih = S.g[e].x;
                aw = S.aw[e];
                beta2 = b2 * ih * ih;
                full = __fsub_rn(tc, ch) >= 0.f && __fadd_rn(tc, ch) <= L;
                if (full) {
                    const float F = KERNEL == URCHIN_KERNEL_M4 ? m4_full_tab(tab, beta2)
                                                               : gt_chord<float>(P, beta2, -ch * ih, ch * ih);
                    if (MODE == MODE_SCATTER) atomicAdd(P.xbar + S.j[e], (double)(S.org[o].coef * (aw.x * F)));
                    else {
                        S.val[p] = F;
                        S.tc[p] = near ? aw.x : aw.y;
                    }
                    if (MODE == MODE_FILL && pos >= 0) static_cast<float*>(P.seg_val)[pos] = aw.x * F;
                    if (MODE == MODE_CHUNK && pos >= 0) P.chunk_seg[pos] = make_int2(S.j[e], __float_as_int(aw.x * F));
                } else {
                    part = true;
                    clip = (__fsub_rn(tc, ch) < 0.f ? kPQClipLo : 0) | (__fadd_rn(tc, ch) > L ? kPQClipHi : 0);
                    u1 = (fmaxf(0.f, tc - ch) - tc) * ih;
                    u2 = (fminf(L, tc + ch) - tc) * ih;
                }
            }
        }
        const unsigned fw = __ballot_sync(0xffffffffu, full);
        if constexpr (!kStored) {
            const unsigned hw = __ballot_sync(0xffffffffu, hit && !near);
            if (lane == 0) S.hit[p0 >> 5] = hw;
        }
        if (MODE == MODE_COUNT) continue;
        if (lane == 0) S.full[p0 >> 5] = fw;
        const unsigned pb = __ballot_sync(0xffffffffu, part);
        if (!pb && !drain) continue;
        if (part) {
            const int i = (qn.part_head + qn.part + __popc(pb & ((1u << lane) - 1u))) & (kPQ - 1);
            pq->item[i] = make_float4(beta2, u1, u2, MODE == MODE_SCATTER ? S.org[o].coef : aw.y);
            if (Queue::kAux) pq->aux[i] = make_int4(S.j[e], (int)(uint32_t)pos, __float_as_int(aw.x), 0);
            if (NF && !Queue::kAux) pq->A[i] = aw.x;
            if constexpr (k3) pq->w23[i] = S.w23[e];
            pq->owner[i] = o | (near ? kPQNear : 0) | clip | (kStored ? pos_hi(pos) : 0);
        }
        qn.part += __popc(pb);
        __syncwarp();
        // (at the end of the rays, drain, what is left: fewer than 32)
        if (qn.part >= 32 || (drain && qn.part > 0))
            flush_partials<KERNEL, XMODE, NF>(P, tab, pq, qn, min(qn.part, 32), k);
        if (drain) break;
    }
    __syncwarp();
    if (c) {
        if (!kStored) k.nhit += (unsigned)__popc(flag_bits(S.hit, off, c));
        if (MODE != MODE_COUNT && MODE != MODE_SCATTER) {
            unsigned far = 0xffffffffu;
            if (NF) far = flag_bits(S.hit, off, c);
            for (unsigned m = flag_bits(S.full, off, c); m; m &= m - 1u) {
                const int i = __ffs(m) - 1;
                const float F = S.val[off + i], w = S.tc[off + i];
                if constexpr (k3) {
                    const float2 q = S.w23[S.pair[off + i] >> 5];
                    Kahan::add_product(k.sum2, k.comp2, q.x, F);
                    Kahan::add_product(k.sum3, k.comp3, q.y, F);
                }
                if (!NF || ((far >> i) & 1u)) Kahan::add_product(k.sum, k.comp, w, F);
                else Kahan::add_product(k.near, k.near_c, w, F);
            }
        }
    }
    __syncwarp();
}

__device__ __forceinline__ double half_chord(float h, double b2)
{
    return sqrt(__fma_rn((double)h, (double)h, -b2));
}

// The same in double: hits go to the queues of full and of partial chords.
template <int KERNEL, int MODE, bool NF, typename Queue, typename St>
__device__ __forceinline__ void pairs_f64(const TraceParams& P, const double2* lt, Queue* hq, Queued& qn,
                                          unsigned long long* stash, St& S, unsigned mm, bool drain, double dx,
                                          double dy, double dz, double L, Sink<double>& k, unsigned& err)
{
    constexpr bool kStored = MODE == MODE_FILL;
    const int lane = threadIdx.x & 31;
    const int c = __popc(mm);
    int off = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, off, d);
        if (lane >= d) off += y;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= c;
    {
        int i = off;
        for (unsigned m = mm; m; m &= m - 1u) S.pair[i++] = (uint16_t)(((__ffs(m) - 1) << 5) | lane);
    }
    __syncwarp();
    if constexpr (kStored) {
        for (int p0 = 0; p0 < total; p0 += 32) {
            const int p = p0 + lane;
            bool hit = false, near = false, full = false;
            if (p < total) {
                const int pr = S.pair[p], e = pr >> 5, o = pr & 31;
                double b2, tc = 0.0;
                hit = decide(S, e, o, dx, dy, dz, L, b2, tc, full);
                if (hit) {
                    near = NF && is_near(S.near_o[o], S.q[e], tc, half_chord(S.q[e].w, b2));
                    S.val[p] = b2;
                    S.tc[p] = tc;
                }
            }
            const unsigned fw = __ballot_sync(0xffffffffu, hit && full);
            const unsigned ha = __ballot_sync(0xffffffffu, hit), hw = __ballot_sync(0xffffffffu, hit && !near);
            if (lane == 0) {
                S.any[p0 >> 5] = ha;
                S.hit[p0 >> 5] = hw;
                S.full[p0 >> 5] = fw;
            }
        }
        __syncwarp();
        const unsigned hm = c ? flag_bits(S.hit, off, c) : 0u;
        k.nhit += (unsigned)__popc(hm);
        S.lane_hits[lane] = hm;
        S.lane_off[lane] = off;
        assign_positions<MODE>(P, stash, S, __popc(hm), k, err);
        __syncwarp();
    }
    for (int p0 = 0; p0 < total || drain; p0 += 32) {
        const int p = p0 + lane;
        bool hit = false, near = false, full = false;
        int e = 0, o = 0;
        double b2 = 0.0, tc = 0.0;
        int64_t pos = -1;
        if (p < total) {
            const int pr = S.pair[p];
            e = pr >> 5;
            o = pr & 31;
            if constexpr (kStored) {
                hit = (S.any[p0 >> 5] >> lane) & 1u;
                if (hit) {
                    b2 = S.val[p];
                    tc = S.tc[p];
                    full = (S.full[p0 >> 5] >> lane) & 1u;
                    near = NF && !((S.hit[p0 >> 5] >> lane) & 1u);
                    if (!near) {
                        pos = hit_position<MODE>(S, p, o);
                        if (pos >= 0) store_index(P, pos, S.j[e]);
                    }
                }
            } else {
                hit = decide(S, e, o, dx, dy, dz, L, b2, tc, full);
                full = full && hit;
                if (hit) near = NF && is_near(S.near_o[o], S.q[e], tc, half_chord(S.q[e].w, b2));
            }
        }
        if constexpr (!kStored) {
            const unsigned hw = __ballot_sync(0xffffffffu, hit && !near);
            if (lane == 0) S.hit[p0 >> 5] = hw;
        }
        if (MODE == MODE_COUNT) continue;
        const unsigned fb = __ballot_sync(0xffffffffu, full), pb = __ballot_sync(0xffffffffu, hit && !full);
        const unsigned lt_mask = (1u << lane) - 1u;
        if (hit) {
            const int kind = full ? 0 : 1, i = (full ? qn.full_head + qn.full + __popc(fb & lt_mask)
                                                     : qn.part_head + qn.part + __popc(pb & lt_mask)) & (kPQ - 1);
            hq->b2[kind][i] = b2;
            if (!full) hq->tc[i] = tc;
            hq->h[kind][i] = S.q[e].w;
            hq->ih[kind][i] = S.ih[e];
            hq->j[kind][i] = S.j[e];
            hq->owner[kind][i] = o | (near ? kPQNear : 0);
            if (kStored) hq->pos[kind][i] = pos;
        }
        qn.full += __popc(fb);
        qn.part += __popc(pb);
        __syncwarp();
        if (qn.full >= 32 || (drain && qn.full > 0))
            flush_hits<KERNEL, MODE, NF, 0>(P, lt, hq, S, qn.full, qn.full_head, min(qn.full, 32), L, k);
        if (qn.part >= 32 || (drain && qn.part > 0))
            flush_hits<KERNEL, MODE, NF, 1>(P, lt, hq, S, qn.part, qn.part_head, min(qn.part, 32), L, k);
        if (drain) break;
    }
    __syncwarp();
    if (!kStored && c) k.nhit += (unsigned)__popc(flag_bits(S.hit, off, c));
    __syncwarp();
}

// The tree walk of one packet: next() gives the blocks of 32 spheres that the
// beam may reach, in their order, one after the other.
struct Walk {
    int lev, node;                // current entry: number `node` of level `lev`
    unsigned mask;                // its children still to be entered
    unsigned pend;                // lane l holds level l's mask while its subtrees are walked
    unsigned visits;
    bool fresh;                   // the current entry's children have not been tested

    __device__ __forceinline__ void children(const TraceParams& P, const Beam& B)
    {
        const int c = 32 * node + (int)(threadIdx.x & 31);
        bool pass = false;
        if (c < P.lev_cnt[lev - 1]) {
            const float4* b = P.boxes + 2 * ((int64_t)P.lev_off[lev - 1] + c);
            const float4 lo = __ldg(b), hi = __ldg(b + 1);
            pass = beam_box(B, lo, hi);
        }
        mask = __ballot_sync(0xffffffffu, pass);
        ++visits;
        fresh = false;
    }

    __device__ __forceinline__ void start(const TraceParams& P)
    {
        lev = P.n_lev;
        node = 0;
        mask = pend = visits = 0u;
        fresh = true;
    }

    // false at the end of the walk
    __device__ __forceinline__ bool next(const TraceParams& P, const Beam& B, int& ref, int& cnt)
    {
        for (;;) {
            if (fresh) children(P, B);
            if (mask == 0u) {
                if (lev == P.n_lev) return false;
                ++lev;
                node >>= 5;
                mask = __shfl_sync(0xffffffffu, pend, lev);
                continue;
            }
            const int c = __ffs(mask) - 1;
            mask &= mask - 1u;
            if (lev == 1) {
                ref = 32 * (32 * node + c);
                cnt = min(32, P.n - ref);
                return true;
            }
            if ((int)(threadIdx.x & 31) == lev) pend = mask;
            node = 32 * node + c;
            --lev;
            fresh = true;
        }
    }
};

// One image of the packet's rays: walk, stage, filter, evaluate (file comment);
// with drain, no image but the queued partial chords (so that the loop holds
// one copy of that code).
template <typename Real, int KERNEL, int XMODE, bool NF, typename Queue, typename St>
__device__ __forceinline__ void packet_image(const TraceParams& P, const unsigned char* tab, const Beam& B, St& S,
                                             Queue* pq, Queued& qn, unsigned long long* stash, float3 pt,
                                             float Lf, Real dx, Real dy, Real dz, bool live, bool drain,
                                             Sink<Real>& sk, unsigned& err, unsigned& nvisit)
{
    constexpr int MODE = XMODE & 7;
    constexpr bool k3 = (XMODE & kThree) != 0;
    const Real L = Real(P.l_ray);
    const int lane = threadIdx.x & 31;
    constexpr bool kF32 = sizeof(Real) == 4;
    constexpr bool kWantW = kF32 && MODE != MODE_COUNT && MODE != MODE_SCATTER;
    constexpr bool kWantA = kF32 && MODE != MODE_COUNT && (MODE != MODE_TAU || NF);
    Walk W;
    W.start(P);
    int ref = 0, cnt = 0;            // the current block (none at first) while the next one is on its way
    bool more = !drain;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 aw = make_float2(0.f, 0.f), w23 = make_float2(0.f, 0.f);
    auto fetch = [&](int r, int c) {
        if (lane < c && r >= 0 && r + lane < P.n) {
            q = __ldg(P.xyzh + r + lane);
            if (kWantA) aw.x = __ldg(P.A32 + r + lane);
            if (kWantW) aw.y = __ldg(P.w32 + r + lane);
            if (k3) w23 = make_float2(__ldg(P.w32_2 + r + lane), __ldg(P.w32_3 + r + lane));
        }
    };
    int ns = 0;                      // spheres in the block being filled
    for (;;) {
        const bool last = !more;
        unsigned pm = 0u;
        float su = 0.f, sv = 0.f, stt = 0.f, shh = 0.f;
        const float4 cq = q;
        const float2 caw = aw, cw23 = w23;
        const int cj = ref + lane;
        if (!last) {
            // sphere (one per lane) against the beam; the next block of spheres is on its way meanwhile
            bool pass = false;
            if (lane < cnt) {
                const float4 c4 = B.c, a4 = B.e1, b4 = B.e2, d4 = B.d;
                const float rx = cq.x - c4.x, ry = cq.y - c4.y, rz = cq.z - c4.z;
                su = rx * a4.x + ry * a4.y + rz * a4.z;
                sv = rx * b4.x + ry * b4.y + rz * b4.z;
                stt = rx * d4.x + ry * d4.y + rz * d4.z;
                const float hh = cq.w * 1.00001f + d4.w + 4e-6f * (fabsf(rx) + fabsf(ry) + fabsf(rz));
                shh = hh * hh;
                const float du = fmaxf(fabsf(su) - a4.w, 0.f), dv = fmaxf(fabsf(sv) - b4.w, 0.f),
                            dt = fmaxf(fabsf(stt) - c4.w, 0.f);
                pass = !(fmaf(dt, dt, fmaf(dv, dv, du * du)) >= shh) && cj >= 0 && cj < P.n;
            }
            pm = __ballot_sync(0xffffffffu, pass);
            more = W.next(P, B, ref, cnt);
            if (more) fetch(ref, cnt);
            if (pm == 0u) continue;
        }
        const int rank = __popc(pm & ((1u << lane) - 1u)), pc = __popc(pm);
        auto stage = [&](int at) {
            S.u[at] = su;
            S.v[at] = sv;
            S.t[at] = stt;
            S.hh[at] = shh;
            S.q[at] = cq;
            S.j[at] = cj;
            if constexpr (kF32) {
                if (kWantA || kWantW) S.aw[at] = caw;
                if constexpr (k3) S.w23[at] = cw23;
            }
        };
        const bool mine = (pm >> lane) & 1u;
        const int room = 32 - ns;
        if (mine && rank < room) stage(ns + rank);
        if (!last && pc < room) {
            ns += pc;
            continue;
        }
        // the block is full (or the walk over): the lanes' candidates in it
        const int m = last ? ns : 32;
        __syncwarp();
        {
            const float h = lane < m ? S.q[lane].w : 1.f;
            if constexpr (kF32) S.g[lane] = make_float2(MODE == MODE_COUNT ? 0.f : 1.f / h, __fmul_rn(h, h));
            else if (MODE != MODE_COUNT) S.ih[lane] = 1.0 / (double)h;
        }
        unsigned mask = candidates(S, m, pt.x, pt.y, pt.z, Lf);
        if (live) sk.ntest += (unsigned)m;
        else mask = 0u;
        // as many spheres at a time as their pairs fit: all, half, a quarter or an eighth
        const int total = __reduce_add_sync(0xffffffffu, __popc(mask));
        int step = 32;
        while (total > St::kPairs && step > 4) {
            step >>= 1;
            int most = 0;
            for (int e0 = 0; e0 < 32; e0 += step)
                most = max(most, (int)__reduce_add_sync(0xffffffffu, __popc(mask & (((1u << step) - 1u) << e0))));
            if (most <= St::kPairs) break;
        }
#pragma unroll 1
        for (int e0 = 0; (total > 0 || drain) && e0 < 32; e0 += step) {
            const unsigned mm = step == 32 ? mask : mask & (((1u << step) - 1u) << e0);
            if constexpr (kF32)
                pairs_f32<KERNEL, XMODE, NF>(P, reinterpret_cast<const float2*>(tab), pq, qn, stash, S, mm, drain, dx,
                                            dy, dz, L, sk, err);
            else
                pairs_f64<KERNEL, MODE, NF>(P, reinterpret_cast<const double2*>(tab), pq, qn, stash, S, mm, drain, dx, dy,
                                            dz, L, sk, err);
        }
        __syncwarp();                // the block's readers are done
        if (last) break;
        ns = pc - room;
        if (mine && rank >= room) stage(rank - room);
    }
    nvisit += W.visits;
    __syncwarp();
}

// The images a of one axis, lo <= a < lo + n, whose particles (bounds [rl, rh]
// + a L) a beam over [c - h, c + h] may reach; m covers the roundings of the
// shifted bounds and origins.
__device__ __forceinline__ void image_range(float c, float h, float rl, float rh, float L, float m, int nimg, int& lo,
                                            int& n)
{
    m += 2e-6f * (fabsf(c) + h);
    lo = max(-nimg, (int)ceilf((c - h - m - rh) / L));
    n = max(0, min(nimg, (int)floorf((c + h + m - rl) / L)) - lo + 1);
}

// Shift of image i of a beam, in ascending order of (x, y, z).
__device__ __forceinline__ int3 image_shift(int64_t i, const int* lo, int ny, int nz)
{
    if (i <= 0x7fffffff) {
        const unsigned u = (unsigned)i, q = u / (unsigned)nz, x = q / (unsigned)ny;
        return make_int3(lo[0] + (int)x, lo[1] + (int)(q - x * (unsigned)ny), lo[2] + (int)(u - q * (unsigned)nz));
    }
    const int64_t q = i / nz, x = q / ny;
    return make_int3(lo[0] + (int)x, lo[1] + (int)(q - x * ny), lo[2] + (int)(i - q * nz));
}

// A packet's origins usually fit in a few smoothing lengths, but some packets
// straddle a gap of the origins' order (a jump of the Morton curve, a sparse
// sample of origins), and one beam around all of them would sweep much of the
// box: such packets are traced as several beams, each of the origins within
// kBeamReach smoothing lengths (across) of its first one.  A ray's sums do not
// depend on the rays that share its beam.
constexpr float kBeamReach = 5.f;

template <typename Real, int KERNEL, int XMODE, bool NF, typename Queue, typename St>
__device__ __forceinline__ void ray_column(const TraceParams& P, const unsigned char* tab, Beam* beam, St& S,
                                           Queue* pq, Queued& qn, unsigned long long* stash, float4 o, Real dx,
                                           Real dy, Real dz, bool live, Sink<Real>& sk, unsigned& err,
                                           unsigned& nvisit)
{
    constexpr int MODE = XMODE & 7;
    const int lane = threadIdx.x & 31;
    const float Lf = P.l_beam;
    const int nimg = P.periodic ? P.nimg : 0;
    constexpr bool kQueue = MODE != MODE_COUNT;
    float3 pt = make_float3(0.f, 0.f, 0.f);
    unsigned left = __ballot_sync(0xffffffffu, live);
    while (left || (kQueue && (qn.part > 0 || qn.full > 0))) {
        const bool drain = !left;
        bool in = false;
        if (!drain) {
            const int a = __ffs(left) - 1;
            const float rx = o.x - __shfl_sync(0xffffffffu, o.x, a), ry = o.y - __shfl_sync(0xffffffffu, o.y, a),
                        rz = o.z - __shfl_sync(0xffffffffu, o.z, a), w = kBeamReach * __shfl_sync(0xffffffffu, o.w, a);
            const float along = rx * (float)dx + ry * (float)dy + rz * (float)dz;
            const float across2 = rx * rx + ry * ry + rz * rz - along * along;
            in = ((left >> lane) & 1u) && (lane == a || (across2 <= w * w && fabsf(along) <= 0.5f * Lf + w));
        }
        const unsigned lv = __ballot_sync(0xffffffffu, in);
        left &= ~lv;
        // the images of the box that the unshifted beam may reach, 32 at a
        // time, then one after the other in ascending order; away from the faces
        // that is the box itself, with the same beam
        bool have_beam = false;
        for (int b = 0;; ++b) {
            unsigned im = 1u;
            if (nimg > 0 && !drain) {
                pt = make_beam<Real>(beam, lv, in, Real(o.x), Real(o.y), Real(o.z), (float)dx, (float)dy, (float)dz, Lf);
                const float Lb = (float)P.Lbox, m1 = 2e-6f * (Lb + fabsf(P.root_lo[0]) + fabsf(P.root_hi[0]) + fabsf(P.root_lo[1]) +
                                                              fabsf(P.root_hi[1]) + fabsf(P.root_lo[2]) + fabsf(P.root_hi[2]));
                const float4 bc = beam->c, bo = beam->o;
                int lo[3], nx, ny, nz;
                image_range(bc.x, bo.x, P.root_lo[0], P.root_hi[0], Lb, m1, nimg, lo[0], nx);
                image_range(bc.y, bo.y, P.root_lo[1], P.root_hi[1], Lb, m1, nimg, lo[1], ny);
                image_range(bc.z, bo.z, P.root_lo[2], P.root_hi[2], Lb, m1, nimg, lo[2], nz);
                const int64_t images = (int64_t)nx * ny * nz;
                if (lane == 0) {
                    S.img_lo[0] = lo[0];
                    S.img_lo[1] = lo[1];
                    S.img_lo[2] = lo[2];
                    S.img_n[0] = ny;
                    S.img_n[1] = nz;
                    S.img_batches = (int)min((images + 31) >> 5, (int64_t)0x7fffffff);
                }
                __syncwarp();
                have_beam = images == 1 && lo[0] == 0 && lo[1] == 0 && lo[2] == 0;
                if (!have_beam) {
                    const int64_t i = (int64_t)b * 32 + lane;
                    bool pass = false;
                    if (i < images) {
                        const int3 a = image_shift(i, lo, ny, nz);
                        const float ax = (float)a.x * Lb, ay = (float)a.y * Lb, az = (float)a.z * Lb;
                        const float m = 1e-6f * (fabsf(ax) + fabsf(ay) + fabsf(az) + Lb);
                        pass = beam_box(*beam,
                                        make_float4(P.root_lo[0] + ax - m, P.root_lo[1] + ay - m, P.root_lo[2] + az - m, 0.f),
                                        make_float4(P.root_hi[0] + ax + m, P.root_hi[1] + ay + m, P.root_hi[2] + az + m, 0.f));
                    }
                    im = __ballot_sync(0xffffffffu, pass);
                }
            }
            for (; im; im &= im - 1u) {
                int3 a = make_int3(0, 0, 0);
                if (nimg > 0 && !drain) a = image_shift((int64_t)b * 32 + __ffs(im) - 1, S.img_lo, S.img_n[0], S.img_n[1]);
                // images of the particles at r_j + a L are reached by shifting the
                // origin to r_i - a L
                const Real sx = Real(o.x) - Real(a.x) * Real(P.Lbox);
                const Real sy = Real(o.y) - Real(a.y) * Real(P.Lbox);
                const Real sz = Real(o.z) - Real(a.z) * Real(P.Lbox);
                S.org[lane] = Origin<Real>{sx, sy, sz, sk.coef};
                if (NF) {
                    S.near_o[lane][0] = (double)o.x - (double)a.x * P.Lbox;
                    S.near_o[lane][1] = (double)o.y - (double)a.y * P.Lbox;
                    S.near_o[lane][2] = (double)o.z - (double)a.z * P.Lbox;
                }
                if (!drain && !have_beam)
                    pt = make_beam<Real>(beam, lv, in, sx, sy, sz, (float)dx, (float)dy, (float)dz, Lf);
                packet_image<Real, KERNEL, XMODE, NF>(P, tab, *beam, S, pq, qn, stash, pt, Lf, dx, dy, dz, in,
                                                     drain, sk, err, nvisit);
            }
            if (nimg == 0 || drain || b + 1 >= S.img_batches) break;
        }
    }
}

// k_trace's shared memory: per warp the work space, the beam, the block of
// chunks (MODE_CHUNK) and the queue of partial chords (FP64: of hits) in modes
// that evaluate chords; the M4 table (FP64: of logarithms).  The same for any
// number of directions (192 of them, 4608 B a block, left two blocks of three on
// an SM): a packet reads its own from global memory.
constexpr size_t kSmShared = 228 * 1024;      // an SM's shared memory, of which a block takes
constexpr size_t kBlockShared = 1024;         // this much beside its own
template <typename Real, int KERNEL, int XMODE, bool NF>
struct TraceLayout {
    static constexpr int MODE = XMODE & 7;
    static constexpr bool kF32 = sizeof(Real) == 4;
    static constexpr bool kQueue = MODE != MODE_COUNT;
    static constexpr bool kTable = kQueue && KERNEL == URCHIN_KERNEL_M4;
    static constexpr bool kStored = MODE == MODE_FILL || MODE == MODE_CHUNK;
    using St = Staged<Real, XMODE, NF>;
    using Queue = std::conditional_t<kF32, PartQueue<XMODE, NF>, HitQueue<kStored, NF>>;
    // warps per block and blocks per SM (k_trace's comment)
    static constexpr int kWarps = (XMODE & kWide) ? 14 : 8;
    static constexpr int kBlocks = (XMODE & (kWide | kThree)) || !kF32 ? 2 : 3;
    static constexpr size_t up(size_t b) { return (b + 15) & ~size_t(15); }
    static constexpr size_t kBeam = up(sizeof(St) * kWarps);
    static constexpr size_t kStashAt = up(kBeam + sizeof(Beam) * kWarps);
    static constexpr size_t kTab = up(kStashAt + kWarps * 2 * sizeof(unsigned long long));
    static constexpr size_t kQueueAt =
        up(kTab + (!kTable ? 0 : kF32 ? sizeof(float2) * (kKTab + 1) : sizeof(double2) * kLogTab));
    static constexpr size_t kBytes = up(kQueueAt + (kQueue ? sizeof(Queue) * kWarps : 0));
    static_assert(kBlocks * (kBytes + kBlockShared) <= kSmShared, "shared memory for the blocks of an SM");
};
static_assert(alignof(Staged<double, 2, true>) <= 32 && sizeof(Staged<float, 4, false>) % 16 == 0, "shared layout");

// Bound by instruction issue (80 % of the slots for plain columns, 73 % with the
// lists; 1/5 of the stalls waiting for shared memory, DRAM idle but for the
// lists): 29 warp instructions per crossed sphere on the 96^3 log-normal box with
// 32 origins per beam, 36 with the lists, against 45 and 46 (128^3) when every lane
// tested every staged sphere exactly, and 14 on a halo's long rays (21).  The pair
// list keeps the exact test and the chords at 30 of 32 lanes (16 to 21 when
// every lane took its own next candidate).  The traversal's loop has to fit
// the instruction cache: with two copies of the partial chords' code in it the
// list-keeping form stalled on fetches for half its time (256^3 box: solve
// 1168 ms, with one copy 893; 806 ms now with the tree of full blocks, the ring
// queue and one beam away from the faces).  All rays of the 128^3 box 102 ms
// before -> 63.7, of the 262144-particle halo 44.1 -> 28.8.
// Three blocks of 8 warps per SM (80 registers a thread).  Plain columns of many
// rays: two blocks of 14 (72 registers; one M4 table for 14 warps leaves the
// shared memory for 28 warps).  128^3 box: 28 warps 63.7 ms, 24 warps 67.8, 20
// warps (96 registers) 72.0, 16 warps (128, no spills) 76.8, 32 warps (64) 66.1;
// 262144-particle halo 30.2 -> 28.8 ms; but the 16^3 lattice's 3072 packets 0.33
// -> 0.36 ms, unevenly spread in blocks of 14.  The other FP32 modes need more
// shared memory per warp (list-keeping 128^3 solve 101.9 ms, with 26 warps
// 103.6; transpose of the 65536-particle halo 6.3 ms with 16 to 24 warps).
// FP64: bound by the FP64 pipe (85 % busy on the 16^3 lattice, 84 % on a 32^3 box
// with G_t, at 22 and 26 of 32 lanes; 17 before the queues of full and partial
// chords), two blocks; with queues and table logarithms the
// 16^3 lattice solve 18.3 -> 11.0 ms (82 ms with every lane testing every staged
// sphere), 24^3 box 10.7 -> 5.0 ms, 8000-particle halo 13.1 -> 8.4 ms, 9973 x 48
// rays of the 48^3 box (G_t) 25.3 -> 18.7 ms (277).
template <typename Real, int KERNEL, int XMODE, bool NF>
__global__ void __launch_bounds__(32 * TraceLayout<Real, KERNEL, XMODE, NF>::kWarps, TraceLayout<Real, KERNEL, XMODE, NF>::kBlocks)
k_trace(TraceParams P)
{
    constexpr int MODE = XMODE & 7;
    constexpr bool k3 = (XMODE & kThree) != 0;
    using Lay = TraceLayout<Real, KERNEL, XMODE, NF>;
    constexpr bool kQueue = Lay::kQueue;
    extern __shared__ __align__(32) unsigned char smem[];
    const int wid = threadIdx.x >> 5;
    typename Lay::St& st = reinterpret_cast<typename Lay::St*>(smem)[wid];
    Beam* beam = reinterpret_cast<Beam*>(smem + Lay::kBeam) + wid;
    unsigned long long* stash = reinterpret_cast<unsigned long long*>(smem + Lay::kStashAt) + 2 * wid;
    unsigned char* s_tab = smem + Lay::kTab;
    typename Lay::Queue* pq = reinterpret_cast<typename Lay::Queue*>(smem + Lay::kQueueAt) + wid;
    if (kQueue) {
        pq->own[threadIdx.x & 31] = 0u;
        if (NF) pq->own[(threadIdx.x & 31) + kPQNear] = 0u;
    }
    Queued qn{0, 0, 0, 0};
    if ((threadIdx.x & 31) == 0) {
        stash[0] = 0ull;
        stash[1] = 0ull;
    }
    if (Lay::kTable && Lay::kF32)
        for (int t = threadIdx.x; t <= kKTab; t += blockDim.x) reinterpret_cast<float2*>(s_tab)[t] = P.ktab[t];
    if (Lay::kTable && !Lay::kF32) log_table(reinterpret_cast<double2*>(s_tab));
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned long long total = (unsigned long long)P.n_chunks * (unsigned long long)P.R;
    unsigned err = 0;
    unsigned long long hits = 0, tests = 0, visits = 0;
    for (;;) {
        unsigned task = 0;
        if (lane == 0) task = atomicAdd(P.counter, 1u);
        task = __shfl_sync(0xffffffffu, task, 0);
        if ((unsigned long long)task >= total) break;
        const int k = (int)(task / P.n_chunks);
        const int64_t chunk = (int64_t)(task % P.n_chunks);
        const int64_t slot = chunk * P.packet + lane;
        // every lane takes part in the packet's votes; lanes past the end of
        // the origin list (and, in the transpose, rays with a zero
        // coefficient) are carried along without a segment
        bool live = lane < P.packet && slot < P.n_items;
        const bool mine = live;
        const int64_t item = !live ? 0 : (P.order ? (int64_t)P.order[(int64_t)k * P.n_items + slot] : slot);
        const int32_t org = live ? (P.items ? P.items[item] : (int32_t)item) : 0;
        float4 o = __ldg(P.xyzh + org);
        const double* dir = P.dirs + 3 * k;
        Real dx = Real(__ldg(dir)), dy = Real(__ldg(dir + 1)), dz = Real(__ldg(dir + 2));
        unsigned nvisit = 0;
        Sink<Real> sk{};
        // stored-segment rows are indexed by direction and Morton slot (rows
        // of particles not in the item list stay empty)
        const int64_t ray = (int64_t)k * P.n + org;
        sk.ray = ray;
        sk.coff = kChunk;
        sk.cur = kNoChunk;
        const int64_t orow = live ? (P.out_row ? (int64_t)P.out_row[item] : item) : 0;
        if (live && MODE == MODE_FILL) {
            sk.pos = (int64_t)P.row_ptr[ray];
            sk.end = (int64_t)P.row_ptr[ray + 1];
        }
        if (live && MODE == MODE_SCATTER) {
            sk.coef = static_cast<const Real*>(P.coef)[orow * P.row_stride + (int64_t)k * P.k_stride];
            live = sk.coef != Real(0);
        }
        ray_column<Real, KERNEL, XMODE, NF>(P, s_tab, beam, st, pq, qn, stash, o, dx, dy, dz, live, sk, err,
                                           nvisit);
        if (mine) {
            hits += sk.nhit;
            tests += sk.ntest;
            visits += nvisit;
            if (MODE == MODE_COUNT || MODE == MODE_CHUNK || (MODE == MODE_TAU && P.counts))
                P.counts[ray] = (sk.nhit + (unsigned)kSegPad - 1u) / (unsigned)kSegPad * (unsigned)kSegPad;
            if (MODE != MODE_COUNT && MODE != MODE_SCATTER) {
                if (MODE == MODE_CHUNK && sk.coff < kChunk) {
                    // zero entries up to a multiple of kSegPad (inside the chunk)
                    for (; (sk.coff & (kSegPad - 1)) != 0; ++sk.coff)
                        P.chunk_seg[(int64_t)sk.cur * kChunk + sk.coff] = make_int2(0, 0);
                }
                if (MODE == MODE_FILL) {
                    // the padding (fewer than kSegPad entries) holds zero values
                    if (sk.end - sk.pos >= kSegPad || sk.pos > sk.end) err |= kStSegment;
                    else
                        for (int64_t q = sk.pos; q < sk.end; ++q) {
                            store_index(P, q, 0);
                            static_cast<Real*>(P.seg_val)[q] = Real(0);
                        }
                }
                // full and partial chords are summed apart, each in an order that
                // depends on the ray alone (not on the rays sharing its warp)
                static_cast<Real*>(P.out)[orow * P.row_stride + (int64_t)k * P.k_stride] =
                    (sk.sum + sk.psum) - (sk.comp + sk.pcomp);
                if constexpr (k3) {
                    const int64_t at = orow * P.row_stride + (int64_t)k * P.k_stride;
                    P.out_2[at] = (sk.sum2 + sk.psum2) - (sk.comp2 + sk.pcomp2);
                    P.out_3[at] = (sk.sum3 + sk.psum3) - (sk.comp3 + sk.pcomp3);
                }
                if (NF) {
                    const int64_t at = P.near_k_stride > 0 ? (int64_t)org + (int64_t)k * P.near_k_stride
                                                           : orow * P.row_stride + (int64_t)k * P.k_stride;
                    static_cast<Real*>(P.out_near)[at] = sk.near;
                }
            }
        }
    }
    if (err && P.status) atomicOr(P.status, err);
    if (P.hits) {
        for (int o = 16; o > 0; o >>= 1) {
            hits += __shfl_xor_sync(0xffffffffu, hits, o);
            tests += __shfl_xor_sync(0xffffffffu, tests, o);
            visits += __shfl_xor_sync(0xffffffffu, visits, o);
        }
        if (lane == 0) {
            atomicAdd(P.hits, hits);
            atomicAdd(P.hits + 1, tests);
            atomicAdd(P.hits + 2, visits);
        }
    }
}

template <typename Real, int KERNEL, int MODE, bool NF>
int launch_one(const TraceParams& P, cudaStream_t s)
{
    const void* fn = (const void*)k_trace<Real, KERNEL, MODE, NF>;
    using Lay = TraceLayout<Real, KERNEL, MODE, NF>;
    const size_t smem = Lay::kBytes;
    URCHIN_TRY(allow_shared(fn, smem, smem));
    int grid = 0;
    URCHIN_TRY(grid_for(fn, 32 * Lay::kWarps, smem, &grid));
    const int64_t tasks = P.n_chunks * P.R;
    const int64_t need = (tasks + Lay::kWarps - 1) / Lay::kWarps;
    if (need < grid) grid = (int)std::max<int64_t>(need, 1);
    k_trace<Real, KERNEL, MODE, NF><<<grid, 32 * Lay::kWarps, smem, s>>>(P);
    URCHIN_TRY(launched());
    return URCHIN_OK;
}

template <typename Real, int KERNEL>
int dispatch_k(const TraceParams& P, int mode, bool nf, cudaStream_t s)
{
    if (P.w32_2) {
        if constexpr (sizeof(Real) == 4) {
            if (!nf && mode == MODE_CHUNK) return launch_one<float, KERNEL, MODE_CHUNK | kThree, false>(P, s);
            if (!nf && mode == MODE_TAU) return launch_one<float, KERNEL, MODE_TAU | kThree, false>(P, s);
        }
        return set_error(URCHIN_ERR_ARG, "trace: three tracers need FP32 columns without the near/far split");
    }
    if (nf) {
        if (mode == MODE_COUNT) return launch_one<Real, KERNEL, MODE_COUNT, true>(P, s);
        if (mode == MODE_FILL) return launch_one<Real, KERNEL, MODE_FILL, true>(P, s);
        if (mode == MODE_SCATTER) return set_error(URCHIN_ERR_ARG, "trace: no transpose with the near/far split");
        if (mode == MODE_CHUNK) return set_error(URCHIN_ERR_ARG, "trace: no chunked segment lists with the near/far split");
        return launch_one<Real, KERNEL, MODE_TAU, true>(P, s);
    }
    if (mode == MODE_COUNT) return launch_one<Real, KERNEL, MODE_COUNT, false>(P, s);
    if (mode == MODE_FILL) return launch_one<Real, KERNEL, MODE_FILL, false>(P, s);
    if (mode == MODE_SCATTER) return launch_one<Real, KERNEL, MODE_SCATTER, false>(P, s);
    if (mode == MODE_CHUNK) {
        if constexpr (sizeof(Real) == 4) return launch_one<Real, KERNEL, MODE_CHUNK, false>(P, s);
        return set_error(URCHIN_ERR_ARG, "trace: chunked segment lists are FP32 only");
    }
    if constexpr (sizeof(Real) == 4) {
        // enough packets for two per warp of the wide form
        int dev = 0, sms = 0;
        URCHIN_TRY_CUDA(cudaGetDevice(&dev));
        URCHIN_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (P.n_chunks * P.R >= (int64_t)sms * 56) return launch_one<float, KERNEL, MODE_TAU | kWide, false>(P, s);
    }
    return launch_one<Real, KERNEL, MODE_TAU, false>(P, s);
}

int dispatch_mode(const TraceParams& P, int precision, int kernel, int mode, bool nf, cudaStream_t s)
{
    if (precision == URCHIN_F64) {
        if (kernel == URCHIN_KERNEL_GT) return dispatch_k<double, URCHIN_KERNEL_GT>(P, mode, nf, s);
        return dispatch_k<double, URCHIN_KERNEL_M4>(P, mode, nf, s);
    }
    if (kernel == URCHIN_KERNEL_GT) return dispatch_k<float, URCHIN_KERNEL_GT>(P, mode, nf, s);
    return dispatch_k<float, URCHIN_KERNEL_M4>(P, mode, nf, s);
}

}  // namespace

// Full-chord M4 integral in double from the antiderivatives above:
// K(t) = 2 H(c), H(c) = Fo(c) [+ Fi(s) - Fo(s) when t < 1/4].
static double m4_full_host(double t)
{
    if (t >= 1.0) return 0.0;
    const double c = std::sqrt(1.0 - t);
    const double lb = t > 0.0 ? 0.5 * std::log(t) : 0.0;
    const double Lc = t > 0.0 ? std::log(c + 1.0) - lb : 0.0;
    double H = c * (0.5 + 3.25 * t) - (3.0 * t + 0.75 * t * t) * Lc;
    if (t < 0.25) {
        const double sv = std::sqrt(0.25 - t);
        const double Ls = t > 0.0 ? std::log(sv + 0.5) - lb : 0.0;
        H += -sv * (0.25 + 6.5 * t) + (3.0 * t + 3.0 * t * t) * Ls;
    }
    return 2.0 * H;
}

void m4_full_table(float2* out)
{
    const double h = 1e-5;
    for (int i = 0; i <= kKTab; ++i) {
        const double t = (double)i / kKTab;
        double d;
        if (t < 2 * h) d = (-3.0 * m4_full_host(t) + 4.0 * m4_full_host(t + h) - m4_full_host(t + 2 * h)) / (2 * h);
        else if (t > 1.0 - 2 * h) d = (3.0 * m4_full_host(t) - 4.0 * m4_full_host(t - h) + m4_full_host(t - 2 * h)) / (2 * h);
        else d = (m4_full_host(t + h) - m4_full_host(t - h)) / (2 * h);
        out[i] = make_float2((float)m4_full_host(t), (float)(d / kKTab));
    }
}

// Length of the segments that the filters see: l_ray, rounded up, but for
// isolated particles no more than the diagonal of their bounds, beyond which a
// ray from one of them meets none.  The filters' margins grow with the length,
// and with l_ray a million times the particles' extent they passed every sphere
// (4000-particle halo, l_ray 1e9 kpc: 2.0 ms, here 0.6, and quadratic in n).
static float beam_length(const urchin_bvh* b, double l_ray)
{
    const double l = l_ray * 1.000001 + 1e-30;
    if (b->periodic) return (float)l;
    double d2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double e = (double)b->root_hi[a] - (double)b->root_lo[a];
        d2 += e * e;
    }
    return (float)std::min(l, std::sqrt(d2) * 1.00001);
}

int launch_trace(const TraceJob& job, cudaStream_t s)
{
    if (job.n_items <= 0) return URCHIN_OK;
    const urchin_bvh* b = job.bvh;
    TraceParams P;
    P.ktab = b->ktab;
    P.boxes = b->boxes;
    P.n_lev = b->n_lev;
    for (int l = 0; l < kMaxLevels; ++l) {
        P.lev_off[l] = b->lev_off[l];
        P.lev_cnt[l] = b->lev_cnt[l];
    }
    P.n = (int)b->n;
    P.xyzh = b->xyzh;
    P.w32 = job.w32;
    P.w64 = job.w64;
    P.dirs = job.dirs_dev;
    P.R = job.R;
    P.l_ray = job.l_ray;
    P.l_beam = beam_length(b, job.l_ray);
    P.items = job.items;
    P.n_items = job.n_items;
    P.row_stride = job.row_stride;
    P.k_stride = job.k_stride;
    P.out_row = job.out_row;
    P.out = job.out;
    P.counter = job.counter;
    P.status = job.status;
    P.hits = job.hits;
    P.periodic = b->periodic;
    P.Lbox = b->L;
    // every image within l_ray + h_max of the box can reach the segment
    P.nimg = b->periodic ? (int)std::ceil((job.l_ray + (double)b->hmax) / b->L) : 0;
    for (int a = 0; a < 3; ++a) {
        P.root_lo[a] = b->root_lo[a];
        P.root_hi[a] = b->root_hi[a];
    }
    GtConst g = gt_constants();
    P.gt_t2 = g.t2;
    P.gt_t = g.t;
    P.gt_pref = g.pref;
    {
        // 32 origins per packet share most spheres; few rays are spread over
        // more warps instead, down to 8 per packet, while 3/4 of the 24 warps an
        // SM holds (FP64, whose evaluation outweighs the walk: all) would be
        // idle.  9^3 lattice, 12 rays: 32, 16, 8, 4 per packet 0.49, 0.34, 0.27,
        // 0.26 ms; 16^3: 0.43, 0.34, 0.38, 0.47 ms; FP64 9^3: 3.3, 1.9, 1.24,
        // 1.37 ms.
        int dev = 0, sms = 0;
        URCHIN_TRY_CUDA(cudaGetDevice(&dev));
        URCHIN_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const int64_t enough = (int64_t)sms * (job.precision == URCHIN_F64 ? 24 : 18);
        P.packet = 32;
        while (P.packet > 8 && (job.n_items + P.packet - 1) / P.packet * job.R < enough) P.packet >>= 1;
    }
    P.n_chunks = (job.n_items + P.packet - 1) / P.packet;
    if ((unsigned long long)P.n_chunks * (unsigned long long)job.R >= 0xffffffffull)
        return set_error(URCHIN_ERR_ARG, "trace: too many rays for one launch");
    URCHIN_TRY_CUDA(cudaMemsetAsync(job.counter, 0, sizeof(unsigned), s));
    P.counts = job.counts;
    P.row_ptr = job.row_ptr;
    P.seg_col = job.seg_col;
    P.seg_lo = job.seg_lo;
    P.seg_hi = job.seg_hi;
    P.seg_val = job.seg_val;
    P.A32 = b->A32;
    P.A64 = b->A64;
    P.coef = job.coef;
    P.xbar = job.xbar;
    P.order = job.order;
    P.out_near = job.out_near;
    P.near_k_stride = job.near_k_stride;
    P.chunk_head = job.chunk_head;
    P.chunk_next = job.chunk_next;
    P.chunk_counter = job.chunk_counter;
    P.chunk_cap = job.chunk_cap;
    P.chunk_seg = job.chunk_seg;
    P.w32_2 = job.w32_2;
    P.w32_3 = job.w32_3;
    P.out_2 = job.out_2;
    P.out_3 = job.out_3;
    if ((job.w32_2 != nullptr) != (job.w32_3 && job.out_2 && job.out_3))
        return set_error(URCHIN_ERR_ARG, "trace: three tracers need two more weights and outputs");
    if (job.near_far && !job.out_near && job.mode != MODE_COUNT)
        return set_error(URCHIN_ERR_ARG, "trace: near/far split without a near-column output");
    if (job.mode == MODE_FILL && !job.seg_col && !(job.seg_lo && (job.seg_hi ? b->n <= (int64_t(1) << 24) : b->n <= (int64_t(1) << 16))))
        return set_error(URCHIN_ERR_ARG, "trace: segment fill without a particle-index array");
    if (job.mode == MODE_CHUNK && (!job.chunk_head || !job.chunk_next || !job.chunk_counter || !job.counts ||
                                   !job.chunk_seg || job.chunk_cap == 0 || job.chunk_cap > 0xffffffffull))
        return set_error(URCHIN_ERR_ARG, "trace: chunked segment lists need heads, links, a counter and counts");
    return dispatch_mode(P, job.precision, job.kernel, job.mode, job.near_far != 0, s);
}

namespace {

// Every third bit of a 64-bit word from the low 21 bits of v (the standard
// Morton interleave).
__device__ __forceinline__ uint64_t spread21(uint32_t v)
{
    uint64_t x = v & 0x1fffffu;
    x = (x | x << 32) & 0x001f00000000ffffull;
    x = (x | x << 16) & 0x001f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

// keys of the items for directions k0 + blockIdx.y: the Morton code of
// (u, v, t / E) in the frame (e1, e2, d), 11 bits each over the widest of the
// three extents of the box (the last bit, of t, dropped)
__global__ void k_ray_keys(const float4* __restrict__ xyzh, const int32_t* __restrict__ items, int64_t n_items,
                           const double* __restrict__ dirs, int k0, float3 c, float3 ext, float inv_E,
                           uint32_t* __restrict__ keys, int32_t* __restrict__ vals)
{
    const int k = k0 + blockIdx.y;
    const float dx = (float)dirs[3 * k], dy = (float)dirs[3 * k + 1], dz = (float)dirs[3 * k + 2];
    // e1 perpendicular to d, from the coordinate axis least aligned with it
    float ax = 0.f, ay = 0.f, az = 0.f;
    if (fabsf(dx) <= fabsf(dy) && fabsf(dx) <= fabsf(dz)) ax = 1.f;
    else if (fabsf(dy) <= fabsf(dz)) ay = 1.f;
    else az = 1.f;
    float e1x = dy * az - dz * ay, e1y = dz * ax - dx * az, e1z = dx * ay - dy * ax;
    const float r = rsqrtf(e1x * e1x + e1y * e1y + e1z * e1z);
    e1x *= r;
    e1y *= r;
    e1z *= r;
    const float e2x = dy * e1z - dz * e1y, e2y = dz * e1x - dx * e1z, e2z = dx * e1y - dy * e1x;
    const float su = fabsf(e1x) * ext.x + fabsf(e1y) * ext.y + fabsf(e1z) * ext.z;
    const float sv = fabsf(e2x) * ext.x + fabsf(e2y) * ext.y + fabsf(e2z) * ext.z;
    const float st = (fabsf(dx) * ext.x + fabsf(dy) * ext.y + fabsf(dz) * ext.z) * inv_E;
    const float inv = 2048.f / fmaxf(fmaxf(fmaxf(su, sv), st), 1e-30f);
    auto q11 = [](float f) { return (uint32_t)fminf(fmaxf(f, 0.f), 2047.f); };
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_items;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float4 p = __ldg(xyzh + (items ? items[i] : (int32_t)i));
        const float rx = p.x - c.x, ry = p.y - c.y, rz = p.z - c.z;
        const float u = (rx * e1x + ry * e1y + rz * e1z + 0.5f * su) * inv;
        const float v = (rx * e2x + ry * e2y + rz * e2z + 0.5f * sv) * inv;
        const float t = ((rx * dx + ry * dy + rz * dz) * inv_E + 0.5f * st) * inv;
        const uint64_t code = (spread21(q11(u)) << 2) | (spread21(q11(v)) << 1) | spread21(q11(t));
        keys[(int64_t)blockIdx.y * n_items + i] = (uint32_t)(code >> 1);
        vals[(int64_t)blockIdx.y * n_items + i] = (int32_t)i;
    }
}

size_t order_bytes(int64_t n_items, int64_t g)
{
    Layout lay;
    lay.take(sizeof(uint32_t) * (size_t)(g * n_items));
    lay.take(radix_tmp_bytes(n_items, g));
    return lay.bytes;
}

// directions sorted at a time
int64_t order_batch(int64_t n_items, int R)
{
    return std::max<int64_t>(1, std::min<int64_t>(R, kRayOrderBatch / std::max<int64_t>(n_items, 1)));
}

}  // namespace

// One direction of a list just below kRadixLarge can need more than all of a
// longer one.
size_t ray_order_tmp_bytes(int64_t n_items, int R)
{
    return std::max(order_bytes(n_items, order_batch(n_items, R)), order_bytes(std::min(n_items, kRadixLarge - 1), 1));
}

double ray_order_elongation(const urchin_bvh* b, double l_ray)
{
    const double hg = b->hgeo > 0.f ? (double)b->hgeo : 1.0;
    return std::min(64.0, std::max(1.0, l_ray / (2.0 * hg)));
}

int ray_order(const urchin_bvh* b, const int32_t* items, int64_t n_items, const double* dirs_dev, int R, double l_ray,
              int32_t* order, void* tmp, size_t tmp_bytes, cudaStream_t s)
{
    if (n_items <= 0) return URCHIN_OK;
    // as many directions at a time as the work space holds (it may be sized for another number of items)
    int64_t g = order_batch(n_items, R);
    while (g > 1 && order_bytes(n_items, g) > tmp_bytes) --g;
    if (order_bytes(n_items, g) > tmp_bytes) return set_error(URCHIN_ERR_ARG, "ray_order: work space too small");
    Layout lay;
    const size_t o_k = lay.take(sizeof(uint32_t) * (size_t)(g * n_items));
    const size_t o_t = lay.take(radix_tmp_bytes(n_items, g));
    uint32_t* keys = reinterpret_cast<uint32_t*>(static_cast<char*>(tmp) + o_k);
    void* rt = static_cast<char*>(tmp) + o_t;
    const double E = ray_order_elongation(b, l_ray);
    const float3 c = make_float3(0.5f * (b->root_lo[0] + b->root_hi[0]), 0.5f * (b->root_lo[1] + b->root_hi[1]),
                                 0.5f * (b->root_lo[2] + b->root_hi[2]));
    const float3 ext = make_float3(b->root_hi[0] - b->root_lo[0], b->root_hi[1] - b->root_lo[1],
                                   b->root_hi[2] - b->root_lo[2]);
    const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_items + 255) / 256, 4096));
    for (int k = 0; k < R; k += (int)g) {
        const int m = (int)std::min<int64_t>(g, R - k);
        int32_t* vals = order + (size_t)k * n_items;
        k_ray_keys<<<dim3(gx, (unsigned)m), 256, 0, s>>>(b->xyzh, items, n_items, dirs_dev, k, c, ext, (float)(1.0 / E),
                                                         keys, vals);
        URCHIN_TRY(launched());
        URCHIN_TRY(radix_sort_pairs(keys, vals, n_items, 32, rt, s, m));
    }
    return URCHIN_OK;
}

// w[s] = A[s] x[perm[s]]
__global__ void k_weights(const float* __restrict__ A32, const double* __restrict__ A64,
                          const int32_t* __restrict__ perm, const double* __restrict__ x, int64_t n,
                          float* w32, double* w64)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        double xv = x[perm[s]];
        if (w64) w64[s] = A64[s] * xv;
        if (w32) w32[s] = (float)(A64[s] * xv);
    }
}

int launch_weights(const urchin_bvh* b, const double* x_orig, float* w32, double* w64, cudaStream_t s)
{
    unsigned grid = (unsigned)std::min<int64_t>((b->n + 255) / 256, 4096);
    k_weights<<<grid, 256, 0, s>>>(b->A32, b->A64, b->perm, x_orig, b->n, w32, w64);
    URCHIN_TRY(launched());
    return URCHIN_OK;
}

// origins (original indices) -> Morton slots; an index out of range flags
// the status word and maps to slot 0
__global__ void k_map_origins(const int32_t* __restrict__ origins, const int32_t* __restrict__ inv,
                              int64_t n_orig, int64_t n, int32_t* items, unsigned* status)
{
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n_orig;
         o += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = origins[o];
        if (i < 0 || i >= n) {
            atomicOr(status, kStOrigin);
            items[o] = 0;
        } else {
            items[o] = inv[i];
        }
    }
}

int launch_map_origins(const urchin_bvh* bvh, const int32_t* origins, int64_t n_orig, int32_t* items,
                       unsigned* status, cudaStream_t s)
{
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_orig + 255) / 256, 4096));
    k_map_origins<<<grid, 256, 0, s>>>(origins, bvh->inv, n_orig, bvh->n, items, status);
    return launched();
}

}  // namespace urchin

namespace urchin {
namespace {

// Argument checks shared by the column entry points (status 1 = valid no-op)
int check_trace_args(const char* fn, const urchin_bvh* bvh, const void* x, const double* dirs, int R, double l_ray,
                     const int32_t* origins, int64_t n_orig, int kernel, int precision, const void* buf)
{
    if (!bvh || !x || !dirs) return set_error(URCHIN_ERR_ARG, "%s: NULL bvh, input or dirs", fn);
    if (R < 1 || R > URCHIN_MAX_RAYS)
        return set_error(URCHIN_ERR_ARG, "%s: R = %d out of range [1, %d]", fn, R, URCHIN_MAX_RAYS);
    if (!(l_ray >= 0.0) || !std::isfinite(l_ray))
        return set_error(URCHIN_ERR_ARG, "%s: l_ray must be finite and >= 0", fn);
    if (kernel != URCHIN_KERNEL_M4 && kernel != URCHIN_KERNEL_GT)
        return set_error(URCHIN_ERR_ARG, "%s: unknown kernel %d", fn, kernel);
    if (precision != URCHIN_F32 && precision != URCHIN_F64)
        return set_error(URCHIN_ERR_ARG, "%s: unknown precision %d", fn, precision);
    if (n_orig < 0) return set_error(URCHIN_ERR_ARG, "%s: n_orig < 0", fn);
    if (n_orig == 0) return 1;
    if (!origins && n_orig != bvh->n) return set_error(URCHIN_ERR_ARG, "%s: origins NULL requires n_orig == n", fn);
    if (!buf) return set_error(URCHIN_ERR_ARG, "%s: output or cotangent array is NULL", fn);
    for (int i = 0; i < 3 * R; ++i)
        if (!std::isfinite(dirs[i])) return set_error(URCHIN_ERR_ARG, "%s: non-finite direction", fn);
    for (int k = 0; k < R; ++k) {
        double nn = dirs[3 * k] * dirs[3 * k] + dirs[3 * k + 1] * dirs[3 * k + 1] + dirs[3 * k + 2] * dirs[3 * k + 2];
        if (std::fabs(nn - 1.0) > 1e-6)
            return set_error(URCHIN_ERR_ARG, "%s: direction %d is not a unit vector", fn, k);
    }
    return URCHIN_OK;
}

// x_bar[perm[s]] += xm[s]
__global__ void k_unpermute_add(const int32_t* __restrict__ perm, const double* __restrict__ xm, int64_t n,
                                double* x_bar)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x)
        x_bar[perm[s]] += xm[s];
}

}  // namespace
}  // namespace urchin

namespace urchin {
namespace {

int trace_columns_impl(const char* fn, const urchin_bvh* bvh, const double* x, const double* dirs, int R,
                       double l_ray, const int32_t* origins, int64_t n_orig, int kernel, int precision,
                       void* tau_out, void* near_out, cudaStream_t s)
{
    {
        const int c = check_trace_args(fn, bvh, x, dirs, R, l_ray, origins, n_orig, kernel, precision, tau_out);
        if (c != URCHIN_OK) return c > 0 ? URCHIN_OK : c;
    }
    const int64_t n = bvh->n;
    const bool f64 = precision == URCHIN_F64;
    Layout lay;
    size_t o_ctr = lay.take(2 * sizeof(unsigned));
    size_t o_dirs = lay.take(sizeof(double) * 3 * (size_t)R);
    size_t o_w = lay.take((f64 ? sizeof(double) : sizeof(float)) * (size_t)n);
    size_t o_items = lay.take(origins ? sizeof(int32_t) * (size_t)n_orig : 0);
    const bool ordered = n_orig >= (origins ? kRayOrderMinSample : kRayOrderMinItems);
    size_t o_ord = lay.take(ordered ? sizeof(int32_t) * (size_t)R * (size_t)n_orig : 0);
    size_t o_otmp = lay.take(ordered ? ray_order_tmp_bytes(n_orig, R) : 0);
    Scratch scr;
    URCHIN_TRY(scr.alloc(lay.bytes, s));
    unsigned* ctr = scr.at<unsigned>(o_ctr);
    URCHIN_TRY_CUDA(cudaMemsetAsync(ctr, 0, 2 * sizeof(unsigned), s));
    URCHIN_TRY_CUDA(cudaMemcpyAsync(scr.at<double>(o_dirs), dirs, sizeof(double) * 3 * (size_t)R,
                                    cudaMemcpyHostToDevice, s));
    URCHIN_TRY(launch_weights(bvh, x, f64 ? nullptr : scr.at<float>(o_w), f64 ? scr.at<double>(o_w) : nullptr, s));
    TraceJob job{};
    job.bvh = bvh;
    job.w32 = f64 ? nullptr : scr.at<float>(o_w);
    job.w64 = f64 ? scr.at<double>(o_w) : nullptr;
    job.dirs_dev = scr.at<double>(o_dirs);
    job.R = R;
    job.l_ray = l_ray;
    job.n_items = n_orig;
    job.row_stride = R;
    job.k_stride = 1;
    job.out = tau_out;
    job.kernel = kernel;
    job.precision = precision;
    job.counter = ctr;
    job.status = ctr + 1;
    if (origins) {
        int32_t* items = scr.at<int32_t>(o_items);
        URCHIN_TRY(launch_map_origins(bvh, origins, n_orig, items, ctr + 1, s));
        job.items = items;
        job.out_row = nullptr;
    } else {
        // all particles, in Morton order for coherence; row = original index
        job.items = nullptr;
        job.out_row = bvh->perm;
    }
    if (ordered) {
        URCHIN_TRY(ray_order(bvh, job.items, n_orig, job.dirs_dev, R, l_ray, scr.at<int32_t>(o_ord),
                             scr.at<void>(o_otmp), ray_order_tmp_bytes(n_orig, R), s));
        job.order = scr.at<int32_t>(o_ord);
    }
    job.near_far = near_out ? 1 : 0;
    job.out_near = near_out;
    job.near_k_stride = 0;                      // same layout as tau_out
    URCHIN_TRY(launch_trace(job, s));
    unsigned st = 0;
    URCHIN_TRY_CUDA(cudaMemcpyAsync(&st, ctr + 1, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    scr.release();
    URCHIN_TRY_CUDA(cudaStreamSynchronize(s));
    if (st & kStOrigin) return set_error(URCHIN_ERR_ARG, "%s: origin index out of range", fn);
    return URCHIN_OK;
}

}  // namespace
}  // namespace urchin

extern "C" int urchin_trace_columns(const urchin_bvh* bvh, const double* x, const double* dirs, int R,
                                    double l_ray, const int32_t* origins, int64_t n_orig, int kernel,
                                    int precision, void* tau_out, urchin_stream_t stream)
{
    urchin::clear_error();
    return urchin::trace_columns_impl("urchin_trace_columns", bvh, x, dirs, R, l_ray, origins, n_orig, kernel,
                                      precision, tau_out, nullptr, (cudaStream_t)stream);
}

extern "C" int urchin_trace_columns_nearfar(const urchin_bvh* bvh, const double* x, const double* dirs, int R,
                                            double l_ray, const int32_t* origins, int64_t n_orig, int kernel,
                                            int precision, void* tau_far_out, void* tau_near_out,
                                            urchin_stream_t stream)
{
    urchin::clear_error();
    if (n_orig > 0 && !tau_near_out)
        return urchin::set_error(URCHIN_ERR_ARG, "urchin_trace_columns_nearfar: tau_near_out is NULL");
    return urchin::trace_columns_impl("urchin_trace_columns_nearfar", bvh, x, dirs, R, l_ray, origins, n_orig,
                                      kernel, precision, tau_far_out, tau_near_out, (cudaStream_t)stream);
}

extern "C" int urchin_trace_columns_vjp(const urchin_bvh* bvh, const double* dirs, int R, double l_ray,
                                        const int32_t* origins, int64_t n_orig, int kernel, int precision,
                                        const void* tau_bar, double* x_bar, urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    cudaStream_t s = (cudaStream_t)stream;
    {
        const int c = check_trace_args("urchin_trace_columns_vjp", bvh, tau_bar ? tau_bar : (const void*)dirs,
                                       dirs, R, l_ray, origins, n_orig, kernel, precision, x_bar);
        if (c != URCHIN_OK) return c > 0 ? URCHIN_OK : c;
        if (!tau_bar) return set_error(URCHIN_ERR_ARG, "urchin_trace_columns_vjp: tau_bar is NULL");
    }
    const int64_t n = bvh->n;
    Layout lay;
    size_t o_ctr = lay.take(2 * sizeof(unsigned));
    size_t o_dirs = lay.take(sizeof(double) * 3 * (size_t)R);
    size_t o_xm = lay.take(sizeof(double) * (size_t)n);
    size_t o_items = lay.take(origins ? sizeof(int32_t) * (size_t)n_orig : 0);
    const bool ordered = n_orig >= (origins ? kRayOrderMinSample : kRayOrderMinItems);
    size_t o_ord = lay.take(ordered ? sizeof(int32_t) * (size_t)R * (size_t)n_orig : 0);
    size_t o_otmp = lay.take(ordered ? ray_order_tmp_bytes(n_orig, R) : 0);
    Scratch scr;
    URCHIN_TRY(scr.alloc(lay.bytes, s));
    unsigned* ctr = scr.at<unsigned>(o_ctr);
    double* xm = scr.at<double>(o_xm);
    URCHIN_TRY_CUDA(cudaMemsetAsync(ctr, 0, 2 * sizeof(unsigned), s));
    URCHIN_TRY_CUDA(cudaMemsetAsync(xm, 0, sizeof(double) * (size_t)n, s));
    URCHIN_TRY_CUDA(cudaMemcpyAsync(scr.at<double>(o_dirs), dirs, sizeof(double) * 3 * (size_t)R,
                                    cudaMemcpyHostToDevice, s));
    TraceJob job{};
    job.bvh = bvh;
    job.dirs_dev = scr.at<double>(o_dirs);
    job.R = R;
    job.l_ray = l_ray;
    job.n_items = n_orig;
    job.row_stride = R;
    job.k_stride = 1;
    job.kernel = kernel;
    job.precision = precision;
    job.counter = ctr;
    job.status = ctr + 1;
    job.mode = 3;
    job.coef = tau_bar;
    job.xbar = xm;
    if (origins) {
        int32_t* items = scr.at<int32_t>(o_items);
        URCHIN_TRY(launch_map_origins(bvh, origins, n_orig, items, ctr + 1, s));
        job.items = items;
        job.out_row = nullptr;
    } else {
        job.items = nullptr;
        job.out_row = bvh->perm;
    }
    if (ordered) {
        URCHIN_TRY(ray_order(bvh, job.items, n_orig, job.dirs_dev, R, l_ray, scr.at<int32_t>(o_ord),
                             scr.at<void>(o_otmp), ray_order_tmp_bytes(n_orig, R), s));
        job.order = scr.at<int32_t>(o_ord);
    }
    URCHIN_TRY(launch_trace(job, s));
    unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4096));
    k_unpermute_add<<<grid, 256, 0, s>>>(bvh->perm, xm, n, x_bar);
    URCHIN_TRY(launched());
    unsigned st = 0;
    URCHIN_TRY_CUDA(cudaMemcpyAsync(&st, ctr + 1, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    scr.release();
    URCHIN_TRY_CUDA(cudaStreamSynchronize(s));
    if (st & kStOrigin) return set_error(URCHIN_ERR_ARG, "urchin_trace_columns_vjp: origin index out of range");
    return URCHIN_OK;
}
