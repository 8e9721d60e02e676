// cher_hits.cu -- the production kernel (steps a1-a5: generate_propagate in
// flat layers) and the adjoint's screening pass.
//
// Only 1-2 % of the bunches of a shower cross a telescope sphere.  A step's
// photons lie on one Cherenkov cone, so the azimuths around the step at which
// a photon can come near any sphere follow from the step alone
// (ring_setup, ring_sectors): a mask over 128 equal sectors, conservative by a bound on
// everything that moves an arrival line (refraction, the step's length, the
// arithmetic).  What is left per bunch:
//   * a step whose mask is empty has its bunches counted and nothing else;
//   * of the other steps' bunches only the Philox word of the azimuth is
//     drawn, and the bunch is dropped when its sector is not in the mask;
//   * the rest (1.2-1.5 times the number of crossings) are queued and
//     propagated 32 at a time, with the arithmetic of every other kernel.
// A step that could lose a bunch on the way (upward, out of the tables'
// height or zenith range), or whose bound does not hold, has all sectors set,
// so every counter and record is what propagating all bunches gives.
//
// Each warp works alone: it collects steps (32 lanes, one step each) until
// up to kCap of them have sectors to serve, works through their bunches in
// windows of 32, and goes on; there is no CTA barrier.
//
// What bounds it.  A vertical 1 TeV shower emits 32 bunches a step; 40 % of
// its steps have a sector to serve, 43 % of the bunches are drawn, 2.5 % are
// propagated and 1.8 % cross a sphere (60 deg: 57 / 69 / 2.5 / 1.1 %; 256
// showers over 2 x 2 km: 20 / 21 / 1.4 / 1.0 %).  So the time is in the steps
// (yield, bound, telescopes) and in the drawn Philox words, not in the
// propagation, and issue slots bound the FP32 kernel: on GB300, 2e6 steps,
// 62-68 % of them used with 30 of 64 warps resident (64 registers; the rest is
// waiting for the steps' and telescopes' loads), FP64 pipe 21-33 %, DRAM
// 81-90 bytes a step (the step is 64, a crossing's record 40).  The FP64 kernel
// is bound by its pipe (83 % busy: the yields' chains and the propagation).
// Per launch, against the kernel that propagated every bunch:
//   2e6 steps, vertical 1 TeV, 19 spheres     FP32   745 -> 279 us
//   2e7 steps, 256 showers, 100 spheres       FP32  6870 -> 1704 us
//   3e6 steps, 60 deg, 100 spheres            FP32   685 -> 488 us
//   2e5 steps, vertical 100 GeV, 19 spheres   FP64  1477 -> 156 us
//   3e5 steps with spectra                    FP32   234 -> 134 us
// Where rings pass many telescopes the bound costs
// more than it saves, and launches over such arrays take the kernel that
// propagates all bunches (k_probe, below).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "cher_internal.h"
#include "cher_path.cuh"

namespace cher {
namespace {

// Steps that a warp holds in shared memory while it works through their
// bunches: collecting stops when fewer than 32 places are left.
constexpr int kCap = 45;
constexpr int kPer = 2;               // consecutive bunches of a step per lane
constexpr int kQueue = 128;           // queued bunches per warp (a ring)
// Steps for the FP64 chain that make a group of their own (2e6 steps, 1 TeV:
// 285 us; the chain in the group where they come up 333; 20 to 32: 284 - 286).
constexpr int kSetAside = 16;
constexpr int kNear = 8;              // telescopes near one step's ring
constexpr int kSectors = 128;         // equal azimuth sectors of a cone
constexpr int kMaskWords = kSectors / 32;
static_assert(kQueue >= 31 + 32 * kPer, "a window's bunches fit behind the queued ones");

// ------------------------------------------------------------------------
// The azimuths of a step's cone that can reach a sphere.
//
// A bunch's arrival line passes the point A = E + g(p) A_x at the emission
// height (E the emission point, p the photon's direction on the cone, g(p) =
// n_e/n_o p_h sec^3(theta_o), A_x the table's horizontal correction: this is
// the kernel's ground point put back up along the arrival direction) with the
// direction p' = p + delta(p), delta the bend by Snell's law.  With A_0 and
// delta_0 those of the step's midpoint and axis, the distance of the line
// from a centre C is at least
//     |V x p| - M,   V = (C - A_0) - |C - A_0| delta_0,
// where M bounds the rest: the wander of E along the step (half its length
// times the angle between the step and the line), of g A_x and of delta over
// the cone (their derivatives along the cone, at the largest zenith on it,
// times the cone's angle), of n along the step, and the arithmetic (5 cm plus
// 1e-5 rad sec^2, and the rounding of the coordinates, which grows with them:
// KParams::Cull).  p = cos_c u + sin_c (cos phi e1 + sin phi e2), and with
// a = V.u, b = (V.e1, V.e2)
//     |V x p| >= | sin_c a (cos phi, sin phi) - cos_c b |
// (the distance of the two directions' gnomonic projections), so a crossing
// of a sphere of radius R needs
//     sin^2((phi - phi_b) / 2) <= (rho^2 - (r_c - r_k)^2) / (4 r_c r_k),
// rho = R + M, r_c = sin_c a, r_k = cos_c |b|.  Spheres come from a grid of
// centres through the bounding box of the ring that the cone leaves on the
// ground.
// ------------------------------------------------------------------------
// Per step, what the test of one telescope needs (64 bytes, in shared memory:
// the pairs of a group's steps and telescopes that pass the first test are
// worked on by full warps).
struct alignas(16) Ring {
    float4 a;      // A_0 (x, y, z above h_obs), mean sine of the cone
    float4 d;      // delta_0, M's constant part
    float4 u;      // axis, M per metre of distance
    float4 e;      // azimuth basis e1 (x, y); rho = (R + M) e.z + e.w a
};

// The kernels: BOUND as described above; LARGE, the same for arrays of more than
// 128 telescopes, which looks at the words of the box's x range only (a kernel of
// its own: the code costs BOUND 2 % where it gives nothing); DIRECT, which
// propagates the bunches of all steps, for launches where the bound would cost
// more than it saves (the array is dense, the rings are long, the steps at the
// edges of the tables: k_probe).
enum : int { BOUND = 0, DIRECT = 1, LARGE = 2 };
enum : int { REACH_NONE = 0, REACH_RING = 1, REACH_ALL = 2 };

// What the first test of one telescope needs besides (32 bytes, behind the
// Ring): the axis's ground point, the distance to it times the cone's sine,
// rho <= R fac + c1; the slack of r_k^2 and the axis's arrival direction.
struct alignas(16) Near {
    float4 p;      // P (x, y), sm a_0, c1
    float4 w;      // u' (x, y, z), E
};

struct Box {
    uint32_t bins;                // of the telescopes' centres: x0, x1 + 1, y0, y1 + 1
    float sec_lo, sec_hi;         // bounds of 1 / cos(theta_o) over the step's bunches
};

// A step's coordinate from the middle of the array, which is a float: the FP32
// path's ground points start from the rounded coordinate, so the difference is
// formed from that (two FP64 subtractions a step cost 2 % of a launch).
template <class R>
__device__ __forceinline__ float from_middle(double x, double o, float of) {
    if constexpr (std::is_same<R, float>::value) return __double2float_rn(x) - of;
    else return __double2float_rn(x - o);
}

// Sets up a step's ring; REACH_ALL where the bound does not hold or a bunch
// may be dropped on its way to the ground.  (Written without early returns:
// the lanes of a group stay together.)
template <int MODE, bool DS>
__device__ __forceinline__ int ring_setup(const KParams &p, float x0, float y0, float dz0, float L,
                                          float ux, float uy, float uz, float eta, float sinc_lo,
                                          float sinc_hi, Ring &G, Near &N, Box &B) {
    // (x0, y0: from the middle of the array); the rounding of coordinates
    const float err = p.cull.err_m * (fmaxf(fabsf(x0), p.cull.ex) + fmaxf(fabsf(y0), p.cull.ey)) +
                      p.cull.err_0;
    const float su2 = ux * ux + uy * uy;
    // the step points down, is a unit vector, and its cone is narrow
    bool ok = (uz < 0.0f) & (fabsf(su2 + uz * uz - 1.0f) <= 4e-6f) & (sinc_hi <= 0.25f);
    // the azimuth basis of prep_step; where rounding could make the two
    // differ in the choice for a vertical step, all sectors
    ok = ok & !((su2 <= 1e-19f) & (su2 > 1e-21f));
    const bool tilted = su2 > 1e-19f;
    const float isu = rsqrtf(tilted ? su2 : 1.0f);
    const float e1x = tilted ? -uy * isu : 1.0f, e1y = tilted ? ux * isu : 0.0f;
    const float su = tilted ? su2 * isu * 1.000001f : 1e-9f, cu = -uz;
    const float th = 1.011f * sinc_hi;                       // >= the cone's angle
    const float cch = sqrtf(1.0f - sinc_hi * sinc_hi);
    const float s_hi = su * cch + cu * sinc_hi + 1e-6f;      // the largest zenith on the cone
    ok = ok & (cu * cch - su * sinc_hi > 0.05f);
    const float half = 0.5f * L, dzm = dz0 + half * uz;
    const float edge = 0.1f + 2e-6f * fabsf(dz0);
    ok = ok & (dz0 + L * uz >= edge) & (dz0 <= p.f.dH_max - edge);
    // Snell at the step's midpoint, and its range over step and band
    const float rm1 = (eta - p.f.eta_o) * p.f.inv_np1o;
    const float k_hi = DS ? p.f.kap[0] : 1.0f, k_lo = DS ? p.f.kap_lo : 1.0f;
    const float rmk = rm1 * (0.5f * (k_hi + k_lo));
    const float drat = p.f.eta_slope * (half + 0.05f) * k_hi;
    const float dkap = DS ? fabsf(rm1) * (k_hi - k_lo) : 0.0f;
    const float bend = (fabsf(rm1) * k_hi + drat) * 1.001f;
    const float so_hi = s_hi * (1.0f + bend);
    const float q_hi = so_hi * so_hi;
    ok = ok & (q_hi <= p.f.q_max * 0.9999f - 1e-6f);
    const float sec_hi = rsqrtf(1.0f - q_hi) * 1.00001f, sec2 = sec_hi * sec_hi;
    const float rat = 1.0f + rmk;
    const float qu = su2 * rat * rat, sec = rsqrtf(1.0f - qu);
    const float dx = rmk * ux, dy = rmk * uy;
    const float dz = su2 * rmk * (2.0f + rmk) * sec * __frcp_rn(1.0f + cu * sec);
    // the table's horizontal correction for the axis
    float A;
    {
        const float fj = dzm * p.f.inv_dht, fk = qu * p.f.inv_dq;
        int jj = static_cast<int>(fj), kk = static_cast<int>(fk);
        jj = min(max(jj, 0), p.H - 2);
        kk = min(max(kk, 0), p.Z - 2);
        const float a = fj - static_cast<float>(jj), b = fk - static_cast<float>(kk);
        const int n0 = dbg_index(p, jj * p.Z + kk, int64_t(p.H - 1) * p.Z - 1, DBG_TAB);
        const float2 *T = p.cull.tab32 + n0;
        const float v00 = __ldg(T).x, v01 = __ldg(T + 1).x;
        const float v10 = __ldg(T + p.Z).x, v11 = __ldg(T + p.Z + 1).x;
        const float v0 = v00 + a * (v10 - v00), v1 = v01 + a * (v11 - v01);
        A = v0 + b * (v1 - v0);
    }
    if (DS) A *= 0.5f * (k_hi + k_lo);
    const float g = rat * sec * sec * sec;
    const float lead = half + A * g;
    const float X0 = x0 + lead * ux, Y0 = y0 + lead * uy;
    const float sm = 0.5f * (sinc_lo + sinc_hi);
    const float spread = DS ? 0.56f * (sinc_hi - sinc_lo) : 0.0f;
    // bounds: of A_x over the step and the cone (with a wavelength-dependent
    // index, over the band: it scales with kappa up to 10 %), of the line's
    // point (mo, metres) and direction (mw, radians)
    float dA = p.cull.ax_sq * (2.02f * su * th + 1.02f * th * th) + p.cull.ax_sh * (half + 0.05f);
    if (DS) dA += fabsf(A) * (0.1f + (k_hi - k_lo));
    const float mA = 1.02f * (fabsf(A) + dA) * sec2 * (3.0f * sec2 - 2.0f) * th + g * su * dA;
    const float bs = bend * sec_hi;
    const float mo = 0.06f + err + half * (sinc_hi + 1.1f * bs) + mA;
    const float mw = (1e-5f + 2.2f * bend * th) * sec2 + (1.1f * drat + dkap) * sec_hi + bs * bs;
    const float fac = 1.002f + 1.5f * bs;
    G.a = make_float4(X0, Y0, dzm, sm);
    G.d = make_float4(dx, dy, dz, mo);
    G.u = make_float4(ux, uy, uz, mw);
    G.e = make_float4(e1x, e1y, fac, spread);
    // (rounded down by 1e-6 of itself and 1e-6, as s_hi up: at 83 deg 1 / cos
    // moves by 66 times the sine's relative error)
    const float su_lo = tilted ? su2 * isu * 0.999999f : 0.0f;
    const float s_lo = fmaxf(su_lo * cch - cu * sinc_hi - 1e-6f, 0.0f) * (1.0f - bend);
    B.sec_lo = ok ? rsqrtf(1.0f - s_lo * s_lo) * 0.99999f : 0.0f;
    B.sec_hi = ok ? sec_hi : 1e30f;        // (0 .. 1e30: decides no transmission draw)
    // the ring on the ground: within sec^2 th (along the azimuth) and sec th
    // (across) of the axis's point per metre of height, so in a box around it
    const float r_max = MODE == MODE_SCREEN ? p.cull.r_cut : p.cull.r_max;
    const float dist = dzm + half;
    const float slack = dist * sec2 * mw + mA + err + 1.0f + 0.02f * L +
                        (1.01f * r_max + p.cull.z_max) * sec_hi;
    const float across = 1.03f * th * dist * sec_hi, along = across * sec_hi;
    const float ca = fabsf(e1y), sa = fabsf(e1x);        // the step's azimuth
    const float bwx = along * ca + across * sa + slack, bwy = along * sa + across * ca + slack;
    const float a0 = sec * dzm, t = rat * a0;
    const float Px = X0 + t * ux, Py = Y0 + t * uy;
    const float bx = (Px - p.cull.x0) * p.cull.inv_bx, by = (Py - p.cull.y0) * p.cull.inv_by;
    const int b0 = max(__float2int_rd(bx - bwx * p.cull.inv_bx), 0);
    const int b1 = min(__float2int_rd(bx + bwx * p.cull.inv_bx), kCullBins - 1);
    const int b2 = max(__float2int_rd(by - bwy * p.cull.inv_by), 0);
    const int b3 = min(__float2int_rd(by + bwy * p.cull.inv_by), kCullBins - 1);
    B.bins = static_cast<uint32_t>(b0) | static_cast<uint32_t>(b1 + 1) << 8 |
             static_cast<uint32_t>(b2) << 16 | static_cast<uint32_t>(b3 + 1) << 24;
    // first test, around the arrival direction u' = u + delta_0 with w = C -
    // A_0 (|w / |w| - u'| is the distance of V / |V| from u), in coordinates
    // D = C - P: w.u' = a_0 + D.u' and |w|^2 - (w.u')^2 = D^2 - (D.u')^2; rho
    // at the largest distance in the box, and the rounding of the squares
    const float w_max = a0 + 1.42f * fmaxf(bwx, bwy) + half + p.cull.z_max;
    const float c1 = mo * fac + 0.1f + (mw * fac + spread + 2.5f * bs * sinc_hi) * w_max;
    N.p = make_float4(Px, Py, sm * a0, c1);
    N.w = make_float4(ux + dx, uy + dy, uz + dz, 4e-6f * (bwx * bwx + bwy * bwy));
    // a step well above every sphere: no line comes to one from behind or from
    // the side (the tests below take a = w.u' > 0 and far from the cone's side)
    ok = ok & (dzm > p.cull.z_max + 2.5f * (r_max * fac + c1));
    return !ok ? REACH_ALL : (b0 <= b1 && b2 <= b3 ? REACH_RING : REACH_NONE);
}

// The first test of one telescope: the ring passes by it.
template <int MODE>
__device__ __forceinline__ bool ring_near(const KParams &p, float sm, float fac, float cm2,
                                          const float4 P, const float4 U, const float4 T) {
    const float dx = T.x - P.x, dy = T.y - P.y;
    const float dz = MODE == MODE_SCREEN ? 0.0f : T.z;
    const float dot = dx * U.x + dy * U.y + dz * U.z;
    const float rk2 = cm2 * (dx * dx + dy * dy + dz * dz - dot * dot);
    const float rc = sm * dot + P.z;
    const float rho = (MODE == MODE_SCREEN ? p.cull.r_cut : T.w) * fac + P.w;
    const float far = rc + rho, near = fmaxf(rc - rho, 0.0f);
    return (rk2 <= far * far + U.w) & (rk2 >= near * near - U.w);
}

// The sectors at which the ring can reach one telescope, first and number
// (kSectors: all, 0: none).
template <int MODE>
__device__ __forceinline__ int2 ring_sectors(const KParams &p, const Ring &G, const float4 T) {
    const float wx = T.x - G.a.x, wy = T.y - G.a.y;
    const float wz = (MODE == MODE_SCREEN ? 0.0f : T.z) - G.a.z;
    const float wl = sqrtf(wx * wx + wy * wy + wz * wz);
    const float vx = wx - wl * G.d.x, vy = wy - wl * G.d.y, vz = wz - wl * G.d.z;
    const float a = vx * G.u.x + vy * G.u.y + vz * G.u.z;
    if (!(a > 0.5f * wl)) return make_int2(0, kSectors);     // beside or behind the step
    const float sm = G.a.w, e1x = G.e.x, e1y = G.e.y;
    const float e2x = -G.u.z * e1y, e2y = G.u.z * e1x, e2z = G.u.x * e1y - G.u.y * e1x;
    const float b1 = vx * e1x + vy * e1y;
    const float b2 = vx * e2x + vy * e2y + vz * e2z;
    const float cm = sqrtf(1.0f - sm * sm);
    const float rk = cm * sqrtf(b1 * b1 + b2 * b2), rc = sm * a;
    const float rad = MODE == MODE_SCREEN ? p.cull.r_cut : T.w;
    const float rho = (rad + G.d.w + G.u.w * wl) * G.e.z + G.e.w * a;
    const float d = rc - rk;
    if (fabsf(d) > rho) return make_int2(0, 0);              // the ring passes it by
    const float num = (rho - d) * (rho + d), den = 4.0f * rc * rk;
    if (!(num < 0.99f * den)) return make_int2(0, kSectors); // all around
    // asin(y) <= y + 0.19 y^3 up to y = 1/2, <= pi/2 y beyond
    const float y = sqrtf(num / den);
    const float w = y < 0.5f ? y + 0.19f * y * y * y : 1.570797f * y;
    constexpr float kSect = kSectors / 6.28318530717958647692f;
    const float mid = atan2f(b2, b1) * kSect, dw = 2.0f * w * kSect + 0.03f;
    const int k0 = __float2int_rd(mid - dw), k1 = __float2int_rd(mid + dw);
    return make_int2(k0 & (kSectors - 1), min(k1 - k0 + 1, kSectors));
}

// Rare work kept out of the loops' code: the FP64 chain of a step that the
// screen left open, and the production profile.
__device__ __noinline__ void exact_call(const KParams &p, double z0, double len, double ekin,
                                        float uz, YieldF &y) {
    exact_yield(p, z0, len, ekin, uz, y);
}
__device__ __noinline__ void exact_disp_call(const KParams &p, double z0, double len, double ekin,
                                             float uz, YieldF &y, SegD<float> &D) {
    exact_yield_disp(p, z0, len, ekin, uz, y, D);
}
template <class R>
__device__ __noinline__ void profile_call(const KParams &p, int64_t i, R N) {
    profile_step<R>(p, i, N);
}

// sines of the cone over the band: the constant index's, or those of the
// smallest and largest kappa (from beta n - 1 = beta (eta kappa - x_th))
__device__ __forceinline__ float cone_sine(float beta, float eta, float kap, float x_th) {
    const float b = beta * (eta * kap - x_th);
    return b > 0.0f ? sqrtf(b * (2.0f + b)) / (1.0f + b) : 0.0f;
}

// ------------------------------------------------------------------------
// A warp's shared memory: its collected steps and its queue of bunches.
// ------------------------------------------------------------------------
template <class R, bool DS>
struct Spectra {
    SegD<R> segd[kCap];
    __device__ __forceinline__ SegD<R> *at(int s) { return segd + s; }
};
template <class R>
struct Spectra<R, false> {
    __device__ __forceinline__ SegD<R> *at(int) { return nullptr; }
};
template <bool TR>
struct SecRange {
    float2 sec[kCap];             // bounds of 1 / cos(theta_o)
};
template <>
struct SecRange<false> {};

// A queued bunch: a step has at most 2^22 bunches, so one word holds it (the
// screening pass takes bunch counts from the caller, and two words).
struct QueueHits {
    uint32_t v;
    __device__ __forceinline__ void set(int s, int j) { v = (static_cast<uint32_t>(s) << 22) | static_cast<uint32_t>(j); }
    __device__ __forceinline__ int place() const { return static_cast<int>(v >> 22); }
    __device__ __forceinline__ int bunch() const { return static_cast<int>(v & 0x3fffffu); }
};
struct QueueScreen {
    int s, j;
    __device__ __forceinline__ void set(int s_, int j_) { s = s_; j = j_; }
    __device__ __forceinline__ int place() const { return s; }
    __device__ __forceinline__ int bunch() const { return j; }
};

template <class R, class Entry, bool TR, bool DS>
struct alignas(16) WarpSmem : Spectra<R, DS>, SecRange<TR> {
    Seg<R> seg[kCap + 1];         // (one past the last: read, never used)
    uint32_t mask[kCap + 1][kMaskWords];
    int64_t step[kCap];
    union {
        Entry queue[kQueue];      // (place of the step, bunch of the step)
        uint16_t near[kNear][32]; // while collecting: each lane's telescopes
    };
    int64_t exact[kSetAside + 32];  // steps whose yield the FP64 chain decides
    int nb[kCap + 1];             // bunches of each place
    int off[kCap + 33];           // first piece (kPer bunches) of each place, the
                                  // total, no more
    unsigned long long n_emit, n_bunch;   // emitting steps and their bunches
    unsigned drop[6];             // bunches dropped, by status; [0]: invalid steps
};

// Word w of the telescopes in a box of bins.
__device__ __forceinline__ uint32_t box_telescopes(const KParams &p, uint32_t bins, int w) {
    const int nw = p.cull.words;
    const uint32_t *X = p.cull.bins + w, *Y = X + (kCullBins + 1) * nw;
    return __ldg(X + (bins >> 8 & 0xffu) * nw) & ~__ldg(X + (bins & 0xffu) * nw) &
           __ldg(Y + (bins >> 24) * nw) & ~__ldg(Y + (bins >> 16 & 0xffu) * nw);
}

// The words of a large array, which is sorted by x, that a box's x range
// touches.  False where the box holds more telescopes, estimated from its two
// ranges, than testing them can save on nb bunches.
__device__ __forceinline__ bool box_words(const KParams &p, uint32_t bins, int nb, int &w0, int &w1) {
    w1 = p.cull.words;
    const uint32_t *X = p.cull.bins + 2 * (kCullBins + 1) * w1, *Y = X + kCullBins + 1;
    const uint32_t x0 = __ldg(X + (bins & 0xffu)), x1 = __ldg(X + (bins >> 8 & 0xffu));
    const uint32_t ny = __ldg(Y + (bins >> 24)) - __ldg(Y + (bins >> 16 & 0xffu));
    w0 = static_cast<int>(x0 >> 5);
    w1 = static_cast<int>((x1 + 31u) >> 5);
    return (x1 - x0) * ny <= static_cast<uint32_t>(p.n_tel) * min(6u * nb + 16u, 65536u);
}

// inclusive prefix sum over the warp
__device__ __forceinline__ int warp_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// The place of the piece 32 win + lane, moving s_cur on to the window's end.
// Places start at distinct pieces, so the starts inside the window are one bit
// each (a shift by 32 or more gives 0); lanes past the last piece get the
// empty place behind the last.
template <class W>
__device__ __forceinline__ int place_at(W &w, int &s_cur, int win, int lane, unsigned below) {
    unsigned bit;
    asm("shl.b32 %0, 1, %1;" : "=r"(bit) : "r"(w.off[s_cur + 1 + lane] - win * 32));
    const unsigned starts = __reduce_or_sync(kFull, bit);
    const int s = s_cur + __popc(starts & (below * 2u + 1u));
    s_cur += __popc(starts);
    return s;
}

// A bunch past the tables' range: queued for the fallback pass.
template <class R>
__device__ __forceinline__ void defer(const KParams &p, const Consts<R> &c, const BunchOut<R> &o,
                                      bool live, R w, int64_t gstep, int j, int lane,
                                      unsigned below) {
    const bool dq = live && o.status == ST_DEFER;
    const unsigned qm = __ballot_sync(kFull, dq);
    if (!qm) return;
    const int leader = __ffs(qm) - 1;
    unsigned long long at0 = 0;
    if (lane == leader)
        at0 = atomicAdd(p.fb_count, static_cast<unsigned long long>(__popc(qm)));
    at0 = __shfl_sync(kFull, at0, leader);
    const unsigned long long at = at0 + __popc(qm & below);
    if (dq && at < static_cast<unsigned long long>(p.fb_cap)) {
        FbEntry<R> e;
        e.xe = o.X; e.ye = o.Y; e.he = c.h_obs + o.he; e.dh = o.he; e.te = o.t;
        e.hx = o.cx; e.hy = o.cy; e.s_obs = o.cz; e.c2 = o.c2; e.lam = o.lam;
        e.w = w;
        e.kap = o.kap;
        e.key = (static_cast<uint64_t>(gstep) << 32) | static_cast<uint32_t>(j);
        e.step_hi = static_cast<uint32_t>(static_cast<uint64_t>(gstep) >> 32);
        static_cast<FbEntry<R> *>(p.fb_list)[dbg_index(p, static_cast<int64_t>(at), p.fb_cap,
                                                       DBG_FB)] = e;
    }
}

// While a group is worked on, the places past cnt are free: place cnt + lane
// holds the lane's Ring and Near, and its mask collects the sectors; the pairs
// that pass the first test (two a lane at a time) are listed where the free
// places' offsets will be.
template <class W>
__device__ __forceinline__ Ring *ring_at(W &w, int place) {
    return reinterpret_cast<Ring *>(&w.seg[place]);
}
template <class W>
__device__ __forceinline__ Near *near_at(W &w, int place) {
    return reinterpret_cast<Near *>(reinterpret_cast<unsigned char *>(&w.seg[place]) + sizeof(Ring));
}
constexpr int kPairs = 64;
template <class W>
__device__ __forceinline__ uint32_t &pair_at(W &w, int q) {
    return reinterpret_cast<uint32_t *>(w.off + kCap - 32)[q];
}
static_assert(sizeof(Ring) + sizeof(Near) <= sizeof(Seg<float>), "a free place holds both");
static_assert(kCap - 32 + kPairs <= kCap + 33, "the pairs fit the free places' offsets");

template <class R, int MODE, bool TR, int FB, bool DS, int KIND>
__device__ __forceinline__ void hits(const KParams &p) {
    if (p.choice && (*p.choice < 0.0f) != (KIND == DIRECT)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    // (volatile: kept in registers instead of read again from the special
    // registers at every use)
    int lane, tid;
    unsigned below;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(below));
    // with the transmission draw every bunch has to be decided
    constexpr bool kDraw = TR && MODE == MODE_HITS && KIND != DIRECT;
    constexpr int kSpan = KIND == DIRECT ? 1 : kPer;     // bunches of a piece
    using Entry = typename std::conditional<MODE == MODE_HITS, QueueHits, QueueScreen>::type;
    using Warp = WarpSmem<R, Entry, kDraw, DS>;
    Warp &W = reinterpret_cast<Warp *>(smem)[tid >> 5];
    if (lane < 6) W.drop[lane] = 0u;

    Consts<R> c;
    R np1o;
    make_consts<R>(p, c, np1o);
    if (lane == 0) W.n_emit = W.n_bunch = 0ull;
    unsigned st_hits = 0, st_over = 0;

    // Groups of p.group steps: the first is the warp's own number, the others
    // come from the counter, asked for one ahead (the atomic's latency passes
    // while the warp works).  One group per request: with up to eight, 3e6
    // steps at 60 deg took 513 us instead of 496, 2e7 steps of 256 showers
    // 1732 instead of 1667.
    const unsigned n_warps = gridDim.x * (blockDim.x >> 5), n_groups = p.n_groups;
    unsigned claim = blockIdx.x * (blockDim.x >> 5) + (tid >> 5) - n_warps;

    int n_exact = 0;
    for (bool more = true; more;) {
        // ---- collect steps with sectors to serve -------------------------------
        int cnt = 0, tot = 0;
        do {
            // A group: the next steps, or, once kSetAside wait (or
            // nothing else is left), the steps whose bunch count the FP32
            // screen could not settle: one lane in twenty, which would hold
            // up its group on the FP64 pipe nearly every time.
            bool listed = n_exact >= kSetAside;
            unsigned cur = 0;
            if (!listed) {
                cur = n_warps + __shfl_sync(kFull, claim, 0);
                if (cur < n_groups) {
                    if (lane == 0)
                        claim = p.tile_counter ? atomicAdd(p.tile_counter, 1u) : n_groups - n_warps;
                } else {
                    if (n_exact == 0) { more = false; break; }
                    listed = true;
                }
            }
            int64_t i;
            bool have;
            if (listed) {
                const int first = max(n_exact - 32, 0);
                have = lane < n_exact - first;
                i = have ? W.exact[first + lane] : 0;
                n_exact = first;
            } else {
                // (the streams' first groups, then their second ones, ...)
                if (p.streams > 1) cur = cur % p.streams * (n_groups / p.streams) + cur / p.streams;
                i = int64_t(cur) * p.group + lane;
                have = lane < p.group && i < p.n;
            }
            using YT = typename std::conditional<std::is_same<R, float>::value, YieldF,
                                                 Yield>::type;
            YT y;
            y.nb = 0;
            SegD<R> D;
            Box B;
            int kind = REACH_NONE;
            bool open = false;
            if (have) {
                const double z0 = __ldg(p.z0 + i), len = __ldg(p.len + i), ekin = __ldg(p.ekin + i);
                const R uz = load_dir<R>(p.uz, i);
                if constexpr (std::is_same<R, float>::value) {
                    if (listed) {
                        if constexpr (DS) exact_disp_call(p, z0, len, ekin, uz, y, D);
                        else exact_call(p, z0, len, ekin, uz, y);
                    } else if constexpr (DS) {
                        open = !screen_yield_disp(p, step_valid<R>(p, i), z0, len, ekin, uz, y, D);
                    } else {
                        open = !screen_yield(p, step_valid<R>(p, i), z0, len, ekin, uz, y);
                    }
                } else {
                    const bool ok = step_valid<R>(p, i);
                    if constexpr (DS) step_yield_disp<R>(p, ok, z0, len, ekin, uz, y, D);
                    else step_yield(p, ok, z0, len, ekin, uz, y);
                }
                if (!open) {
                    if constexpr (MODE == MODE_SCREEN) {
                        // the adjoint freezes the sub-step structure
                        if (p.nb_frozen) {
                            const int nf = __ldg(p.nb_frozen + i);
                            y.nb = (y.s2 > 0.0 && nf > 0) ? nf : 0;
                        } else {
                            p.y_nb[i] = y.nb;
                        }
                    }
                    if constexpr (MODE == MODE_HITS) {
                        if (p.prof && y.nb > 0) profile_call<R>(p, i, static_cast<R>(y.N));
                    }
                    if (!y.valid) atomicAdd(&W.drop[0], 1u);
                }
                if (KIND != DIRECT && !open && y.nb > 0) {
                    float ux, uy, uzf, eta, s_lo, s_hi;
                    if constexpr (std::is_same<R, float>::value) {
                        ux = load_dir<R>(p.ux, i);
                        uy = load_dir<R>(p.uy, i);
                        uzf = uz;
                        eta = y.eta;
                    } else {
                        ux = d2f_rn(load_dir<R>(p.ux, i));
                        uy = d2f_rn(load_dir<R>(p.uy, i));
                        uzf = d2f_rn(uz);
                        eta = d2f_rn(y.eta);
                    }
                    if constexpr (DS) {
                        const float beta = static_cast<float>(D.beta), xt = static_cast<float>(D.x_th);
                        s_lo = cone_sine(beta, eta, p.f.kap_lo, xt);
                        s_hi = cone_sine(beta, eta, p.f.kap[0], xt) * 1.0001f + 1e-6f;
                    } else if constexpr (std::is_same<R, float>::value) {
                        s_lo = s_hi = sqrtf(y.s2);
                    } else {
                        s_lo = s_hi = sqrtf(d2f_rn(y.s2));
                    }
                    kind = ring_setup<MODE, DS>(p, from_middle<R>(__ldg(p.x0 + i), p.cull.ox, p.cull.oxf),
                                                from_middle<R>(__ldg(p.y0 + i), p.cull.oy, p.cull.oyf),
                                                __double2float_rn(z0) - p.f.h_obs,
                                                __double2float_rn(len), ux, uy, uzf,
                                                eta, s_lo, s_hi,
                                                *ring_at(W, cnt + lane), *near_at(W, cnt + lane), B);
                }
            }
            if constexpr (std::is_same<R, float>::value) {
                if (!listed) {
                    const unsigned om = __ballot_sync(kFull, open);
                    if (open) W.exact[n_exact + __popc(om & below)] = i;
                    n_exact += __popc(om);
                }
            }
            const int nb = open ? 0 : y.nb;
            if constexpr (MODE == MODE_HITS) {
                const unsigned emit = __popc(__ballot_sync(kFull, nb > 0));
                const unsigned sum = __reduce_add_sync(kFull, static_cast<unsigned>(nb));
                if (lane == 0) {
                    W.n_emit += emit;
                    W.n_bunch += sum;
                }
            }

            uint32_t mask[kMaskWords], any = 0u;
            if constexpr (KIND != DIRECT) {
                // the telescopes near each lane's ring (32 to a word, from the box
                // by the bins' prefix masks), then the sectors of those pairs
#pragma unroll
                for (int w = 0; w < kMaskWords; ++w) W.mask[cnt + lane][w] = 0u;
                int n_near = 0, w0 = 0, w1 = p.cull.words;
                if constexpr (KIND == LARGE)
                    if (kind == REACH_RING && !box_words(p, B.bins, nb, w0, w1)) kind = REACH_ALL;
                if (kind == REACH_RING) {
                    const Ring *G = ring_at(W, cnt + lane);
                    const Near *N = near_at(W, cnt + lane);
                    const float sm = G->a.w, fac = G->e.z, cm2 = 1.0f - sm * sm;
                    const float4 P = N->p, U = N->w;
                    for (int w = w0; w < w1; ++w) {
                        uint32_t cand = box_telescopes(p, B.bins, w);
                        while (cand) {
                            const int m = w * 32 + __ffs(cand) - 1;
                            cand &= cand - 1u;
                            const bool in = ring_near<MODE>(
                                p, sm, fac, cm2, P, U,
                                __ldg(p.cull.tel + dbg_index(p, m, p.n_tel, DBG_GRID)));
                            if (in) W.near[n_near & (kNear - 1)][lane] = static_cast<uint16_t>(m);
                            n_near += in;
                        }
                    }
                    if (n_near > kNear) {
                        kind = REACH_ALL;
                        n_near = 0;
                    }
                }
                __syncwarp();
                // two telescopes a lane at a time: one round of full lanes for the
                // usual 19 - 30 pairs of a group
                for (int k0 = 0; __any_sync(kFull, n_near > k0); k0 += 2) {
                    int n_pairs = 0;
#pragma unroll
                    for (int k = k0; k < k0 + 2; ++k) {
                        const unsigned has = __ballot_sync(kFull, n_near > k);
                        if (n_near > k)
                            pair_at(W, n_pairs + __popc(has & below)) =
                                static_cast<uint32_t>(cnt + lane) << 16 | W.near[k][lane];
                        n_pairs += __popc(has);
                    }
                    __syncwarp();
                    for (int q = lane; q < n_pairs; q += 32) {
                        const uint32_t e = pair_at(W, q);
                        const int at = static_cast<int>(e >> 16);
                        const int2 sec = ring_sectors<MODE>(p, *ring_at(W, at),
                                                            __ldg(p.cull.tel + (e & 0xffffu)));
                        // sectors sec.x .. sec.x + sec.y - 1 around the circle, word by word
                        for (int s = sec.x, n = sec.y; n > 0;) {
                            const int b = s & 31, m = min(32 - b, n);
                            atomicOr(&W.mask[at][(s >> 5) & (kMaskWords - 1)],
                                     (m == 32 ? kFull : (1u << m) - 1u) << b);
                            s += m;
                            n -= m;
                        }
                    }
                    __syncwarp();
                }
#pragma unroll
                for (int w = 0; w < kMaskWords; ++w) {
                    mask[w] = kind == REACH_ALL ? kFull : W.mask[cnt + lane][w];
                    any |= mask[w];
                }
                __syncwarp();
            }
            const bool keep = nb > 0 && (KIND == DIRECT || kDraw || any != 0u);
            const unsigned kept = __ballot_sync(kFull, keep);
            const int np = (nb + kSpan - 1) / kSpan;
            const int v = warp_scan(keep ? np : 0, lane);
            if (keep) {
                const int s = dbg_index(p, cnt + __popc(kept & below), kCap, DBG_SMEM);
                W.off[s] = tot + v - np;
                W.nb[s] = nb;
                if constexpr (KIND != DIRECT) {
#pragma unroll
                    for (int w = 0; w < kMaskWords; ++w) W.mask[s][w] = mask[w];
                }
                if constexpr (kDraw) W.sec[s] = make_float2(B.sec_lo, B.sec_hi);
                W.step[s] = i;
                // (what prep_step takes of the yield, until the batch is full)
                W.seg[s].cosc = static_cast<R>(y.g);
                W.seg[s].sinc = static_cast<R>(y.s2);
                W.seg[s].inv_nb = static_cast<R>(y.eta);
                W.seg[s].w = static_cast<R>(y.N);
                if constexpr (DS) *W.at(s) = D;
            }
            cnt += __popc(kept);
            tot += __shfl_sync(kFull, v, 31);
        } while (cnt <= kCap - 32);
        W.off[cnt + 1 + lane] = 0x7fffffff;
        if (lane == 0) W.off[cnt] = tot;
        if (lane < kMaskWords) W.mask[cnt][lane] = 0u;
        if (lane == 0) W.nb[cnt] = 0;
        __syncwarp();
        // their constants, by full warps
        for (int s = lane; s < cnt; s += 32) {
            typename std::conditional<std::is_same<R, float>::value, YieldF, Yield>::type y;
            y.nb = W.nb[s];
            y.g = W.seg[s].cosc;
            y.s2 = W.seg[s].sinc;
            y.eta = W.seg[s].inv_nb;
            y.N = W.seg[s].w;
            prep_step<R>(p, W.step[s], y, W.seg[s]);
        }
        __syncwarp();

        // ---- their bunches: 32 pieces of kPer at a time ------------------------
        const int nwin = (tot + 31) >> 5;
        int s_cur = 0, head = 0, queued = 0, win = 0;
        for (;;) {
            for (; win < nwin && queued < 32; ++win) {
                const int s = place_at(W, s_cur, win, lane, below);
                const int sc = dbg_index(p, s, kCap + 1, DBG_SMEM);
                const Seg<R> &S = W.seg[sc];
                const int j0 = (win * 32 + lane - W.off[sc]) * kSpan, left = W.nb[sc] - j0;
                if constexpr (KIND == DIRECT) {
                    // all are propagated as they come; those that cross a
                    // sphere, few of them, are queued to be propagated again and
                    // recorded by full warps
                    const bool live = left > 0;
                    BunchOut<R> o;
                    o.status = -1;
                    o.zg = R(0);
                    if (live) {
                        bunch<R, TR, FB, DS>(p, c, S, W.at(sc), j0, o);
                        if (o.status != ST_GROUND && o.status != ST_DEFER)
                            atomicAdd(&W.drop[o.status], 1u);
                    }
                    if constexpr (FB == 1)
                        defer<R>(p, c, o, live, S.w, p.track_base + (live ? W.step[sc] : 0), j0,
                                 lane, below);
                    int s0 = 0, gsel = 0;
                    const bool pass = live && sphere_hits<R>(p, c, o, s0, gsel) != 0u;
                    const unsigned in = __ballot_sync(kFull, pass);
                    if (pass)
                        W.queue[(head + queued + __popc(in & below)) & (kQueue - 1)].set(s, j0);
                    queued += __popc(in);
                    continue;
                }
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const int j = j0 + k;
                    const uint4 x = philox_bunch<R>(p, S, static_cast<uint32_t>(j));
                    bool pass = (W.mask[sc][x.y >> 30] >> ((x.y >> 25) & 31u)) & (k < left);
                    if constexpr (kDraw) {
                        if (k < left) {
                            // the survival draw, with the arrival zenith known
                            // only to the step's range: decided where both ends
                            // of the range agree, propagated otherwise
                            R u0, u2, u3, lam;
                            if constexpr (std::is_same<R, float>::value) {
                                u0 = u01f(x.x); u2 = u01f(x.z); u3 = u01f(x.w);
                            } else {
                                u0 = u01d(x.x); u2 = u01d(x.z); u3 = u01d(x.w);
                            }
                            if constexpr (DS) {
                                R kap, cc, ss;
                                disp_sample<R>(p, *W.at(sc), u2, lam, kap, cc, ss);
                            } else {
                                lam = R(1) / (c.lam_inv1 - u2 * c.lam_dinv);
                            }
                            const R fl = (static_cast<R>(j) + u0) * S.inv_nb * S.L;
                            const R tau = trans_tau<R>(p, lam, c.h_obs + (S.dz0 + fl * S.uz));
                            const float2 sec = W.sec[sc];
                            R p_lo, p_hi;
                            if constexpr (std::is_same<R, float>::value) {
                                p_lo = __expf(-(tau * sec.y));
                                p_hi = __expf(-(tau * sec.x));
                            } else {
                                p_lo = exp(-(tau * static_cast<R>(sec.y)));
                                p_hi = exp(-(tau * static_cast<R>(sec.x)));
                            }
                            // (a depth past the precision's range makes the
                            // probabilities NaN where the zenith is unbounded:
                            // propagated)
                            const bool gone = u3 >= p_hi * R(1.00002);
                            const bool stays = u3 < p_lo * R(0.99998);
                            if (gone) atomicAdd(&W.drop[ST_ABSORBED], 1u);
                            pass = !gone && (pass || !stays);
                        }
                    }
                    const unsigned in = __ballot_sync(kFull, pass);
                    if (pass)
                        W.queue[(head + queued + __popc(in & below)) & (kQueue - 1)].set(s, j);
                    queued += __popc(in);
                }
            }
            // ---- propagate the queued ones, full warps (the rest at the end) ------
            if (queued == 0) break;
            {
                __syncwarp();
                const int n = min(queued, 32);
                const bool live = lane < n;
                BunchOut<R> o;
                o.status = -1;
                o.zg = R(0);
                int s = 0, j = 0;
                if (live) {
                    const Entry e = W.queue[(head + lane) & (kQueue - 1)];
                    s = dbg_index(p, e.place(), kCap, DBG_SMEM);
                    j = e.bunch();
                }
                __syncwarp();          // read before the places are used again
                if (live) {
                    bunch<R, TR, FB, DS>(p, c, W.seg[s], W.at(s), j, o);
                    if (KIND != DIRECT && o.status != ST_GROUND && o.status != ST_DEFER)
                        atomicAdd(&W.drop[o.status], 1u);
                }
                head = (head + n) & (kQueue - 1);
                queued -= n;
                if constexpr (MODE == MODE_SCREEN) {
                    // list the bunch if it lands near a telescope centre
                    if (live && o.status == ST_GROUND) {
                        const R rc2 = std::is_same<R, float>::value ? static_cast<R>(p.f.rcut2)
                                                                    : static_cast<R>(p.rcut2);
                        for (int k = 0; k < p.n_tel; ++k) {
                            R tx, ty, tz;
                            tel_xyz<R>(p, k, tx, ty, tz);
                            const R ex = o.X - tx, ey = o.Y - ty;
                            if (ex * ex + ey * ey < rc2) {
                                const unsigned long long at = atomicAdd(p.list_count, 1ull);
                                if (at < static_cast<unsigned long long>(p.list_cap))
                                    p.list[at] = (static_cast<uint64_t>(W.step[s]) << 32) |
                                                 static_cast<uint32_t>(j);
                                break;
                            }
                        }
                    }
                    continue;
                }
                const int64_t gstep = p.track_base + W.step[s];
                const uint64_t key = (static_cast<uint64_t>(gstep) << 32) | static_cast<uint32_t>(j);
                if constexpr (FB == 1 && KIND != DIRECT)
                    defer<R>(p, c, o, live, W.seg[s].w, gstep, j, lane, below);
                int s0 = 0, gsel = 0;
                const unsigned hm = live ? sphere_hits<R>(p, c, o, s0, gsel) : 0u;
                const R np1 = DS ? R(1) + o.kap * c.eta_o : np1o;
                const R w = W.seg[s].w, lam = o.lam, t = o.t;
                record_hits<R>(p, o, hm, s0, gsel,
                               [w, key, lam, t](R &w_, uint64_t &k_, R &l_, R &t_) {
                                   w_ = w;
                                   k_ = key;
                                   l_ = lam;
                                   t_ = t;
                               },
                               np1, lane, st_hits, st_over);
            }
        }
        __syncwarp();
    }

    unsigned long long *S = p.stats;
    if (MODE == MODE_HITS && S) {
        if (blockIdx.x == 0 && tid == 0)
            atomicAdd(S + CHER_STAT_STEPS, static_cast<unsigned long long>(p.n));
        __syncwarp();
        unsigned drop = lane >= ST_UPWARD && lane <= ST_ABSORBED ? W.drop[lane] : 0u;
        if (drop) {
            const int idx = lane == ST_UPWARD  ? CHER_STAT_UPWARD
                            : lane == ST_BELOW ? CHER_STAT_BELOW_OBS
                            : lane == ST_ABOVE ? CHER_STAT_ABOVE_MAX
                            : lane == ST_ANGLE ? CHER_STAT_ANGLE
                                               : CHER_STAT_ABSORBED;
            atomicAdd(S + idx, static_cast<unsigned long long>(drop));
        }
        drop = __reduce_add_sync(kFull, drop);
        if (lane == 0) {
            if (W.drop[0]) atomicAdd(S + CHER_STAT_INVALID, static_cast<unsigned long long>(W.drop[0]));
            if (W.n_emit) {
                atomicAdd(S + CHER_STAT_EMITTING, W.n_emit);
                atomicAdd(S + CHER_STAT_BUNCHES, W.n_bunch);
                // reached the ground = generated - dropped
                atomicAdd(S + CHER_STAT_GROUND, W.n_bunch - drop);
            }
        }
        flush_stat(S, CHER_STAT_HITS, st_hits);
        flush_stat(S, CHER_STAT_OVERFLOW, st_over);
    }
}

// One instantiation for every block size: 64 registers in FP32 (1024 threads
// per SM; none spilled but 4 bytes with the transmission draw or the fallback),
// up to 148 in FP64.  With spectra (128-step blocks only) 72: seven CTAs per SM
// with 24 - 36 bytes spilled against eight with more, 144 -> 136 us at 3e5 steps.
template <class R, int MODE, bool TR, int FB, bool DS, int KIND>
__global__ void __launch_bounds__(DS ? 128 : 512, std::is_same<R, float>::value ? (DS ? 7 : 2) : 1)
    k_hits(const __grid_constant__ KParams p) {
    hits<R, MODE, TR, FB, DS, KIND>(p);
}

// Whether the bound saves more than it costs (p.choice, less than 0: no), from
// one step per warp, spread evenly over the list, its lanes sharing the
// telescopes.  In instructions of a warp per bunch, from both kernels' times over
// the arrays below: propagating one costs 10; with the bound 2 for drawing it (5
// with the transmission draw), 50 if its azimuth is in a sector (the records'
// waits for their places among them), 22 where the step has all sectors; a step
// 3, and 3 a telescope of its box.
// FP32, 2e6 vertical (1e6 at 60 deg, 3e5 at 69 deg) steps, us per launch, the
// bound / all bunches / chosen (10 - 14 more than the kernel alone):
//   64 spheres of 8 m over 300 x 300 m                   1092 /  965 /  979
//   256 of 6 m over 500 x 500 m                          1205 /  965 /  978
//   1000 of 6 m over 2 x 2 km, vertical; 60 deg     565 / 810 / 578; 985 / 370 / 383
//   4096 of 6 m over 8 x 8 km, vertical; 60 deg     298 / 735 / 310; 520 / 323 / 335
//   100 over 2 x 2 km at 69 deg, tables to 70 with the fallback    211 / 160 / 173
//   64 of 8 m over 300 x 300 m, 2e5 steps with spectra     239 /  240 /  253
// (before the choice, all words of a large array looked at: 870 and 1285 us over
// the 1000, 1150 and 1352 over the 4096; the kernel that always propagated all
// took 947, 980, 848 and 362, 752 and 334, 164, 237).
template <bool DS>
__global__ void __launch_bounds__(256) k_probe(const __grid_constant__ KParams p) {
    __shared__ float s_gain[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t w = int64_t(blockIdx.x) * 8 + warp;
    const int64_t i = w * (p.n / (int64_t(gridDim.x) * 8));
    float gain = 0.0f;
    YieldF y;
    y.nb = 0;
    SegD<float> D;
    const double z0 = __ldg(p.z0 + i), len = __ldg(p.len + i), ekin = __ldg(p.ekin + i);
    const double x0 = __ldg(p.x0 + i), y0 = __ldg(p.y0 + i);
    const float ux = load_dir<float>(p.ux, i), uy = load_dir<float>(p.uy, i);
    const float uz = load_dir<float>(p.uz, i);
    const bool valid = step_valid<float>(p, i);
    // (a step that the screen leaves open has few bunches)
    bool open;
    if constexpr (DS) open = !screen_yield_disp(p, valid, z0, len, ekin, uz, y, D);
    else open = !screen_yield(p, valid, z0, len, ekin, uz, y);
    if (!open && y.nb > 0) {
        float s_lo, s_hi;
        if constexpr (DS) {
            s_lo = cone_sine(D.beta, y.eta, p.f.kap_lo, D.x_th);
            s_hi = cone_sine(D.beta, y.eta, p.f.kap[0], D.x_th);
        } else {
            s_lo = s_hi = sqrtf(y.s2);
        }
        Ring G;
        Near N;
        Box B;
        int kind = ring_setup<MODE_HITS, DS>(p, from_middle<float>(x0, p.cull.ox, p.cull.oxf),
                                             from_middle<float>(y0, p.cull.oy, p.cull.oyf),
                                             __double2float_rn(z0) - p.f.h_obs,
                                             __double2float_rn(len), ux, uy, uz, y.eta, s_lo, s_hi,
                                             G, N, B);
        int tests = 0, near = 0, w0 = 0, w1 = p.cull.words;
        float sectors = 0.0f;
        if (kind == REACH_RING && w1 > kCullFewWords && !box_words(p, B.bins, y.nb, w0, w1))
            kind = REACH_ALL;
        if (kind == REACH_RING) {
            uint32_t mask[kMaskWords] = {};
            const float sm = G.a.w;
            for (int v = w0; v < w1; ++v) {
                const uint32_t cand = box_telescopes(p, B.bins, v);
                tests += 1 + __popc(cand);
                if (!(cand >> lane & 1u)) continue;
                const float4 T = __ldg(p.cull.tel + v * 32 + lane);
                if (!ring_near<MODE_HITS>(p, sm, G.e.z, 1.0f - sm * sm, N.p, N.w, T)) continue;
                ++near;
                const int2 sec = ring_sectors<MODE_HITS>(p, G, T);
                for (int k = sec.x; k < sec.x + sec.y; ++k) {
#pragma unroll
                    for (int q = 0; q < kMaskWords; ++q)
                        if ((k >> 5 & (kMaskWords - 1)) == q) mask[q] |= 1u << (k & 31);
                }
            }
            if (__reduce_add_sync(kFull, static_cast<unsigned>(near)) > kNear) kind = REACH_ALL;
#pragma unroll
            for (int q = 0; q < kMaskWords; ++q)
                sectors += static_cast<float>(__popc(__reduce_or_sync(kFull, mask[q])));
        }
        const float queued = kind == REACH_ALL ? 22.0f : 50.0f / kSectors * sectors;
        const float drawn = p.trans ? 5.0f : queued > 0.0f ? 2.0f : 0.0f;
        gain = static_cast<float>(y.nb) * (10.0f - drawn - queued) - 3.0f - 3.0f * tests;
    }
    if (lane == 0) s_gain[warp] = gain;
    __syncthreads();
    if (tid == 0) {
        for (int k = 1; k < 8; ++k) gain += s_gain[k];
        atomicAdd(p.choice, gain);
    }
}

template <class R, int MODE, bool DS, int KIND>
const void *pick(bool tr, bool fb) {
    if constexpr (MODE == MODE_SCREEN) {
        if constexpr (DS) {
            return nullptr;
        } else {
            return tr ? reinterpret_cast<const void *>(&k_hits<R, MODE, true, 0, false, KIND>)
                      : reinterpret_cast<const void *>(&k_hits<R, MODE, false, 0, false, KIND>);
        }
    } else {
        if (fb)
            return tr ? reinterpret_cast<const void *>(&k_hits<R, MODE, true, 1, DS, KIND>)
                      : reinterpret_cast<const void *>(&k_hits<R, MODE, false, 1, DS, KIND>);
        return tr ? reinterpret_cast<const void *>(&k_hits<R, MODE, true, 0, DS, KIND>)
                  : reinterpret_cast<const void *>(&k_hits<R, MODE, false, 0, DS, KIND>);
    }
}

template <class R>
const void *pick_mode(int mode, bool tr, bool fb, bool ds) {
    if (mode == MODE_SCREEN) return ds ? pick<R, MODE_SCREEN, true, BOUND>(tr, fb)
                                       : pick<R, MODE_SCREEN, false, BOUND>(tr, fb);
    return ds ? pick<R, MODE_HITS, true, BOUND>(tr, fb) : pick<R, MODE_HITS, false, BOUND>(tr, fb);
}

}  // namespace

namespace {
constexpr int kOptions = kTransBit | kFbBit | kDispBit | kCurvBit | kDirectBit | kProbeBit |
                         kLargeBit;
}

bool hits_kernel_serves(int mode) {
    const int m = mode & ~kOptions;
    return !(mode & kCurvBit) && (m == MODE_HITS || m == MODE_SCREEN);
}

const void *hits_kernel(bool fp32, int mode) {
    const bool tr = (mode & kTransBit) != 0, fb = (mode & kFbBit) != 0, ds = (mode & kDispBit) != 0;
    const int m = mode & ~kOptions;
    if (mode & (kDirectBit | kProbeBit | kLargeBit)) {      // (crossings of the FP32 path only)
        if (!fp32 || m != MODE_HITS) return nullptr;
        if (mode & kProbeBit)
            return ds ? reinterpret_cast<const void *>(&k_probe<true>)
                      : reinterpret_cast<const void *>(&k_probe<false>);
        if (mode & kDirectBit)
            return ds ? pick<float, MODE_HITS, true, DIRECT>(tr, fb)
                      : pick<float, MODE_HITS, false, DIRECT>(tr, fb);
        return ds ? pick<float, MODE_HITS, true, LARGE>(tr, fb)
                  : pick<float, MODE_HITS, false, LARGE>(tr, fb);
    }
    return fp32 ? pick_mode<float>(m, tr, fb, ds) : pick_mode<double>(m, tr, fb, ds);
}

namespace {
template <class R, class Entry>
size_t warp_bytes(bool tr, bool ds) {
    return ds ? (tr ? sizeof(WarpSmem<R, Entry, true, true>) : sizeof(WarpSmem<R, Entry, false, true>))
              : (tr ? sizeof(WarpSmem<R, Entry, true, false>) : sizeof(WarpSmem<R, Entry, false, false>));
}
}  // namespace

size_t hits_smem_bytes(bool fp32, int mode, int block) {
    const int m = mode & ~kOptions;
    // (the draw's bounds of the steps: not where every bunch is propagated)
    const bool tr = m == MODE_HITS && (mode & kTransBit) != 0 && !(mode & (kDirectBit | kProbeBit)), ds = (mode & kDispBit) != 0;
    const size_t w = m == MODE_HITS ? (fp32 ? warp_bytes<float, QueueHits>(tr, ds)
                                            : warp_bytes<double, QueueHits>(tr, ds))
                                    : (fp32 ? warp_bytes<float, QueueScreen>(tr, ds)
                                            : warp_bytes<double, QueueScreen>(tr, ds));
    return w * (block / 32);
}

}  // namespace cher
