// stencil64.cu -- FP64 heat7 and wave25 window kernels on sm_103a.
//
// The paper ran its fields in double precision (Section VI).  These kernels
// update the planes [z0, z1) of FP64 ring windows (plane z in slot
// (z + zbase) mod nslot; a dense field is the ring with nslot = nz, zbase =
// 0) with zero ghosts outside the grid, one step per launch:
//   heat7:  u' = u + r (sum of the 6 neighbours - 6u)
//   wave25: L = 3 c0 p + sum_m c_m (sum of the 6 neighbours m cells away),
//           p' = kappa L + (2p - p_prev)  (+ the source amplitude)
//
// GB300 has two FP64 lanes per SM and clock, 1/32 of its integer ALU rate
// (measured: 0.06 against 2 warp instructions per clock and SM), so a stencil
// in FP64 instructions (7 per heat7 point, 27 per wave25 point) takes 112 and
// 432 SM clocks per warp whatever the memory does.  The neighbour sums
// therefore run in 64-bit integer arithmetic: each value is kept as its
// 53-bit significand (left-justified in 64 bits) and its biased exponent; a
// thread shifts the values of its two points' stencils to the largest exponent
// among them, with 5 (heat7) or 6 (wave25) bits below that value's last place
// and rounded to nearest, and adds them without rounding.  The wave's weights
// are its FP64 coefficients as 53-bit integers.  One conversion and two FMAs in
// FP64 finish the point.
// Against the FP64 sequence the sum carries no rounding but the shifts' (each
// at most 2^-58 of the stencil's largest value, wave25 2^-59 in its unit) and
// one at its end.  By CPU emulation against 113 bits (24 x 20 x 20, r = 1/6) the
// error over the FP64 instructions' is 0.6 to 0.8 for wave25 from 8 to 12800
// steps, and for heat7, whose two FMAs set it, 0.8 to 0.9 up to 50 steps and 0.9
// to 1.07 at 200 to 800, on smooth, rough, positive, steep and isolated fields;
// f(-u) = -f(u) as in FP64 instructions (see the GPU tests).
//
// Stencils that the integer form does not hold as exactly as FP64 would take
// the FP64 instructions instead, per thread: infinities, NaN, a largest
// exponent outside [kELo, kEHi] (results near overflow or below 1e-270), and
// values so far apart that the sum's unit exceeds 2^-53 of every value that the
// point sums (wave25: of their shares of the sum).  A result depends only
// on the values of its thread's two stencils (and the exponents of the pairs
// beside them, which hold one value more), so windows of a slab and whole
// fields give the same bits.
//
// A warp owns a 64-point row segment, two points per thread (16-byte double2
// accesses); each value is converted once by the thread that loads it (halo
// rows by the CTA that needs them) and its neighbours read it from shared
// memory (double buffered, one barrier per plane), each load issued one plane
// ahead of its use.  heat7 keeps its z-neighbours in registers; wave25 keeps
// its nine planes' own values in shared memory, which leaves 80 registers and
// 24 warps per SM.
//
// Measured, us per step at 384^3 (G point-steps/s), FP64 instructions against
// integer sums: wave25 3200 (17.7) and 1066 (53); heat7 775 (73) and 344
// (165).  wave25 took 839 with shifts cut off and 16-bit rational weights: a
// tenth more instructions for the rounding, twice the multiplies for the
// weights.  White noise: wave25 1067, heat7 478, where some lane of most warps
// takes the FP64 instructions.  Where all do, the sums are run in vain: values
// 2^60 apart 960 -> 1220 (heat7; also a point release at r = 1/6 and a
// half-empty checkerboard) and 3800 -> 4320 (wave25).  A wave from rest, whose
// steep precursors take them in part: 0.85 ms per 256^3 step over its first 100.
// A fallback for heat7 in integers at the neighbours' own exponent would be
// faster, but rounds so seldom that its error on a point release grows to 1.35
// of the FP64 instructions' after 800 steps.  Bound now:
// wave25 by the ALU pipe and shared-memory wavefronts, heat7 by the FP64 pipe
// (61 %) and the ALU pipe with 28 warps per SM.
#include <type_traits>

#include "stencil_common.cuh"

namespace ooc {

using namespace sten;

namespace {

constexpr int kTY64 = 4;  // heat7 rows per CTA
constexpr int kSeg64 = 2 * kTX;
constexpr int kWTY64 = 8;  // wave25 rows per CTA
constexpr int kWR = 4;
constexpr double kD0 = -205.0 / 72.0, kD1 = 8.0 / 5.0, kD2 = -1.0 / 5.0, kD3 = 8.0 / 315.0, kD4 = -1.0 / 560.0;

// Biased exponents of the stencil's largest value that the integer form takes.
constexpr uint32_t kELo = 128, kEHi = 1900;

__device__ __forceinline__ double heat_pt64(double c, double xl, double xr, double up, double dn, double zm,
                                            double zp, double r)
{
    const double t = __dadd_rn(__dadd_rn(__dadd_rn(xl, xr), __dadd_rn(up, dn)), __dadd_rn(zm, zp));
    return __fma_rn(r, __fma_rn(-6.0, c, t), c);
}

__device__ __forceinline__ double2 ldg2(const double *p) { return __ldg(reinterpret_cast<const double2 *>(p)); }

// A pair of doubles as significands at the pair's exponent (the larger of the
// two biased exponents): |x| = m * 2^(e - 1085), 0 <= m < 2^63, held as m and,
// for a negative x, as ~m.  A zero takes the implicit one too: its exponent
// shifts it out.  e is 0 only where both values are zero.
//
// The ones' complement makes the shifts odd functions of x.  An arithmetic
// shift of ~m is the complement of that of m, and y + (y & 1) takes y and ~y to
// opposite even numbers, |x| rounded to the nearest (a tie away from zero).  A
// shift of -m would be cut off towards minus infinity, an error of one sign
// that adds up over the steps: on a point release at r = 1/6, heat7's error
// was 1.9 times the FP64 instructions' after 200 steps and 2.5 times after 800
// (1.0 so), and f(-u) differed from -f(u) (CPU emulation of the kernel's
// integers against 113 bits, 24 x 20 x 20).
struct Fx2 {
    long long a, b;
    uint32_t e;
};

__device__ __forceinline__ long long sar64(long long v, uint32_t s)  // shifts past 63 leave the sign
{
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}

__device__ __forceinline__ long long fx_mant(uint32_t hi, uint32_t lo, uint32_t d)
{
    unsigned long long m = (((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo) << 10;
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(d));  // shifts past 63 give 0
    return (long long)m ^ (long long)((int)hi >> 31);
}

__device__ __forceinline__ int fx_odd(long long y) { return (int)((uint32_t)y & 1u); }
// the even number that y stands for
__device__ __forceinline__ long long fx_even(long long y) { return y + fx_odd(y); }

__device__ __forceinline__ Fx2 to_fx(double2 v)
{
    const uint32_t h0 = (uint32_t)__double2hiint(v.x), h1 = (uint32_t)__double2hiint(v.y);
    const uint32_t e0 = (h0 >> 20) & 0x7FFu, e1 = (h1 >> 20) & 0x7FFu;
    uint32_t e = max(e0, e1);
    if (e == 0u)  // 1 for subnormals, so that 0 means zeros
        e = (unsigned long long)(__double_as_longlong(v.x) | __double_as_longlong(v.y)) << 1 != 0ull ? 1u : 0u;
    return Fx2{fx_mant(h0, (uint32_t)__double2loint(v.x), e - e0), fx_mant(h1, (uint32_t)__double2loint(v.y), e - e1),
               e};
}

// Above kFxBig when |v| >= 2^54 (also of several of these ORed together: when
// one of their values is).  Then a rounded shift is off by at most 2^-54 of v.
constexpr uint32_t kFxBig = (1u << 23) - 1;
__device__ __forceinline__ uint32_t fx_big(long long v) { return (uint32_t)(v >> 32) + (1u << 22); }

// v * 2^k for a nonzero double far from both ends of the range
__device__ __forceinline__ double scale_exp(double v, int k)
{
    const int hi = __double2hiint(v), lo = __double2loint(v);
    return (hi | lo) == 0 ? v : __hiloint2double(hi + (k << 20), lo);
}

template <int V>
using IC = std::integral_constant<int, V>;

// Slots of consecutive planes: the slot of plane z + d from the slot of z.
__device__ __forceinline__ int slot_at(int s, int d, int nslot)
{
    s += d;
    s %= nslot;
    return s < 0 ? s + nslot : s;
}

// The two points at (x, y, z) in FP64 instructions, values read from memory.
// Any exponent, infinities and NaN.
__device__ __noinline__ double2 heat_pair_f64(const double *in, int s, int nslot, int64_t plane, int64_t off,
                                              int64_t nx, int64_t ny, int64_t nz, int64_t x, int64_t y, int64_t z,
                                              double r)
{
    const double2 z2 = make_double2(0.0, 0.0);
    const double *p = in + (int64_t)s * plane + off;
    const double2 c = ldg2(p);
    const double2 row = make_double2(x >= 1 ? __ldg(p - 1) : 0.0, x + 2 < nx ? __ldg(p + 2) : 0.0);
    const double2 up = y >= 1 ? ldg2(p - nx) : z2, dn = y + 1 < ny ? ldg2(p + nx) : z2;
    const double2 zm = z >= 1 ? ldg2(in + (int64_t)slot_at(s, -1, nslot) * plane + off) : z2;
    const double2 zp = z + 1 < nz ? ldg2(in + (int64_t)slot_at(s, 1, nslot) * plane + off) : z2;
    return make_double2(heat_pt64(c.x, row.x, c.y, up.x, dn.x, zm.x, zp.x, r),
                        heat_pt64(c.y, c.x, row.y, up.y, dn.y, zm.y, zp.y, r));
}

__global__ void __launch_bounds__(kTX *kTY64, 7)
    heat7_f64_kernel(const double *__restrict__ in, double *__restrict__ out, int nslot, int64_t zbase, Grid3 g,
                     int64_t z0, int64_t z1, int64_t zchunk, double r)
{
    // a row: the 32 pairs, the pair left of the row in column 0 and the pair
    // right of it in column 33
    __shared__ longlong2 tm[2][kTY64 + 2][kTX + 2];
    __shared__ uint32_t te[2][kTY64 + 2][kTX + 2];
    const int lane = threadIdx.x, ty = threadIdx.y;
    const int64_t gx = (g.nx + kSeg64 - 1) / kSeg64;
    const int64_t xs = (int64_t)(blockIdx.x % gx) * kSeg64;
    const int64_t x2 = xs + 2 * lane;
    const int64_t y0 = (int64_t)(blockIdx.x / gx) * kTY64;
    const int64_t y = y0 + ty;
    const int64_t za = z0 + (int64_t)blockIdx.y * zchunk;
    const int cnt = (int)(min(za + zchunk, z1) - za);
    const int64_t nz = g.nz, plane = g.plane;
    const bool inside = x2 < g.nx && y < g.ny;
    const int64_t off = inside ? y * g.nx + x2 : 0;
    // halo pairs: the first and last warp take the rows above and below, a
    // middle warp the 2 kTY64 pairs beyond the rows' ends
    const bool edge = ty == 0 || ty == kTY64 - 1, side = ty == kTY64 / 2;
    const int hr = ty == 0 ? 0 : (ty == kTY64 - 1 ? kTY64 + 1 : 1 + (lane >> 1));
    const int hc = edge ? lane + 1 : (lane & 1) * (kTX + 1);
    const int64_t yh = y0 + hr - 1, xh = xs + 2 * (hc - 1);
    const bool halo = edge || (side && lane < 2 * kTY64);
    const bool hin = halo && yh >= 0 && yh < g.ny && xh >= 0 && xh < g.nx;
    const int64_t hoff = hin ? yh * g.nx + xh : 0;
    const double2 z2 = make_double2(0.0, 0.0);
    int s0 = (int)ring_slot(za, zbase, nslot);  // slot of plane z
    int s1 = wrap_add(s0, 1, nslot);
    const double *p0 = in + (int64_t)s0 * plane, *p1 = in + (int64_t)s1 * plane;
    double2 cur = inside ? ldg2(p0 + off) : z2;
    Fx2 fm = to_fx((inside && za >= 1) ? ldg2(in + (int64_t)slot_at(s0, -1, nslot) * plane + off) : z2);
    Fx2 fc = to_fx(cur);
    double2 nxt = (inside && za + 1 < nz) ? ldg2(p1 + off) : z2;
    double2 hv = hin ? ldg2(p0 + hoff) : z2;
    // offsets of the planes z and z + 1; planes from za to the grid's end
    int64_t o0 = (int64_t)s0 * plane, o1 = (int64_t)s1 * plane;
    const int left = (int)min(nz - za, (int64_t)1 << 30);
    const double *in_own = in + off, *in_halo = in + hoff;
    double *out_own = out + off;
#pragma unroll 2
    for (int i = 0; i < cnt; ++i) {
        const int s2 = wrap_add(s1, 1, nslot);
        const int64_t o2 = s2 == 0 ? 0 : o1 + plane;
        const int b = i & 1;
        tm[b][ty + 1][lane + 1] = make_longlong2(fc.a, fc.b);
        te[b][ty + 1][lane + 1] = fc.e;
        if (halo) {
            const Fx2 h = to_fx(hv);
            tm[b][hr][hc] = make_longlong2(h.a, h.b);
            te[b][hr][hc] = h.e;
        }
        // the next planes' loads, a plane ahead of their use
        const double2 nn = (inside && i + 2 < left) ? ldg2(in_own + o2) : z2;
        hv = (hin && i + 1 < left) ? ldg2(in_halo + o1) : z2;
        const Fx2 fp = to_fx(nxt);
        __syncthreads();
        const longlong2 up = tm[b][ty][lane + 1], dn = tm[b][ty + 2][lane + 1];
        const uint32_t eu = te[b][ty][lane + 1], ed = te[b][ty + 2][lane + 1];
        const long long xl = tm[b][ty + 1][lane].y, xr = tm[b][ty + 1][lane + 2].x;
        const uint32_t el = te[b][ty + 1][lane], er = te[b][ty + 1][lane + 2];
        const uint32_t E = max(max(max(fm.e, fc.e), max(fp.e, eu)), max(max(ed, el), er));
        double2 o;
        const bool zeros = E == 0u;
        bool exact = E >= kELo && E <= kEHi;
        {  // run by every thread (branches around it cost more than they save)
            const uint32_t et = E + 4u;
            const long long ca = sar64(fc.a, et - fc.e), cb = sar64(fc.b, et - fc.e);
            const long long za = sar64(fm.a, et - fm.e), zb = sar64(fm.b, et - fm.e);
            const long long wa = sar64(fp.a, et - fp.e), wb = sar64(fp.b, et - fp.e);
            const long long ua = sar64(up.x, et - eu), ub = sar64(up.y, et - eu);
            const long long da = sar64(dn.x, et - ed), db = sar64(dn.y, et - ed);
            const long long la = sar64(xl, et - el), rb = sar64(xr, et - er);
            // the six that are summed: the FP64 sequence rounds at their size,
            // not at c's, and a large c among tiny neighbours is what a point
            // release at r = 1/6 consists of
            const uint32_t biga = fx_big(cb) | fx_big(za) | fx_big(wa) | fx_big(ua) | fx_big(da) | fx_big(la);
            const uint32_t bigb = fx_big(ca) | fx_big(zb) | fx_big(wb) | fx_big(ub) | fx_big(db) | fx_big(rb);
            exact = zeros || (exact && biga > kFxBig && bigb > kFxBig);
            const int na = (fx_odd(za) + fx_odd(wa) + fx_odd(ua)) + (fx_odd(da) + fx_odd(la) + fx_odd(cb));
            const int nb = (fx_odd(zb) + fx_odd(wb) + fx_odd(ub)) + (fx_odd(db) + fx_odd(rb) + fx_odd(ca));
            const long long sa = (za + wa) + (ua + da) + (la + cb) + na;
            const long long sb = (zb + wb) + (ub + db) + (rb + ca) + nb;
            const int k = (int)E - 1081;
            // The sum is rounded before 6 c comes off: kept whole, sum - 6 c is
            // any multiple n of c's last bit, and with r = RN(1/6) < 1/6 an
            // n = 3 (mod 6), just short of a tie, always rounds towards c, a
            // bias that adds up (error of 8 steps 1.03e-16, of 32 3.5e-16; so 7.7e-17 and
            // 8.1e-17, in FP64 instructions 1.0e-16 and 1.05e-16).
            const double ta = zeros ? 0.0 : scale_exp(__ll2double_rn(sa), k);
            const double tb = zeros ? 0.0 : scale_exp(__ll2double_rn(sb), k);
            o.x = __fma_rn(r, __fma_rn(-6.0, cur.x, ta), cur.x);
            o.y = __fma_rn(r, __fma_rn(-6.0, cur.y, tb), cur.y);
        }
        if (!exact && inside) {
            o = heat_pair_f64(in, s0, nslot, plane, off, g.nx, g.ny, nz, x2, y, za + i, r);
        }
        if (inside)
            *reinterpret_cast<double2 *>(out_own + o0) = o;
        fm = fc;
        fc = fp;
        cur = nxt;
        nxt = nn;
        s0 = s1;
        s1 = s2;
        o0 = o1;
        o1 = o2;
    }
}

// One wave25 point in FP64 instructions: its x-neighbours xm/xp[m-1] at +-m,
// y and z likewise.
__device__ __forceinline__ double wave_lap64(double c, const double (&xm)[kWR], const double (&xp)[kWR],
                                             const double (&ym)[kWR], const double (&yp)[kWR], const double (&zm)[kWR],
                                             const double (&zp)[kWR])
{
    const double cf[kWR] = {kD1, kD2, kD3, kD4};
    double lap = __dmul_rn(3.0 * kD0, c);
#pragma unroll
    for (int m = 0; m < kWR; ++m) {
        const double s = __dadd_rn(__dadd_rn(__dadd_rn(xm[m], xp[m]), __dadd_rn(ym[m], yp[m])),
                                   __dadd_rn(zm[m], zp[m]));
        lap = __fma_rn(cf[m], s, lap);
    }
    return lap;
}

// L at the two points (x, y, z) and (x + 1, y, z) in FP64 instructions,
// values read from memory.
__device__ __noinline__ double2 wave_lap_pair_f64(const double *in, int s, int nslot, int64_t plane, int64_t off,
                                                  int64_t nx, int64_t ny, int64_t nz, int64_t x, int64_t y, int64_t z)
{
    const double *p = in + (int64_t)s * plane + off;
    double row[2 * kWR + 2], ym[2][kWR], yp[2][kWR], zm[2][kWR], zp[2][kWR];
#pragma unroll
    for (int j = 0; j < 2 * kWR + 2; ++j) {
        const int64_t xj = x - kWR + j;
        row[j] = xj >= 0 && xj < nx ? __ldg(p - kWR + j) : 0.0;
    }
#pragma unroll
    for (int m = 1; m <= kWR; ++m) {
        const double2 z2 = make_double2(0.0, 0.0);
        const double2 a = y >= m ? ldg2(p - m * nx) : z2, b = y + m < ny ? ldg2(p + m * nx) : z2;
        const double2 c = z >= m ? ldg2(in + (int64_t)slot_at(s, -m, nslot) * plane + off) : z2;
        const double2 d = z + m < nz ? ldg2(in + (int64_t)slot_at(s, m, nslot) * plane + off) : z2;
        ym[0][m - 1] = a.x, ym[1][m - 1] = a.y;
        yp[0][m - 1] = b.x, yp[1][m - 1] = b.y;
        zm[0][m - 1] = c.x, zm[1][m - 1] = c.y;
        zp[0][m - 1] = d.x, zp[1][m - 1] = d.y;
    }
    double l[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const double xm[kWR] = {row[i + 3], row[i + 2], row[i + 1], row[i]};
        const double xp[kWR] = {row[i + 5], row[i + 6], row[i + 7], row[i + 8]};
        l[i] = wave_lap64(row[i + kWR], xm, xp, ym[i], yp[i], zm[i], zp[i]);
    }
    return make_double2(l[0], l[1]);
}

// The weights are the FP64 coefficients 3 c0, c1 .. c4 themselves, as integers
// (53 bits each), so that the sum carries the operator that FP64 instructions
// carry.  (The rational coefficients, 5040 c_m in 16 bits, differ from it by
// some 1e-16 in the same way at every step: the error of 200 steps on rough
// fields was 2.8 times the FP64 instructions', of 800 steps 5.2 times; 0.75 and
// 0.77 with these weights, by CPU emulation against 113 bits.)  The values at
// distance m are held in units of 2^kU(m) last bits (0, 2, 5 and 9, about the
// inverse of their coefficient), so that where a field rises steeply (ahead of
// a wave front a value four cells away is many orders larger) the large far
// values, which weigh little, don't push the near ones out; the weights take
// the units up.
//
// A weight is kWE bits left-justified and split as hi 2^31 + lo, lo in
// [-2^30, 2^30); a sum S is even and split as hi 2^32 + 2 lo, so that all four
// partial products are of signed words.
__host__ __device__ constexpr int kU(int m) { return m == 4 ? 9 : (m == 3 ? 5 : (m == 2 ? 2 : 0)); }
constexpr int kWE = 57;  // weight of 1.0: 2^57
__host__ __device__ constexpr long long wave_weight(int m)
{
    const double c = m == 0 ? 3.0 * kD0 : (m == 1 ? kD1 : (m == 2 ? kD2 : (m == 3 ? kD3 : kD4)));
    return (long long)(c * (double)(1ll << kU(m)) * (double)(1ll << kWE));
}
__host__ __device__ constexpr int wave_wlo(int m)
{
    return (int)(((wave_weight(m) + (1ll << 30)) & 0x7FFFFFFFll) - (1ll << 30));
}
__host__ __device__ constexpr int wave_whi(int m) { return (int)((wave_weight(m) - wave_wlo(m)) / (1ll << 31)); }
// Exact, and the accumulators below hold any sums: |S| <= 2^60 for the centre
// and 6 2^60 at a distance.
constexpr bool wave_weights_fit()
{
    double pos = 0.0, neg = 0.0, lpos = 0.0, lneg = 0.0, mid = 0.0;
    for (int m = 0; m <= 4; ++m) {
        const double c = m == 0 ? 3.0 * kD0 : (m == 1 ? kD1 : (m == 2 ? kD2 : (m == 3 ? kD3 : kD4)));
        if ((double)wave_weight(m) != c * (double)(1ll << kU(m)) * (double)(1ll << kWE) ||
            (long long)wave_whi(m) * (1ll << 31) + wave_wlo(m) != wave_weight(m))
            return false;
        const double h = wave_whi(m), l = wave_wlo(m), al = l < 0.0 ? -l : l;
        (h < 0.0 ? neg : pos) += h < 0.0 ? -h : h;
        (l < 0.0 ? lneg : lpos) += al;
        mid += (m == 0 ? 1.0 : 6.0) * al;
    }
    const double two31 = 2147483648.0, top = 9.2e18;
    return (pos > neg ? pos : neg) * two31 + mid * (two31 / 8.0) + 2.0 * two31 < top && lpos * two31 < top &&
           lneg * two31 < top;
}
static_assert(wave_weights_fit(), "weights");
struct WaveAcc {
    long long h, x, l;  // products of the high words, mixed, of the low words
};

__device__ __forceinline__ long long mad_wide_s(int a, int b, long long c)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
    return c;
}

template <int M>
__device__ __forceinline__ void wave_add(WaveAcc &w, long long s)
{
    constexpr int wh = wave_whi(M), wl = wave_wlo(M);
    const int hi = (int)(s >> 32), lo = (int)((uint32_t)s >> 1);
    w.h = mad_wide_s(hi, wh, w.h);
    w.x = mad_wide_s(lo, wh, w.x);
    w.x = mad_wide_s(hi, wl, w.x);
    w.l = mad_wide_s(lo, wl, w.l);
}

// L in FP64: the sum h 2^62 + x 2^31 + l, cut below 2^59 with the last bit set
// if anything was cut off (which makes the cut an odd function and lets the
// conversion round correctly), is an integer of 2^(E - 1079), below 2^62.1:
// 2^-57 of the stencil's largest value.
__device__ __forceinline__ double wave_finish(const WaveAcc &w, int E)
{
    const long long g = w.x + (w.l >> 31);
    const long long v = (w.h << 3) + (g >> 28);
    const uint32_t rest = ((uint32_t)g & 0x0FFFFFFFu) | ((uint32_t)w.l & 0x7FFFFFFFu);
    return scale_exp(__ll2double_rn(rest != 0u ? v | 1 : v), E - 1079);
}

// Above kW1 when one of the ORed values (held as to_fx holds them) is at least
// 2^54 in magnitude; above kW6 when one of the ORed sums of six (even numbers;
// v + its sign tells s and -s alike) reaches 2^57, so that a value in it
// reaches 2^54.  A value of 2^54 in its unit weighs 0.8 x 2^53 units of the
// sum or more.  At 2^54 the rms error stays below the FP64 instructions' on all
// tested fields (heat7 at 2^53 does not).
constexpr uint32_t kW1 = (1u << 23) - 1, kW6 = (1u << 26) - 1;
__device__ __forceinline__ uint32_t w_one(long long v) { return (uint32_t)(v >> 32) + (1u << 22); }
__device__ __forceinline__ uint32_t w_six(long long v) { return (uint32_t)((v + (v >> 63)) >> 32) + (1u << 25); }

// Shared memory of a wave25 CTA: the row tile of the centre plane (double
// buffered: 4 + TY + 4 rows of 2 + 32 + 2 pairs, the 4 x-neighbours beyond
// each row end in the outer columns) and each thread's own values of the
// planes z-4 .. z+4, plane za + k in slot (k + 4) mod 9.
constexpr int kWQ = 2 * kWR + 1;
struct Wave64Smem {
    longlong2 tm[2][kWTY64 + 2 * kWR][kTX + 4];
    longlong2 qm[kWQ][kWTY64][kTX];
    uint32_t te[2][kWTY64 + 2 * kWR][kTX + 4];
    uint32_t qe[kWQ][kWTY64][kTX];
};

// Leapfrog on FP64 rings: p' = kappa L(p) + (2p - p_prev) written over
// p_prev in place (each point's p_prev is read only by its own thread).
__global__ void __launch_bounds__(kTX *kWTY64, 3)
    wave25_f64_kernel(const double *__restrict__ pin, double *pout, const double *__restrict__ kap, int nslot,
                      int64_t zbase, Grid3 g, int64_t z0, int64_t z1, int64_t zchunk, int64_t sx, int64_t sy,
                      int64_t sz, double w, WaveSrcTable tab)
{
    extern __shared__ __align__(16) unsigned char w64_smem[];
    Wave64Smem &sm = *reinterpret_cast<Wave64Smem *>(w64_smem);
    const int lane = threadIdx.x, ty = threadIdx.y;
    const int64_t gx = (g.nx + kSeg64 - 1) / kSeg64;
    const int64_t xs = (int64_t)(blockIdx.x % gx) * kSeg64;
    const int64_t x2 = xs + 2 * lane;
    const int64_t y0 = (int64_t)(blockIdx.x / gx) * kWTY64;
    const int64_t y = y0 + ty;
    const int64_t za = z0 + (int64_t)blockIdx.y * zchunk;
    const int cnt = (int)(min(za + zchunk, z1) - za);
    const int64_t nz = g.nz, plane = g.plane;
    const bool inside = x2 < g.nx && y < g.ny;
    const int64_t off = inside ? y * g.nx + x2 : 0;
    // each warp takes one halo row (four above, four below)
    const int64_t yh = ty < kWR ? y0 - kWR + ty : y0 + kWTY64 + (ty - kWR);
    const int hrow_t = ty < kWR ? ty : ty + kWTY64;
    const bool hrow = x2 < g.nx && yh >= 0 && yh < g.ny;
    const int64_t hoff = hrow ? yh * g.nx + x2 : 0;
    // the third warp also takes the two pairs beyond each end of the rows
    static_assert(kWTY64 == 2 * kWR, "one halo row per warp, one lane per pair beyond the rows' ends");
    const int xrow = lane >> 2;
    const bool side = ty == 2;
    const int xr = kWR + xrow, xc = (lane & 3) < 2 ? (lane & 3) : kTX + (lane & 3);
    const int64_t xe = xs + 2 * (xc - 2), ye = y0 + xrow;
    const bool xhalo = side && xe >= 0 && xe < g.nx && ye < g.ny;
    const int64_t xoff = xhalo ? ye * g.nx + xe : 0;
    const bool src_here = inside && y == sy && (sx == x2 || sx == x2 + 1);
    const double2 z2 = make_double2(0.0, 0.0);

    int s0 = (int)ring_slot(za, zbase, nslot);  // slot of plane z
    int s1 = slot_at(s0, 1, nslot), s5 = slot_at(s0, kWR + 1, nslot);
    auto put = [&](int slot, const Fx2 &v) {
        sm.qm[slot][ty][lane] = make_longlong2(v.a, v.b);
        sm.qe[slot][ty][lane] = v.e;
    };
#pragma unroll
    for (int j = 0; j < kWQ; ++j) {
        const int64_t zj = za - kWR + j;
        put(j, to_fx((inside && zj >= 0 && zj < nz)
                         ? ldg2(pin + (int64_t)slot_at(s0, j - kWR, nslot) * plane + off)
                         : z2));
    }
    int ph = kWR;  // slot of plane z
    double2 hv = hrow ? ldg2(pin + (int64_t)s0 * plane + hoff) : z2;
    double2 xv = xhalo ? ldg2(pin + (int64_t)s0 * plane + xoff) : z2;
    // offsets of the planes z, z + 1 and z + 5; planes from za to the grid's
    // end; the source's plane
    int64_t o0 = (int64_t)s0 * plane, o1 = (int64_t)s1 * plane, o5 = (int64_t)s5 * plane;
    const int left = (int)min(nz - za, (int64_t)1 << 30);
    const int isz = src_here && sz >= za && sz < za + cnt ? (int)(sz - za) : -1;
#pragma unroll 9
    for (int i = 0; i < cnt; ++i) {
        const int b = i & 1;
        const longlong2 cm = sm.qm[ph][ty][lane];
        const uint32_t ce = sm.qe[ph][ty][lane];
        sm.tm[b][ty + kWR][lane + 2] = cm;
        sm.te[b][ty + kWR][lane + 2] = ce;
        {
            const Fx2 h = to_fx(hv);
            sm.tm[b][hrow_t][lane + 2] = make_longlong2(h.a, h.b);
            sm.te[b][hrow_t][lane + 2] = h.e;
        }
        if (side) {
            const Fx2 h = to_fx(xv);
            sm.tm[b][xr][xc] = make_longlong2(h.a, h.b);
            sm.te[b][xr][xc] = h.e;
        }
        // the next plane's halos and the queue's next plane
        const bool more = i + 1 < cnt;
        const int64_t b0 = o0 + off;
        hv = (hrow && more) ? ldg2(pin + hoff + o1) : z2;
        xv = (xhalo && more) ? ldg2(pin + xoff + o1) : z2;
        const double2 qn = (inside && more && i + kWR + 1 < left) ? ldg2(pin + off + o5) : z2;
        // p_prev is overwritten by this kernel: plain loads, not the read-only path
        __syncthreads();
        const int e = lane + 2;  // this thread's pair in the row
        uint32_t ey[2 * kWR], exn[4];
#pragma unroll
        for (int m = 1; m <= kWR; ++m) {
            ey[m - 1] = sm.te[b][ty + kWR - m][e];
            ey[kWR + m - 1] = sm.te[b][ty + kWR + m][e];
        }
        exn[0] = sm.te[b][ty + kWR][e - 2];
        exn[1] = sm.te[b][ty + kWR][e - 1];
        exn[2] = sm.te[b][ty + kWR][e + 1];
        exn[3] = sm.te[b][ty + kWR][e + 2];
        // the largest exponent, each distance's in its unit (the outer row
        // pairs hold a value at distance 3, the inner ones one at 1)
        uint32_t ez[2 * kWR];
        const longlong2 *zq[2 * kWR];
        int E = (int)max(ce, max(exn[1], exn[2])), Z = (int)max(exn[0], exn[3]);
        Z = max(Z, E);  // the largest as it is
        E = max(E, (int)max(exn[0], exn[3]) - kU(3));
#pragma unroll
        for (int j = 0; j < kWR; ++j) {
            const int lo = ph >= j + 1 ? ph - (j + 1) : ph - (j + 1) + kWQ;
            const int hi = ph + j + 1 < kWQ ? ph + j + 1 : ph + j + 1 - kWQ;
            ez[j] = sm.qe[lo][ty][lane];
            ez[kWR + j] = sm.qe[hi][ty][lane];
            zq[j] = &sm.qm[lo][ty][lane];
            zq[kWR + j] = &sm.qm[hi][ty][lane];
            const int em = (int)max(max(ez[j], ez[kWR + j]), max(ey[j], ey[kWR + j]));
            E = max(E, em - kU(j + 1));
            Z = max(Z, em);
        }
        double2 lap = make_double2(0.0, 0.0);
        bool exact = Z == 0;  // all zeros
        {
            // run by every thread: without a branch the values' loads start
            // ahead of the exponents' test
            const bool range = E >= (int)kELo && Z <= (int)kEHi;
            const uint32_t et = (uint32_t)E + 3u;
            WaveAcc wa{0, 0, 0}, wb{0, 0, 0};
            // A row value at distance m of the first point is at m - 1 or
            // m + 1 of the second.  xa[j], xb[j]: at distance j + 1 left and
            // right of the first and of the second point, in that unit.
            const longlong2 l2 = sm.tm[b][ty + kWR][e - 2], l1 = sm.tm[b][ty + kWR][e - 1];
            const longlong2 r1 = sm.tm[b][ty + kWR][e + 1], r2 = sm.tm[b][ty + kWR][e + 2];
            auto at = [&](long long v, uint32_t ev, int m) { return sar64(v, et + (uint32_t)kU(m) - ev); };
            const long long ca = at(cm.x, ce, 0), cb = at(cm.y, ce, 0);
            auto two = [&](long long v, long long q) { return v + q + (fx_odd(v) + fx_odd(q)); };
            const long long xa[kWR] = {two(at(l1.y, exn[1], 1), cb), two(at(l1.x, exn[1], 2), at(r1.x, exn[2], 2)),
                                       two(at(l2.y, exn[0], 3), at(r1.y, exn[2], 3)),
                                       two(at(l2.x, exn[0], 4), at(r2.x, exn[3], 4))};
            const long long xb[kWR] = {two(ca, at(r1.x, exn[2], 1)), two(at(l1.y, exn[1], 2), at(r1.y, exn[2], 2)),
                                       two(at(l1.x, exn[1], 3), at(r2.x, exn[3], 3)),
                                       two(at(l2.y, exn[0], 4), at(r2.y, exn[3], 4))};
            wave_add<0>(wa, fx_even(ca));
            wave_add<0>(wb, fx_even(cb));
            // is the sums' unit small against the values of each point's own
            // stencil (one: beside it, six: sums further out)?
            const uint32_t own = w_one(ca) | w_one(cb);
            uint32_t onea = own, oneb = own, sixa = 1u << 25, sixb = 1u << 25;
            auto taps = [&](auto m_c) {
                constexpr int m = decltype(m_c)::value;
                const longlong2 um = sm.tm[b][ty + kWR - m][e], up = sm.tm[b][ty + kWR + m][e];
                const longlong2 zm = *zq[m - 1], zp = *zq[kWR + m - 1];
                const uint32_t em = ey[m - 1], ep = ey[kWR + m - 1], fm = ez[m - 1], fp = ez[kWR + m - 1];
                const long long ya = at(um.x, em, m), va = at(up.x, ep, m), za = at(zm.x, fm, m), qa = at(zp.x, fp, m);
                const long long yb = at(um.y, em, m), vb = at(up.y, ep, m), zb = at(zm.y, fm, m), qb = at(zp.y, fp, m);
                const int na = (fx_odd(ya) + fx_odd(va)) + (fx_odd(za) + fx_odd(qa));
                const int nb = (fx_odd(yb) + fx_odd(vb)) + (fx_odd(zb) + fx_odd(qb));
                const long long sa = xa[m - 1] + (ya + va) + (za + qa) + na, sb = xb[m - 1] + (yb + vb) + (zb + qb) + nb;
                if (m == 1) {
                    onea |= w_one(ya) | w_one(va) | w_one(za) | w_one(qa);
                    oneb |= w_one(yb) | w_one(vb) | w_one(zb) | w_one(qb);
                }
                sixa |= w_six(sa);
                sixb |= w_six(sb);
                wave_add<m>(wa, sa);
                wave_add<m>(wb, sb);
            };
            taps(IC<4>{});
            taps(IC<3>{});
            taps(IC<2>{});
            taps(IC<1>{});
            lap.x = exact ? 0.0 : wave_finish(wa, E);
            lap.y = exact ? 0.0 : wave_finish(wb, E);
            exact = exact || (range && (onea > kW1 || sixa > kW6) && (oneb > kW1 || sixb > kW6));
        }
        if (!exact && inside) {
            lap = wave_lap_pair_f64(pin, s0, nslot, plane, off, g.nx, g.ny, nz, x2, y, za + i);
        }
        // This plane's other operands, read where they are used (the barrier
        // keeps them here): 12 registers that, held across the sums, spill
        // (384^3 1262 us per step loaded before the sums, 1066 here; with L2
        // prefetches in their old place 1145).
        asm volatile("" ::: "memory");
        const double2 c = inside ? ldg2(pin + b0) : z2;
        const double2 kv = inside ? ldg2(kap + b0) : z2;
        const double2 ppv = inside ? *reinterpret_cast<const double2 *>(pout + b0) : z2;
        double2 o;
        o.x = __fma_rn(kv.x, lap.x, __fma_rn(2.0, c.x, -ppv.x));
        o.y = __fma_rn(kv.y, lap.y, __fma_rn(2.0, c.y, -ppv.y));
        if (i == isz) {
            double ws = w;
            if (tab.w) {  // amplitude of step n = plan time + n_off, from the device table
                const int64_t n = *tab.t + tab.n_off;
                ws = n >= 0 && n < tab.nw ? (double)tab.w[n] : 0.0;
            }
            if (sx == x2)
                o.x = __dadd_rn(o.x, ws);
            else
                o.y = __dadd_rn(o.y, ws);
        }
        if (inside)
            *reinterpret_cast<double2 *>(pout + b0) = o;
        // plane z + 5 into the slot of z - 4 (read by this thread alone)
        ++ph;
        put(ph + kWR < kWQ ? ph + kWR : ph + kWR - kWQ, to_fx(qn));
        ph = ph == kWQ ? 0 : ph;
        s0 = s1;
        s1 = s1 + 1 == nslot ? 0 : s1 + 1;
        s5 = s5 + 1 == nslot ? 0 : s5 + 1;
        o0 = o1;
        o1 = s1 == 0 ? 0 : o1 + plane;
        o5 = s5 == 0 ? 0 : o5 + plane;
    }
}

}  // namespace

cudaError_t launch_heat7_f64_ring(DConstRing in, DRing out, int64_t nx, int64_t ny, int64_t nz, int64_t z0, int64_t z1,
                                  double r, cudaStream_t st)
{
    if (z1 <= z0)
        return cudaSuccess;
    static const int res = resident((const void *)heat7_f64_kernel, kTX * kTY64);  // once, thread-safe
    const int64_t gx = (nx + kSeg64 - 1) / kSeg64, gy = (ny + kTY64 - 1) / kTY64;
    const int64_t chunk = choose_chunk(gx * gy, z1 - z0, 8, 2, res);
    const int64_t gz = (z1 - z0 + chunk - 1) / chunk;
    if (in.nslot != out.nslot || in.zbase != out.zbase || in.base == out.base || in.nslot > (1ll << 30) ||
        gx * gy > 0x7fffffffll)
        return cudaErrorInvalidValue;
    heat7_f64_kernel<<<dim3((unsigned)(gx * gy), (unsigned)gz), dim3(kTX, kTY64), 0, st>>>(
        in.base, out.base, (int)in.nslot, in.zbase, Grid3{nx, ny, nz, nx * ny}, z0, z1, chunk, r);
    return cudaGetLastError();
}

cudaError_t launch_heat7_f64(const double *in, double *out, int64_t nx, int64_t ny, int64_t nz, double r,
                             cudaStream_t st)
{
    return launch_heat7_f64_ring(DConstRing{in, nz, 0}, DRing{out, nz, 0}, nx, ny, nz, 0, nz, r, st);
}

cudaError_t launch_wave25_f64(DConstRing p, DRing pprev_out, DConstRing kappa, int64_t nx, int64_t ny, int64_t nz,
                              int64_t z0, int64_t z1, int64_t sx, int64_t sy, int64_t sz, double w, cudaStream_t st,
                              WaveSrcTable tab)
{
    if (z1 <= z0)
        return cudaSuccess;
    // set once (thread-safe); 0 if the attribute could not be set
    static const int res = []() -> int {
        if (cudaFuncSetAttribute(wave25_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(Wave64Smem)) != cudaSuccess)
            return 0;
        return resident((const void *)wave25_f64_kernel, kTX * kWTY64, sizeof(Wave64Smem));
    }();
    if (res <= 0)
        return cudaErrorInvalidValue;
    const int64_t gx = (nx + kSeg64 - 1) / kSeg64, gy = (ny + kWTY64 - 1) / kWTY64;
    const int64_t chunk = choose_chunk(gx * gy, z1 - z0, 16, 9, res);
    const int64_t gz = (z1 - z0 + chunk - 1) / chunk;
    if (p.nslot != pprev_out.nslot || p.zbase != pprev_out.zbase || p.nslot != kappa.nslot ||
        p.zbase != kappa.zbase || p.base == pprev_out.base || p.nslot > (1ll << 30) || gx * gy > 0x7fffffffll)
        return cudaErrorInvalidValue;
    wave25_f64_kernel<<<dim3((unsigned)(gx * gy), (unsigned)gz), dim3(kTX, kWTY64), sizeof(Wave64Smem), st>>>(
        p.base, pprev_out.base, kappa.base, (int)p.nslot, p.zbase, Grid3{nx, ny, nz, nx * ny}, z0, z1, chunk, sx, sy,
        sz, w, tab);
    return cudaGetLastError();
}

}  // namespace ooc
