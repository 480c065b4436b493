// codec.cu -- FR4 fixed-rate 4x4x4 block codec on sm_103a.
//
// Section IV of the paper asks for a fixed-rate lossy codec: the user fixes
// the bits kept per value, so every compressed unit has a known size and the
// device buffers are preallocated.  FR4 follows the published fixed-rate
// method (Lindstrom, IEEE TVCG 2014): block floating point on 4^3 blocks,
// a reversible integer decorrelating transform, sequency ordering,
// negabinary, and embedded bit-plane coding with group tests.  Its exact
// definition (header, lifting steps, ordering, plane coder, dequantisation)
// is stated in the oracle's codec; this file is an independent GPU
// implementation that must match it bit for bit.
//
// GPU design: one thread per 4^3 block.  The 64 values stay in registers
// (16 coalesced 128-bit loads: neighbouring threads own neighbouring blocks
// along x).  The bit-plane stage turns the 64 negabinary words into 32
// 64-bit plane masks with two in-register 32x32 bit transposes; a plane is
// then coded (code_plane) or parsed (parse_plane) as a whole, its new ones
// together, so that the lanes of a warp, whose blocks have them in different
// planes and numbers, run the same instructions.  The compressed words of a
// warp's blocks are staged in shared memory and move to and from the stream
// with coalesced 16-byte accesses; the plane masks pass through shared memory
// 16 planes at a time.
//
// The kernels are bound by the integer ALU pipe (76-80 % busy, against 22-29 %
// of DRAM), which issues half of what the schedulers do.  56 planes of 1024^2,
// R = 8, 16, 24, us: encode 196, 224, 241 -> 125, 141, 146; decode 196, 236,
// 261 -> 139, 163, 176, against a plane loop that wrote its fields by
// read-modify-write and parsed the new ones segment by segment (22 of 32
// lanes active).  The transform and the transposes alone take 92 and 80 us.
//
// Also here: dense-field kernels for any shape (partial blocks padded with
// the nearest inside value) and the variable-size fixed-precision and
// fixed-accuracy modes, which find their blocks' offsets by a decoupled
// look-back.
#include <utility>

#include "common.cuh"

namespace ooc {

// Set by a kernel whose bounded wait gave up (the variable-size encoder's
// look-back); read and cleared by take_codec_fault().
__device__ unsigned g_codec_fault = 0u;

namespace {

constexpr int kPrec = 26;  // block-floating-point precision (bits)
constexpr int kThreads = 128;
constexpr int kHalfStride = 33;   // words per thread for 16 planes' masks (odd: different banks)
constexpr int kSlack = 8;         // words past a block's 2R that a coder may touch

// ---- sequency order ---------------------------------------------------------
// r-th coefficient of the coding order: sort by level sum of (i, j, k) with
// level (0, 1, 2, 2) per axis, ties by linear index (counting order).
__host__ __device__ constexpr int order_at(int r)
{
    int c = 0;
    for (int s = 0; s <= 6; ++s)
        for (int l = 0; l < 64; ++l) {
            const int li = (l & 3) == 0 ? 0 : ((l & 3) == 1 ? 1 : 2);
            const int lj = ((l >> 2) & 3) == 0 ? 0 : (((l >> 2) & 3) == 1 ? 1 : 2);
            const int lk = (l >> 4) == 0 ? 0 : ((l >> 4) == 1 ? 1 : 2);
            if (li + lj + lk == s) {
                if (c == r)
                    return l;
                ++c;
            }
        }
    return -1;
}

// Negabinary of q is (q + kNB) ^ kNB; the XOR happens in the plane masks
// (to_planes32, from_planes32).
constexpr uint32_t kNB = 0xAAAAAAAAu;

template <int... R>
__device__ __forceinline__ void to_coding_order(uint32_t (&u)[64], const int32_t (&q)[64],
                                                std::integer_sequence<int, R...>)
{
    ((u[R] = (uint32_t)q[std::integral_constant<int, order_at(R)>::value] + kNB), ...);
}

template <int... R>
__device__ __forceinline__ void from_coding_order(int32_t (&q)[64], const uint32_t (&u)[64],
                                                  std::integer_sequence<int, R...>)
{
    ((q[std::integral_constant<int, order_at(R)>::value] = (int32_t)(u[R] - kNB)), ...);
}

// ---- wrapping int32 lifting ---------------------------------------------------
__device__ __forceinline__ int32_t wadd(int32_t a, int32_t b) { return (int32_t)((uint32_t)a + (uint32_t)b); }
__device__ __forceinline__ int32_t wsub(int32_t a, int32_t b) { return (int32_t)((uint32_t)a - (uint32_t)b); }

__device__ __forceinline__ void lift_fwd(int32_t &a0, int32_t &a1, int32_t &a2, int32_t &a3)
{
    int32_t d0 = wsub(a0, a1);
    const int32_t s0 = wadd(a1, d0 >> 1);
    int32_t d1 = wsub(a2, a3);
    const int32_t s1 = wadd(a3, d1 >> 1);
    const int32_t D = wsub(s0, s1);
    const int32_t S = wadd(s1, D >> 1);
    d0 = wsub(d0, D >> 1);
    d1 = wsub(d1, D >> 1);
    a0 = S;
    a1 = D;
    a2 = d0;
    a3 = d1;
}

__device__ __forceinline__ void lift_inv(int32_t &a0, int32_t &a1, int32_t &a2, int32_t &a3)
{
    const int32_t S = a0, D = a1;
    const int32_t d0 = wadd(a2, D >> 1);
    const int32_t d1 = wadd(a3, D >> 1);
    const int32_t s1 = wsub(S, D >> 1);
    const int32_t s0 = wadd(s1, D);
    const int32_t x3 = wsub(s1, d1 >> 1);
    const int32_t x2 = wadd(x3, d1);
    const int32_t x1 = wsub(s0, d0 >> 1);
    const int32_t x0 = wadd(x1, d0);
    a0 = x0;
    a1 = x1;
    a2 = x2;
    a3 = x3;
}

__device__ __forceinline__ void transform_fwd(int32_t (&c)[64])
{
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int b = 4 * y + 16 * z;
            lift_fwd(c[b], c[b + 1], c[b + 2], c[b + 3]);
        }
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 16 * z;
            lift_fwd(c[b], c[b + 4], c[b + 8], c[b + 12]);
        }
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 4 * y;
            lift_fwd(c[b], c[b + 16], c[b + 32], c[b + 48]);
        }
}

__device__ __forceinline__ void transform_inv(int32_t (&c)[64])
{
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 4 * y;
            lift_inv(c[b], c[b + 16], c[b + 32], c[b + 48]);
        }
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 16 * z;
            lift_inv(c[b], c[b + 4], c[b + 8], c[b + 12]);
        }
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int b = 4 * y + 16 * z;
            lift_inv(c[b], c[b + 1], c[b + 2], c[b + 3]);
        }
}

// ---- 32x32 bit transpose of a[OFF .. OFF+31] in registers --------------------
// Afterwards bit i of a[OFF + p] is the former bit p of a[OFF + i].  Each
// stage swaps one bit of the row index with that bit of the column index, so
// the stages commute.  The 16- and 8-bit stages are pure byte moves (one byte
// permute per word), the others a shift and a bit select per word.  With NIN
// (NOUT) the rows of odd index are complemented on the way in (out): the
// negabinary offset's XOR with 0xAAAAAAAA, in the plane masks, for free.
template <int OFF, int J, uint32_t M, bool NIN, bool NOUT>
__device__ __forceinline__ void transpose_stage(uint32_t (&a)[64])
{
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if (!(k & J)) {
            const uint32_t x = a[OFF + k], y = a[OFF + k + J];
            static_assert(J == 1 || (!NIN && !NOUT), "odd rows are one operand of the stage J = 1");
            const uint32_t hi = y << J;
            a[OFF + k] = NIN ? (x & M) | (~hi & ~M) : (x & M) | (hi & ~M);
            const uint32_t lo = x >> J;
            a[OFF + k + J] = NIN ? (lo & M) | (~y & ~M) : (NOUT ? ~((lo & M) | (y & ~M)) : (lo & M) | (y & ~M));
        }
    }
}

template <int OFF>
__device__ __forceinline__ void transpose_stage16(uint32_t (&a)[64])
{
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t lo = a[OFF + k], hi = a[OFF + k + 16];
        a[OFF + k] = __byte_perm(lo, hi, 0x5410);
        a[OFF + k + 16] = __byte_perm(lo, hi, 0x7632);
    }
}

template <int OFF>
__device__ __forceinline__ void transpose_stage8(uint32_t (&a)[64])
{
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if (!(k & 8)) {
            const uint32_t lo = a[OFF + k], hi = a[OFF + k + 8];
            a[OFF + k] = __byte_perm(lo, hi, 0x6240);
            a[OFF + k + 8] = __byte_perm(lo, hi, 0x7351);
        }
    }
}

// Coefficients (plus kNB) to plane masks, and back.
template <int OFF>
__device__ __forceinline__ void to_planes32(uint32_t (&a)[64])
{
    transpose_stage16<OFF>(a);
    transpose_stage8<OFF>(a);
    transpose_stage<OFF, 4, 0x0F0F0F0Fu, false, false>(a);
    transpose_stage<OFF, 2, 0x33333333u, false, false>(a);
    transpose_stage<OFF, 1, 0x55555555u, false, true>(a);
}

template <int OFF>
__device__ __forceinline__ void from_planes32(uint32_t (&a)[64])
{
    transpose_stage<OFF, 1, 0x55555555u, true, false>(a);
    transpose_stage<OFF, 2, 0x33333333u, false, false>(a);
    transpose_stage<OFF, 4, 0x0F0F0F0Fu, false, false>(a);
    transpose_stage8<OFF>(a);
    transpose_stage16<OFF>(a);
}

// ---- bit writer / reader over a thread's shared-memory words ------------------
__device__ __forceinline__ uint32_t low_mask(int l)  // l in [0, 32]
{
    return (uint32_t)((1ull << l) - 1ull);
}

// A block's stream words in shared memory, followed by kZeroWords zero words:
// bits past the budget read as 0, which is what a truncated stream means;
// only the implied-one rule needs the budget.
constexpr int kZeroWords = 4;

__device__ __forceinline__ uint64_t shl64(uint64_t v, int n)  // n >= 0; 0 for n >= 64
{
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}

// The 32 bits from bit position pos on (0 past the block's nwords words).
__device__ __forceinline__ uint32_t bits_at(const uint32_t *w, int nwords, int pos)
{
    const int i = min(pos >> 5, nwords);
    return __funnelshift_r(w[i], w[i + 1], pos);
}

// Bit fields appended to a thread's words in shared memory: the word that
// holds bit `off` keeps its bits below off, and the words behind it are
// written, not read, so the buffer needs no zeros beforehand.  A field's bits
// past its length are zero, so that what is written past the new end is too.
__device__ __forceinline__ void put64(uint32_t *w, int off, uint32_t lo, uint32_t hi)
{
    uint32_t *p = w + (off >> 5);
    const uint32_t k = p[0];
    p[0] = k | __funnelshift_l(0u, lo, off);
    p[1] = __funnelshift_l(lo, hi, off);
    p[2] = __funnelshift_l(hi, 0u, off);
}

__device__ __forceinline__ void put32(uint32_t *w, int off, uint32_t v)
{
    uint32_t *p = w + (off >> 5);
    const uint32_t k = p[0];
    p[0] = k | __funnelshift_l(0u, v, off);
    p[1] = __funnelshift_l(v, 0u, off);
}

// A plane's new ones are written as its bits with every one followed by the
// group bit 1 of the next segment: inserts a one behind each one of `at`
// (a subset of v's, lowest first; the result fits 32 bits).
__device__ __forceinline__ uint32_t insert_ones(uint32_t v, uint32_t at)
{
    do {  // with `at` 0 a pass changes nothing
        const uint32_t a1 = at - 1u, upto = at ^ a1;
        v = (v & upto) | ((v << 1) & ~upto);
        at = (at & a1) << 1;
    } while (at != 0u);
    return v;
}

// ---- one block ----------------------------------------------------------------
// Lowest coded bit plane: 0 at a fixed rate; 32 - P at fixed precision P;
// at fixed accuracy with L = floor(log2 tol), L - (emax - 26) - 4 clamped to
// [0, 32] (the dropped planes then cost at most tol/2 after the inverse
// transform's gain of 2.25 per axis).
__device__ __forceinline__ int plane_floor(int mode, int mparam, int emax)
{
    if (mode == OOC_FR4_PRECISION)
        return 32 - mparam;
    if (mode == OOC_FR4_ACCURACY) {
        const int p = mparam - (emax - kPrec) - 4;
        return p < 0 ? 0 : (p > 32 ? 32 : p);
    }
    return 0;
}

// The bit-plane coder shared by FR4 and FR4D.
//
// Plane p is written as: the refinement bits of the n significant
// coefficients; then, for each new one at offset t past n, a group bit 1, the
// zeros before it and the one itself; then a closing group bit 0 if
// coefficients remain.  When a new one is the last coefficient its one is
// implied and not written.
//
// With rest = the plane's bits past n and tl its highest one, the part after
// the refinement bits is the group bit 1, the bits of rest below tl with
// every one doubled (the one itself and the next segment's group bit 1), and
// the one at tl.  n after the plane is the larger of n and the plane's bit
// length.
struct CodePos {
    int n, off;
};

// New ones that take more than 32 bits: 16 bits of rest at a time.
__device__ __noinline__ CodePos code_long(uint32_t *dst, uint64_t rest, int n, int off)
{
    const int tl = 63 - __clzll((long long)rest), n_new = n + tl + 1;
    put32(dst, off, 1u);
    ++off;
    uint64_t before = rest ^ (1ull << tl);
    for (int i = 0; i < tl; i += 16) {
        const int c = tl - i < 16 ? tl - i : 16;
        const uint32_t v = (uint32_t)before & 0xFFFFu;
        put32(dst, off, insert_ones(v, v));
        off += c + __popc(v);
        before >>= 16;
    }
    if (n_new < 64) {
        put32(dst, off, 1u);
        off += 2;
    }
    return CodePos{n_new, off};
}

// One plane (bits xl of coefficients 0..31, xh of 32..63) from bit `off` on.
__device__ __forceinline__ CodePos code_plane(uint32_t *dst, uint32_t xl, uint32_t xh, int n, int off)
{
    const uint64_t keep = shl64(~0ull, n);
    put64(dst, off, xl & ~(uint32_t)keep, xh & ~(uint32_t)(keep >> 32));
    off += n;
    const int len = xh != 0u ? 64 - __clz((int)xh) : 32 - __clz((int)xl);
    if (n >= 64)
        return CodePos{n, off};
    if (len <= n) {  // the closing group bit; the word of `off` is written already
        return CodePos{n, off + 1};
    }
    const uint32_t s = (uint32_t)((((uint64_t)xh << 32) | xl) >> n);
    const int tl = len - n - 1, bits = tl + __popc(s);  // bits: up to and with the last one
    if (tl > 31 || bits > 30)
        return code_long(dst, (((uint64_t)xh << 32) | xl) >> n, n, off);
    const uint32_t last = 1u << tl;
    uint32_t v = insert_ones(s, s ^ last);
    const bool open = len < 64;
    if (!open)  // the last coefficient's one is implied
        v ^= 1u << (bits - 1);
    put32(dst, off, 1u | (v << 1));
    return CodePos{len, off + bits + (open ? 2 : 0)};
}

__device__ __forceinline__ uint32_t shl32(uint32_t v, int n)  // n >= 0; 0 for n >= 32
{
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}
__device__ __forceinline__ uint32_t shr32(uint32_t v, int n)
{
    uint32_t r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}

// Planes p .. stop, whose masks are at pb[-2 p] and pb[1 - 2 p].  FIRST (the first
// 16 planes of a block): the leading ones take few bits, and as long as a
// plane of every lane's block fits 32 (and the coefficients 32..63 have no one
// yet), it is written as one field.  On smooth fields these are 10 to 12 of
// 28 planes: R = 16 148 -> 141 us, 139 -> 138 on rough ones; in the later
// parts too it gains nothing there and costs 2 %.  All 32 lanes of the warp
// come here and take the same turns of the first loop, so the vote is one of
// the whole warp; a lane without planes (p < stop) or budget left votes for
// going on.  (56 planes of 1024^2, us, against votes of whatever lanes were
// together: R = 16 148 and 151, R = 24 153 and 157, rough 138 and 139; FP64, 24
// of 64 bits, encoded and decoded 848 and 809.)
template <bool FIRST>
__device__ __forceinline__ CodePos code_planes(uint32_t *dst, const uint32_t *pb, int &p, int stop, int budget, CodePos c)
{
#pragma unroll 1
    for (int turns = FIRST ? __reduce_max_sync(0xffffffffu, p - stop + 1) : 0; turns > 0; --turns) {
        const bool more = p >= stop && c.off < budget;
        const uint32_t *pm = pb - 2 * max(p, stop);
        const uint32_t x = pm[0];
        const uint32_t s = shr32(x, c.n);  // new ones; 0: tl = -1, bits = -1
        const int tl = 31 - __clz((int)s), bits = tl + __popc((int)s);
        const bool fits = pm[1] == 0u && c.n + bits + 2 <= 32;
        if (__any_sync(0xffffffffu, more && !fits))
            break;
        if (more) {
            const uint32_t v = insert_ones(s, s ^ (1u << (tl & 31)));
            const uint32_t field = (v << 1) | (s != 0u ? 1u : 0u);
            put32(dst, c.off, (x & ~shl32(~0u, c.n)) | shl32(field, c.n));
            c.off += c.n + bits + 2;
            c.n += tl + 1;
            --p;
        }
    }
#pragma unroll 1
    for (; p >= stop && c.off < budget; --p)
        c = code_plane(dst, pb[-2 * p], pb[1 - 2 * p], c.n, c.off);
    return c;
}

// The words behind the coded bits up to the block's `words`.
__device__ __forceinline__ void clear_tail(uint32_t *dst, int off, int words)
{
    for (int i = (off >> 5) + 1; i < words; ++i)
        dst[i] = 0u;
}

// Encode one block into dst[0 .. words) (a bit budget of 32 words; words =
// 2R at a fixed rate) with the plane range of `mode`.  Called by whole
// warps.  Returns the coded length in bits (exact for the variable-size modes,
// whose budget never binds).  The planes go through shared memory 16 at a time,
// in the part of dst that the coded words have not reached yet: half the shared
// memory of all 32 planes, and none beside the words, for 24 warps per SM at
// any rate up to 32 and in the variable-size modes (with 33 words of their own per thread it was 16 warps
// at R = 24, 157 us against 144, and 16 in the variable-size encoder, 512^3 at
// tolerance 1e-4 530 against 475).
//
// Before plane 31 - j at most 73 + 65 j bits are coded (var_block_words), and
// coding it touches words up to (138 + 65 j) / 32 + 1.  Its own two words are
// read before; the next plane's are at kPlanes1 + 2 (j + 1) while j < 16, at
// kPlanes0 + 2 (j - 15) after that, which is further for every j.  A budget of
// `words` ends the coding within 129 bits of it, so that planes behind words +
// 5 are out of reach whatever j is (R = 8: 55 words per thread instead of 71,
// which leaves the loads more of the L1 cache: 130 -> 126 us).  The kernel
// that reads single values takes kPlanes0 at any budget (!TIGHT): it has no
// register left for the variable (128 x 253 x 515 at R = 16: 43 against 45).
constexpr int kPlanes1 = 5, kPlanes0 = 38;  // planes 31 .. 16 and 15 .. 0
template <bool TIGHT>
__host__ __device__ constexpr int planes0_at(int words)
{
    return TIGHT && words + 6 < kPlanes0 ? words + 6 : kPlanes0;
}
constexpr bool planes_clear()
{
    for (int j = 0; j < 32; ++j)
        if ((138 + 65 * j) / 32 + 1 >= (j < 16 ? kPlanes1 + 2 * (j + 1) : kPlanes0 + 2 * (j - 15)))
            return false;
    return (73 + 65 * 16) / 32 < kPlanes0;  // the second half's planes behind the first half's words
}
static_assert(planes_clear(), "coded words stay below the planes that are yet to be coded");
template <bool TIGHT>
__device__ __forceinline__ int encode_block(uint32_t (&v)[64], int words, int mode, int mparam, uint32_t *dst)
{
    // the largest magnitude, three values per instruction (any NaN gives one
    // with the same exponent)
    float top = 0.0f;
#pragma unroll
    for (int i = 0; i < 64; i += 2)
        asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(top) : "f"(__uint_as_float(v[i])), "f"(__uint_as_float(v[i + 1])));
    const uint32_t mx = __float_as_uint(top);
    const int budget = 32 * words;
    auto zeros = [&] {
        dst[0] = 0u;
        if (mode == OOC_FR4_RATE)
            clear_tail(dst, 0, words);
        return 1;
    };
    if (!__any_sync(0xffffffffu, mx != 0u))
        return zeros();
    const int emax = (int)(mx >> 23) - 126;  // largest frexp exponent, >= -126
    const int pmin = plane_floor(mode, mparam, emax);

    // q = trunc(x * 2^(26 - emax)), with the power of two split in two
    // normal factors; the first product is exact whenever the result can be
    // nonzero, the second is exact or already below 1.
    const int kk = kPrec - emax;
    const int k1 = kk >> 1, k2 = kk - k1;
    const float s1 = __int_as_float((k1 + 127) << 23);
    const float s2 = __int_as_float((k2 + 127) << 23);
    int32_t q[64];
#pragma unroll
    for (int i = 0; i < 64; ++i)
        q[i] = __float2int_rz(__fmul_rn(__fmul_rn(__uint_as_float(v[i]), s1), s2));

    transform_fwd(q);
    to_coding_order(v, q, std::make_integer_sequence<int, 64>{});
    to_planes32<0>(v);   // v[p]      = bits p of coefficients 0..31
    to_planes32<32>(v);  // v[32 + p] = bits p of coefficients 32..63
    // the leading planes without a one (up to 8 of them), a group bit 0 each
    int skip = 8;
#pragma unroll
    for (int i = 7; i >= 0; --i)
        skip = (v[31 - i] | v[63 - i]) != 0u ? i : skip;
    skip = min(skip, 32 - pmin);
    dst[0] = 1u | ((uint32_t)((emax + 127) & 0xFF) << 1);
    dst[1] = 0u;
    CodePos c{0, 9 + skip};
    int p = mx != 0u ? 31 - skip : -1;  // a block of zeros has no planes
    auto code_half = [&](auto base_c) {  // planes base + 15 .. base
        constexpr int base = decltype(base_c)::value;
        const int stop = max(pmin, base);
        const uint32_t *pb = dst + (base != 0 ? kPlanes1 : planes0_at<TIGHT>(words)) + 2 * (15 + base);
        c = code_planes<base != 0>(dst, pb, p, stop, budget, c);
    };
    auto keep_half = [&](uint32_t *pm, auto at_c) {  // the plane that is coded first comes first
        constexpr int at = decltype(at_c)::value;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            pm[2 * (15 - i)] = v[at + i];
            pm[2 * (15 - i) + 1] = v[32 + at + i];
        }
    };
    keep_half(dst + kPlanes1, std::integral_constant<int, 16>{});
    code_half(std::integral_constant<int, 16>{});
    keep_half(dst + planes0_at<TIGHT>(words), std::integral_constant<int, 0>{});
    code_half(std::integral_constant<int, 0>{});
    if (mx == 0u)
        return zeros();
    if (mode == OOC_FR4_RATE)
        clear_tail(dst, c.off, words);
    return c.off;
}

struct Plane {
    uint32_t xl, xh;  // bits of coefficients 0..31 and 32..63
    int n, pos;       // significant coefficients and stream position behind it
};

// A plane's new ones, segment by segment, from the group bit at `pos` on: a
// group bit 1, zeros, a one; a 0 group bit ends the plane.  Any stream.
__device__ __noinline__ Plane parse_segments(const uint32_t *w, int nwords, int n, int pos)
{
    uint64_t X = 0ull;
    for (;;) {
        const uint32_t wv = bits_at(w, nwords, pos);
        if ((wv & 1u) == 0u) {  // group test: nothing more in this plane
            ++pos;
            break;
        }
        const int len = 63 - n;  // explicit scan bits at most (after the group bit)
        uint32_t sc = wv >> 1;   // 31 of them
        int t = __ffs((int)sc) - 1;
        if (sc == 0u && len > 31) {  // a longer scan
            const int mm = len - 31 < 32 ? len - 31 : 32;
            sc = bits_at(w, nwords, pos + 32) & low_mask(mm);
            t = 30 + __ffs((int)sc);
        }
        if (sc != 0u && t < len) {
            X |= 1ull << (n + t);
            n += t + 1;
            pos += t + 2;
            continue;
        }
        // the scan bits are zero: the last coefficient's one is implied
        if (pos + 1 + len <= 32 * nwords) {
            X |= 1ull << 63;
            n = 64;
        }
        pos += 1 + len;
        break;
    }
    return Plane{(uint32_t)X, (uint32_t)(X >> 32), n, pos};
}

// One bit plane of a block: `n` refinement bits of the significant
// coefficients, then the new ones (see code_planes for the form).
//
// The new ones of a plane are found together.  Past the first group bit the
// stream holds the plane's bits with every one followed by the group bit of
// the next segment, so in a run of ones they alternate: value, group, value
// ..; the plane ends after the first run of odd length, whose last one has
// the group bit 0 behind it.  Runs that start on an even bit are told from
// the others by one addition that ripples through them (`ec`), which gives
// every group one at once (`gr`); removing those below the end leaves the
// plane's bits.  A plane has few new ones (20 in the 32 planes of a block of
// the benchmark's field), but some lane of a warp has some in nearly every
// plane, so all lanes go through it.  A plane whose end does not lie in the
// 32-bit window, or that reaches the last coefficient (once per block), is
// parsed by parse_segments.
__device__ __forceinline__ Plane parse_plane(const uint32_t *w, int nwords, int n, int pos)
{
    const uint32_t *p = w + (pos >> 5);
    const uint32_t a0 = p[0], a1 = p[1], a2 = p[2];
    const int at = pos + n;
    const uint32_t *ps = w + (at >> 5);
    const uint32_t s = __funnelshift_r(ps[0], ps[1], at);  // from the group bit on
    const bool rest = n < 64, has = (s & 1u) != 0u && rest;
    const uint32_t sc = has ? s >> 1 : 0u;
    const uint32_t ec = sc + (sc & ~(sc << 1) & 0x55555555u);  // starts of runs: a one after a zero
    const uint32_t gr = sc & (ec ^ 0xAAAAAAAAu);
    const uint32_t odd = sc & ~(sc >> 1) & ~gr;  // value ones with a group bit 0 behind (bit 30: perhaps)
    const uint32_t upto = odd ^ (odd - 1u);      // bits up to the first of them
    uint32_t v = sc & upto, g = gr & upto;
    const int k = __popc(upto);
    const int nv = k - __popc(g);  // coefficients scanned
    const uint64_t keep = shl64(~0ull, n);  // of the refinement bits: those below
    Plane r;
    r.xl = __funnelshift_r(a0, a1, pos) & ~(uint32_t)keep;
    r.xh = __funnelshift_r(a1, a2, pos) & ~(uint32_t)(keep >> 32);
    r.n = has ? n + nv : n;
    r.pos = at + (has ? k + 2 : (rest ? 1 : 0));  // with both group bits
    if (has && (k > 30 || n + nv > 63)) {
        const Plane t = parse_segments(w, nwords, n, at);
        r.xl |= t.xl;
        r.xh |= t.xh;
        r.n = t.n;
        r.pos = t.pos;
        return r;
    }
    // take the group ones out, lowest first; the first removal without a test
    // (with no group one left it changes nothing)
    do {
        const uint32_t g1 = g - 1u, below = g1 & ~g;
        v = (v & below) | ((v >> 1) & ~below);
        g = (g & g1) >> 1;
    } while (g != 0u);
    const uint64_t y = shl64(v, n);
    r.xl |= (uint32_t)y;
    r.xh |= (uint32_t)(y >> 32);
    return r;
}

// Decode one block of `nwords` words (2R at a fixed rate), held in shared
// memory with kZeroWords zeros behind, with the plane range of `mode`.  The
// planes are parsed 16 at a time into the thread's 32 words at pm and taken
// from there into registers, half transposed: half the shared memory of all
// 32 planes, for 24 warps per SM up to R = 16 (16 with all planes) and 20 above.
__device__ __forceinline__ void decode_block(const uint32_t *w, int nwords, int mode, int mparam, float (&out)[64],
                                             uint32_t *pm)
{
    const int budget = 32 * nwords;
    const uint32_t w0 = w[0];
    if ((w0 & 1u) == 0u) {
#pragma unroll
        for (int i = 0; i < 64; ++i)
            out[i] = 0.0f;
        return;
    }
    const int emax = (int)((w0 >> 1) & 0xFFu) - 127;
    const int pmin = plane_floor(mode, mparam, emax);
    // the leading planes without a one, a group bit 0 each (up to 16 of them)
    const uint32_t lead = __funnelshift_r(w0, w[1], 9) | 0x10000u;
    const int skip = min(__ffs((int)lead) - 1, budget - 9);
    int pos = 9 + skip, n = 0, p = 31 - skip;
    auto parse_half = [&](int base) {  // planes base + 15 .. base
        const int stop = max(pmin, base);
        uint32_t *pb = pm - base;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            pm[i] = 0u;
#pragma unroll 1
        for (; p >= stop && pos < budget; --p) {
            const Plane r = parse_plane(w, nwords, n, pos);
            pb[p] = r.xl;
            pb[16 + p] = r.xh;
            n = r.n;
            pos = r.pos;
        }
    };
    uint32_t u[64];
    parse_half(16);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        u[16 + i] = pm[i];
        u[48 + i] = pm[16 + i];
    }
    parse_half(0);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        u[i] = pm[i];
        u[32 + i] = pm[16 + i];
    }
    const int k = emax - kPrec;
    from_planes32<0>(u);
    from_planes32<32>(u);
    int32_t q[64];
    from_coding_order(q, u, std::make_integer_sequence<int, 64>{});
    transform_inv(q);
    // x = RN(RN(q) * 2^(emax - 26)): one exact or correctly rounded scaling.
    const bool split = k < -126;
    const float sa = __int_as_float(((split ? k + 64 : k) + 127) << 23);
#pragma unroll
    for (int i = 0; i < 64; ++i)
        out[i] = __fmul_rn(__int2float_rn(q[i]), sa);
    if (split) {
        const float sb = __int_as_float((-64 + 127) << 23);
#pragma unroll
        for (int i = 0; i < 64; ++i)
            out[i] = __fmul_rn(out[i], sb);
    }
}

// Words per block in the decoder's shared memory: odd, so that the threads'
// blocks start in different banks.
__host__ __device__ constexpr int decode_stride(int words) { return (words + kZeroWords) | 1; }

// A warp's `nv` consecutive blocks of `words` words from the stream at `src`
// into its part of shared memory.
__device__ __forceinline__ void stage_blocks(const uint32_t *__restrict__ src, int nv, int words, int stride,
                                             uint32_t *dst)
{
    const int lane = threadIdx.x & 31;
    if ((words & 3) == 0 && ((uintptr_t)src & 15) == 0) {
        // chunk c of 4 words is words 4 (c mod q) .. of block c / q
        const int q = words >> 2;
        int blk = lane / q, ch = lane - blk * q;
        const int step_blk = 32 / q, step_ch = 32 - step_blk * q;
        for (int c = lane; c < nv * q; c += 32) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src) + c);
            uint32_t *d = dst + blk * stride + 4 * ch;
            d[0] = v.x;
            d[1] = v.y;
            d[2] = v.z;
            d[3] = v.w;
            blk += step_blk;
            ch += step_ch;
            if (ch >= q) {
                ch -= q;
                ++blk;
            }
        }
    } else {
        int blk = lane / words, wd = lane - blk * words;
        const int step_blk = 32 / words, step_wd = 32 - step_blk * words;
        for (int o = lane; o < nv * words; o += 32) {
            dst[blk * stride + wd] = __ldg(src + o);
            blk += step_blk;
            wd += step_wd;
            if (wd >= words) {
                wd -= words;
                ++blk;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kZeroWords; ++i)
        dst[lane * stride + words + i] = 0u;
    __syncwarp();
}

// ---- kernels ------------------------------------------------------------------
// Words per block in the encoder's shared memory: odd, so that the threads'
// blocks start in different banks.
__host__ __device__ constexpr int encode_stride64(int words) { return (words + kSlack) | 1; }
template <bool TIGHT>
__host__ __device__ constexpr int encode_stride(int words)  // with room for the planes in them
{
    const int p = planes0_at<TIGHT>(words) + 32;
    return words + kSlack > p ? (words + kSlack) | 1 : p | 1;
}

// A warp's `nv` consecutive blocks of `words` words from its part of shared
// memory to the stream at `dst`.
__device__ __forceinline__ void store_blocks(uint32_t *dst, int nv, int words, int stride, const uint32_t *src)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if ((words & 3) == 0 && ((uintptr_t)dst & 15) == 0) {
        // chunk c of 4 words is words 4 (c mod q) .. of block c / q
        const int q = words >> 2;
        int blk = lane / q, ch = lane - blk * q;
        const int step_blk = 32 / q, step_ch = 32 - step_blk * q;
        for (int c = lane; c < nv * q; c += 32) {
            const uint32_t *w = src + blk * stride + 4 * ch;
            reinterpret_cast<uint4 *>(dst)[c] = make_uint4(w[0], w[1], w[2], w[3]);
            blk += step_blk;
            ch += step_ch;
            if (ch >= q) {
                ch -= q;
                ++blk;
            }
        }
        return;
    }
    int blk = lane / words, wd = lane - blk * words;
    const int step_blk = 32 / words, step_wd = 32 - step_blk * words;
    for (int o = lane; o < nv * words; o += 32) {
        dst[o] = src[blk * stride + wd];
        blk += step_blk;
        wd += step_wd;
        if (wd >= words) {
            wd -= words;
            ++blk;
        }
    }
}

__global__ void __launch_bounds__(kThreads, 6) fr4_encode_kernel(ConstRing in, int64_t nx, int64_t ny, int64_t z0,
                                                                 int64_t nblk, int rate, uint32_t *__restrict__ out)
{
    extern __shared__ uint32_t smem[];  // each thread's block
    const int words = 2 * rate, stride = encode_stride<true>(words);
    const int64_t b = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t first = b - (threadIdx.x & 31);
    if (first >= nblk)
        return;
    const int64_t own = min(b, nblk - 1);  // lanes past the end code the last block too
    uint32_t *mine = smem + threadIdx.x * stride;
    uint32_t v[64];
    const int64_t nbx = nx >> 2, nby = ny >> 2;
    const int64_t bx = own % nbx, t2 = own / nbx, by = t2 % nby, bz = t2 / nby;
    const int64_t slot = ring_slot(z0 + 4 * bz, in.zbase, in.nslot);
    const float *p = in.base + (slot * ny + 4 * by) * nx + 4 * bx;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 f = __ldg(reinterpret_cast<const float4 *>(p + ((int64_t)k * ny + j) * nx));
            v[16 * k + 4 * j + 0] = __float_as_uint(f.x);
            v[16 * k + 4 * j + 1] = __float_as_uint(f.y);
            v[16 * k + 4 * j + 2] = __float_as_uint(f.z);
            v[16 * k + 4 * j + 3] = __float_as_uint(f.w);
        }
    encode_block<true>(v, words, OOC_FR4_RATE, 0, mine);
    store_blocks(out + first * words, (int)min(nblk - first, (int64_t)32), words, stride,
                 mine - (threadIdx.x & 31) * stride);
}

// MINB CTAs per SM: 6 (80 registers) up to R = 16; above, where the staged
// blocks leave room for 5, 5 (96 registers).
template <int MINB>
__global__ void __launch_bounds__(kThreads, MINB) fr4_decode_kernel(const uint32_t *__restrict__ in, int64_t nx, int64_t ny,
                                                             int64_t z0, int64_t nblk, int rate, Ring out)
{
    extern __shared__ uint32_t smem[];  // each thread's block
    const int words = 2 * rate, stride = decode_stride(words);
    const int64_t b = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t first = b - (threadIdx.x & 31);
    if (first >= nblk)
        return;
    uint32_t *mine = smem + threadIdx.x * stride;
    stage_blocks(in + first * words, (int)min(nblk - first, (int64_t)32), words, stride,
                 mine - (threadIdx.x & 31) * stride);
    if (b >= nblk)
        return;
    float f[64];
    decode_block(mine, words, OOC_FR4_RATE, 0, f, smem + kThreads * stride + threadIdx.x * kHalfStride);
    const int64_t nbx = nx >> 2, nby = ny >> 2;
    const int64_t bx = b % nbx, t2 = b / nbx, by = t2 % nby, bz = t2 / nby;
    const int64_t slot = ring_slot(z0 + 4 * bz, out.zbase, out.nslot);
    float *p = out.base + (slot * ny + 4 * by) * nx + 4 * bx;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4 *>(p + ((int64_t)k * ny + j) * nx) =
                make_float4(f[16 * k + 4 * j], f[16 * k + 4 * j + 1], f[16 * k + 4 * j + 2], f[16 * k + 4 * j + 3]);
}

// ---- FR4D: the same codec for FP64 fields -------------------------------------
// 58-bit block floating point (emax clamped at -1022, 11 header bits), the
// FR4 lifting in wrapping int64, the same coding order, 64-bit negabinary
// and 64 bit planes through the shared plane coder and parser.  One thread
// owns one block; a CTA of 64 threads keeps each thread's staged words and 16
// planes at a time in shared memory.  The high words' 32 planes are transposed
// and coded first; the low words' only when the budget reaches them (it ends
// about there at 24 of 64 bits on smooth fields).  56 planes of 1024^2, R = 24
// and 32, us, against all 128 plane words per thread in shared memory (8 warps
// per SM): encode 474, 505 -> 333, 348 (12 warps, 168 registers); decode 647,
// 678 -> 455, 479 (16 warps at 128 registers with spills; 12 warps without are
// 4 % slower), with the scaling as an addition to the exponent instead of a
// second FP64 instruction per value.
constexpr int kPrec64 = 58;
constexpr int kThreads64 = 64;
constexpr uint64_t kNB64 = 0xAAAAAAAAAAAAAAAAull;

__device__ __forceinline__ int64_t wadd64(int64_t a, int64_t b) { return (int64_t)((uint64_t)a + (uint64_t)b); }
__device__ __forceinline__ int64_t wsub64(int64_t a, int64_t b) { return (int64_t)((uint64_t)a - (uint64_t)b); }

__device__ __forceinline__ void lift_fwd64(int64_t &a0, int64_t &a1, int64_t &a2, int64_t &a3)
{
    int64_t d0 = wsub64(a0, a1);
    const int64_t s0 = wadd64(a1, d0 >> 1);
    int64_t d1 = wsub64(a2, a3);
    const int64_t s1 = wadd64(a3, d1 >> 1);
    const int64_t D = wsub64(s0, s1);
    const int64_t S = wadd64(s1, D >> 1);
    d0 = wsub64(d0, D >> 1);
    d1 = wsub64(d1, D >> 1);
    a0 = S;
    a1 = D;
    a2 = d0;
    a3 = d1;
}

__device__ __forceinline__ void lift_inv64(int64_t &a0, int64_t &a1, int64_t &a2, int64_t &a3)
{
    const int64_t S = a0, D = a1;
    const int64_t d0 = wadd64(a2, D >> 1);
    const int64_t d1 = wadd64(a3, D >> 1);
    const int64_t s1 = wsub64(S, D >> 1);
    const int64_t s0 = wadd64(s1, D);
    const int64_t x3 = wsub64(s1, d1 >> 1);
    const int64_t x2 = wadd64(x3, d1);
    const int64_t x1 = wsub64(s0, d0 >> 1);
    const int64_t x0 = wadd64(x1, d0);
    a0 = x0;
    a1 = x1;
    a2 = x2;
    a3 = x3;
}

__device__ __forceinline__ void transform_fwd64(int64_t (&c)[64])
{
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int b = 4 * y + 16 * z;
            lift_fwd64(c[b], c[b + 1], c[b + 2], c[b + 3]);
        }
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 16 * z;
            lift_fwd64(c[b], c[b + 4], c[b + 8], c[b + 12]);
        }
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 4 * y;
            lift_fwd64(c[b], c[b + 16], c[b + 32], c[b + 48]);
        }
}

__device__ __forceinline__ void transform_inv64(int64_t (&c)[64])
{
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 4 * y;
            lift_inv64(c[b], c[b + 16], c[b + 32], c[b + 48]);
        }
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int b = x + 16 * z;
            lift_inv64(c[b], c[b + 4], c[b + 8], c[b + 12]);
        }
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int b = 4 * y + 16 * z;
            lift_inv64(c[b], c[b + 1], c[b + 2], c[b + 3]);
        }
}

// coefficient order_at(r) as 64-bit negabinary, split into its low and high
// words
template <int... R>
__device__ __forceinline__ void to_coding_order64(uint32_t (&lo)[64], uint32_t (&hi)[64], const int64_t (&q)[64],
                                                  std::integer_sequence<int, R...>)
{
    ((lo[R] = (uint32_t)((uint64_t)q[std::integral_constant<int, order_at(R)>::value] + kNB64),
      hi[R] = (uint32_t)(((uint64_t)q[std::integral_constant<int, order_at(R)>::value] + kNB64) >> 32)),
     ...);
}

template <int... R>
__device__ __forceinline__ void from_coding_order64(int64_t (&q)[64], const uint32_t (&lo)[64],
                                                    const uint32_t (&hi)[64], std::integer_sequence<int, R...>)
{
    ((q[std::integral_constant<int, order_at(R)>::value] =
          (int64_t)((((uint64_t)hi[R] << 32) | lo[R]) - kNB64)),
     ...);
}

__device__ __forceinline__ uint64_t umax64(uint64_t a, uint64_t b) { return a > b ? a : b; }

__device__ __forceinline__ double pow2d(int k)  // k in [-1022, 1023]
{
    return __longlong_as_double((long long)(k + 1023) << 52);
}

// Encode one FP64 block (bit patterns v) into dst[0 .. words) at a fixed
// rate: words = 2R, a budget of 64R bits.  Called by whole warps.
__device__ __forceinline__ void encode_block64(const uint64_t (&v)[64], int words, uint32_t *dst, uint32_t *pm)
{
    uint64_t mx = 0;
#pragma unroll
    for (int i = 0; i < 64; ++i)
        mx = umax64(mx, v[i] & 0x7FFFFFFFFFFFFFFFull);
    if (!__any_sync(0xffffffffu, mx != 0ull)) {
        dst[0] = 0u;
        clear_tail(dst, 0, words);
        return;
    }
    // largest frexp exponent (biased exponent - 1022; subnormals clamp to -1022)
    const int emax = (int)(mx >> 52) - 1022;
    // q = trunc(x * 2^(58 - emax)) in integer arithmetic on the bits (the
    // FP64 pipe is scarce on this GPU): x = m 2^e with the 53-bit significand
    // m, so |q| = m shifted by e + 58 - emax (left by at most 5, since |x| <
    // 2^emax; right past 63 is 0), then the sign
    const int kk = kPrec64 - emax;
    int64_t q[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) {
        const uint64_t b = v[i];
        const int eb = (int)((b >> 52) & 0x7FFu);
        const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (eb != 0 ? (1ull << 52) : 0ull);
        const int sh = (eb != 0 ? eb - 1075 : -1074) + kk;
        const uint64_t a = sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull);
        q[i] = (b >> 63) ? -(int64_t)a : (int64_t)a;
    }
    transform_fwd64(q);
    uint32_t lo[64], hi[64];
    to_coding_order64(lo, hi, q, std::make_integer_sequence<int, 64>{});
    // the leading planes without a one, a group bit 0 each (up to 32 of them)
    uint32_t any = 0u;
#pragma unroll
    for (int i = 0; i < 64; ++i)
        any |= hi[i] ^ kNB;
    const int skip = min(__clz((int)any), 32 * words - 12);
    dst[0] = 1u | ((uint32_t)(emax + 1023) << 1);
    dst[1] = 0u;
    CodePos c{0, 12 + skip};
    int p = mx != 0ull ? 63 - skip : -1;  // a block of zeros has no planes
    // planes base + 15 .. base, whose masks are in a[at ..] and a[at + 32 ..]
    auto code_part = [&](auto base_c, const uint32_t (&a)[64], auto at_c) {
        constexpr int base = decltype(base_c)::value;
        constexpr int at = decltype(at_c)::value;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            pm[2 * (15 - i)] = a[at + i];
            pm[2 * (15 - i) + 1] = a[32 + at + i];
        }
        const uint32_t *pb = pm + 2 * (15 + base);
        c = code_planes<base == 48>(dst, pb, p, base, 32 * words, c);
    };
    to_planes32<0>(hi);
    to_planes32<32>(hi);
    code_part(std::integral_constant<int, 48>{}, hi, std::integral_constant<int, 16>{});
    code_part(std::integral_constant<int, 32>{}, hi, std::integral_constant<int, 0>{});
    if (c.off < 32 * words) {
        to_planes32<0>(lo);
        to_planes32<32>(lo);
        code_part(std::integral_constant<int, 16>{}, lo, std::integral_constant<int, 16>{});
        code_part(std::integral_constant<int, 0>{}, lo, std::integral_constant<int, 0>{});
    }
    if (mx == 0ull) {
        dst[0] = 0u;
        c.off = 0;
    }
    clear_tail(dst, c.off, words);
}

__device__ __forceinline__ void decode_block64(const uint32_t *w, int nwords, double (&out)[64], uint32_t *pm)
{
    const uint32_t w0 = w[0];
    if ((w0 & 1u) == 0u) {
#pragma unroll
        for (int i = 0; i < 64; ++i)
            out[i] = 0.0;
        return;
    }
    const int emax = (int)((w0 >> 1) & 0x7FFu) - 1023;
    const int budget = 32 * nwords;
    // the leading planes without a one, a group bit 0 each (up to 20 of them)
    const uint32_t lead = __funnelshift_r(w0, w[1], 12) | 0x100000u;
    const int skip = min(__ffs((int)lead) - 1, budget - 12);
    int pos = 12 + skip, n = 0, p = 63 - skip;
    // planes base + 15 .. base into a[at ..] and a[at + 32 ..]
    auto parse_part = [&](int base, uint32_t (&a)[64], auto at_c) {
        constexpr int at = decltype(at_c)::value;
        uint32_t *pb = pm - base;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            pm[i] = 0u;
#pragma unroll 1
        for (; p >= base && pos < budget; --p) {
            const Plane r = parse_plane(w, nwords, n, pos);
            pb[p] = r.xl;
            pb[16 + p] = r.xh;
            n = r.n;
            pos = r.pos;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            a[at + i] = pm[i];
            a[32 + at + i] = pm[16 + i];
        }
    };
    uint32_t lo[64], hi[64];
    parse_part(48, hi, std::integral_constant<int, 16>{});
    parse_part(32, hi, std::integral_constant<int, 0>{});
    from_planes32<0>(hi);
    from_planes32<32>(hi);
    if (pos < budget) {
        parse_part(16, lo, std::integral_constant<int, 16>{});
        parse_part(0, lo, std::integral_constant<int, 0>{});
        from_planes32<0>(lo);
        from_planes32<32>(lo);
    } else {  // the budget ended in the high planes
#pragma unroll
        for (int i = 0; i < 64; ++i)
            lo[i] = kNB;
    }
    int64_t q[64];
    from_coding_order64(q, lo, hi, std::make_integer_sequence<int, 64>{});
    transform_inv64(q);
    // x = RN(RN(q) * 2^(emax - 58)): one exact or correctly rounded scaling.
    // Away from both ends of the range it is an addition to the exponent; the
    // conversion stays on the FP64 pipe (16 clocks per warp each).
    const int k = emax - kPrec64;
    if (k >= -1022 && k <= 960) {
#pragma unroll
        for (int i = 0; i < 64; ++i) {
            const double f = __ll2double_rn((long long)q[i]);
            const int h = __double2hiint(f);
            out[i] = __hiloint2double(h != 0 ? h + (k << 20) : 0, __double2loint(f));
        }
        return;
    }
    const bool split = k < -1022;
    const double sa = pow2d(split ? k + 64 : k), sb = pow2d(-64);
#pragma unroll
    for (int i = 0; i < 64; ++i) {
        double f = __dmul_rn(__ll2double_rn((long long)q[i]), sa);
        if (split)
            f = __dmul_rn(f, sb);
        out[i] = f;
    }
}

__global__ void __launch_bounds__(kThreads64, 6) fr4d_encode_kernel(DConstRing in, int64_t nx, int64_t ny, int64_t z0,
                                                                 int64_t nblk, int rate, uint32_t *__restrict__ out)
{
    extern __shared__ uint32_t smem[];  // each thread's block, then each thread's planes
    const int words = 2 * rate, stride = encode_stride64(words);
    const int64_t b = (int64_t)blockIdx.x * kThreads64 + threadIdx.x;
    const int64_t first = b - (threadIdx.x & 31);
    if (first >= nblk)
        return;
    uint32_t *mine = smem + threadIdx.x * stride;
    uint64_t v[64] = {};
    if (b < nblk) {
        const int64_t nbx = nx >> 2, nby = ny >> 2;
        const int64_t bx = b % nbx, t2 = b / nbx, by = t2 % nby, bz = t2 / nby;
        const int64_t slot = ring_slot(z0 + 4 * bz, in.zbase, in.nslot);
        const double *p = in.base + (slot * ny + 4 * by) * nx + 4 * bx;
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double2 *row = reinterpret_cast<const double2 *>(p + ((int64_t)k * ny + j) * nx);
                const double2 a = __ldg(row), c = __ldg(row + 1);
                v[16 * k + 4 * j + 0] = (uint64_t)__double_as_longlong(a.x);
                v[16 * k + 4 * j + 1] = (uint64_t)__double_as_longlong(a.y);
                v[16 * k + 4 * j + 2] = (uint64_t)__double_as_longlong(c.x);
                v[16 * k + 4 * j + 3] = (uint64_t)__double_as_longlong(c.y);
            }
    }
    encode_block64(v, words, mine, smem + kThreads64 * stride + threadIdx.x * kHalfStride);
    store_blocks(out + first * words, (int)min(nblk - first, (int64_t)32), words, stride,
                 mine - (threadIdx.x & 31) * stride);
}

__global__ void __launch_bounds__(kThreads64, 7) fr4d_decode_kernel(const uint32_t *__restrict__ in, int64_t nx,
                                                                 int64_t ny, int64_t z0, int64_t nblk, int rate,
                                                                 DRing out)
{
    extern __shared__ uint32_t smem[];  // each thread's block and plane words
    const int words = 2 * rate, stride = decode_stride(words);
    const int64_t b = (int64_t)blockIdx.x * kThreads64 + threadIdx.x;
    const int64_t first = b - (threadIdx.x & 31);
    if (first >= nblk)
        return;
    uint32_t *mine = smem + threadIdx.x * stride;
    stage_blocks(in + first * words, (int)min(nblk - first, (int64_t)32), words, stride,
                 mine - (threadIdx.x & 31) * stride);
    if (b >= nblk)
        return;
    double f[64];
    decode_block64(mine, words, f, smem + kThreads64 * stride + threadIdx.x * kHalfStride);
    const int64_t nbx = nx >> 2, nby = ny >> 2;
    const int64_t bx = b % nbx, t2 = b / nbx, by = t2 % nby, bz = t2 / nby;
    const int64_t slot = ring_slot(z0 + 4 * bz, out.zbase, out.nslot);
    double *p = out.base + (slot * ny + 4 * by) * nx + 4 * bx;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            double2 *row = reinterpret_cast<double2 *>(p + ((int64_t)k * ny + j) * nx);
            row[0] = make_double2(f[16 * k + 4 * j], f[16 * k + 4 * j + 1]);
            row[1] = make_double2(f[16 * k + 4 * j + 2], f[16 * k + 4 * j + 3]);
        }
}

size_t smem_bytes64(int rate, bool encoder)
{
    if (!encoder)
        return (size_t)kThreads64 * (decode_stride(2 * rate) + kHalfStride) * sizeof(uint32_t);
    return (size_t)kThreads64 * (encode_stride64(2 * rate) + kHalfStride) * sizeof(uint32_t);
}

cudaError_t ensure_smem_attr64()
{
    // set once per process (thread-safe); the attribute is per function
    static const cudaError_t once = [] {
        cudaError_t e = cudaFuncSetAttribute(fr4d_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem_bytes64(64, true));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fr4d_decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem_bytes64(64, false));
        return e;
    }();
    return once;
}

// ---- dense fields of any shape, fixed rate and variable-size modes -------------
constexpr int kVarWords = 130;  // most words of a variable-size block that a decoder takes

// Most words of a block coded without a budget down to plane pmin: 9 header
// bits; per plane, the refinement and scanned bits are at most one per
// coefficient and the closing group bit one more; every coefficient costs one
// group bit 1.  68 words for all 32 planes.
__host__ __device__ constexpr int var_block_words(int pmin) { return (9 + (32 - pmin) * 65 + 64 + 31) / 32; }

// Block (bx, by, bz) of a dense field; a block reaching past the field takes
// the value of the nearest point inside it (each coordinate clamped).  VEC:
// nx is a multiple of 4 and the field 16-byte aligned, so a row of the block
// is one 16-byte access.
template <bool VEC>
__device__ __forceinline__ void gather_clamped(const float *in, int64_t nx, int64_t ny, int64_t nz, int64_t bx,
                                               int64_t by, int64_t bz, uint32_t (&v)[64])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t z = min(4 * bz + k, nz - 1);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float *row = in + (z * ny + min(4 * by + j, ny - 1)) * nx;
            if (VEC) {
                const float4 f = __ldg(reinterpret_cast<const float4 *>(row + 4 * bx));
                v[16 * k + 4 * j + 0] = __float_as_uint(f.x);
                v[16 * k + 4 * j + 1] = __float_as_uint(f.y);
                v[16 * k + 4 * j + 2] = __float_as_uint(f.z);
                v[16 * k + 4 * j + 3] = __float_as_uint(f.w);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    v[16 * k + 4 * j + i] = __float_as_uint(__ldg(row + min(4 * bx + i, nx - 1)));
            }
        }
    }
}

// The points of block (bx, by, bz) that lie inside the field; VEC as above.
template <bool VEC>
__device__ __forceinline__ void scatter_inside(float *out, int64_t nx, int64_t ny, int64_t nz, int64_t bx, int64_t by,
                                               int64_t bz, const float (&f)[64])
{
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t z = 4 * bz + k, y = 4 * by + j;
            if (z < nz && y < ny) {
                float *row = out + (z * ny + y) * nx + 4 * bx;
                if (VEC) {
                    *reinterpret_cast<float4 *>(row) = make_float4(f[16 * k + 4 * j], f[16 * k + 4 * j + 1],
                                                                   f[16 * k + 4 * j + 2], f[16 * k + 4 * j + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (4 * bx + i < nx)
                            row[i] = f[16 * k + 4 * j + i];
                }
            }
        }
}

inline bool vec_rows(const void *field, int64_t nx) { return nx % 4 == 0 && (uintptr_t)field % 16 == 0; }

// Fixed rate for any shape: `words` words per block, the CTA's output
// staged and written with coalesced stores.
template <bool VEC>
__global__ void __launch_bounds__(kThreads, 6)
    fr4_encode_dense_kernel(const float *__restrict__ in, int64_t nx, int64_t ny, int64_t nz, int64_t nblk, int words,
                            uint32_t *__restrict__ out)
{
    extern __shared__ uint32_t smem[];
    const int stride = encode_stride<VEC>(words);
    const int64_t b = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t first = b - (threadIdx.x & 31);
    if (first >= nblk)
        return;
    const int64_t own = min(b, nblk - 1);  // lanes past the end code the last block too
    uint32_t *mine = smem + threadIdx.x * stride;
    uint32_t v[64];
    const int64_t nbx = (nx + 3) >> 2, nby = (ny + 3) >> 2;
    const int64_t bx = own % nbx, t2 = own / nbx, by = t2 % nby, bz = t2 / nby;
    gather_clamped<VEC>(in, nx, ny, nz, bx, by, bz, v);
    encode_block<VEC>(v, words, OOC_FR4_RATE, 0, mine);
    store_blocks(out + first * words, (int)min(nblk - first, (int64_t)32), words, stride,
                 mine - (threadIdx.x & 31) * stride);
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads, 6)
    fr4_decode_dense_kernel(const uint32_t *__restrict__ in, int64_t nx, int64_t ny, int64_t nz, int64_t nblk,
                            int words, float *__restrict__ out)
{
    extern __shared__ uint32_t smem[];  // each thread's block, then each thread's planes
    const int stride = decode_stride(words);
    const int64_t b = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t first = b - (threadIdx.x & 31);
    if (first >= nblk)
        return;
    uint32_t *mine = smem + threadIdx.x * stride;
    stage_blocks(in + first * words, (int)min(nblk - first, (int64_t)32), words, stride,
                 mine - (threadIdx.x & 31) * stride);
    if (b >= nblk)
        return;
    float f[64];
    decode_block(mine, words, OOC_FR4_RATE, 0, f, smem + kThreads * stride + threadIdx.x * kHalfStride);
    const int64_t nbx = (nx + 3) >> 2, nby = (ny + 3) >> 2;
    const int64_t bx = b % nbx, t2 = b / nbx, by = t2 % nby, bz = t2 / nby;
    scatter_inside<VEC>(out, nx, ny, nz, bx, by, bz, f);
}

// Variable-size: block b is words [index[b], index[b + 1]), clamped to the
// stream and to kVarWords.  A warp stages its blocks one behind the other in
// kVarBuf words (38 per block: 6 CTAs per SM; slots of the largest block's
// size leave 2), those that fit first and the rest in further rounds.
constexpr int kVarBuf = 32 * 38;
static_assert(kVarBuf >= kVarWords + kZeroWords, "any block fits alone");

template <bool VEC>
__global__ void __launch_bounds__(kThreads, 6)
    fr4_decode_var_kernel(const uint32_t *__restrict__ in, int64_t in_words, const uint64_t *__restrict__ index,
                          int64_t nx, int64_t ny, int64_t nz, int64_t nblk, int mode, int mparam,
                          float *__restrict__ out)
{
    extern __shared__ uint32_t smem[];  // the warps' blocks, then each thread's planes
    const int lane = threadIdx.x & 31;
    uint32_t *buf = smem + (threadIdx.x >> 5) * kVarBuf;
    uint32_t *pm = smem + (kThreads / 32) * kVarBuf + threadIdx.x * kHalfStride;
    const int64_t b = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    bool todo = b < nblk;
    const uint32_t *src = in;
    int nw = 0;
    if (todo) {
        uint64_t lo = __ldg(index + b), hi = __ldg(index + b + 1);
        lo = lo < (uint64_t)in_words ? lo : (uint64_t)in_words;
        hi = hi < (uint64_t)in_words ? hi : (uint64_t)in_words;
        const uint64_t n = hi > lo ? hi - lo : 0;
        nw = (int)(n < (uint64_t)kVarWords ? n : (uint64_t)kVarWords);
        src = in + lo;
    }
    const int64_t nbx = (nx + 3) >> 2, nby = (ny + 3) >> 2;
    const int64_t bx = b % nbx, t2 = b / nbx, by = t2 % nby, bz = t2 / nby;
    while (__any_sync(0xffffffffu, todo)) {
        const int need = todo ? nw + kZeroWords : 0;
        int end = need;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, end, d);
            if (lane >= d)
                end += t;
        }
        const bool now = todo && end <= kVarBuf;
        if (now) {
            uint32_t *w = buf + (end - need);
            for (int i = 0; i < nw; ++i)
                w[i] = __ldg(src + i);
#pragma unroll
            for (int i = 0; i < kZeroWords; ++i)
                w[nw + i] = 0u;
            float f[64];
            decode_block(w, nw, mode, mparam, f, pm);
            scatter_inside<VEC>(out, nx, ny, nz, bx, by, bz, f);
        }
        todo = todo && !now;
        __syncwarp();  // the next round's blocks take this one's places
    }
}

// ---- variable-size modes: one pass with a decoupled look-back ---------------------
// Tile t is the kThreads blocks of the t-th CTA to start: an atomic counter
// numbers the CTAs as they begin, so every tile a CTA waits on is already
// running and never waits on a later one.  status[t] holds the tile's state
// in bits 62-63 and a word count in bits 0-61: kTileAgg its own words,
// kTilePrefix the words of tiles 0 .. t, kTileFailed a look-back that gave up.
// Each published value carries everything its reader needs, so relaxed 64-bit
// accesses suffice.  The states are in rising order and are published by
// atomicMax: a tile that gave up also marks the last tile failed, whose word
// the host reads, and that mark stays whatever the last tile publishes later
// (a later tile may have counted the failed one's words before it gave up).
constexpr uint64_t kTileAgg = 1ull << 62, kTilePrefix = 2ull << 62, kTileFailed = 3ull << 62;
constexpr uint64_t kTileValue = (1ull << 62) - 1;
constexpr int kLookbackSpins = 1 << 24;  // about a second of 64 ns sleeps per tile waited on

__device__ __forceinline__ uint64_t ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Block b's words at out + index[b]; index[nblk] = total words.  A block is
// written only if it ends within out_words.  scratch: the tile counter, then
// one status word per tile, all zero at launch.  `cap`: words of shared
// memory for a block (var_block_words of the lowest plane).
template <bool VEC>
__global__ void __launch_bounds__(kThreads, 6)
    fr4_encode_var_kernel(const float *__restrict__ in, int64_t nx, int64_t ny, int64_t nz, int64_t nblk, int mode,
                          int mparam, int cap, uint32_t *__restrict__ out, uint64_t out_words,
                          uint64_t *__restrict__ index, unsigned long long *scratch)
{
    extern __shared__ uint32_t smem[];
    __shared__ uint64_t warp_tot[kThreads / 32];
    __shared__ int64_t s_tile;
    __shared__ uint64_t s_prefix;
    __shared__ int s_fail;
    unsigned long long *status = scratch + 1;
    if (threadIdx.x == 0) {
        s_tile = (int64_t)atomicAdd(scratch, 1ull);
        s_fail = 0;
    }
    __syncthreads();
    const int64_t tile = s_tile;
    const int stride = encode_stride<true>(cap);
    const int64_t b = tile * kThreads + threadIdx.x;
    const int64_t own = min(b, nblk - 1);  // lanes past the end code the last block too
    uint32_t *mine = smem + threadIdx.x * stride;
    uint32_t v[64];
    const int64_t nbx = (nx + 3) >> 2, nby = (ny + 3) >> 2;
    const int64_t bx = own % nbx, t2 = own / nbx, by = t2 % nby, bz = t2 / nby;
    gather_clamped<VEC>(in, nx, ny, nz, bx, by, bz, v);
    const int bits = encode_block<true>(v, cap, mode, mparam, mine);
    const uint64_t nw = b < nblk ? (uint64_t)((bits + 31) >> 5) : 0;
    // exclusive scan of the word counts over the CTA
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t incl = nw;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d)
            incl += t;
    }
    if (lane == 31)
        warp_tot[warp] = incl;
    __syncthreads();
    uint64_t before = incl - nw, total = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        if (w < warp)
            before += warp_tot[w];
        total += warp_tot[w];
    }
    if (warp == 0) {
        // the look-back, 32 tiles at a time: lane l reads tile - 1 - l
        uint64_t prefix = 0;
        bool failed = false;
        if (lane == 0)
            atomicMax(&status[tile], (tile == 0 ? kTilePrefix : kTileAgg) | total);
        for (int64_t j = tile - 1 - lane; tile > 0; j -= 32) {
            uint64_t v = kTilePrefix;  // before tile 0: nothing
            if (j >= 0) {
                v = ld_relaxed_u64(&status[j]);
                for (int spins = 0; (v >> 62) == 0 && spins < kLookbackSpins; ++spins) {
                    __nanosleep(64);
                    v = ld_relaxed_u64(&status[j]);
                }
            }
            const uint64_t state = v & ~kTileValue;
            const uint32_t done = __ballot_sync(0xffffffffu, state == kTilePrefix);
            const uint32_t bad = __ballot_sync(0xffffffffu, state == 0 || state == kTileFailed);
            const int last = done ? __ffs((int)done) - 1 : 31;  // tiles up to the nearest prefix count
            const uint32_t counted = last == 31 ? 0xffffffffu : (2u << last) - 1u;
            if (bad & counted) {
                failed = true;
                break;
            }
            uint64_t sum = lane <= last ? v & kTileValue : 0;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1)
                sum += __shfl_xor_sync(0xffffffffu, sum, d);
            prefix += sum;
            if (done)
                break;
        }
        if (lane == 0) {
            if (failed) {
                atomicMax(&status[tile], kTileFailed);  // later tiles stop at once
                atomicMax(&status[gridDim.x - 1], kTileFailed);
                atomicOr(&g_codec_fault, 1u);
                s_fail = 1;
            } else if (tile > 0) {
                atomicMax(&status[tile], kTilePrefix | (prefix + total));
            }
            s_prefix = prefix;
        }
    }
    __syncthreads();
    if (s_fail || b >= nblk)
        return;
    const uint64_t off = s_prefix + before;
    index[b] = off;
    if (b == nblk - 1)
        index[nblk] = off + nw;
    if (off + nw <= out_words)
        for (uint64_t i = 0; i < nw; ++i)
            out[off + i] = mine[i];
}

size_t dense_smem_bytes(int words, bool encoder, bool vec)
{
    if (!encoder)
        return (size_t)kThreads * (decode_stride(words) + kHalfStride) * sizeof(uint32_t);
    return (size_t)kThreads * (vec ? encode_stride<true>(words) : encode_stride<false>(words)) * sizeof(uint32_t);
}

// Shared memory of the variable-size kernels.
size_t var_encode_smem(int cap) { return dense_smem_bytes(cap, true, true); }
constexpr size_t kVarDecodeSmem = (size_t)((kThreads / 32) * kVarBuf + kThreads * kHalfStride) * sizeof(uint32_t);

cudaError_t ensure_dense_smem_attr()
{
    // set once per process (thread-safe); the attribute is per function
    static const cudaError_t once = [] {
        struct {
            const void *fn;
            size_t bytes;
        } const a[] = {{(const void *)fr4_encode_dense_kernel<false>, dense_smem_bytes(128, true, false)},
                       {(const void *)fr4_encode_dense_kernel<true>, dense_smem_bytes(128, true, false)},
                       {(const void *)fr4_decode_dense_kernel<false>, dense_smem_bytes(128, false, false)},
                       {(const void *)fr4_decode_dense_kernel<true>, dense_smem_bytes(128, false, false)},
                       {(const void *)fr4_encode_var_kernel<false>, var_encode_smem(var_block_words(0))},
                       {(const void *)fr4_encode_var_kernel<true>, var_encode_smem(var_block_words(0))},
                       {(const void *)fr4_decode_var_kernel<false>, kVarDecodeSmem},
                       {(const void *)fr4_decode_var_kernel<true>, kVarDecodeSmem}};
        for (const auto &x : a) {
            const cudaError_t e = cudaFuncSetAttribute(x.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x.bytes);
            if (e != cudaSuccess)
                return e;
        }
        return cudaSuccess;
    }();
    return once;
}

// Shared memory per CTA: the encoder's blocks with the planes in them, or the
// decoder's blocks and then each thread's planes.
size_t smem_bytes(int rate, bool encoder)
{
    if (!encoder)
        return (size_t)kThreads * (decode_stride(2 * rate) + kHalfStride) * sizeof(uint32_t);
    return (size_t)kThreads * encode_stride<true>(2 * rate) * sizeof(uint32_t);
}

cudaError_t ensure_smem_attr()
{
    // set once per process (thread-safe); the attribute is per function
    static const cudaError_t once = [] {
        cudaError_t e = cudaFuncSetAttribute(fr4_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem_bytes(64, true));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fr4_decode_kernel<6>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem_bytes(64, false));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fr4_decode_kernel<5>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem_bytes(64, false));
        return e;
    }();
    return once;
}

}  // namespace

cudaError_t launch_fr4_encode(ConstRing in, int64_t nx, int64_t ny, int64_t z0, int64_t z1, int rate,
                              uint32_t *out, cudaStream_t st)
{
    const int64_t nblk = (nx / 4) * (ny / 4) * ((z1 - z0) / 4);
    if (nblk <= 0)
        return cudaSuccess;
    cudaError_t e = ensure_smem_attr();
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads - 1) / kThreads;
    fr4_encode_kernel<<<(unsigned)grid, kThreads, smem_bytes(rate, true), st>>>(in, nx, ny, z0, nblk, rate, out);
    return cudaGetLastError();
}

cudaError_t launch_fr4_decode(const uint32_t *in, int64_t nx, int64_t ny, int64_t z0, int64_t z1, int rate,
                              Ring out, cudaStream_t st)
{
    const int64_t nblk = (nx / 4) * (ny / 4) * ((z1 - z0) / 4);
    if (nblk <= 0)
        return cudaSuccess;
    cudaError_t e = ensure_smem_attr();
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads - 1) / kThreads;
    if (rate > 16)
        fr4_decode_kernel<5><<<(unsigned)grid, kThreads, smem_bytes(rate, false), st>>>(in, nx, ny, z0, nblk, rate, out);
    else
        fr4_decode_kernel<6><<<(unsigned)grid, kThreads, smem_bytes(rate, false), st>>>(in, nx, ny, z0, nblk, rate, out);
    return cudaGetLastError();
}

cudaError_t launch_fr4d_encode(DConstRing in, int64_t nx, int64_t ny, int64_t z0, int64_t z1, int rate,
                               uint32_t *out, cudaStream_t st)
{
    const int64_t nblk = (nx / 4) * (ny / 4) * ((z1 - z0) / 4);
    if (nblk <= 0)
        return cudaSuccess;
    if (rate < 1 || rate > 64)
        return cudaErrorInvalidValue;
    cudaError_t e = ensure_smem_attr64();
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads64 - 1) / kThreads64;
    fr4d_encode_kernel<<<(unsigned)grid, kThreads64, smem_bytes64(rate, true), st>>>(in, nx, ny, z0, nblk, rate, out);
    return cudaGetLastError();
}

cudaError_t launch_fr4d_decode(const uint32_t *in, int64_t nx, int64_t ny, int64_t z0, int64_t z1, int rate,
                               DRing out, cudaStream_t st)
{
    const int64_t nblk = (nx / 4) * (ny / 4) * ((z1 - z0) / 4);
    if (nblk <= 0)
        return cudaSuccess;
    if (rate < 1 || rate > 64)
        return cudaErrorInvalidValue;
    cudaError_t e = ensure_smem_attr64();
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads64 - 1) / kThreads64;
    fr4d_decode_kernel<<<(unsigned)grid, kThreads64, smem_bytes64(rate, false), st>>>(in, nx, ny, z0, nblk, rate, out);
    return cudaGetLastError();
}

int64_t fr4_blocks(int64_t nx, int64_t ny, int64_t nz) { return ((nx + 3) / 4) * ((ny + 3) / 4) * ((nz + 3) / 4); }

cudaError_t launch_fr4_encode_dense(const float *in, int64_t nx, int64_t ny, int64_t nz, int words, uint32_t *out,
                                    cudaStream_t st)
{
    const int64_t nblk = fr4_blocks(nx, ny, nz);
    if (nblk <= 0)
        return cudaSuccess;
    if (words < 1 || words > 128)
        return cudaErrorInvalidValue;
    cudaError_t e = ensure_dense_smem_attr();
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads - 1) / kThreads;
    const auto kernel = vec_rows(in, nx) ? fr4_encode_dense_kernel<true> : fr4_encode_dense_kernel<false>;
    kernel<<<(unsigned)grid, kThreads, dense_smem_bytes(words, true, vec_rows(in, nx)), st>>>(in, nx, ny, nz, nblk, words, out);
    return cudaGetLastError();
}

cudaError_t launch_fr4_encode_var(const float *in, int64_t nx, int64_t ny, int64_t nz, int mode, int mparam,
                                  uint32_t *out, uint64_t out_words, uint64_t *index, void *scratch, cudaStream_t st)
{
    const int64_t nblk = fr4_blocks(nx, ny, nz);
    if (nblk <= 0)
        return cudaSuccess;
    cudaError_t e = ensure_dense_smem_attr();
    if (e != cudaSuccess)
        return e;
    e = cudaMemsetAsync(scratch, 0, var_scratch_bytes(nblk), st);
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads - 1) / kThreads;
    const int cap = var_block_words(mode == OOC_FR4_PRECISION ? 32 - mparam : 0);
    const auto kernel = vec_rows(in, nx) ? fr4_encode_var_kernel<true> : fr4_encode_var_kernel<false>;
    kernel<<<(unsigned)grid, kThreads, var_encode_smem(cap), st>>>(in, nx, ny, nz, nblk, mode, mparam, cap, out,
                                                                   out_words, index, (unsigned long long *)scratch);
    return cudaGetLastError();
}

cudaError_t take_codec_fault(unsigned *fault)
{
    unsigned v = 0u;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_codec_fault, sizeof(v));
    if (e == cudaSuccess && v != 0u) {
        const unsigned zero = 0u;
        e = cudaMemcpyToSymbol(g_codec_fault, &zero, sizeof(zero));
    }
    *fault = v;
    return e;
}

cudaError_t launch_fr4_decode_dense(const uint32_t *in, int64_t in_words, const uint64_t *index, int64_t nx,
                                    int64_t ny, int64_t nz, int words, int mode, int mparam, float *out,
                                    cudaStream_t st)
{
    const int64_t nblk = fr4_blocks(nx, ny, nz);
    if (nblk <= 0)
        return cudaSuccess;
    cudaError_t e = ensure_dense_smem_attr();
    if (e != cudaSuccess)
        return e;
    const int64_t grid = (nblk + kThreads - 1) / kThreads;
    if (mode == OOC_FR4_RATE) {
        if (words < 1 || words > 128)
            return cudaErrorInvalidValue;
        const auto kernel = vec_rows(out, nx) ? fr4_decode_dense_kernel<true> : fr4_decode_dense_kernel<false>;
        kernel<<<(unsigned)grid, kThreads, dense_smem_bytes(words, false, false), st>>>(in, nx, ny, nz, nblk, words, out);
    } else {
        const auto kernel = vec_rows(out, nx) ? fr4_decode_var_kernel<true> : fr4_decode_var_kernel<false>;
        kernel<<<(unsigned)grid, kThreads, kVarDecodeSmem, st>>>(in, in_words, index, nx, ny, nz, nblk, mode, mparam,
                                                                 out);
    }
    return cudaGetLastError();
}

int64_t var_total_word(int64_t nblk) { return (nblk + kThreads - 1) / kThreads; }

bool var_total(uint64_t word, uint64_t *total)
{
    *total = word & kTileValue;
    return (word & ~kTileValue) == kTilePrefix;
}

// the tile counter and one status word per tile of the variable-size encoder
size_t var_scratch_bytes(int64_t nblk) { return sizeof(uint64_t) * (size_t)((nblk + kThreads - 1) / kThreads + 1); }


}  // namespace ooc
