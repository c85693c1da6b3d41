// Device-side common random generator of the CORE library (sm_100a).
//
// The paper only requires that all machines share a generator of fresh
// N(0, I_d) vectors (Algorithm 1, first step).  Here that generator is
// Philox4x32-10 (Salmon et al., SC'11) followed by Box-Muller:
//   key     = (seed lo, seed hi)
//   counter = (q lo, q hi, j, t)   q = coordinate block k >> 2, j = vector, t = round
//   u(w)    = ((w >> 9) + 1/2) 2^-23
//   pair    = sqrt(-2 ln u(w_even)) * (cos, sin)(2 pi u(w_odd))
// One counter yields xi_j[4q .. 4q+3].  The words are the same in every kernel.
// From them there are two ways to the angle: polynomials, in registers alone
// (the projections of several machines, short reconstructions and rows, those of
// few or very many vectors), and a table in a CTA's shared memory (last section;
// long reconstructions, long single rows).  Each is within 1.2e-6 of Box-Muller,
// so a projection by one and a reconstruction by the other see vectors that
// differ by 2.4e-6 at most.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace core {

constexpr uint32_t kPhiloxMulA = 0xD2511F53u;  // multiplies counter word 0
constexpr uint32_t kPhiloxMulB = 0xCD9E8D57u;  // multiplies counter word 2
constexpr uint32_t kPhiloxKeyA = 0x9E3779B9u;  // key word 0 increment per round
constexpr uint32_t kPhiloxKeyB = 0xBB67AE85u;  // key word 1 increment per round

// Key schedule, expanded once on the host: a[r], b[r] are the key words of round r.  The last word is a
// constant that turn_parts() wants as a run-time value.
constexpr uint32_t kTurnUnder = 0x3F800100u;
struct RoundKeys {
    uint32_t a[10];
    uint32_t b[10];
    uint32_t turn_under;
};

inline RoundKeys expand_keys(uint64_t seed) {
    RoundKeys k;
    uint32_t a = (uint32_t)(seed & 0xFFFFFFFFu), b = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        k.a[r] = a;
        k.b[r] = b;
        a += kPhiloxKeyA;
        b += kPhiloxKeyB;
    }
    k.turn_under = kTurnUnder;
    return k;
}

__device__ __forceinline__ void mul_wide(uint32_t mult, uint32_t x, uint32_t &hi, uint32_t &lo) {
    unsigned long long p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(x), "r"(mult));
    lo = (uint32_t)p;
    hi = (uint32_t)(p >> 32);
}

// One Philox round.
__device__ __forceinline__ void philox_round(uint32_t &c0, uint32_t &c1, uint32_t &c2, uint32_t &c3,
                                             uint32_t ka, uint32_t kb) {
    uint32_t hi_a, lo_a, hi_b, lo_b;
    mul_wide(kPhiloxMulA, c0, hi_a, lo_a);
    mul_wide(kPhiloxMulB, c2, hi_b, lo_b);
    c0 = hi_b ^ c1 ^ ka;
    c1 = lo_b;
    c2 = hi_a ^ c3 ^ kb;
    c3 = lo_a;
}

// Rounds FIRST..9 on a counter that has already been through rounds 0..FIRST-1.
template <int FIRST>
__device__ __forceinline__ void philox_finish(uint32_t &c0, uint32_t &c1, uint32_t &c2, uint32_t &c3,
                                              const RoundKeys &k) {
#pragma unroll
    for (int r = FIRST; r < 10; ++r) philox_round(c0, c1, c2, c3, k.a[r], k.b[r]);
}

// Plain ten-round evaluation (used where speed does not matter).
__device__ __forceinline__ uint4 philox4x32_10(uint32_t q_lo, uint32_t q_hi, uint32_t j, uint32_t t,
                                               const RoundKeys &k) {
    uint32_t c0 = q_lo, c1 = q_hi, c2 = j, c3 = t;
    philox_finish<0>(c0, c1, c2, c3, k);
    return make_uint4(c0, c1, c2, c3);
}

// ---- split evaluation of the first two rounds ------------------------------------
// After round 0 the counter is (hiB(j)^q_hi^a0, loB(j), hiA(q_lo)^t^b0, loA(q_lo)):
// words 0,1 depend only on (j, q_hi), words 2,3 only on (q_lo, t).  Round 1 then
// needs MulA * word0 (a function of j, q_hi) and MulB * word2 (a function of q_lo, t).
// A kernel that keeps j fixed while q varies, or q fixed while j varies, evaluates
// the invariant half once.  The 32x32->64 multiply is the scarcest resource of the
// generator on this GPU (a quarter of the fp32 rate), so this saves real time.

struct JPart {       // depends on (j, q_hi)
    uint32_t x0;     // loB(j) ^ a1: xored with hiB(word 2) gives word 0 after round 1
    uint32_t x2;     // hiA(word 0 after round 0) ^ b1: xored with word 3 gives word 2 after round 1
    uint32_t w3;     // loA(word 0 after round 0) = word 3 after round 1
};

struct QPart {       // depends on (q_lo, t)
    uint32_t hi_b;   // hiB(word 2 after round 0)
    uint32_t lo_b;   // loB(word 2 after round 0) = word 1 after round 1
    uint32_t w3;     // loA(q_lo) = word 3 after round 0
};

__device__ __forceinline__ JPart philox_jpart(uint32_t j, uint32_t q_hi, const RoundKeys &k) {
    uint32_t hi_b, lo_b, hi_a, lo_a;
    mul_wide(kPhiloxMulB, j, hi_b, lo_b);
    uint32_t w0 = hi_b ^ q_hi ^ k.a[0];
    mul_wide(kPhiloxMulA, w0, hi_a, lo_a);
    JPart p;
    p.x0 = lo_b ^ k.a[1];
    p.x2 = hi_a ^ k.b[1];
    p.w3 = lo_a;
    return p;
}

__device__ __forceinline__ QPart philox_qpart(uint32_t q_lo, uint32_t t, const RoundKeys &k) {
    uint32_t hi_a, lo_a;
    mul_wide(kPhiloxMulA, q_lo, hi_a, lo_a);
    uint32_t w2 = hi_a ^ t ^ k.b[0];
    QPart p;
    mul_wide(kPhiloxMulB, w2, p.hi_b, p.lo_b);
    p.w3 = lo_a;
    return p;
}

__device__ __forceinline__ uint4 philox_combine(const JPart &jp, const QPart &qp, const RoundKeys &k) {
    uint32_t c0 = qp.hi_b ^ jp.x0;
    uint32_t c1 = qp.lo_b;
    uint32_t c2 = jp.x2 ^ qp.w3;
    uint32_t c3 = jp.w3;
    philox_finish<2>(c0, c1, c2, c3, k);
    return make_uint4(c0, c1, c2, c3);
}

// ---- Box-Muller ---------------------------------------------------------------------
// One call turns the four words of a counter into four Gaussians.  The two pairs are
// evaluated side by side in packed fp32 (fma.rn.f32x2 and friends), which halves the
// instruction count of the floating-point part.  On this GPU the fp32 pipe also executes
// the wide multiplies of Philox, so the split of the work between pipes matters: bit
// manipulation (integer pipe) is preferred over floating-point arithmetic where both can
// do the job.
//
// Radius.  u = (k + 1/2) 2^-23 is formed exactly by inserting k = w >> 9 under the
// exponent of 1.0 (one funnel shift) and subtracting 1 - 2^-24.  S = sqrt(-log2 u) comes
// from the hardware log2 and square root; r = sqrt(2 ln 2) S, and that constant is folded
// into the sine/cosine polynomials.  The hardware log2 has an absolute error of about
// 2e-7, harmless except when u is close to 1 (log u close to 0): for v = 1 - u < 2^-10
// (v is exact) the series of -log2(1 - v) replaces it.  That case is rare (one radius in
// 1024), so it sits behind a branch tested once per call.
//
// Angle.  theta = 2 pi u = pi (h + f) with h = bit 31 of the word (which half turn) and
// f = (bits 30..9 + 1/2) / 2^22 in (0, 1).  Those 22 bits, doubled plus one, inserted under
// the exponent of 1.0, minus 1.5, are y = f - 1/2 in (-1/2, 1/2) exactly, and
//   cos theta = -(-1)^h sin(pi y),   sin theta = (-1)^h cos(pi y):
// odd/even minimax polynomials in y (the minus sits in the odd one's coefficients), and bit
// 31 is xored into the sign of S.  No integer arithmetic on the word beyond the bit insert.
//
// Worst absolute error over all 2^23 radius words and all 2^23 angle words: 1.2e-6.

constexpr uint32_t kNearOneWord = 0xFFC00000u;   // words with v = 1 - u < 2^-10

// (w & MASK) | under in one instruction: one holds a single constant, so where `under` is known to the compiler it makes two.
template <uint32_t MASK>
__device__ __forceinline__ float insert_bits(uint32_t w, uint32_t under) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(w), "n"(MASK), "r"(under));
    return __uint_as_float(r);
}

__device__ __forceinline__ float2 bm_splat(float c) { return make_float2(c, c); }

// -log2(1 - v) = (v + v^2/2 + v^3/3 + v^4/4 + ...) / ln 2
__device__ __forceinline__ float bm_near_one(float v) {
    float s = fmaf(v, 0.36067376f, 0.48089835f);
    s = fmaf(s, v, 0.72134752f);
    s = fmaf(s, v, 1.44269504f);
    return s * v;
}
__device__ __forceinline__ float2 bm_near_one(float2 v) {
    float2 s = __ffma2_rn(v, bm_splat(0.36067376f), bm_splat(0.48089835f));
    s = __ffma2_rn(s, v, bm_splat(0.72134752f));
    s = __ffma2_rn(s, v, bm_splat(1.44269504f));
    return __fmul2_rn(s, v);
}

// log2 u (negative) of the two radius words of a call (lanes x, y = pair a, pair b) by the
// hardware log2; u itself is returned for the rare correction.
__device__ __forceinline__ float2 bm_log2(uint4 w, float2 &u) {
    u = __fadd2_rn(make_float2(__uint_as_float(__funnelshift_r(w.x, 0x7Fu, 9)),
                               __uint_as_float(__funnelshift_r(w.z, 0x7Fu, 9))),
                   bm_splat(-0.99999994f));
    float2 l;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l.x) : "f"(u.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l.y) : "f"(u.y));
    return l;
}

// l of N calls.  The rare near-one correction of all 2N radii sits behind one test, which leaves the N evaluations in one
// straight-line block for the instruction scheduler.  A warp finds some radius of its 64 N near one in a fifth of the cases,
// but rarely more than one: with EACH the calls are then tested one by one, which suits the kernels that take the angle
// from the table (0.9 % faster; those with the polynomials are 1 to 2 % slower with it).
template <int N, bool EACH>
__device__ __forceinline__ void bm_logs(const uint4 (&w)[N], float2 (&l)[N]) {
    float2 u[N];
    uint32_t top = 0u;
#pragma unroll
    for (int c = 0; c < N; ++c) {
        l[c] = bm_log2(w[c], u[c]);
        top = __vimax3_u32(top, w[c].x, w[c].z);
    }
    if (EACH ? __builtin_expect(top >= kNearOneWord, 0) : top >= kNearOneWord) {
#pragma unroll
        for (int c = 0; c < N; ++c) {
            if constexpr (EACH) {
                if (__builtin_expect(max(w[c].x, w[c].z) >= kNearOneWord, 0)) {
                    const float2 s = bm_near_one(__fadd2_rn(bm_splat(1.0f), make_float2(-u[c].x, -u[c].y)));
                    if (w[c].x >= kNearOneWord) l[c].x = s.x;
                    if (w[c].z >= kNearOneWord) l[c].y = s.y;
                }
            } else {
                if (w[c].x >= kNearOneWord) l[c].x = bm_near_one(1.0f - u[c].x);
                if (w[c].z >= kNearOneWord) l[c].y = bm_near_one(1.0f - u[c].y);
            }
        }
    }
}

// The rest of Box-Muller given l with |l| = -log2 u of the two pairs (the sign of l is ignored:
// the hardware path delivers log2 u < 0, the correction delivers the positive series), as its factors:
// with S = (-1)^h sqrt(-log2 u) the pair is (r cos theta, r sin theta) = ((S y) sp, S cs).  Lanes x, y of
// every member = pair a, pair b.  A consumer that multiplies the values by a number p of its own can let p
// meet S first, ((p S) y) sp and (p S) cs, and save the two products that would form the values; with
// p = 1 that is bit for bit what bm_finish returns.
struct BmParts {
    float2 s;     // (-1)^h sqrt(-log2 u)
    float2 y;     // f - 1/2
    float2 sp;    // -sqrt(2 ln 2) sin(pi y) / y
    float2 cs;    //  sqrt(2 ln 2) cos(pi y)
};

__device__ __forceinline__ BmParts bm_parts(uint4 w, float2 l) {
    BmParts r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.s.x) : "f"(fabsf(l.x)));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.s.y) : "f"(fabsf(l.y)));

    // angles: theta = pi (h + f), h = bit 31 of the word, f = (bits 30..9 + 1/2) / 2^22 in (0, 1).
    // With y = f - 1/2:  cos theta = -(-1)^h sin(pi y),  sin theta = (-1)^h cos(pi y).
    r.y = __fadd2_rn(make_float2(__uint_as_float(((w.y >> 8) & 0x007FFFFEu) | 0x3F800001u),
                                 __uint_as_float(((w.w >> 8) & 0x007FFFFEu) | 0x3F800001u)),
                     bm_splat(-1.5f));
    r.s.x = __uint_as_float(__float_as_uint(r.s.x) ^ (w.y & 0x80000000u));
    r.s.y = __uint_as_float(__float_as_uint(r.s.y) ^ (w.w & 0x80000000u));
    const float2 y2 = __fmul2_rn(r.y, r.y);
    // -sqrt(2 ln 2) sin(pi y) / y and sqrt(2 ln 2) cos(pi y)
    float2 sp = __ffma2_rn(bm_splat(-0.09091975539922714f), y2, bm_splat(0.7041443586349487f));
    sp = __ffma2_rn(sp, y2, bm_splat(-3.0024325847625732f));
    sp = __ffma2_rn(sp, y2, bm_splat(6.08450984954834f));
    r.sp = __ffma2_rn(sp, y2, bm_splat(-3.6989426612854004f));
    float2 cp = __ffma2_rn(bm_splat(0.2591251730918884f), y2, bm_splat(-1.568420648574829f));
    cp = __ffma2_rn(cp, y2, bm_splat(4.778461456298828f));
    cp = __ffma2_rn(cp, y2, bm_splat(-5.810277938842773f));
    r.cs = __ffma2_rn(cp, y2, bm_splat(1.1774100065231323f));
    return r;
}

__device__ __forceinline__ float4 bm_finish(uint4 w, float2 l) {
    const BmParts r = bm_parts(w, l);
    const float2 zs = __fmul2_rn(r.s, r.cs);                       // r sin theta
    const float2 zc = __fmul2_rn(__fmul2_rn(r.s, r.y), r.sp);      // r cos theta
    return make_float4(zc.x, zs.x, zc.y, zs.y);
}

// N calls at once.
template <int N>
__device__ __forceinline__ void box_muller4xN(const uint4 (&w)[N], float4 (&z)[N]) {
    float2 l[N];
    bm_logs<N, false>(w, l);
#pragma unroll
    for (int c = 0; c < N; ++c) z[c] = bm_finish(w[c], l[c]);
}

// The factors of N calls.
template <int N>
__device__ __forceinline__ void box_muller_parts(const uint4 (&w)[N], BmParts (&r)[N]) {
    float2 l[N];
    bm_logs<N, false>(w, l);
#pragma unroll
    for (int c = 0; c < N; ++c) r[c] = bm_parts(w[c], l[c]);
}

__device__ __forceinline__ float4 box_muller4(uint4 w) {
    const uint4 ws[1] = {w};
    float4 zs[1];
    box_muller4xN<1>(ws, zs);
    return zs[0];
}

// ---- Box-Muller with the angle from a table ----------------------------------------------
// Long launches take sine and cosine from a table of kTurnEntries angles in shared memory (64 KB): the 13 top bits of the
// word name the entry, the other ten bits used an angle delta of at most pi/8192 about its middle, and
//   cos(theta) = C - S delta,   sin(theta) = S + C delta.
// What is left out, 1 - cos(delta) <= 7.4e-8, is met by its mean in the scale of the entries.  Every integer and every fp32
// instruction costs the schedulers two cycles here (scalar fp32: one; wide multiplies: two of their four; loads from shared
// memory: about one), so it is their number that counts: 3 integer, 2.5 fp32 instructions and a load per angle in place of
// 3 and 6.5.  116 -> 108 cycles per counter in the reconstruction, and closer to Box-Muller than the polynomials: rms error
// 7.5e-8 against 1.02e-7, worst 1.2e-6 as there.  The two integer instructions that cut out the fraction are one where its upper bits
// come from a kernel parameter (insert_bits): 107.4 -> 105.6 cycles, d = 2.5e7, m = 256: 4607 -> 4536 us; the same in the angles
// of the polynomials made the tcgen05 projection 3 to 6 % slower and changed nothing elsewhere.  (A copy of 512 entries per lane, free of bank conflicts but in need of
// second-order terms: 117.  Two loads of 4 bytes instead of one of 8, the products packed: 110.  4096 entries: rms error 1.27e-7.)
//
// The table comes without the factor kTurnScale = sqrt(2 ln 2): values below 1 are twice as finely spaced, and the factor is
// applied where a sum ends.  Its fp32 rounding, and the bias of the hardware's log2 and square root (the radius is 1.5e-7
// too small at first order, of which 3e-8 is best taken back: more makes the longest radii worse), are in the entries.
constexpr int kTurnBits = 13;
constexpr int kTurnEntries = 1 << kTurnBits;
constexpr int kTurnBytes = kTurnEntries * 8;
constexpr float kTurnScale = 1.1774100225154747f;

constexpr double turn_series(double x, double term, int k) {      // x^k/k! - x^(k+2)/(k+2)! + ...
    double sum = 0.0;
    for (; k < 40; k += 2) {
        sum += term;
        term = -term * x * x / ((k + 1) * (k + 2));
    }
    return sum;
}
// The entries are made in place by an angle addition: 256 coarse angles in two floats each, 32 fine ones (cosine minus one).
constexpr int kTurnFine = 32;
struct TurnSeed {
    float4 coarse[kTurnEntries / kTurnFine];      // {C, C's remainder, S, S's remainder}
    float2 fine[kTurnFine];                       // {cos - 1, sin}
};
constexpr TurnSeed make_turn_seed() {
    constexpr double pi = 3.14159265358979323846, delta = pi / kTurnEntries;
    constexpr double scale = 1.17741002251547469101 / (double)kTurnScale * (1.0 - delta * delta / 6.0) * (1.0 + 3e-8);
    TurnSeed t{};
    for (int h = 0; h < kTurnEntries / kTurnFine; ++h) {
        const double a = 2.0 * pi * (h + 0.5) / (kTurnEntries / kTurnFine) - pi;        // series in (-pi, pi), then negated
        const double c = -scale * turn_series(a, 1.0, 0), s = -scale * turn_series(a, a, 1);
        t.coarse[h].x = (float)c;
        t.coarse[h].y = (float)(c - (double)t.coarse[h].x);
        t.coarse[h].z = (float)s;
        t.coarse[h].w = (float)(s - (double)t.coarse[h].z);
    }
    for (int l = 0; l < kTurnFine; ++l) {
        const double a = 2.0 * pi * (l + 0.5 - kTurnFine / 2) / kTurnEntries;
        t.fine[l].x = (float)-(a * a / 2.0 - a * a * a * a / 24.0);
        t.fine[l].y = (float)turn_series(a, a, 1);
    }
    return t;
}
static __device__ const TurnSeed kTurnSeed = make_turn_seed();

// Filled by WARPS warps of a CTA; the caller synchronises.  A warp reads its coarse angles in one load, a lane each.
template <int WARPS>
__device__ __forceinline__ void fill_turn_table(float2 *table, int warp, int lane) {
    constexpr int kCoarse = kTurnEntries / kTurnFine, kMine = (kCoarse + WARPS - 1) / WARPS;
    static_assert(kMine <= 32, "a coarse angle per lane");
    const float2 f = __ldg(&kTurnSeed.fine[lane]);
    const float4 mine = __ldg(&kTurnSeed.coarse[min(warp + lane * WARPS, kCoarse - 1)]);
#pragma unroll 4
    for (int i = 0; i < kMine; ++i) {
        const int h = warp + i * WARPS;
        const float4 g = make_float4(__shfl_sync(0xffffffffu, mine.x, i), __shfl_sync(0xffffffffu, mine.y, i),
                                     __shfl_sync(0xffffffffu, mine.z, i), __shfl_sync(0xffffffffu, mine.w, i));
        // C cos - S sin = C + (C (cos - 1) - S sin + C's remainder): what is rounded before the last sum is small
        if (h < kCoarse)
            table[h * kTurnFine + lane] = make_float2(g.x + fmaf(g.x, f.x, fmaf(-g.z, f.y, g.y)), g.z + fmaf(g.z, f.x, fmaf(g.x, f.y, g.w)));
    }
}

// The four values of a call are kTurnScale times (s c, s n) of pair a (lanes x) and of pair b (lanes y).
struct TurnParts {
    float2 s;     // sqrt(-log2 u)
    float2 c;     // cosine
    float2 n;     // sine
};
__device__ __forceinline__ TurnParts turn_parts(uint4 w, float2 l, const float2 *table, const RoundKeys &k) {
    constexpr uint32_t kFraction = ((1u << (32 - kTurnBits)) - 1u) & ~511u;
    constexpr float kUnit = (float)(1u << (32 - kTurnBits)) / 8388608.0f;               // an entry's share of the mantissa
    constexpr float kSlope = 6.283185307179586f / kTurnEntries / kUnit;
    const float2 ta = table[w.y >> (32 - kTurnBits)], tb = table[w.w >> (32 - kTurnBits)];
    const float2 f = make_float2(insert_bits<kFraction>(w.y, k.turn_under), insert_bits<kFraction>(w.w, k.turn_under));
    const float2 delta = __ffma2_rn(f, bm_splat(kSlope), bm_splat(-(1.0f + 0.5f * kUnit) * kSlope));
    TurnParts r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.s.x) : "f"(fabsf(l.x)));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.s.y) : "f"(fabsf(l.y)));
    r.c = make_float2(fmaf(-ta.y, delta.x, ta.x), fmaf(-tb.y, delta.y, tb.x));
    r.n = make_float2(fmaf(ta.x, delta.x, ta.y), fmaf(tb.x, delta.y, tb.y));
    return r;
}

}  // namespace core
