// Device flow graphs of the Cordic-based Loeffler 8-point DCT (Sec. 2.5.2,
// Fig. 1) and its transpose: the forward graph on exact integers in float32,
// the inverse in int32 registers.
//
// Forward graph (standard Loeffler structure, four stages in series):
//   stage 1  s_n = x_n + x_{7-n}, d_n = x_n - x_{7-n}
//   stage 2  even e0 = s0+s3, e3 = s0-s3, e1 = s1+s2, e2 = s1-s2;
//            odd  (a4,a7) = rot(d3,d0,3pi/16), (a5,a6) = rot(d2,d1,pi/16)
//   stage 3  Y0 = e0+e1, Y4 = e0-e1, (Y2,Y6) = rot(e2,e3,3pi/8);
//            b4 = a4+a6, b6 = a4-a6, b7 = a7+a5, b5 = a7-a5
//   stage 4  Y1 = b7+b4, Y7 = b7-b4, Y3 = b5, Y5 = b6
// Every rot() is a CORDIC block of kN shift-add micro-rotations
// (a, b) <- (a + s (b >> i), b - s (a >> i)), i = 1..kN, arithmetic shifts;
// 3pi/8 is the exact quarter turn (a, b) -> (b, -a) followed by a CORDIC
// rotation of -pi/8.  The sqrt(2) factors of stage 4 and the CORDIC gain are
// not computed: the quantiser and dequantiser tables absorb them.
//
// The inverse graph is the transpose: steps in reverse order, butterflies
// unchanged, each micro-rotation with -s in ascending i, and the quarter
// turn's transpose (a, b) -> (-b, a).
#pragma once
#include "dctgb_spec.h"


namespace dctgb {

// acc + (v >> I) with an arithmetic (floor) shift: one instruction of the
// integer ALU, acc - (v >> I) two.  (A mad.hi.s32 computes the same value, the
// high word of v * 2^(32-I), at about a quarter of that rate: dct_int_peak.)
template <int I>
__device__ __forceinline__ int add_shr(int acc, int v) {
    return acc + (v >> I);
}

template <int I>
__device__ __forceinline__ int sub_shr(int acc, int v) {
    return acc - (v >> I);
}

// Micro-rotations I..kN with the directions of MASK (bit i set: s_i = +1):
// (a, b) <- (a + s_i (b >> i), b - s_i (a >> i)) from the pre-step values.
template <unsigned MASK, int I>
__device__ __forceinline__ void cordic_fwd_from(int& a, int& b) {
    if constexpr (I <= kN) {
        int na, nb;
        if constexpr ((MASK >> I) & 1u) {
            na = add_shr<I>(a, b);
            nb = sub_shr<I>(b, a);
        } else {
            na = sub_shr<I>(a, b);
            nb = add_shr<I>(b, a);
        }
        a = na;
        b = nb;
        cordic_fwd_from<MASK, I + 1>(a, b);
    }
}

// Transposed micro-rotations: the same shifts with -s_i, ascending i.
template <unsigned MASK, int I>
__device__ __forceinline__ void cordic_tr_from(int& a, int& b) {
    if constexpr (I <= kN) {
        int na, nb;
        if constexpr ((MASK >> I) & 1u) {
            na = sub_shr<I>(a, b);
            nb = add_shr<I>(b, a);
        } else {
            na = add_shr<I>(a, b);
            nb = sub_shr<I>(b, a);
        }
        a = na;
        b = nb;
        cordic_tr_from<MASK, I + 1>(a, b);
    }
}

// Constants added to a pair (a, b).
struct FltBias {
    long long a, b;
};

// ---- Transposed rotations, one instruction per half micro-rotation --------
// The ALU computes acc + (v >> i) and (v >> i) - acc in one instruction
// (measured), but acc - (v >> i), which every micro-rotation has in one of
// its halves, takes two.  So a and b are held with signs and offsets known at
// compile time, A = sa a + ka and B = sb b + kb, and the half
// a' = a + s floor(b / 2^i) becomes
//   A' = A + (B >> i)  (sign kept)      when sb = sa s,
//   A' = (B >> i) - A  (sign flipped)   when sb = -sa s,
// and likewise b' = b - s floor(a / 2^i) from the old A.  B >> i is exact for
// it when it is sb floor(b / 2^i) plus a constant: with sb = 1 that needs
// kb = 0 (mod 2^i); with sb = -1, floor((kb - b) / 2^i) = -floor((b - kb +
// 2^i - 1) / 2^i) needs kb = -1 (mod 2^i).  Every step maps the offsets by an
// integer matrix with odd determinant, so the conditions of steps 1..N have
// exactly one solution for the starting pair modulo 2^(1 + .. + N); the
// compiler finds it below.  The offsets stay below 2^22 and the inverse
// graph's nodes below 1.17e9, so nothing overflows.  A pass then takes 64
// instructions per 8 values (36 shift-adds, 28 additions that either pipe can
// do) instead of 75; 8192 x 8192 + 4K 4:2:0 measured: inverse from stored
// codes 100.5 us against 103.6 us, fused 138.4 against 140.4 us.
struct TrState {
    long long ka, kb;
    int sa, sb;
    bool ok;
};
constexpr TrState tr_run(unsigned mask, long long ka, long long kb, int upto) {
    int sa = 1, sb = 1;
    for (int i = 1; i <= upto; ++i) {
        const int s = (mask >> i) & 1u ? -1 : 1;      // transposed: -s_i
        const long long m = 1LL << i;
        if ((sb > 0 ? kb : kb + 1) % m != 0 || (sa > 0 ? ka : ka + 1) % m != 0) return {0, 0, 0, 0, false};
        const long long cb = sb > 0 ? kb / m : (kb + 1) / m - 1;
        const long long ca = sa > 0 ? ka / m : (ka + 1) / m - 1;
        const bool fa = sb != sa * s, fb = sa != -s * sb;
        ka = (fa ? -ka : ka) + cb;
        kb = (fb ? -kb : kb) + ca;
        sa = fa ? -sa : sa;
        sb = fb ? -sb : sb;
    }
    return {ka, kb, sa, sb, true};
}
constexpr bool kTrOffsets = kN <= 6;
// Starting offsets, lifted step by step: the solution of steps 1..i-1 is known
// modulo 2^(1 + .. + i-1), and step i picks its next i bits of each.
constexpr FltBias tr_start(unsigned mask) {
    if (!kTrOffsets) return {0, 0};
    long long ka = 0, kb = 0;
    int bits = 0;
    for (int i = 1; i <= kN; ++i) {
        bool found = false;
        for (long long x = 0; x < (1LL << i) && !found; ++x)
            for (long long y = 0; y < (1LL << i) && !found; ++y)
                if (tr_run(mask, ka + (x << bits), kb + (y << bits), i).ok) {
                    ka += x << bits;
                    kb += y << bits;
                    found = true;
                }
        bits += i;
    }
    const long long m = 1LL << bits;
    return {ka >= m / 2 ? ka - m : ka, kb >= m / 2 ? kb - m : kb};
}

// A transposed rotation block: run() takes a + start.a and b + start.b and
// leaves sa * a' + ka and sb * b' + kb (end).  Other CORDIC counts run the
// plain form with no offsets.
template <unsigned MASK>
struct TrRotation {
    static constexpr FltBias start = tr_start(MASK);
    static constexpr TrState end = kTrOffsets ? tr_run(MASK, start.a, start.b, kN) : TrState{0, 0, 1, 1, true};
    static_assert(end.ok, "no starting offsets for a transposed rotation");
    template <int I, int SA, int SB>
    static __device__ __forceinline__ void steps(int& a, int& b) {
        if constexpr (I <= kN) {
            constexpr int s = (MASK >> I) & 1u ? -1 : 1;
            constexpr bool fa = SB != SA * s, fb = SA != -s * SB;
            const int na = fa ? (b >> I) - a : a + (b >> I);
            const int nb = fb ? (a >> I) - b : b + (a >> I);
            a = na;
            b = nb;
            steps<I + 1, fa ? -SA : SA, fb ? -SB : SB>(a, b);
        }
    }
    static __device__ __forceinline__ void run(int& a, int& b) {
        if constexpr (kTrOffsets) steps<1, 1, 1>(a, b);
        else cordic_tr_from<MASK, 1>(a, b);
    }
};

// ---- Forward graph in float32 --------------------------------------------
// The forward graph's nodes are integers below 2^20, so they are exact in
// float32: its additions and floor shifts run on the FMA pipes, which take a
// float operation in half the time of an integer shift or add (measured: 0.26
// clocks and SM for an FFMA against 0.51 for a shift-add, a permute or an
// integer multiply-add).  Two vectors run at once in the packed form
// (add.f32x2, fma.f32x2): a packed operation holds the FMA pipe for two, so
// the rate is the same, but the code is half as long.  8192 x 8192 + 4K 4:2:0,
// coefficients out, one lane per block: 83.0 us with integer additions and
// float micro-rotations 2..N, 74.8 us with everything in plain float32, 66.7
// us packed; the fused two-lane kernel 152.7 us plain, 140.4 us packed.
//
// Floor shifts.  Every float32 of magnitude in [2^23, 2^24) is an integer,
// and a fused multiply-add rounds its exact result once.  Hold a and b as the
// floats A = alpha + a and B = beta + b, with compile-time biases alpha, beta
// in that range (either sign) and beta * 2^-i, alpha * 2^-i integers; then
//   fma round-down(B,  2^-i, A) = (alpha + beta 2^-i) + a + floor(b / 2^i)
//   fma round-up  (A, -2^-i, B) = (beta - alpha 2^-i) + b - floor(a / 2^i)
// exactly, as long as the results stay in the range: one operation per half
// micro-rotation.  The biases follow the micro-rotations themselves (without
// floors), so the schedule below is fixed per rotation block and checked at
// compile time against the forward graph's node bound.  Step 1 (a 26.6
// degree turn) would carry every bias pair out of the range, so it starts
// from unbiased values and brings the biases in:
//   fma round-down(b,  1/2, alpha) = alpha + floor(b / 2), then + a
//   fma round-up  (a, -1/2, beta)  = beta - floor(a / 2),  then + b
// with both sums exact (integers of magnitude below 2^24).  In the row pass
// a and b are multiples of 2^kP = 16, so steps 1 and 2 round nothing and are
// one linear map: two plain fused multiply-adds per output, biases included.
constexpr long long kFwdNodeBound = 1LL << 20;   // |node| of the forward graph
                                                 // at kP = 4 (interval
                                                 // propagation: 719380)
constexpr bool kFltForward = kN <= 6;             // biases need 2^(2+..+kN) | alpha

// Bias pair before micro-rotation i (2 <= i <= kN + 1) of a block with
// directions MASK that starts step 2 with (a0, b0).
__host__ __device__ constexpr FltBias flt_bias(unsigned mask, long long a0, long long b0, int i) {
    long long a = a0, b = b0;
    for (int j = 2; j < i; ++j) {
        const long long da = b / (1LL << j), db = a / (1LL << j);
        if ((mask >> j) & 1u) {
            a += da;
            b -= db;
        } else {
            a -= da;
            b += db;
        }
    }
    return {a, b};
}

constexpr bool flt_in_range(long long x) {
    const long long m = x < 0 ? -x : x;
    return m - kFwdNodeBound >= (1LL << 23) && m + kFwdNodeBound < (1LL << 24);
}

constexpr bool flt_schedule_ok(unsigned mask, long long a0, long long b0) {
    for (int i = 2; i <= kN + 1; ++i) {
        const FltBias p = flt_bias(mask, a0, b0, i);
        if (!flt_in_range(p.a) || !flt_in_range(p.b)) return false;
        if (i <= kN && (p.a % (1LL << i) != 0 || p.b % (1LL << i) != 0)) return false;
    }
    return true;
}

// Starting biases (multiples of 2^20), chosen by exhaustive search for the
// widest margin; one table serves kN = 3..6.
constexpr long long kFltUnit = 1LL << 20;
constexpr long long kFltOddUpperA = -13 * kFltUnit, kFltOddUpperB = 10 * kFltUnit;
constexpr long long kFltOddLowerA = -14 * kFltUnit, kFltOddLowerB = -10 * kFltUnit;
constexpr long long kFltEvenA = -13 * kFltUnit, kFltEvenB = 10 * kFltUnit;
static_assert(!kFltForward || (flt_schedule_ok(kSigOddUpper, kFltOddUpperA, kFltOddUpperB) &&
                               flt_schedule_ok(kSigOddLower, kFltOddLowerA, kFltOddLowerB) &&
                               flt_schedule_ok(kSigEven, kFltEvenA, kFltEvenB)),
              "float micro-rotation bias schedule leaves the exact-integer range");

// Two float32 in a 64-bit register pair, and the packed instructions.
struct f2 {
    unsigned long long v;
};
__device__ __forceinline__ f2 f2_pack(float x, float y) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ f2 f2_splat(float k) { return f2_pack(k, k); }
__device__ __forceinline__ float2 f2_unpack(f2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma_rn(f2 a, float k, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(f2_splat(k).v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma_rd(f2 a, float k, f2 c) {
    f2 r;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(f2_splat(k).v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma_ru(f2 a, float k, f2 c) {
    f2 r;
    asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(f2_splat(k).v), "l"(c.v));
    return r;
}

// Micro-rotations I..kN on biased values.
template <unsigned MASK, int I>
__device__ __forceinline__ void cordic_fwd_flt_from(f2& a, f2& b) {
    if constexpr (I <= kN) {
        constexpr float sc = 1.0f / float(1 << I);   // exact power of two
        f2 na, nb;
        if constexpr ((MASK >> I) & 1u) {
            na = f2_fma_rd(b, sc, a);     // a + floor(b / 2^I)
            nb = f2_fma_ru(a, -sc, b);    // b - floor(a / 2^I)
        } else {
            na = f2_fma_ru(b, -sc, a);    // a - floor(b / 2^I)
            nb = f2_fma_rd(a, sc, b);     // b + floor(a / 2^I)
        }
        a = na;
        b = nb;
        cordic_fwd_flt_from<MASK, I + 1>(a, b);
    }
}

// A rotation block on unbiased integers in float32; run() leaves the
// schedule's final biases (end) on the results.  ROW: the row pass (inputs
// multiples of 2^kP).
template <unsigned MASK, long long A0, long long B0>
struct FltRotation {
    static constexpr FltBias end = flt_bias(MASK, A0, B0, kN + 1);
    template <bool ROW>
    static __device__ __forceinline__ void run(f2& a, f2& b) {
        f2 fa, fb;
        if constexpr (ROW) {
            static_assert(kP >= 3 && kN >= 2, "steps 1 and 2 must be exact");
            constexpr float s1 = (MASK >> 1) & 1u ? 1.0f : -1.0f, s2 = (MASK >> 2) & 1u ? 1.0f : -1.0f;
            constexpr float c = 1.0f - s1 * s2 / 8.0f, k = s1 / 2.0f + s2 / 4.0f;
            constexpr FltBias e = flt_bias(MASK, A0, B0, 3);
            fa = f2_fma_rn(a, c, f2_fma_rn(b, k, f2_splat((float)e.a)));
            fb = f2_fma_rn(b, c, f2_fma_rn(a, -k, f2_splat((float)e.b)));
            cordic_fwd_flt_from<MASK, 3>(fa, fb);
        } else {
            if constexpr ((MASK >> 1) & 1u) {
                fa = a + f2_fma_rd(b, 0.5f, f2_splat((float)A0));
                fb = b + f2_fma_ru(a, -0.5f, f2_splat((float)B0));
            } else {
                fa = a + f2_fma_ru(b, -0.5f, f2_splat((float)A0));
                fb = b + f2_fma_rd(a, 0.5f, f2_splat((float)B0));
            }
            cordic_fwd_flt_from<MASK, 2>(fa, fb);
        }
        a = fa;
        b = fb;
    }
};
using RotOddUpper = FltRotation<kSigOddUpper, kFltOddUpperA, kFltOddUpperB>;
using RotOddLower = FltRotation<kSigOddLower, kFltOddLowerA, kFltOddLowerB>;
using RotEven = FltRotation<kSigEven, kFltEvenA, kFltEvenB>;

__device__ __forceinline__ void loeffler8_fwd(int (&v)[8]);

// Sample k of a little-endian word as the float 2^19 + (p << kP): at 2^19 the
// last mantissa bit counts 2^-4, so the byte goes straight into the second
// mantissa byte (one byte permute).  The level-shifted sample (p - 128) << kP
// is that less kPixBias; the graph is linear up to the rotations and its
// differences cancel the bias, so only Y0 has to take it off (eight times).
static_assert(kP == 4, "the sample encoding places the byte at a unit of 2^kP");
constexpr float kPixBias = 524288.0f + 2048.0f;
template <int K>
__device__ __forceinline__ float pix_float(uint32_t word) {
    return __int_as_float(__byte_perm(word, 0x49000000u, 0x7404u | (K << 4)));
}

// Forward 8-point graph between its first stage (s[n] = x[n] + x[7-n], d[n] =
// x[n] - x[7-n]) and its last additions.
struct FwdNodes {
    f2 e0, e1, y2, y6, a4, a5, a6, a7;   // y2 and y6 still biased (RotEven::end)
};
template <bool ROW>
__device__ __forceinline__ FwdNodes fwd_nodes(const f2 (&s)[4], const f2 (&d)[4]) {
    FwdNodes n;
    n.e0 = s[0] + s[3];
    n.e1 = s[1] + s[2];
    n.y2 = s[0] - s[3];
    n.y6 = s[2] - s[1];                // quarter turn of (e2, e3): (e3, -e2)
    RotEven::run<ROW>(n.y2, n.y6);
    n.a4 = d[3];
    n.a7 = d[0];
    RotOddUpper::run<ROW>(n.a4, n.a7);
    n.a4 = n.a4 + f2_splat((float)-RotOddUpper::end.a);
    n.a7 = n.a7 + f2_splat((float)-RotOddUpper::end.b);
    n.a5 = d[2];
    n.a6 = d[1];
    RotOddLower::run<ROW>(n.a5, n.a6);
    n.a5 = n.a5 + f2_splat((float)-RotOddLower::end.a);
    n.a6 = n.a6 + f2_splat((float)-RotOddLower::end.b);
    return n;
}
// The last additions of one vector: y[k] <- Y_k.
template <bool ROW>
__device__ __forceinline__ void fwd_last(float e0, float e1, float y2, float y6, float a4, float a5, float a6, float a7,
                                         float (&y)[8]) {
    const float b4 = __fadd_rn(a4, a6), b7 = __fadd_rn(a7, a5), y0 = __fadd_rn(e0, e1);
    y[0] = ROW ? __fadd_rn(y0, -8.0f * kPixBias) : y0;
    y[4] = __fsub_rn(e0, e1);
    y[2] = __fadd_rn(y2, (float)-RotEven::end.a);
    y[6] = __fadd_rn(y6, (float)-RotEven::end.b);
    y[1] = __fadd_rn(b7, b4);
    y[7] = __fsub_rn(b7, b4);
    y[3] = __fsub_rn(a7, a5);
    y[5] = __fsub_rn(a4, a6);
}

// Forward 8-point graph of two vectors in float32 (in place: v[k] <- Y_k).
// ROW: they come from pix_float; else they hold unbiased integers.  Packed
// between the first and the last additions: those run unpacked, so that each
// vector stays in registers of its own (rows for 16-byte stores, columns out
// of row registers) without moves.
template <bool ROW>
__device__ __forceinline__ void fwd_two(float (&v0)[8], float (&v1)[8]) {
    if constexpr (!kFltForward) {       // CORDIC counts without a bias schedule
        int w0[8], w1[8];
        const float bias = ROW ? -kPixBias : 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            w0[i] = __float2int_rn(__fadd_rn(v0[i], bias));
            w1[i] = __float2int_rn(__fadd_rn(v1[i], bias));
        }
        loeffler8_fwd(w0);
        loeffler8_fwd(w1);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v0[i] = __int2float_rn(w0[i]);
            v1[i] = __int2float_rn(w1[i]);
        }
    } else {
        f2 s[4], d[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            s[n] = f2_pack(__fadd_rn(v0[n], v0[7 - n]), __fadd_rn(v1[n], v1[7 - n]));
            d[n] = f2_pack(__fsub_rn(v0[n], v0[7 - n]), __fsub_rn(v1[n], v1[7 - n]));
        }
        const FwdNodes n = fwd_nodes<ROW>(s, d);
        const float2 e0 = f2_unpack(n.e0), e1 = f2_unpack(n.e1), y2 = f2_unpack(n.y2), y6 = f2_unpack(n.y6);
        const float2 a4 = f2_unpack(n.a4), a5 = f2_unpack(n.a5), a6 = f2_unpack(n.a6), a7 = f2_unpack(n.a7);
        fwd_last<ROW>(e0.x, e1.x, y2.x, y6.x, a4.x, a5.x, a6.x, a7.x, v0);
        fwd_last<ROW>(e0.y, e1.y, y2.y, y6.y, a4.y, a5.y, a6.y, a7.y, v1);
    }
}

// Samples of one row (two little-endian words) for the row pass.
__device__ __forceinline__ void pix_row(const uint32_t (&w)[2], float (&y)[8]) {
    y[0] = pix_float<0>(w[0]);
    y[1] = pix_float<1>(w[0]);
    y[2] = pix_float<2>(w[0]);
    y[3] = pix_float<3>(w[0]);
    y[4] = pix_float<0>(w[1]);
    y[5] = pix_float<1>(w[1]);
    y[6] = pix_float<2>(w[1]);
    y[7] = pix_float<3>(w[1]);
}

// N vectors, two at a time.
template <bool ROW, int N>
__device__ __forceinline__ void fwd_vectors(float (&v)[N][8]) {
    static_assert(N % 2 == 0, "vectors go in pairs");
#pragma unroll
    for (int i = 0; i < N; i += 2) fwd_two<ROW>(v[i], v[i + 1]);
}

template <unsigned MASK>
__device__ __forceinline__ void cordic_fwd(int& a, int& b) { cordic_fwd_from<MASK, 1>(a, b); }

// Forward 8-point graph on v[0..7] in integers (in place: v[k] <- Y_k), for
// CORDIC counts without a float bias schedule (kN > 6).
__device__ __forceinline__ void loeffler8_fwd(int (&v)[8]) {
    const int s0 = v[0] + v[7], d0 = v[0] - v[7];
    const int s1 = v[1] + v[6], d1 = v[1] - v[6];
    const int s2 = v[2] + v[5], d2 = v[2] - v[5];
    const int s3 = v[3] + v[4], d3 = v[3] - v[4];
    const int e0 = s0 + s3, e3 = s0 - s3;
    const int e1 = s1 + s2, e2 = s1 - s2;
    int a4 = d3, a7 = d0;
    cordic_fwd<kSigOddUpper>(a4, a7);
    int a5 = d2, a6 = d1;
    cordic_fwd<kSigOddLower>(a5, a6);
    int y2 = e3, y6 = -e2;             // quarter turn of (e2, e3)
    cordic_fwd<kSigEven>(y2, y6);
    const int b4 = a4 + a6, b6 = a4 - a6;
    const int b7 = a7 + a5, b5 = a7 - a5;
    v[0] = e0 + e1;
    v[4] = e0 - e1;
    v[2] = y2;
    v[6] = y6;
    v[1] = b7 + b4;
    v[7] = b7 - b4;
    v[3] = b5;
    v[5] = b6;
}

// c ? x + y : x - y with a compile-time choice.
template <bool C>
__device__ __forceinline__ unsigned add_if(unsigned x, unsigned y) { return C ? x + y : x - y; }

// Transposed (inverse) 8-point graph on v[0..7] (in place: v[n] <- x_n).
// The inputs carry a constant Z (the bits a float dequantiser leaves, see
// dequant_bits), which comes off, and the rotations' starting offsets go in,
// through the three-input additions of the first stage.  Their final offsets
// come off in six additions of their own rather than as a third input of the
// last eight and four: three-input additions issue only on the integer ALU,
// which the shift-adds already fill (measured 105.6 against 100.5 us, inverse
// from stored codes).  dc is added to v[0].
template <int Z>
__device__ __forceinline__ void loeffler8_inv(int (&v)[8], int dc) {
    using Up = TrRotation<kSigOddUpper>;
    using Lo = TrRotation<kSigOddLower>;
    using Ev = TrRotation<kSigEven>;
    constexpr unsigned z = (unsigned)Z;
    const unsigned v0 = v[0], v1 = v[1], v3 = v[3], v4 = v[4], v5 = v[5], v7 = v[7];
    const unsigned t = v1 + v7, u = v1 - v7;
    int a7 = (int)(t + v3 + ((unsigned)Up::start.b - 3u * z)), a5 = (int)(t - v3 + ((unsigned)Lo::start.a - z));
    int a4 = (int)(u + v5 + ((unsigned)Up::start.a - z)), a6 = (int)(u - v5 + ((unsigned)Lo::start.b + z));
    const unsigned e0 = v0 + v4 - 2u * z + (unsigned)dc, e1 = v0 - v4 + (unsigned)dc;
    int p = (int)((unsigned)v[2] + ((unsigned)Ev::start.a - z)), q = (int)((unsigned)v[6] + ((unsigned)Ev::start.b - z));
    Ev::run(p, q);                     // e3 = p, e2 = -q (transposed quarter turn)
    Up::run(a4, a7);                   // -> (d3, d0)
    Lo::run(a5, a6);                   // -> (d2, d1)
    // signs and offsets come off: the signs in the additions that follow
    constexpr bool sp = Ev::end.sa > 0, sq = Ev::end.sb > 0;
    constexpr bool s4 = Up::end.sa > 0, s7 = Up::end.sb > 0, s5 = Lo::end.sa > 0, s6 = Lo::end.sb > 0;
    if constexpr (kTrOffsets) {
        p = (int)((unsigned)p - (unsigned)Ev::end.ka);
        q = (int)((unsigned)q - (unsigned)Ev::end.kb);
        a4 = (int)((unsigned)a4 - (unsigned)Up::end.ka);
        a7 = (int)((unsigned)a7 - (unsigned)Up::end.kb);
        a5 = (int)((unsigned)a5 - (unsigned)Lo::end.ka);
        a6 = (int)((unsigned)a6 - (unsigned)Lo::end.kb);
    }
    const unsigned s0 = add_if<sp>(e0, (unsigned)p), s3 = add_if<!sp>(e0, (unsigned)p);
    const unsigned s1 = add_if<!sq>(e1, (unsigned)q), s2 = add_if<sq>(e1, (unsigned)q);
    v[0] = (int)add_if<s7>(s0, (unsigned)a7);
    v[7] = (int)add_if<!s7>(s0, (unsigned)a7);
    v[1] = (int)add_if<s6>(s1, (unsigned)a6);
    v[6] = (int)add_if<!s6>(s1, (unsigned)a6);
    v[2] = (int)add_if<s5>(s2, (unsigned)a5);
    v[5] = (int)add_if<!s5>(s2, (unsigned)a5);
    v[3] = (int)add_if<s4>(s3, (unsigned)a4);
    v[4] = (int)add_if<!s4>(s3, (unsigned)a4);
}

}  // namespace dctgb
