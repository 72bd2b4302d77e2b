// F-engine with the first transform stage on the tensor cores: 4-bit unpack
// -> optional gain/delay -> K-point real FFT -> the corner-turned workspace.
//
// Paper: Sec. 1 (split each stream into channels with an FFT), Sec. 4
// (forward, unnormalised float FFT; conversion of its output before the
// cross-multiply), Sec. 2.1 (a phase applied per stream before accumulation).
//
// K = N1 M, n = M n1 + n2, k = k1 + N1 k2:
//   y[k1][n2] = sum_{n1 < N1} x[M n1 + n2] W_N1^{n1 k1}          (stage 1)
//   X[k]      = sum_{n2 < M} W_M^{n2 k2} (W_K^{n2 k1} y[k1][n2])  (stage 2)
// Stage 1 is a real transform of the samples themselves, N1 x N1 real numbers
// (k1 = 1 .. N1/2 - 1 complex, k1 = 0 and N1/2 real), done by mma.sync
// (m16n8k16): the samples are small integers, exact in FP16, and each matrix
// element is hi + 2^-12 lo with both parts multiples of 2^-11, so every
// product and every sum of a stage-1 accumulator is an exact multiple of
// 2^-11 below 2^21 of them: the tensor core rounds nothing, and
// y = fma(lo, 2^-12, hi) has one rounding.  (The elements are exact to 2^-24.)
// For M >= 16 (K >= 512) stage 1 is folded first: even k1 take x[n1] + x[n1 +
// N1/2], odd k1 the differences (exact, one packed add per pair of MMA
// operands), which halves the matrix and its MMAs; an m-tile then holds k1 of
// one parity.
// Stage 2 is the twiddle and an M-point DFT per k1 on the FP32 pipes.  As y
// comes from the real samples, k1 = 1 .. N1/2 - 1 gives X[k] for k < K/2 (k2 <
// M/2) and conj X[K - k] for the rest: all channels but the multiples of N1/2
// appear without a real-to-complex split.
//
// Fragment layouts make the exchange between the stages free.  Rows of an
// m-tile are Re (row g) and Im (row g + 8) of 8 k1 (k1_of); the 8 columns are
// 8 frames; one MMA set per n2.  A lane (g = lane / 4, c = lane % 4) thus ends
// with y[k1][n2] of frames 2c and 2c + 1 for every n2, in registers: no shared
// memory, no shuffles.  The sample operand wants, per lane, pairs of n1 of one
// frame and n2: two nibbles of equal position in two words, one PRMT and one
// LOP3 away from the packed bytes.  A nibble u = v + 8 becomes the FP16
// subnormal u 2^-24 (or 16 u 2^-24 from a high nibble: odd n2), which the MMA
// takes as it is; the twiddles carry 2^24 (2^20 for odd n2).  The offset of 8
// is the same for every n1 and n2, so it drops out of every row but k1 = 0 (the
// others sum to zero exactly) and, in row k1 = 0, out of every channel
// but X[0]: that row's twiddles are 1 and its first butterflies add and
// subtract integers, so its differences lose the offset exactly before any
// other factor.  X[0] has it subtracted after stage 2.
//
// k1 = 0 and N1/2 share the row pair g = 0 of m-tile 0 as real sequences.  Its
// lanes swap them so that one complex transform holds the k1 = 0 sequences of
// both frames and the other the k1 = N1/2 ones (times W_K^{n2 N1/2}), and
// separate the two frames afterwards from Z[k2] and its mirror, both in the
// lane's registers.
//
// What bounds it: issue slots and register ports -- mma.sync and FP32
// instructions do not overlap fully here (4 HMMA + 32 FFMA per warp take 1.4
// times the longer of the two), so the stage-1 MMAs cost about a quarter of
// the time before the fold -- at 12-16 warps per SM (64 accumulators per
// lane).  190-250 warp instructions per 512 samples (unfolded) against 453 of
// the FP32 radix-16 kernel.
// Measured per pass (GB300, before -> now):
//   K = 256,  N = 64,  16384 frames: FP32 mode 4152 -> 230 us, FP16 4099 -> 179
//             (before: the general radix-2 kernel, one frame at a time);
//   K = 512,  N = 44,  16384 frames: FP16 337 -> 263 us (unfolded 284), FP8
//             344 -> 274 (295; 294 for the first pass of an integration, whose
//             first 3072 frames take the FP32 FFT); FP32 mode 346 against 369
//             here: the FP32 kernel stays there;
//   K = 1024, N = 256, 4096 frames: FP16 1236 -> 960 us (1130), FP8 977 (1062);
//             FP32 mode 1374 against 1449 here, the FP32 kernel stays;
//   K = 2048, N = 64,  4096 frames: FP16 1001 -> 695 us (728), FP8 700 (757),
//             FP32 mode 1124 -> 901 (877).
#include "corr_internal.h"
#include "fengine_k512.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <type_traits>

namespace gbcorr {
namespace {

using namespace fk;

// ------------------------------------------------------ stage-1 matrix (host)

constexpr int round_abs(double v) { return v >= 0.0 ? (int)(v + 0.5) : -(int)(-v + 0.5); }
// FP16 bits of q 2^-11 2^-sh for |q| <= 2048, sh = 0 or 4 (always exact).
constexpr uint32_t half_bits(int q, int sh) {
    uint32_t sign = 0;
    if (q < 0) {
        sign = 0x8000u;
        q = -q;
    }
    if (q == 0) return 0;
    int e = 0;
    while ((2 << e) <= q) ++e;                      // 2^e <= q < 2^(e+1)
    const int ex = e - 11 - sh;                     // exponent of the value
    const uint32_t man = e <= 10 ? (uint32_t)q << (10 - e) : (uint32_t)q >> 1;
    if (ex >= -14) return sign | ((uint32_t)(ex + 15) << 10) | (man & 0x3ffu);
    return sign | ((uint32_t)q << (13 - sh));       // subnormal: q 2^(13 - sh) 2^-24
}

// cos and sin of 2 pi m / K by their Taylor series on [0, pi/4] (20 terms:
// below 1e-17), from an exact integer angle.
constexpr double kPi = 3.14159265358979323846;
constexpr double taylor(double x, bool sine) {
    double t = sine ? x : 1.0, s = t;
    for (int i = sine ? 1 : 0; i < 20; i += 2) {
        t *= -x * x / ((i + 1) * (i + 2));
        s += t;
    }
    return s;
}
constexpr double cos_k(int m, int K) {
    m &= K - 1;
    if (2 * m > K) m = K - m;                        // [0, pi]
    const bool neg = 4 * m > K;
    if (neg) m = K / 2 - m;                          // [0, pi/2]
    const double v = 8 * m <= K ? taylor(2.0 * kPi * m / K, false)
                                : taylor(2.0 * kPi * (K / 4.0 - m) / K, true);
    return neg ? -v : v;
}

// Folded stage 1 (M >= 16): the matrix takes x[n1] + x[n1 + N1/2] for even k1
// and x[n1] - x[n1 + N1/2] for odd k1, half the columns; m-tiles hold k1 of one
// parity.
constexpr bool folded(int M) { return M >= 16; }
// k1 of row g of m-tile mt.
__host__ __device__ constexpr int k1_of(bool fold, int mt, int g) {
    return fold ? 16 * (mt >> 1) + 2 * g + (mt & 1) : 8 * mt + g;
}

// A fragments (row-major m16 x k16) of the stage-1 matrix, per m-tile, k-tile,
// part (hi, lo 2^12) and lane.  PAIR: K = N1 (M = 1), where the two
// samples of a pair come from the two nibbles of one byte and the odd one is
// 16 times larger: its columns are divided by 16.
template <int N1, bool PAIR, bool FOLD>
struct WFrag {
    static constexpr int KT = N1 / 16 / (FOLD ? 2 : 1);
    uint4 v[N1 / 16][KT][2][32];
};

constexpr int w_part(int N1, bool fold, int row16, int mt, int n1, int hl) {
    const int g = row16 & 7, im = row16 >> 3;
    const int k1 = k1_of(fold, mt, g);
    double w = 0.0;
    if (k1 == 0)
        w = im ? ((n1 & 1) ? -1.0 : 1.0) : 1.0;     // k1 = 0 and k1 = N1/2, both real
    else
        w = im ? cos_k(k1 * n1 + N1 / 4, N1) : cos_k(k1 * n1, N1);     // -sin : cos
    const int hi = round_abs(w * 2048.0);
    return hl ? round_abs((w * 2048.0 - hi) * 4096.0) : hi;
}

template <int N1, bool PAIR, bool FOLD>
constexpr WFrag<N1, PAIR, FOLD> make_wfrag() {
    WFrag<N1, PAIR, FOLD> f{};
    for (int mt = 0; mt < N1 / 16; ++mt)
        for (int kt = 0; kt < f.KT; ++kt)
            for (int hl = 0; hl < 2; ++hl)
                for (int lane = 0; lane < 32; ++lane) {
                    uint32_t r[4] = {0, 0, 0, 0};
                    for (int e = 0; e < 4; ++e) {
                        const int row = (lane >> 2) + 8 * (e & 1);
                        const int n1 = 16 * kt + 2 * (lane & 3) + 8 * (e >> 1);
                        r[e] = half_bits(w_part(N1, FOLD, row, mt, n1, hl), 0) |
                               (half_bits(w_part(N1, FOLD, row, mt, n1 + 1, hl), PAIR ? 4 : 0) << 16);
                    }
                    f.v[mt][kt][hl][lane].x = r[0];
                    f.v[mt][kt][hl][lane].y = r[1];
                    f.v[mt][kt][hl][lane].z = r[2];
                    f.v[mt][kt][hl][lane].w = r[3];
                }
    return f;
}

__device__ constexpr auto kW16p = make_wfrag<16, true, false>();
__device__ constexpr auto kW32p = make_wfrag<32, true, false>();
__device__ constexpr auto kW32 = make_wfrag<32, false, false>();
__device__ constexpr auto kW32f = make_wfrag<32, false, true>();
__device__ constexpr auto kW64f = make_wfrag<64, false, true>();

template <int N1, int M>
__device__ __forceinline__ const uint4* wfrag(int mt, int kt, int hl, int lane) {
    if constexpr (M == 1 && N1 == 16) return &kW16p.v[mt][kt][hl][lane];
    else if constexpr (M == 1) return &kW32p.v[mt][kt][hl][lane];
    else if constexpr (N1 == 64) return &kW64f.v[mt][kt][hl][lane];
    else if constexpr (folded(M)) return &kW32f.v[mt][kt][hl][lane];
    else return &kW32.v[mt][kt][hl][lane];
}

// Twiddles [mt][p][j][g]: W_K^{j (k1 + N1 p)}, k1 of the row, as (re a, re b,
// im a, im b) for the lane's two transforms: frames a and b, equal but in the
// special row (m-tile 0, g = 0), whose second transform is k1 = N1/2; times
// 2^24 (2^20 for odd j: high nibbles), half of it in the special row (the
// separation of its two frames).
template <int N1, int M>
struct TwTab {
    static constexpr int MT = N1 / 16, MC = M < 16 ? M : 16, Q = M / MC;
    float4 v[MT][Q * MC * 8];
};
template <int N1, int M>
constexpr TwTab<N1, M> make_tw() {
    using T = TwTab<N1, M>;
    T f{};
    for (int mt = 0; mt < T::MT; ++mt)
        for (int p = 0; p < T::Q; ++p)
            for (int j = 0; j < T::MC; ++j)
                for (int g = 0; g < 8; ++g) {
                    const bool sp = M > 1 && mt == 0 && g == 0;
                    const int k1 = k1_of(folded(M), mt, g);
                    const int ma = j * (k1 + N1 * p);
                    const int mb = j * ((sp ? N1 / 2 : k1) + N1 * p);
                    const double s = ((j & 1) ? 1048576.0 : 16777216.0) * (sp ? 0.5 : 1.0);
                    float4& o = f.v[mt][(p * T::MC + j) * 8 + g];
                    o.x = (float)(s * cos_k(ma, N1 * M));
                    o.y = (float)(s * cos_k(mb, N1 * M));
                    o.z = (float)(s * cos_k(ma + N1 * M / 4, N1 * M));
                    o.w = (float)(s * cos_k(mb + N1 * M / 4, N1 * M));
                }
    return f;
}
template <int N1, int M>
__device__ constexpr TwTab<N1, M> kTw = make_tw<N1, M>();

// ------------------------------------------------------------ device pieces

__device__ __forceinline__ void mma16816(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1,
                                         float c0, float c1, float c2, float c3) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2),
          "f"(c3));
}

__device__ __forceinline__ void stmatrix4(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2,
                                          uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr),
                 "r"(r0), "r"(r1), "r"(r2), "r"(r3)
                 : "memory");
}
__device__ __forceinline__ void stmatrix2(uint32_t addr, uint32_t r0, uint32_t r1) {
    asm volatile("stmatrix.sync.aligned.m8n8.x2.shared.b16 [%0], {%1,%2};" ::"r"(addr), "r"(r0),
                 "r"(r1)
                 : "memory");
}

// half2 (lo half = a)
__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t sub_h2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// The FP32 values minus the FP16 pair rounded from them (exact)
__device__ __forceinline__ float2 minus_h2(float a, float b, uint32_t h) {
    float2 r;
    asm("{.reg .f16 l, u, m;\n mov.b32 {l, u}, %2;\n mov.b16 m, 0xBC00;\n"
        " fma.rn.f32.f16 %0, l, m, %3;\n fma.rn.f32.f16 %1, u, m, %4;}"
        : "=f"(r.x), "=f"(r.y)
        : "r"(h), "f"(a), "f"(b));
    return r;
}

// Complex values of two transforms side by side: re = (re a, re b), im alike.
// Every operation on them is one packed FP32x2 instruction per part.  (The
// FP32 rate of three-operand packed FMAs is lower than of scalar ones here,
// 2.6 against 3.9 lanes' worth per clock and SM, but the register pairs and
// half the issue slots win: K = 256 FP32 mode 230 against 241 us, K = 1024
// FP16 1078 against 1138 us per pass with scalar arithmetic.)
struct C2 {
    float2 re, im;
};
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
    return __ffma2_rn(a, b, c);
}
__device__ __forceinline__ C2 operator+(C2 a, C2 b) { return {vadd(a.re, b.re), vadd(a.im, b.im)}; }
__device__ __forceinline__ C2 operator-(C2 a, C2 b) { return {vsub(a.re, b.re), vsub(a.im, b.im)}; }
__device__ __forceinline__ C2 add_mi(C2 a, C2 b) { return {vadd(a.re, b.im), vsub(a.im, b.re)}; }   // a - i b
__device__ __forceinline__ C2 add_i(C2 a, C2 b) { return {vsub(a.re, b.im), vadd(a.im, b.re)}; }    // a + i b
// a (c - i s)
__device__ __forceinline__ C2 rot(C2 a, float c, float s) {
    return {vfma(f2(s), a.im, vmul(f2(c), a.re)), vfma(f2(-s), a.re, vmul(f2(c), a.im))};
}
// a (x + i y)
__device__ __forceinline__ C2 mul(C2 a, float2 x, float2 y) {
    return {vfma(a.re, x, vmul(a.im, make_float2(-y.x, -y.y))), vfma(a.re, y, vmul(a.im, x))};
}

// 4-point forward DFT in place; MI: x2 stands for -i x2; CONJ: the outputs
// x2 and x3 are conjugated.
template <bool MI, bool CONJ>
__device__ __forceinline__ void dft4p(C2& x0, C2& x1, C2& x2, C2& x3) {
    const C2 t0 = MI ? add_mi(x0, x2) : x0 + x2, t1 = MI ? add_i(x0, x2) : x0 - x2;
    const C2 t2 = x1 + x3, d = x1 - x3;
    x0 = t0 + t2;
    x1 = add_mi(t1, d);
    x2 = {vsub(t0.re, t2.re), CONJ ? vsub(t2.im, t0.im) : vsub(t0.im, t2.im)};
    x3 = {vsub(t1.re, d.im), vadd(t1.im, d.re)};
    if (CONJ) x3.im = make_float2(-x3.im.x, -x3.im.y);
}

// M-point forward DFT in registers, natural order in and out; the upper half
// of the outputs conjugated (M > 1).
template <int M>
__device__ __forceinline__ void dftp(C2 (&x)[M]) {
    constexpr float c8 = 0.923879532511286756f, s8 = 0.382683432365089772f;   // pi/8
    constexpr float r2 = 0.707106781186547524f;
    if constexpr (M == 16) {
        // radix 4 x 4: columns j2, twiddles W16^{j2 m1}, rows m1
#pragma unroll
        for (int j2 = 0; j2 < 4; ++j2) dft4p<false, false>(x[j2], x[4 + j2], x[8 + j2], x[12 + j2]);
        x[5] = rot(x[5], c8, s8);
        x[6] = rot(x[6], r2, r2);
        x[7] = rot(x[7], s8, c8);
        x[9] = rot(x[9], r2, r2);
        x[11] = rot(x[11], -r2, r2);
        x[13] = rot(x[13], s8, c8);
        x[14] = rot(x[14], -r2, r2);
        x[15] = rot(x[15], -c8, -s8);
        dft4p<false, true>(x[0], x[1], x[2], x[3]);
        dft4p<false, true>(x[4], x[5], x[6], x[7]);
        dft4p<true, true>(x[8], x[9], x[10], x[11]);       // x[10] W16^4 = -i x[10]
        dft4p<false, true>(x[12], x[13], x[14], x[15]);
        // x[4 m1 + m2] holds X[m1 + 4 m2]
        C2 y[16];
#pragma unroll
        for (int m1 = 0; m1 < 4; ++m1)
#pragma unroll
            for (int m2 = 0; m2 < 4; ++m2) y[m1 + 4 * m2] = x[4 * m1 + m2];
#pragma unroll
        for (int q = 0; q < 16; ++q) x[q] = y[q];
    } else if constexpr (M == 8) {
        // radix 2 x 4: E from the even, O from the odd points
        dft4p<false, false>(x[0], x[2], x[4], x[6]);
        dft4p<false, false>(x[1], x[3], x[5], x[7]);
        const C2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
        const C2 o0 = x[1], o1 = rot(x[3], r2, r2), o2 = x[5], o3 = rot(x[7], -r2, r2);
        x[0] = e0 + o0;
        x[1] = e1 + o1;
        x[2] = add_mi(e2, o2);
        x[3] = e3 + o3;
        x[4] = {vsub(e0.re, o0.re), vsub(o0.im, e0.im)};
        x[5] = {vsub(e1.re, o1.re), vsub(o1.im, e1.im)};
        x[6] = add_i(e2, o2);
        x[6].im = make_float2(-x[6].im.x, -x[6].im.y);
        x[7] = {vsub(e3.re, o3.re), vsub(o3.im, e3.im)};
    } else if constexpr (M == 4) {
        dft4p<false, true>(x[0], x[1], x[2], x[3]);
    } else if constexpr (M == 2) {
        const C2 a = x[0], b = x[1];
        x[0] = a + b;
        x[1] = {vsub(a.re, b.re), vsub(b.im, a.im)};
    }
}

// lop3 (t & m) ^ x with the mask in a register: written as C, the compiler
// makes two instructions with immediates of it.
__device__ __forceinline__ uint32_t and_xor(uint32_t t, uint32_t m, uint32_t x) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x6a;" : "=r"(r) : "r"(t), "r"(m), "r"(x));
    return r;
}
__device__ __forceinline__ uint32_t reg_const(uint32_t v) {
    uint32_t r;
    asm volatile("mov.b32 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
// Shared-memory loads kept where they are written: hoisted, the twiddles of a
// whole transform would need 60 registers at once.
__device__ __forceinline__ uint4 lds128(const void* p) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(tc::smem_u32(p)));
    return v;
}
__device__ __forceinline__ uint2 lds64(const void* p) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(tc::smem_u32(p)));
    return v;
}
__device__ __forceinline__ float4 lds128f(const void* p) {
    const uint4 v = lds128(p);
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}
// 16 bytes global -> shared; zeros when !valid
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}

constexpr int kMmaThreads = 128;    // 4 warps of 8 frames: one 32-frame block
constexpr int kMmaFrames = 32;

template <int N1, int M, int MTC>
struct MmaShape {
    static constexpr int K = N1 * M, C = K / 2;
    static constexpr int MT = N1 / 16;               // m-tiles (8 values of k1 each)
    static constexpr int MTG = MT / MTC;             // CTAs that share a block's m-tiles
    static constexpr int KB = 8 * MTC;               // adjacent channels of a slot in a CTA
    static constexpr int H = M > 1 ? M / 2 : 1;      // slots of a half (k < K/2; the conjugated ones)
    static constexpr int HV = M > 1 ? 2 : 1;         // halves
    static constexpr int ROWS = M * KB;              // channels per antenna of a CTA
    static constexpr int MC = M < 16 ? M : 16;       // points of the in-register DFT
    static constexpr int Q = M / MC;                 // radix step before it (M = 32: 2)
    static constexpr int TW = MTC * Q * MC * 8;      // twiddles per antenna
    static constexpr bool kFold = folded(M);         // half the matrix columns
    static constexpr int KT = N1 / 16 / (kFold ? 2 : 1);
    static constexpr bool kAsync = K >= 512;         // samples through shared memory
    static constexpr int kRaw = kAsync ? K / 2 : 0;  // bytes of a frame in the sample buffer
    static constexpr int row_bytes(int out) {        // a channel's Re and Im, 32 frames, one plane
        return out == SPEC_F32 ? 256 : (out == SPEC_F8 ? 64 : (out == kOutDebug ? 0 : 128));
    }
    // Bytes of a slot of the conjugated half for m-tile 0 alone (part7, part1):
    // the box of the k1 = N1/2 channel starts on a 128-byte boundary, as a TMA
    // box must, so FP8's 64-byte channels leave one place free before it.
    static constexpr int split_slot(int out) { return out == SPEC_F8 ? 640 : KB * row_bytes(out); }
    static constexpr int unit_bytes(int out) {       // staging of an antenna
        return (out == SPEC_F16X2 ? 2 : 1) *
               (H * KB * row_bytes(out) + (HV > 1 ? H * (MTG > 1 ? split_slot(out) : KB * row_bytes(out)) : 0));
    }
    static size_t smem(int out, bool corr, int an, int ns) {
        const size_t rows = (size_t)ROWS * an;
        return (out == kOutDebug ? 0 : 1024) + (size_t)ns * an * unit_bytes(out) +
               kMmaFrames * kRaw + ((size_t)an * TW + MTC * KT * 64) * sizeof(float4) + (corr ? rows * sizeof(float4) : 0) +
               (out == SPEC_F16 || out == SPEC_F8 ? rows * sizeof(float2) : 0);
    }
};

// Channel of slot k2 and row g: k1 + N1 k2 below K/2, and for the upper slots,
// which hold conj X[K - k], K - k (the k1 = N1/2 channels in the special row).
template <int N1, int M>
__device__ __forceinline__ int mma_channel(int mt, int k2, int g) {
    const int k1 = k1_of(folded(M), mt, g);
    if (M == 1 || k2 < M / 2) return k1 + N1 * k2;
    return N1 * (M - k2) - (k1 == 0 ? N1 / 2 : k1);
}

// Output tensor maps of the workspace, five dimensions: the frames of a tile
// (FP16: of an antenna's Re and Im rows, adjacent in memory), rows (FP16:
// antennas), channel mod N1, channel / N1, tile (the lo plane's follow the hi
// plane's).  full: KB channels x the H slots of a half; for a CTA that holds
// m-tile 0 alone the conjugated half has 7 adjacent channels and the k1 = N1/2
// one apart (part7, part1; one slot each).
struct OutMaps {
    CUtensorMap full, odd, part7, part1;
};

// Units of work: 32-frame blocks of AN antennas, all m-tiles (M < 16) or one.
// Persistent CTAs take contiguous ranges of an antenna's frame blocks, so the
// tables and matrix fragments are loaded once or twice per launch, and the
// next unit's samples are fetched while this one is transformed.  The CTAs
// with one range's different m-tiles share its samples through L2.  Results
// are staged in shared memory and written by TMA: one instruction per 8 KB
// instead of the address arithmetic, loads and stores of a store phase.
template <int N1, int M, int MTC, int OUT, bool CORR, int MINB, int NS>
__global__ void __launch_bounds__(kMmaThreads, MINB)
fengine_mma(const __grid_constant__ FengineArgs a, const __grid_constant__ OutMaps maps, int AN,
            int nfb, int64_t units) {
    using Sh = MmaShape<N1, M, MTC>;
    constexpr int K = Sh::K, C = Sh::C, KT = Sh::KT, MC = Sh::MC, Q = Sh::Q, KB = Sh::KB;
    constexpr int NB = N1 / 8;                         // sample pairs per lane and n2
    constexpr bool kFold = Sh::kFold;
    constexpr bool DEBUG = OUT == kOutDebug;
    constexpr bool kScaled = OUT == SPEC_F16 || OUT == SPEC_F8;
    constexpr bool kAsync = Sh::kAsync;
    constexpr int kRowB = Sh::row_bytes(OUT), kRaw = Sh::kRaw;
    constexpr int kPlanes = OUT == SPEC_F16X2 ? 2 : 1;
    constexpr int kHalfB = Sh::H * KB * kRowB;         // bytes of a half's box
    constexpr int kUnitB = Sh::unit_bytes(OUT);        // of an antenna
    extern __shared__ __align__(128) unsigned char smem_raw[];

    const int tid = threadIdx.x;
    const int lane = tid & 31, w = tid >> 5;
    const int g = lane >> 2, c = lane & 3;
    const int mt0 = (int)(blockIdx.x % Sh::MTG) * MTC;
    const unsigned G = gridDim.x / Sh::MTG, bx = blockIdx.x / Sh::MTG;
    const int64_t u_end = units * (bx + 1) / G;
    int64_t un = units * bx / G;                       // unit = antenna group * nfb + frame block
    if (un >= u_end) return;

    // staging ([antenna][plane][half][slot][channel], the boxes of the output
    // maps), the sample buffer, and per antenna of the group the twiddles
    // (times its pre-scale), corrections and scales in slot order
    const int rows = AN * Sh::ROWS;
    // (aligned by an offset: a rounded pointer would lose its address space)
    unsigned char* smem = smem_raw + (DEBUG ? 0u : (0u - tc::smem_u32(smem_raw)) & 1023u);
    unsigned char* raw = smem + (size_t)NS * AN * kUnitB;
    float4* tw = reinterpret_cast<float4*>(raw + kMmaFrames * kRaw);
    float4* corr_tab = tw + AN * Sh::TW + MTC * KT * 64;   // (re, re, im, im)
    float2* sc_tab = reinterpret_cast<float2*>(corr_tab + (CORR ? rows : 0));   // (s, s)
    const uint32_t stg0 = tc::smem_u32(smem);
    const int wu = __shfl_sync(0xffffffffu, w, 0);     // warp index, uniform
    const int lo_tile = kPlanes == 2 ? (int)(a.plane_stride / ((int64_t)C * 2 * a.N) >> 5) : 0;
    const bool split = Sh::MTG > 1 && mt0 == 0;        // conjugated half as part7 + part1 (M >= 16)
    // Position of row r (= g) of m-tile ml among the KB channels of a slot, and
    // in the conjugated half, which runs backwards: with all m-tiles in the
    // CTA k1 = N1/2 comes first, with m-tile 0 alone last (part1).
    auto pos_up = [](int ml, int r) { return 8 * ml + r; };
    auto pos_dn = [](int ml, int r) { return Sh::MTG == 1 ? (KB - 8 * ml - r) & (KB - 1) : 7 - r; };

    // Packed samples of the lane's frame (as an operand column): for each pair
    // (n1, n1 + 1), n1 = 8 b + 2 c, and n2 = 16 q .. 16 q + 15, words X and Z.
    // M >= 16: the warp's 8 frames go through its own rows of the sample
    // buffer (cp.async: no registers held while in flight); shorter
    // transforms load their few words directly.
    uint32_t X[NB][2], Z[NB][2];
    const int fstride = a.N * (K / 2);                 // bytes from one frame's record to the next
    constexpr int kFL = K == 512 ? 16 : 32;            // lanes per frame of a 512-byte fetch step
    auto lane_src = [&](int64_t s, int i) {            // records of frame s .. of antenna i
        const uint8_t* p = a.in + (s + 8 * w) * fstride + (int64_t)i * (K / 2);
        return kAsync ? p + (lane / kFL) * fstride + (lane % kFL) * 16 : p + g * fstride + c * M;
    };
    // 16-byte chunks of a frame are XOR-ed so that the lanes of a take() spread
    // over the banks
    auto raw_xor = [](int f) { return M == 16 ? (f & 1) << 2 : f & 1; };
    auto fetch = [&](const uint8_t* p, int nv) {   // nv: valid frames of the block
        if constexpr (kAsync) {
            const uint32_t wraw_s = tc::smem_u32(raw + 8 * w * kRaw);
#pragma unroll
            for (int e = 0; e < K / 128; ++e) {        // 8 frames of K/2 bytes, 512 bytes a step
                const int f = 32 * e / (K / 32), b = 32 * e % (K / 32);
                const bool v = 8 * w + f + lane / kFL < nv;
                const int fl = f + lane / kFL;
                cp_async16z(wraw_s + fl * kRaw + 16 * ((b + lane % kFL) ^ raw_xor(fl)),
                            v ? p + f * fstride + 16 * b : a.in, v);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        } else {
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                X[b][0] = Z[b][0] = 0u;
                const uint8_t* r = p + 4 * M * b;
                if (8 * w + g < nv) {
                    if constexpr (M == 8) {
                        const uint2 x = __ldg(reinterpret_cast<const uint2*>(r));
                        X[b][0] = x.x, Z[b][0] = x.y;
                    } else if constexpr (M == 4) {
                        X[b][0] = __ldg(reinterpret_cast<const uint32_t*>(r));
                    } else if constexpr (M == 2) {
                        X[b][0] = __ldg(reinterpret_cast<const unsigned short*>(r));
                    } else {
                        X[b][0] = __ldg(r);
                    }
                }
            }
        }
    };
    auto take = [&](int n8) {                          // words of n2 = 8 n8 .. from the sample buffer
        const unsigned char* p0 = raw + (8 * w + g) * kRaw;
        const int sw = raw_xor(g);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if constexpr (M == 32) {
                const int ch = 2 * (4 * b + c);
                const uint2 x = lds64(p0 + 16 * (ch ^ sw) + 4 * n8);
                const uint2 z = lds64(p0 + 16 * ((ch + 1) ^ sw) + 4 * n8);
                X[b][0] = x.x, X[b][1] = x.y, Z[b][0] = z.x, Z[b][1] = z.y;
            } else {
                const uint4 x = lds128(p0 + 16 * ((4 * b + c) ^ sw));
                X[b][0] = x.x, X[b][1] = x.y, Z[b][0] = x.z, Z[b][1] = x.w;
            }
        }
    };

    static_assert(MTC <= 2 && (MTC == 1 || MTC == N1 / 16), "m-tiles of a CTA: one, or both");
    static_assert(kFold == (Sh::MTG > 1) && kFold == kAsync, "one m-tile per CTA: folded");
    uint4* wtab = reinterpret_cast<uint4*>(tw + AN * Sh::TW);   // [m-tile][kt][hi, lo][lane]
    for (int e = tid; e < MTC * KT * 64; e += kMmaThreads)
        wtab[e] = __ldg(wfrag<N1, M>(mt0, 0, 0, 0) + e);
    const uint32_t mlo = reg_const(0x000F000Fu), mhi = reg_const(0x00F000F0u);

    int ag = (int)(un / nfb);
    int fb = (int)(un - (int64_t)ag * nfb);
    int tab = -1;                                      // antenna group of the tables
    auto valid_frames = [&](int b) { return (int)min((int64_t)kMmaFrames, a.S - (int64_t)b * kMmaFrames); };
    const uint8_t* src = lane_src((int64_t)fb * kMmaFrames, ag * AN);
    fetch(src, valid_frames(fb));
    __syncthreads();                                   // the matrix fragments
    int sb = 0;                                        // staging buffer of this unit

#pragma unroll 1
    for (; un < u_end; ++un) {
        const int i0 = ag * AN;
        const int an = kAsync ? 1 : min(AN, a.N - i0);
        unsigned char* stg_p = smem + (NS > 1 ? sb * AN * kUnitB : 0);
        const uint32_t stg = stg0 + (NS > 1 ? sb * AN * kUnitB : 0);
        if (tab != ag) {
            __syncthreads();                           // nobody reads the old tables
            tab = ag;
            for (int ai = 0; ai < an; ++ai) {
                const float post = OUT == SPEC_F16X2 ? __ldg(a.split + i0 + ai) : 1.0f;
                const float4* t0 = &kTw<N1, M>.v[mt0][0];
                for (int e = tid; e < Sh::TW; e += kMmaThreads) {
                    const float4 t = __ldg(t0 + e);
                    tw[ai * Sh::TW + e] = OUT == SPEC_F16X2 ? make_float4(t.x * post, t.y * post, t.z * post, t.w * post) : t;
                }
            }
            if (CORR || kScaled)
                for (int e = tid; e < an * Sh::ROWS; e += kMmaThreads) {
                    const int ai = e / Sh::ROWS, r = e - ai * Sh::ROWS;
                    const int k = mma_channel<N1, M>(mt0 + r / (8 * M), (r >> 3) % M, r & 7);
                    if (CORR) {
                        const float2 t = __ldg(a.corr + (int64_t)(i0 + ai) * C + k);
                        corr_tab[e] = make_float4(t.x, t.x, t.y, t.y);
                    }
                    if (kScaled) sc_tab[e] = f2(__ldg(a.scale + (int64_t)(i0 + ai) * C + k));
                }
        }
        bool fresh = true;                             // nothing staged in this unit yet

        // One m-tile of one antenna; SP: m-tile 0, whose row g = 0 is special.
        // ODD (folded): k1 odd.
        auto unit = [&](auto sp, auto odd, int ml, int ai) {
                constexpr bool SP = decltype(sp)::value;
                [[maybe_unused]] constexpr bool ODD = decltype(odd)::value;
                [[maybe_unused]] const int mt = SP ? 0 : mt0 + ml;
                const bool special = SP && g == 0;
                if constexpr (kAsync) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                }
                // ------------ stage 1: y[n2] of frames 2c (a) and 2c + 1 (b)
                uint4 W[2][KT];                        // the m-tile's matrix fragments
#pragma unroll
                for (int kt = 0; kt < KT; ++kt) {
                    W[0][kt] = lds128(wtab + ((ml * KT + kt) * 2) * 32 + lane);
                    W[1][kt] = lds128(wtab + ((ml * KT + kt) * 2 + 1) * 32 + lane);
                }
                C2 y[M];
#pragma unroll
                for (int n2 = 0; n2 < M; ++n2) {
                    const int j = n2 & 15;
                    if (kAsync && j == 0) take(n2 >> 3);
                    uint32_t B[NB];
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        uint32_t t;
                        [[maybe_unused]] const int by = (j & 7) >> 1;
                        if constexpr (M >= 8)
                            t = __byte_perm(X[b][j >> 3], Z[b][j >> 3], 0x4400 + 0x1111 * by);
                        else if constexpr (M == 4)
                            t = __byte_perm(X[b][0], 0u, 0x2200 + 0x1111 * by);
                        else if constexpr (M == 2)
                            t = __byte_perm(X[b][0], 0u, 0x1100);
                        else
                            t = X[b][0] * 0x00010001u;
                        if (M == 1)
                            B[b] = (t & 0x00F0000Fu) ^ 0x00800008u;
                        else if (j & 1)
                            B[b] = and_xor(t, mhi, 0x00800080u);
                        else
                            B[b] = and_xor(t, mlo, 0x00080008u);
                    }
                    if constexpr (kFold) {             // exact: subnormals add as integers
#pragma unroll
                        for (int b = 0; b < NB / 2; ++b)
                            B[b] = ODD ? sub_h2(B[b], B[b + NB / 2]) : B[b] + B[b + NB / 2];
                    }
                    float h[4], l[4];
                    mma16816(h, W[0][0], B[0], B[1], 0.f, 0.f, 0.f, 0.f);
                    mma16816(l, W[1][0], B[0], B[1], 0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int kt = 1; kt < KT; ++kt) {
                        mma16816(h, W[0][kt], B[2 * kt], B[2 * kt + 1], h[0], h[1], h[2], h[3]);
                        mma16816(l, W[1][kt], B[2 * kt], B[2 * kt + 1], l[0], l[1], l[2], l[3]);
                    }
                    constexpr float e12 = 1.0f / 4096.0f;
                    y[n2].re = vfma(make_float2(l[0], l[1]), f2(e12), make_float2(h[0], h[1]));
                    y[n2].im = vfma(make_float2(l[2], l[3]), f2(e12), make_float2(h[2], h[3]));
                }
                // the next samples, in flight during stage 2
                if (kAsync) __syncwarp();
                if (ai + 1 < an)
                    fetch(src + (ai + 1) * (K / 2), valid_frames(fb));
                else if (ml + 1 < MTC)
                    fetch(src, valid_frames(fb));
                else if (un + 1 < u_end)
                    fetch(fb + 1 < nfb ? src + kMmaFrames * (int64_t)fstride : lane_src(0, (ag + 1) * AN),
                          valid_frames(fb + 1 < nfb ? fb + 1 : 0));
                if (fresh) {                           // the tables are there, the staging is free
                    if (!DEBUG) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(NS - 1) : "memory");
                    __syncthreads();
                    fresh = false;
                }

                // ------------ stage 2
                if constexpr (SP) {
                    // row g = 0: frames a and b of k1 = 0 become the parts of
                    // transform a, those of k1 = N1/2 of transform b; with
                    // M = 1 the latter is the dropped Nyquist term
                    if (special) {
#pragma unroll
                        for (int n = 0; n < M; ++n) {
                            if (M == 1) {
                                y[n].im = f2(0.f);
                            } else {
                                const float t = y[n].re.y;
                                y[n].re.y = y[n].im.x;
                                y[n].im.x = t;
                            }
                        }
                    }
                }
                const float4* tm = tw + (ai * MTC + ml) * (Q * MC * 8) + g;
                if constexpr (Q == 2) {
                    // radix 2 over n2 and n2 + 16 (p = k2 mod 2)
                    const float2 pa = __ldg(a.twiddle + ((16 * k1_of(kFold, mt, g)) & (K - 1)));
                    const float2 pb = SP && special ? __ldg(a.twiddle + ((16 * (N1 / 2)) & (K - 1))) : pa;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const C2 t = mul(y[16 + j], make_float2(pa.x, pb.x), make_float2(pa.y, pb.y));
                        y[16 + j] = y[j] - t;
                        y[j] = y[j] + t;
                    }
                }
                C2 x[M];
#pragma unroll
                for (int p = 0; p < Q; ++p) {
                    C2 v[MC];
                    const float4 t0 = lds128f(tm + p * MC * 8);    // j = 0
                    v[0] = {vmul(y[16 * p].re, make_float2(t0.x, t0.y)),
                            vmul(y[16 * p].im, make_float2(t0.x, t0.y))};
#pragma unroll
                    for (int j = 1; j < MC; ++j) {
                        const float4 t = lds128f(tm + (p * MC + j) * 8);
                        v[j] = mul(y[16 * p + j], make_float2(t.x, t.y), make_float2(t.z, t.w));
                    }
                    dftp<MC>(v);
#pragma unroll
                    for (int m = 0; m < MC; ++m) x[p + Q * m] = v[m];
                }
                // x[k2] for k2 < M/2, conj x[k2] above
                if (SP && special) {
                    // transform a = DFT of (frame a + i frame b) for k1 = 0, b
                    // the same for k1 = N1/2 (halved by the twiddles): separate
                    // the frames; X[0] loses the samples' offset of 8
                    const float dc = tm[0].x * (8.0f * K * (M > 1 ? 2 : 1) / 16777216.0f);
                    if constexpr (M > 1) {
                        float2 hold = make_float2(x[0].re.x, -x[0].im.x);   // conj of transform a's mirror
#pragma unroll
                        for (int k2 = 0; k2 < M / 2; ++k2) {
                            C2& lo = x[k2];
                            C2& up = x[M - 1 - k2];
                            const float2 z1 = make_float2(lo.re.x, lo.im.x), m1 = hold;
                            const float2 z2 = make_float2(up.re.y, up.im.y), m2 = make_float2(lo.re.y, lo.im.y);
                            hold = make_float2(up.re.x, up.im.x);
                            lo.re = make_float2(z1.x + m1.x, z1.y - m1.y);
                            lo.im = make_float2(z1.y + m1.y, m1.x - z1.x);
                            up.re = make_float2(z2.x + m2.x, m2.y - z2.y);
                            up.im = make_float2(z2.y + m2.y, z2.x - m2.x);
                        }
                    }
                    x[0].re = make_float2(x[0].re.x - dc, x[0].re.y - dc);
                }

                // ------------ corrections, scales, conversion and staging
                const int row0 = (ai * MTC + ml) * M * 8;  // tables: [antenna][m-tile][slot][g]
                unsigned char* ust = stg_p + ai * kUnitB;
                // stmatrix: this lane addresses row lane % 8 of matrix lane / 8.
                // A channel's 128 bytes are [plane][32 frames] in 16-byte
                // chunks, XOR-ed by the 128-byte line mod 8 (the maps' swizzle)
                const int mi = lane >> 3, mg = lane & 7;
                const int step = OUT == SPEC_F16X2 ? kUnitB / 2 : (M > 2 ? KB * 128 : 0);   // mi >> 1
                const uint32_t chunk = (mi & 1) * 4 + w;
                const uint32_t up = stg + ai * kUnitB + pos_up(ml, mg) * 128 +
                                    ((chunk ^ (pos_up(ml, mg) & 7)) << 4) + (mi >> 1) * step;
                const uint32_t dn = stg + ai * kUnitB + kHalfB + pos_dn(ml, mg) * 128 +
                                    ((chunk ^ (pos_dn(ml, mg) & 7)) << 4) +
                                    (mi >> 1) * (OUT == SPEC_F16X2 ? step : -step);
                const int pu = pos_up(ml, g);
                const int pd = pos_dn(ml, g) + (OUT == SPEC_F8 && SP && Sh::MTG > 1 && g == 0 ? 1 : 0);
                constexpr int dslot = SP && Sh::MTG > 1 ? Sh::split_slot(OUT) : KB * kRowB;
#pragma unroll
                for (int k2 = 0; k2 < M; ++k2) {
                    const bool desc = M > 1 && k2 >= M / 2;
                    [[maybe_unused]] const int slot = desc ? M - 1 - k2 : k2;   // within its half
                    if (CORR) {
                        const float4 t = corr_tab[row0 + 8 * k2 + g];
                        x[k2] = mul(x[k2], make_float2(t.x, t.y), make_float2(t.z, t.w));
                    }
                    if (kScaled) {
                        const float2 s = sc_tab[row0 + 8 * k2 + g];
                        x[k2] = {vmul(x[k2].re, s), vmul(x[k2].im, s)};
                    }
                    const float2 R = x[k2].re, I = x[k2].im;
                    if constexpr (DEBUG) {
                        const int64_t s = (int64_t)fb * kMmaFrames + 8 * w + 2 * c;
                        float2* o = a.debug_out + ((int64_t)(i0 + ai) * a.S + s) * C + mma_channel<N1, M>(mt, k2, g);
                        if (s < a.S) o[0] = make_float2(R.x, I.x);
                        if (s + 1 < a.S) o[C] = make_float2(R.y, I.y);
                    } else if constexpr (OUT == SPEC_F16X2) {
                        // matrices (Re hi, Im hi, Re lo, Im lo)
                        const uint32_t hr = pack_h2(R.x, R.y), hm = pack_h2(I.x, I.y);
                        const float2 lr = minus_h2(R.x, R.y, hr), lm = minus_h2(I.x, I.y, hm);
                        stmatrix4((desc ? dn : up) + slot * KB * 128, hr, hm, pack_h2(lr.x, lr.y),
                                  pack_h2(lm.x, lm.y));
                    } else if constexpr (OUT == SPEC_F16) {
                        if (M <= 2) {
                            stmatrix2((desc ? dn : up) + slot * KB * 128, pack_h2(R.x, R.y), pack_h2(I.x, I.y));
                        } else if (k2 & 1) {               // with the slot before it
                            const C2 o = x[k2 - 1];
                            stmatrix4((desc ? dn + (slot + 1) * KB * 128 : up + (slot - 1) * KB * 128),
                                      pack_h2(o.re.x, o.re.y), pack_h2(o.im.x, o.im.y),
                                      pack_h2(R.x, R.y), pack_h2(I.x, I.y));
                        }
                    } else {
                        // FP32: [Re, Im] lines of 32 frames, 128-byte swizzle;
                        // FP8: [Re, Im] of 32 bytes, 32-byte swizzle
                        if constexpr (OUT == SPEC_F32) {
                            const int r = (desc ? pd : pu) + slot * KB;
                            unsigned char* d = ust + (desc ? kHalfB : 0) + r * kRowB;
                            const int ch = 2 * w + (c >> 1);
                            d += 8 * (c & 1);
                            *reinterpret_cast<float2*>(d + ((ch ^ ((2 * r) & 7)) << 4)) = R;
                            *reinterpret_cast<float2*>(d + 128 + ((ch ^ ((2 * r + 1) & 7)) << 4)) = I;
                        } else {
                            const int o = desc ? kHalfB + slot * dslot + pd * 64 : (slot * KB + pu) * 64;
                            unsigned char* d = ust + o + (((w >> 1) ^ ((o >> 7) & 1)) << 4) + 8 * (w & 1) + 2 * c;
                            *reinterpret_cast<__nv_fp8x2_storage_t*>(d) =
                                __nv_cvt_float2_to_fp8x2(R, __NV_SATFINITE, __NV_E4M3);
                            *reinterpret_cast<__nv_fp8x2_storage_t*>(d + 32) =
                                __nv_cvt_float2_to_fp8x2(I, __NV_SATFINITE, __NV_E4M3);
                        }
                    }
                }
        };
        if constexpr (MTC == 1) {
            for (int ai = 0; ai < an; ++ai) {
                if (mt0 == 0)
                    unit(std::true_type{}, std::false_type{}, 0, ai);
                else if (kFold && (mt0 & 1))
                    unit(std::false_type{}, std::bool_constant<kFold>{}, 0, ai);
                else if (!kFold || Sh::MT > 2)
                    unit(std::false_type{}, std::false_type{}, 0, ai);
            }
        } else {
#pragma unroll 1
            for (int ai = 0; ai < an; ++ai) unit(std::true_type{}, std::false_type{}, 0, ai);
#pragma unroll 1
            for (int ai = 0; ai < an; ++ai) unit(std::false_type{}, std::false_type{}, 1, ai);
        }
        if constexpr (!DEBUG) {
            // the staged boxes go out by TMA, one lane of each warp issuing
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (tc::elect_one()) {
                constexpr int tsh = OUT == SPEC_F8 ? 7 : 5;
                const int64_t s = a.s_base + (int64_t)fb * kMmaFrames;
                const int tile = (int)(s >> tsh), x = (int)(s & ((1 << tsh) - 1));
                for (int e = wu; e < an * kPlanes * Sh::HV; e += 4) {
                    const int half = e % Sh::HV, pl = e / Sh::HV % kPlanes, ai = e / (kPlanes * Sh::HV);
                    const uint32_t sm = stg + ai * kUnitB + pl * (kUnitB / kPlanes) + half * kHalfB;
                    const int row = OUT == SPEC_F16X2 || OUT == SPEC_F16 ? i0 + ai : 2 * (i0 + ai);
                    const int t = tile + pl * lo_tile;
                    // (folded: maps of every second channel)
                    const CUtensorMap* full = kFold && (mt0 & 1) ? &maps.odd : &maps.full;
                    if (half == 0)
                        tc::tma_store_5d(full, sm, x, row, kFold ? 8 * (mt0 >> 1) : 8 * mt0, 0, t);
                    else if (!split)
                        tc::tma_store_5d(full, sm, x, row,
                                         kFold ? N1 / 2 - 7 - 8 * (mt0 >> 1) - (mt0 & 1) : N1 / 2, 0, t);
                    else
                        for (int sl = 0; sl < Sh::H; ++sl) {
                            const uint32_t ss = sm + sl * Sh::split_slot(OUT);
                            tc::tma_store_5d(&maps.part7, ss, x, row, N1 / 2 - 7, sl, t);
                            tc::tma_store_5d(&maps.part1, ss + (OUT == SPEC_F8 ? 512 : 7 * kRowB), x, row, N1 / 4, sl, t);
                        }
                }
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
        if (NS > 1) sb ^= 1;
        src += kMmaFrames * (int64_t)fstride;
        if (++fb == nfb) {
            fb = 0;
            ++ag;
            src = lane_src(0, ag * AN);
        }
    }
    if (!DEBUG) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// The output maps of a launch (see OutMaps).
template <int N1, int M, int MTC>
cudaError_t make_maps(const FengineArgs& a, OutMaps& m) {
    using Sh = MmaShape<N1, M, MTC>;
    if (!tc::get_encoder()) return cudaErrorNotSupported;
    const bool pairs = a.spec_type == SPEC_F16X2 || a.spec_type == SPEC_F16;
    const int eb = spec_elem_bytes(a.spec_type);
    const cuuint64_t T = (cuuint64_t)1 << spec_tile_shift(a.spec_type);
    const cuuint64_t rowb = 2 * (cuuint64_t)a.N * T * eb;        // one channel
    const cuuint64_t tiles = spec_planes(a.spec_type) == 2
                                 ? 2 * (cuuint64_t)(a.plane_stride / ((int64_t)Sh::C * 2 * a.N)) / T
                                 : ((cuuint64_t)(a.s_base + a.S_pad) + T - 1) / T;
    const cuuint64_t dims[5] = {pairs ? 2 * T : T, pairs ? (cuuint64_t)a.N : 2 * (cuuint64_t)a.N,
                                (cuuint64_t)(M == 1 || Sh::kFold ? N1 / 2 : N1), (cuuint64_t)Sh::H, tiles};
    const cuuint64_t str[4] = {(pairs ? 2 : 1) * T * eb, (Sh::kFold ? 2 : 1) * rowb, N1 * rowb, Sh::C * rowb};
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const CUtensorMapDataType dt = eb == 4   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : eb == 2 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                             : CU_TENSOR_MAP_DATA_TYPE_UINT8;
    const CUtensorMapSwizzle sw = eb == 1 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_128B;
    auto enc = [&](CUtensorMap& t, cuuint32_t nch, cuuint32_t nsl, cuuint64_t first = 0) {
        const cuuint32_t box[5] = {pairs ? 64u : 32u, pairs ? 1u : 2u, nch, nsl, 1};
        return tc::get_encoder()(&t, dt, 5, static_cast<char*>(a.spec) + first, dims, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                                 CU_TENSOR_MAP_L2_PROMOTION_NONE,
                                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    bool ok = enc(m.full, Sh::KB, Sh::H);
    if (Sh::kFold) ok = ok && enc(m.odd, Sh::KB, Sh::H, rowb) && enc(m.part7, 7, 1) && enc(m.part1, 1, 1);
    return ok ? cudaSuccess : cudaErrorInvalidValue;
}

// NARROW: only the FP16 and FP8 outputs.
template <int N1, int M, int MTC, int MINB, int NS, bool NARROW>
cudaError_t launch_shape(const FengineArgs& a, cudaStream_t st) {
    using Sh = MmaShape<N1, M, MTC>;
    const bool dbg = a.debug_out != nullptr;
    const int64_t fr = dbg ? a.S : a.S_pad;
    if (fr <= 0) return cudaSuccess;
    const int out = dbg ? kOutDebug : a.spec_type;
    // antennas per unit: short transforms share a unit's set-up
    const int AN = std::min(a.N, Sh::kAsync ? 1 : 16 / M);
    const int64_t nfb = (fr + kMmaFrames - 1) / kMmaFrames;
    const int64_t units = nfb * ((a.N + AN - 1) / AN);
    if (nfb > 0x7fffffff) return cudaErrorInvalidValue;
    const size_t smem = Sh::smem(out, a.corr != nullptr, AN, NS);
    OutMaps maps{};
    if (!dbg) {
        const cudaError_t e = make_maps<N1, M, MTC>(a, maps);
        if (e != cudaSuccess) return e;
    }
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int dev = 0, nsm = 0, occ = 0;
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kMmaThreads, smem);
        if (e != cudaSuccess) return e;
        const int64_t slots = (int64_t)nsm * std::max(occ, 1) / Sh::MTG;
        const int64_t ranges = std::max<int64_t>(1, std::min(units, slots));
        kern<<<(unsigned)(ranges * Sh::MTG), kMmaThreads, smem, st>>>(a, maps, AN, (int)nfb, units);
        return cudaGetLastError();
    };
    auto go2 = [&](auto plain, auto corrected) { return a.corr ? go(corrected) : go(plain); };
#define GBCORR_MMA(OUT)                                                 \
    go2(fengine_mma<N1, M, MTC, OUT, false, MINB, NS>, \
        fengine_mma<N1, M, MTC, OUT, true, MINB, NS>)
    switch (out) {
        case SPEC_F16: return GBCORR_MMA(SPEC_F16);
        case SPEC_F8: return GBCORR_MMA(SPEC_F8);
        default: break;
    }
    if constexpr (!NARROW) {
        switch (out) {
            case kOutDebug: return GBCORR_MMA(kOutDebug);
            case SPEC_F32: return GBCORR_MMA(SPEC_F32);
            case SPEC_F16X2: return GBCORR_MMA(SPEC_F16X2);
            default: break;
        }
    }
#undef GBCORR_MMA
    return cudaErrorInvalidValue;
}

}  // namespace

// One E4M3 rounding that falls the other way moves a visibility by up to ~0.45
// of a sample's power, 0.45 / (T sqrt(2 / N + 1 / T)) of the rms visibility of T
// spectra: in short integrations the two kinds of kernel, equally accurate,
// differ by 1e-3 of it (N = 44, T = 2048) to 4e-3 (N = 11, T = 120).  So an FP8
// integration starts on the FP32 FFTs, and its frames go over to the others
// where 2 T^2 / N + T = 420000 (N = 44: 3072 frames), from where it stays below
// 7e-4.  The line is one of the integration's frames, not of the pushes: the
// same samples round alike however they are pushed.  FP16's roundings are 64
// times finer.
int64_t fp8_fft_frames(int N) {
    int64_t T = kSpecPad;
    while (2.0 * (double)T * T / N + T < 420000.0) T += kSpecPad;
    return T;
}

bool fengine_mma_serves(const FengineArgs& a) {
    if (a.K < 16 || a.K > 2048) return false;
    if (a.spec_type == SPEC_F8 && !a.debug_out && a.pos < fp8_fft_frames(a.N)) return false;
    if (a.stable && (a.spec_type == SPEC_F32 || a.spec_type == SPEC_F16X2)) return false;
    // bytes of the widest load: one pair of n1, at least a cp.async for K >= 512
    const uintptr_t align = a.K >= 512 ? 16 : (a.K <= 32 ? 1 : a.K / 32);
    if (reinterpret_cast<uintptr_t>(a.in) % align) return false;
    if ((a.K == 512 || a.K == 1024) && (a.debug_out || (a.spec_type != SPEC_F16 && a.spec_type != SPEC_F8)))
        return false;
    // (without tensor maps only FP32 outputs exist: the other types' handles need them)
    return a.debug_out || tc::get_encoder();
}

cudaError_t launch_fengine_mma(const FengineArgs& a, cudaStream_t st) {
    switch (a.K) {
        case 16: return launch_shape<16, 1, 1, 4, 1, false>(a, st);
        case 32: return launch_shape<32, 1, 2, 4, 1, false>(a, st);
        case 64: return launch_shape<32, 2, 2, 4, 1, false>(a, st);
        case 128: return launch_shape<32, 4, 2, 4, 1, false>(a, st);
        case 256: return launch_shape<32, 8, 2, 4, 1, false>(a, st);
        case 512: return launch_shape<32, 16, 1, 4, 2, true>(a, st);
        case 1024: return launch_shape<64, 16, 1, 4, 2, true>(a, st);
        case 2048: return launch_shape<64, 32, 1, 2, 1, false>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gbcorr
