// rick_dft.cuh -- in-register and in-shared-memory length-N DFTs shared by the
// transform kernels (rick_fft.cu, rick_cols.cu); the algorithm is described at
// the head of rick_fft.cu.
#pragma once

#include <cmath>
#include <vector>

#include "rick_internal.cuh"

namespace rick {

namespace {

// cos(2 pi k / 32) for 0 <= k <= 8, from the values of cos(pi k / 16)
__host__ __device__ constexpr float quarter32(int k) {
    return k == 0 ? 1.0f
         : k == 1 ? 0.98078528040323044913f
         : k == 2 ? 0.92387953251128675613f
         : k == 3 ? 0.83146961230254523708f
         : k == 4 ? 0.70710678118654752440f
         : k == 5 ? 0.55557023301960222474f
         : k == 6 ? 0.38268343236508977173f
         : k == 7 ? 0.19509032201612826785f
         : 0.0f;
}

__host__ __device__ constexpr float cos32(int k) {
    return (k & 31) <= 8    ? quarter32(k & 31)
         : (k & 31) <= 16 ? -quarter32(16 - (k & 31))
         : (k & 31) <= 24 ? -quarter32((k & 31) - 16)
                            : quarter32(32 - (k & 31));
}

__host__ __device__ constexpr float sin32(int k) { return cos32(k - 8); }

// cos(2 pi k / 64) for 0 <= k <= 16 (cos(pi k / 32), from the FP64 values)
__host__ __device__ constexpr float quarter64(int k) {
    return k == 0 ? 1.0f
         : k == 1 ? 0.99518472667219692873f
         : k == 2 ? 0.98078528040323043058f
         : k == 3 ? 0.95694033573220882438f
         : k == 4 ? 0.92387953251128673848f
         : k == 5 ? 0.88192126434835504956f
         : k == 6 ? 0.83146961230254523567f
         : k == 7 ? 0.77301045336273699338f
         : k == 8 ? 0.70710678118654757274f
         : k == 9 ? 0.63439328416364548779f
         : k == 10 ? 0.55557023301960228867f
         : k == 11 ? 0.47139673682599780857f
         : k == 12 ? 0.38268343236508983729f
         : k == 13 ? 0.29028467725446233105f
         : k == 14 ? 0.19509032201612833135f
         : k == 15 ? 0.09801714032956077016f
         : 0.0f;
}

__host__ __device__ constexpr float cos64(int k) {
    return (k & 63) <= 16   ? quarter64(k & 63)
         : (k & 63) <= 32 ? -quarter64(32 - (k & 63))
         : (k & 63) <= 48 ? -quarter64((k & 63) - 32)
                            : quarter64(64 - (k & 63));
}

__host__ __device__ constexpr float sin64(int k) { return cos64(k - 16); }

// Complex add and subtract as one packed two-lane FP32 instruction each
// (add/sub.rn.f32x2, sm_100 and later): the same IEEE round-to-nearest results
// as two scalar instructions, half the issue slots -- the butterflies are
// mostly adds, and the transform kernels are issue-bound.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
    uint64_t ra = *reinterpret_cast<uint64_t*>(&a), rb = *reinterpret_cast<uint64_t*>(&b), rd;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    return *reinterpret_cast<float2*>(&rd);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    uint64_t ra = *reinterpret_cast<uint64_t*>(&a), rb = *reinterpret_cast<uint64_t*>(&b), rd;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    return *reinterpret_cast<float2*>(&rd);
}
__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * (s i), s = +1 (INV) or -1
template <bool INV>
__device__ __forceinline__ float2 mul_si(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// v * e^(s 2 pi i e / R) for compile-time e and R <= 32 (after unrolling), s = +1 (INV) or -1
template <bool INV>
__device__ __forceinline__ float2 twiddle_const(float2 v, int e, int R) {
    const int k = (e * (32 / R)) & 31;   // in 32nds of a turn
    if (k == 0) return v;
    if (k == 8) return mul_si<INV>(v);
    if (k == 16) return make_float2(-v.x, -v.y);
    if (k == 24) return mul_si<!INV>(v);
    const float c = cos32(k), s = INV ? sin32(k) : -sin32(k);
    return make_float2(fmaf(v.x, c, -v.y * s), fmaf(v.x, s, v.y * c));
}

// v * e^(s 2 pi i k / 64) for compile-time k (after unrolling), s = +1 (INV) or -1
template <bool INV>
__device__ __forceinline__ float2 twiddle64(float2 v, int k) {
    k &= 63;
    if (k == 0) return v;
    if (k == 16) return mul_si<INV>(v);
    if (k == 32) return make_float2(-v.x, -v.y);
    if (k == 48) return mul_si<!INV>(v);
    const float c = cos64(k), s = INV ? sin64(k) : -sin64(k);
    return make_float2(fmaf(v.x, c, -v.y * s), fmaf(v.x, s, v.y * c));
}

// In-register length-R DFT, X[f] = sum_t a[t] e^(s 2 pi i t f / R), natural order.
template <int R, bool INV>
struct Dft;

template <bool INV>
struct Dft<2, INV> {
    static __device__ __forceinline__ void run(float2* a) {
        const float2 x = a[0], y = a[1];
        a[0] = cadd(x, y);
        a[1] = csub(x, y);
    }
};

template <bool INV>
struct Dft<4, INV> {
    static __device__ __forceinline__ void run(float2* a) {
        const float2 t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]);
        const float2 t2 = cadd(a[1], a[3]), t3 = mul_si<INV>(csub(a[1], a[3]));
        a[0] = cadd(t0, t2);
        a[2] = csub(t0, t2);
        a[1] = cadd(t1, t3);
        a[3] = csub(t1, t3);
    }
};

// R = 4 S: X[f0 + 4 f1] = sum_{t1 < S} W_S^(t1 f1) [W_R^(t1 f0) sum_{t2 < 4} a[t1 + S t2] W_4^(t2 f0)]
template <int R, bool INV>
struct Dft {
    static_assert(R == 8 || R == 16 || R == 32, "radix");
    static constexpr int S = R / 4;
    static __device__ __forceinline__ void run(float2* a) {
        float2 y[R];  // y[f0 S + t1]
#pragma unroll
        for (int t1 = 0; t1 < S; ++t1) {
            float2 b[4] = {a[t1], a[t1 + S], a[t1 + 2 * S], a[t1 + 3 * S]};
            Dft<4, INV>::run(b);
#pragma unroll
            for (int f0 = 0; f0 < 4; ++f0) y[f0 * S + t1] = twiddle_const<INV>(b[f0], t1 * f0, R);
        }
#pragma unroll
        for (int f0 = 0; f0 < 4; ++f0) {
            Dft<S, INV>::run(y + f0 * S);
#pragma unroll
            for (int f1 = 0; f1 < S; ++f1) a[f0 + 4 * f1] = y[f0 * S + f1];
        }
    }
};

__device__ __forceinline__ int skew(int a) { return a + (a >> 4); }
// skew(a + 16 k) = skew(a) + 17 k: an offset that is a multiple of 16 becomes
// a constant added to the skewed base, so unrolled accesses at base + 16 k
// need no address arithmetic of their own
__host__ __device__ constexpr int skew16(int k16) { return k16 + k16 / 16; }

template <int LOG2N>
struct Shape {
    static constexpr int N = 1 << LOG2N;
    static constexpr int T = N / 16;                 // threads per transform
    static constexpr int kR16 = LOG2N / 4;            // radix-16 stages
    static constexpr int kLastR = 1 << (LOG2N % 4);   // 1: the last stage is radix 16
    static constexpr int kArray = N + N / 16;         // skewed array length
    // radix-16 stages with twiddles (all but a last radix-16 stage)
    static constexpr int kTwStages = kLastR == 1 ? kR16 - 1 : kR16;
    // butterfly groups t1 of stage s, table entries per t1 (stage 0: 4 powers,
    // the others: all 15), and the offset of the stage's table
    __host__ __device__ static constexpr int stage_cnt(int s) { return (N / 16) >> (4 * s); }
    __host__ __device__ static constexpr int stage_per(int s) { return s == 0 ? 4 : 15; }
    __host__ __device__ static constexpr int stage_off(int s) {
        int o = 0;
        for (int i = 0; i < s; ++i) o += stage_per(i) * stage_cnt(i);
        return o;
    }
    static constexpr int kTw = stage_off(kTwStages);  // twiddle table entries
    // 128 (LOG2N = 7) only for the four-step column pass at N = 16384
    static_assert(LOG2N >= 7 && LOG2N <= 14, "128 <= N <= 16384");
};

// Radix-16 stage s (M = 16^s, not the last stage): a holds the butterfly's
// inputs u + (N/16) t2 for u = b; the DFT, the twiddles W_N^(t1 f0 M) from the
// stage's table sw (stage 0: sw[j cnt + t1] = W^(2^j t1 M), j < 4, the other
// powers formed from them; later stages, whose t1 takes few values, hold all
// fifteen: sw[(f0 - 1) cnt + t1] = W^(t1 f0 M)) and the stores t1 16 M + g +
// M f0 into buf.
template <int LOG2N, bool INV>
__device__ __forceinline__ void radix16_out(float2 (&a)[16], int b, int s, float2* buf,
                                            const float2* tw) {
    using Sh = Shape<LOG2N>;
    Dft<16, INV>::run(a);
    const int log2M = 4 * s;
    const int M = 1 << log2M;
    const int t1 = b >> log2M, g = b & (M - 1);
    const int base = (t1 << (log2M + 4)) + g;
    // output f0 goes to base + M f0: for M >= 16 (M f0 a multiple of 16) and
    // for M = 1 (base a multiple of 16, f0 < 16) its skewed index is
    // skew(base) plus a constant
    float2* out = buf + skew(base);
    auto at = [&](int f0) -> float2& { return M == 1 ? out[f0] : out[skew16(M * f0)]; };
    // t1 = 0: the table holds W^0 = 1 exactly, and a * 1 = a exactly
    const int cnt = Sh::stage_cnt(s);
    const float2* sw = tw + Sh::stage_off(s) + t1;
    if (Sh::stage_per(s) == 15) {
        at(0) = a[0];
#pragma unroll
        for (int f0 = 1; f0 < 16; ++f0) {
            float2 w = sw[(f0 - 1) * cnt];
            if (!INV) w.y = -w.y;
            at(f0) = cmulf(a[f0], w);
        }
        return;
    }
    float2 w[16];
    w[1] = sw[0];
    w[2] = sw[cnt];
    w[4] = sw[2 * cnt];
    w[8] = sw[3 * cnt];
    if (!INV) {
        w[1].y = -w[1].y;
        w[2].y = -w[2].y;
        w[4].y = -w[4].y;
        w[8].y = -w[8].y;
    }
    w[3] = cmulf(w[2], w[1]);
    w[5] = cmulf(w[4], w[1]);
    w[6] = cmulf(w[4], w[2]);
    w[7] = cmulf(w[4], w[3]);
#pragma unroll
    for (int f0 = 9; f0 < 16; ++f0) w[f0] = cmulf(w[8], w[f0 - 8]);
    at(0) = a[0];
#pragma unroll
    for (int f0 = 1; f0 < 16; ++f0) at(f0) = cmulf(a[f0], w[f0]);
}

// Stage 0 (M = 1) of the inverse transform whose 16 inputs of thread b all
// carry one more factor sc (the split row pass's e^(+2 pi i r b / N)): the
// factor is moved past the butterfly, so output f0 is multiplied by
// sc W^(b f0) -- the products formed from sc and the stage's four table
// powers -- instead of every input by sc (31 complex multiplies instead of 42).
template <int LOG2N>
__device__ __forceinline__ void radix16_first_scaled(float2 (&a)[16], int b, float2* buf, const float2* tw,
                                                     float2 sc) {
    using Sh = Shape<LOG2N>;
    Dft<16, true>::run(a);
    const int cnt = Sh::stage_cnt(0);
    const float2* sw = tw + Sh::stage_off(0) + b;   // t1 = b
    const float2 w1 = sw[0], w2 = sw[cnt], w4 = sw[2 * cnt], w8 = sw[3 * cnt];
    float2 w[16];
    w[0] = sc;
    w[1] = cmulf(sc, w1);
    w[2] = cmulf(sc, w2);
    w[3] = cmulf(w[1], w2);
    w[4] = cmulf(sc, w4);
#pragma unroll
    for (int f0 = 5; f0 < 8; ++f0) w[f0] = cmulf(w[f0 - 4], w4);
    w[8] = cmulf(sc, w8);
#pragma unroll
    for (int f0 = 9; f0 < 16; ++f0) w[f0] = cmulf(w[f0 - 8], w8);
    float2* out = buf + skew(16 * b);   // outputs 16 b + f0
#pragma unroll
    for (int f0 = 0; f0 < 16; ++f0) out[f0] = cmulf(a[f0], w[f0]);
}

// The middle radix-16 stages (all but the first, which starts from registers,
// and the last) on buf, in place: loads, barrier, compute and stores, barrier.
template <int LOG2N, bool INV>
__device__ __forceinline__ void middle_stages(float2* buf, int b, const float2* tw) {
    using Sh = Shape<LOG2N>;
    constexpr int kMiddle = Sh::kTwStages - 1;
    const float2* in = buf + skew(b);   // inputs b + T t2, T a multiple of 16
#pragma unroll
    for (int s = 1; s <= kMiddle; ++s) {
        float2 a[16];
#pragma unroll
        for (int t2 = 0; t2 < 16; ++t2) a[t2] = in[skew16(Sh::T * t2)];
        __syncthreads();
        radix16_out<LOG2N, INV>(a, b, s, buf, tw);
        __syncthreads();
    }
}

// The last stage (radix kLastR, or 16), M = N/R, no twiddles: x[j] = X[b + (N/16) j].
template <int LOG2N, bool INV>
__device__ __forceinline__ void last_stage(const float2* buf, int b, float2 (&x)[16]) {
    using Sh = Shape<LOG2N>;
    constexpr int R = Sh::kLastR == 1 ? 16 : Sh::kLastR;
    constexpr int NB = 16 / R;          // butterflies per thread
    constexpr int M = Sh::N / R;
    const float2* in = buf + skew(b);   // T i + M t2 is a multiple of 16
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        float2 a[R];
#pragma unroll
        for (int t2 = 0; t2 < R; ++t2) a[t2] = in[skew16(Sh::T * i + M * t2)];
        Dft<R, INV>::run(a);
        // output u + M f0 = b + T (i + NB f0)
#pragma unroll
        for (int f0 = 0; f0 < R; ++f0) x[i + NB * f0] = a[f0];
    }
}

// One whole transform of the array whose first stage inputs a[t2] = x[b + T t2]
// are in registers; on return x[j] = X[b + T j].  buf is free on entry and
// holds the last stage's input on return (a barrier is needed before reuse).
template <int LOG2N, bool INV>
__device__ __forceinline__ void transform(float2 (&a)[16], float2* buf, int b, const float2* tw,
                                          float2 (&x)[16]) {
    radix16_out<LOG2N, INV>(a, b, 0, buf, tw);
    __syncthreads();
    middle_stages<LOG2N, INV>(buf, b, tw);
    last_stage<LOG2N, INV>(buf, b, x);
}

template <int LOG2N>
__device__ __forceinline__ void load_tables(const float2* __restrict__ twid, float2* tw, int tid, int nthreads) {
    for (int i = tid; i < Shape<LOG2N>::kTw; i += nthreads) tw[i] = __ldg(twid + i);
}

}  // namespace

}  // namespace rick
