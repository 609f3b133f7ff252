// rick_learn.cu -- training objective of the learned support-4 kernel.
//
// A fixed visibility sample (one observation's u, v, w and weights) is placed
// once (FP64, the same rules as the gridder) and sorted by w-plane.  For each
// training field (point sources on pixel centres) the kernels
//   1. predict the visibilities from the sources (Eq. 1),
//   2. evaluate at probe pixels both the w-stacking image that the gridder,
//      FFT and phase screen would produce with the current tap table (Eq. 2,
//      Eq. 3, written per visibility as in the oracle's per-pixel form) and
//      the direct Fourier inversion of the same visibilities,
//   3. form the loss sum_P (I_P - D_P)^2 / sum_P D_P^2, and
//   4. back-propagate it to the tap table (bilinear lattice, per plane),
// after which rick_mlp_backward carries the table gradient into the network.
// The table holds a correction added to the support-4 Kaiser-Bessel taps (so a
// zero table is the Kaiser-Bessel kernel); its gradient is the tap gradient.
//
// Phases: with x = u fov + N/2 the continuous cell position, u l_p =
// (x - N/2)(p - N/2)/N turns.  x - N/2 = X + f with X integer, so the turn is
// (X (p - N/2) mod N)/N + f (p - N/2)/N: exact integer reduction (N is a power of
// two: a mask) plus a term below half a turn, which FP32 carries to ~3e-8 turns.
//
// The work is (visibility, probe) pairs, 64 probes a visibility, bound by
// instruction issue.  Per pair the forward pass needs one phasor of the footprint's
// first cell, e^(2 pi i (i0 p + j0 q)/N) -- shared by the image term and the direct
// inversion, whose phases differ from it by a constant of the probe, the terms of the
// cell fractions (below half a turn each) and w (n - 1), formed in FP32: an error of
// 1e-7 |w (n - 1)| turns -- and the taps' two polynomials in the probe's unit steps (-1) e^(2 pi
// i p/N), whose powers are the probe's constants (rounded from FP64 on the host).
// A thread of the forward pass owns one probe and walks visibilities staged in
// shared memory, so its sums stay in registers; a thread of the backward pass owns
// one visibility and walks the probes.  I - D is a small difference of I and D, so the
// loss magnifies the rounding of the two sums: a thread's FP32 sums cover one staged
// block (32 terms) and go on in FP64 from there to the loss.  RMS relative error of the
// loss against 64 bits over 6 to 8 seeds, at 2 M / 200 k / 20 k visibilities: FP32 sums
// throughout 4.6e-6 / 1.5e-5 / 7.1e-6 (a warp reduction per pair 1.2e-5 / 1.7e-5 /
// 2.2e-6), now 1.9e-6 / 2.7e-6 / 7.6e-7.  Measured on GB300 (N = 2048, 2 M
// visibilities, 64 probes, lattice 32) against one visibility a thread in the
// forward pass with a warp reduction per pair, 64-bit remainders and four phasors:
// forward 3.37 -> 0.65 ms, backward 2.19 -> 0.39 ms, prediction of a field's sources
// 0.6 -> 0.1 ms (each with FP32 sums throughout); a training step of four fields
// 25.2 -> 4.96 ms, 4.75 of it before the FP64 sums.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "rick_internal.cuh"

namespace rick {
void set_error_message(const char* msg);
int64_t mlp_param_count(int H);
}

using namespace rick;

namespace {

constexpr int kMaxProbes = 64;
constexpr int kMaxSources = 64;
constexpr int kLearnS = 4;

struct __align__(16) LearnVis {
    int i0, j0, k, pad;
    float fx, fy, w, W;
};

// Constants of a probe pixel (p, q): the powers 1..3 of -e^(2 pi i p / N) and of
// -e^(2 pi i q / N), (p - N/2)/N and (q - N/2)/N, n - 1, the turns by which the
// direct inversion's phasor is ahead of the footprint's (DftTurn below), and the
// scales of the image, (-1)^(p+q) n / (C(p) C(q)), and of the inversion, n.
struct __align__(16) Probe {
    float2 sx[3], sy[3];
    int p, q;
    float pn, qn;
    float delta, turn, scale_img, scale_dft;
};

struct LearnConst {
    int N, Nw, L, nvis, ns, np;
    float inv_wsum;
};

// ---- placement --------------------------------------------------------------

__global__ void k_learn_place(const double* __restrict__ uvw, const float* __restrict__ weight,
                              int64_t nvis, int N, int Nw, double fov, double w_min,
                              double w_scale, LearnVis* __restrict__ out, int* __restrict__ status,
                              unsigned* __restrict__ plane_count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nvis) return;
    LearnVis v = {0, 0, -1, 0, 0.f, 0.f, 0.f, 0.f};
    int st = 0;
    const float W = weight[i];
    if (W != 0.0f && isfinite(W)) {
        const double u = uvw[3 * i], vv = uvw[3 * i + 1], w = uvw[3 * i + 2];
        const double x = __dadd_rn(__dmul_rn(u, fov), 0.5 * N);
        const double y = __dadd_rn(__dmul_rn(vv, fov), 0.5 * N);
        const double sx = __dsub_rn(x, 0.5 * kLearnS), sy = __dsub_rn(y, 0.5 * kLearnS);
        const double flx = floor(sx), fly = floor(sy);
        if (isfinite(x) && isfinite(y) && isfinite(w) && flx >= -1.0 && fly >= -1.0 &&
            flx + kLearnS <= N - 1 && fly + kLearnS <= N - 1) {
            v.i0 = (int)flx + 1;
            v.j0 = (int)fly + 1;
            v.fx = (float)__dsub_rn(sx, flx);
            v.fy = (float)__dsub_rn(sy, fly);
            int k = 0;
            if (Nw > 1) {
                double kf = floor(__dmul_rn(__dsub_rn(w, w_min), w_scale));
                kf = fmin(fmax(kf, 0.0), (double)(Nw - 1));
                k = (int)kf;
            }
            v.k = k;
            v.w = (float)w;
            v.W = W;
            st = 1;
            atomicAdd(&plane_count[k], 1u);
        } else {
            st = -1;
        }
    }
    out[i] = v;
    status[i] = st;
}

__global__ void k_learn_sort(const LearnVis* __restrict__ in, int64_t nvis,
                             unsigned* __restrict__ cursor, LearnVis* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nvis) return;
    const LearnVis v = in[i];
    if (v.k < 0) return;
    out[atomicAdd(&cursor[v.k], 1u)] = v;
}

// ---- per field ---------------------------------------------------------------

__device__ __forceinline__ float2 turn_phasor(float t) {  // exp(2 pi i t), t reduced first
    float s, c;
    sincospif(2.0f * (t - rintf(t)), &s, &c);
    return make_float2(c, s);
}

// (X * P mod N)/N + f P / N, in turns, for integer X, P and f in [0, 1); N a power
// of two, so that the product modulo 2^32 keeps the remainder
__device__ __forceinline__ float cell_turns(int X, int P, float f, int N) {
    const float inv = 1.0f / (float)N;   // exact
    const uint32_t r = ((uint32_t)X * (uint32_t)P) & (uint32_t)(N - 1);
    return (float)r * inv + f * (float)P * inv;
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// The turns of u l for a source at pixel offset P = p - N/2 (any real p):
// with P = Pi + Pf (Pi integer, 0 <= Pf < 1), (X + f)(Pi + Pf)/N is the exact
// integer reduction of X Pi plus f Pi/N plus (X + f) Pf / N, each below half a
// turn in magnitude.
__device__ __forceinline__ float source_turns(int X, float P, float f, int N) {
    const float Pi = floorf(P);
    return cell_turns(X, (int)Pi, f, N) + ((float)X + f) * (P - Pi) * (1.0f / (float)N);
}

// V_j W_j for the field: sources src[s] = (P_s, Q_s, A_s / n_s, delta_s) with
// P_s = p_s - N/2, Q_s = q_s - N/2 (pixel offsets from the centre; p_s, q_s
// continuous positions in pixels).
__global__ void k_learn_predict(const LearnVis* __restrict__ vis, LearnConst C,
                                const float4* __restrict__ src, float2* __restrict__ wv) {
    __shared__ float4 s_src[kMaxSources];
    for (int s = threadIdx.x; s < C.ns; s += blockDim.x) s_src[s] = src[s];
    __syncthreads();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= C.nvis) return;
    const LearnVis v = vis[j];
    const int X = v.i0 - 1 + kLearnS / 2 - C.N / 2, Y = v.j0 - 1 + kLearnS / 2 - C.N / 2;
    float2 acc = make_float2(0.f, 0.f);
    for (int s = 0; s < C.ns; ++s) {
        const float4 q = s_src[s];
        const float t = source_turns(X, q.x, v.fx, C.N) + source_turns(Y, q.y, v.fy, C.N) + v.w * q.w;
        const float2 e = turn_phasor(-t);  // Eq. 1: exp(-2 pi i (u l + v m + w (n - 1)))
        acc.x += q.z * e.x;
        acc.y += q.z * e.y;
    }
    wv[j] = make_float2(v.W * acc.x, v.W * acc.y);
}

// The support-4 Kaiser-Bessel taps as polynomials in 2f - 1 (fitted on the host).
struct KbTaps {
    float coef[4][kPolyDegree + 1];
};

__device__ __forceinline__ float kb_tap(const KbTaps& K, int a, float t) {
    float acc = K.coef[a][kPolyDegree];
#pragma unroll
    for (int q = kPolyDegree - 1; q >= 0; --q) acc = fmaf(acc, t, K.coef[a][q]);
    return acc;
}

// Taps of visibility v: the Kaiser-Bessel products plus the correction
// interpolated (bilinearly) from the table, t[b*4 + a].
__device__ __forceinline__ void learn_taps(const float* __restrict__ table, int L, const LearnVis& v,
                                           const KbTaps& K, float* t) {
    const float X = v.fx * L, Y = v.fy * L;
    const int ix = min((int)X, L - 1), iy = min((int)Y, L - 1);
    const float ax = X - ix, ay = Y - iy;
    const size_t row = (size_t)(L + 1);
    const float* t00 = table + (((size_t)v.k * row + iy) * row + ix) * 16;
    const float* t01 = t00 + row * 16;
    const float w00 = (1.f - ax) * (1.f - ay), w10 = ax * (1.f - ay), w01 = (1.f - ax) * ay, w11 = ax * ay;
    const float tx = fmaf(2.0f, v.fx, -1.0f), ty = fmaf(2.0f, v.fy, -1.0f);
    float gx[4], gy[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        gx[a] = kb_tap(K, a, tx);
        gy[a] = kb_tap(K, a, ty);
    }
#pragma unroll
    for (int q = 0; q < 16; ++q)
        t[q] = gx[q & 3] * gy[q >> 2] + w00 * __ldg(t00 + q) + w10 * __ldg(t00 + 16 + q) +
               w01 * __ldg(t01 + q) + w11 * __ldg(t01 + 16 + q);
}

// (-1)^(i0+j0) e^(2 pi i (i0 p + j0 q)/N): the checkerboard sign is half a turn, and
// the turn an exact multiple of 1/N
__device__ __forceinline__ float2 cell_phasor(int i0, int j0, int p, int q, int N, float inv_half_n) {
    const uint32_t m = (uint32_t)i0 * (uint32_t)p + (uint32_t)j0 * (uint32_t)q + (uint32_t)((i0 + j0) & 1) * (uint32_t)(N / 2);
    float s, c;
    sincospif((float)(m & (uint32_t)(N - 1)) * inv_half_n, &s, &c);
    return make_float2(c, s);
}

constexpr size_t kSharedMax = 227 * 1024;   // shared memory of a CTA at most
constexpr int kFwdVis = 128;   // visibilities staged at a time
constexpr int kFwdRow = 6;     // float4 of a staged visibility: 16 taps, (W V, fx, fy), (w, i0, j0, k)

// I_P and D_P summed over all visibilities (out[2P], out[2P + 1]): eight warps,
// four pairs of them taking a quarter of the staged visibilities each, lane l of a
// pair's first and second warp the probes l and 32 + l.
template <bool STAGED>
__global__ void __launch_bounds__(256)
k_learn_forward(const LearnVis* __restrict__ vis, const float2* __restrict__ wv,
                const float* __restrict__ table, LearnConst C, KbTaps K, const Probe* __restrict__ probes,
                const float2* __restrict__ ph, double* __restrict__ out) {
    extern __shared__ __align__(16) float4 s_vis[];   // kFwdVis rows, then (STAGED) the phasors e^(2 pi i w_k delta_P)
    float2* s_ph = reinterpret_cast<float2*>(s_vis + kFwdVis * kFwdRow);
    __shared__ double2 s_acc[4][kMaxProbes];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int P = (warp & 1) * 32 + (tid & 31), quarter = warp >> 1;
    if (STAGED)
        for (int i = tid; i < C.Nw * kMaxProbes; i += 256) s_ph[i] = ph[i];
    Probe pr = {};
    if (P < C.np) pr = probes[P];
    const bool idle = (warp & 1) * 32 >= C.np;
    const float inv_half_n = 2.0f / (float)C.N;
    double img64 = 0.0, dft64 = 0.0;
    for (int base = blockIdx.x * kFwdVis; base < C.nvis; base += gridDim.x * kFwdVis) {
        __syncthreads();   // the previous visibilities have been read (and the phasors are there)
        if (tid < kFwdVis) {
            float4* row = s_vis + tid * kFwdRow;
            float taps[16];
            LearnVis v = {0, 0, 0, 0, 0.f, 0.f, 0.f, 0.f};
            float2 w2 = make_float2(0.f, 0.f);
            if (base + tid < C.nvis) {
                v = vis[base + tid];
                w2 = wv[base + tid];
                learn_taps(table, C.L, v, K, taps);
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q) taps[q] = 0.f;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) row[q] = make_float4(taps[4 * q], taps[4 * q + 1], taps[4 * q + 2], taps[4 * q + 3]);
            row[4] = make_float4(w2.x, w2.y, v.fx, v.fy);
            row[5] = make_float4(v.w, __int_as_float(v.i0), __int_as_float(v.j0), __int_as_float(v.k));
        }
        __syncthreads();
        if (idle) continue;
        const float4* row = s_vis + quarter * (kFwdVis / 4) * kFwdRow;
        float img = 0.f, dft = 0.f;
#pragma unroll 2
        for (int r = 0; r < kFwdVis / 4; ++r, row += kFwdRow) {
            const float4 a = row[4], b = row[5];
            const float2 e = cell_phasor(__float_as_int(b.y), __float_as_int(b.z), pr.p, pr.q, C.N, inv_half_n);
            const float2 c = cmulf(make_float2(a.x, a.y), e);   // W V times the first cell's phasor
            float2 g[4];   // the taps' polynomial in x, row by row
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 t = row[q];
                g[q].x = fmaf(t.w, pr.sx[2].x, fmaf(t.z, pr.sx[1].x, fmaf(t.y, pr.sx[0].x, t.x)));
                g[q].y = fmaf(t.w, pr.sx[2].y, fmaf(t.z, pr.sx[1].y, t.y * pr.sx[0].y));
            }
            float2 S = g[0];
#pragma unroll
            for (int q = 1; q < 4; ++q) {
                S.x = fmaf(g[q].x, pr.sy[q - 1].x, fmaf(-g[q].y, pr.sy[q - 1].y, S.x));
                S.y = fmaf(g[q].x, pr.sy[q - 1].y, fmaf(g[q].y, pr.sy[q - 1].x, S.y));
            }
            const int at = __float_as_int(b.w) * kMaxProbes + P;
            const float2 u = cmulf(c, STAGED ? s_ph[at] : __ldg(ph + at));
            img = fmaf(u.x, S.x, fmaf(-u.y, S.y, img));
            // the direct inversion: the rest of its turn, |w (n - 1)| + 1.5 at most
            const float2 d = turn_phasor(fmaf(a.z, pr.pn, fmaf(a.w, pr.qn, fmaf(b.x, pr.delta, pr.turn))));
            dft = fmaf(c.x, d.x, fmaf(-c.y, d.y, dft));
        }
        img64 += img;
        dft64 += dft;
    }
    s_acc[quarter][P] = make_double2(img64, dft64);
    __syncthreads();
    if (tid < C.np) {
        double2 t = s_acc[0][tid];
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            t.x += s_acc[q][tid].x;
            t.y += s_acc[q][tid].y;
        }
        const Probe& o = probes[tid];
        atomicAdd(&out[2 * tid], (double)o.scale_img * t.x * (double)C.inv_wsum);
        atomicAdd(&out[2 * tid + 1], (double)o.scale_dft * t.y * (double)C.inv_wsum);
    }
}

// loss = sum (I - D)^2 / sum D^2; ge[P] = dloss/dI_P (scaled by 1/sum W, which
// the backward kernel's per-visibility terms omit); idft[2P], idft[2P + 1] = I_P, D_P
// rounded.  One warp, two probes a lane.
__global__ void k_learn_loss(const double* __restrict__ sums, int np, float inv_wsum,
                             float* __restrict__ idft, float* __restrict__ loss, float* __restrict__ ge) {
    const int lane = threadIdx.x;
    double e[2], num = 0.0, den = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int P = lane + 32 * h;
        const double i = P < np ? sums[2 * P] : 0.0, d = P < np ? sums[2 * P + 1] : 0.0;
        if (P < np) {
            idft[2 * P] = (float)i;
            idft[2 * P + 1] = (float)d;
        }
        e[h] = i - d;
        num += e[h] * e[h];
        den += d * d;
    }
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    den = fmax(den, 1e-30);
    if (lane == 0) *loss = (float)(num / den);
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (lane + 32 * h < np) ge[lane + 32 * h] = (float)(2.0 * e[h] / den * inv_wsum);
}

// *p += v, as one reduction of four floats where the caller's table is 16-byte aligned
__device__ __forceinline__ void add4(float* p, float4 v, bool aligned16) {
    if (aligned16) {
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                     : "memory");
    } else {
        atomicAdd(p, v.x);
        atomicAdd(p + 1, v.y);
        atomicAdd(p + 2, v.z);
        atomicAdd(p + 3, v.w);
    }
}

// d loss / d table: per visibility the 16 tap gradients sum_P ge_P scale_P Re(W V
// e^(2 pi i w_k delta_P) E_x(i0 + a) E_y(j0 + b)), spread bilinearly onto the lattice
// of its plane by vector reductions in L2 (16 of four floats a visibility; FP32
// shared-memory atomics are compare-and-swap loops).
template <bool STAGED>
__global__ void __launch_bounds__(256)
k_learn_backward(const LearnVis* __restrict__ vis, const float2* __restrict__ wv, LearnConst C,
                 const Probe* __restrict__ probes, const float2* __restrict__ ph, const float* __restrict__ ge,
                 float* __restrict__ table_grad, bool aligned16) {
    __shared__ __align__(16) float4 s_step[kMaxProbes][3];   // sx[0..2], sy[0..2]
    __shared__ int2 s_pq[kMaxProbes];
    extern __shared__ float2 s_gph[];             // STAGED: ge_P scale_P e^(2 pi i w_k delta_P)
    __shared__ float s_g[kMaxProbes];             // otherwise: ge_P scale_P
    for (int i = threadIdx.x; i < C.np; i += blockDim.x) {
        const Probe o = probes[i];
        s_step[i][0] = make_float4(o.sx[0].x, o.sx[0].y, o.sx[1].x, o.sx[1].y);
        s_step[i][1] = make_float4(o.sx[2].x, o.sx[2].y, o.sy[0].x, o.sy[0].y);
        s_step[i][2] = make_float4(o.sy[1].x, o.sy[1].y, o.sy[2].x, o.sy[2].y);
        s_pq[i] = make_int2(o.p, o.q);
        if (!STAGED) s_g[i] = ge[i] * o.scale_img;
    }
    for (int i = threadIdx.x; STAGED && i < C.Nw * kMaxProbes; i += blockDim.x) {
        const int P = i % kMaxProbes;
        const float g = P < C.np ? ge[P] * probes[P].scale_img : 0.f;
        s_gph[i] = make_float2(g * ph[i].x, g * ph[i].y);
    }
    __syncthreads();
    const float inv_half_n = 2.0f / (float)C.N;
    const int L1 = C.L + 1;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < C.nvis; j += gridDim.x * blockDim.x) {
        const LearnVis v = vis[j];
        const float2 w2 = wv[j];
        const float2* gph = STAGED ? s_gph + v.k * kMaxProbes : ph + (size_t)v.k * kMaxProbes;
        float gt[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) gt[q] = 0.f;
#pragma unroll 2
        for (int P = 0; P < C.np; ++P) {
            const int2 pq = s_pq[P];
            const float4 s0 = s_step[P][0], s1 = s_step[P][1], s2 = s_step[P][2];
            const float2 e = cell_phasor(v.i0, v.j0, pq.x, pq.y, C.N, inv_half_n);
            float2 f = gph[P];
            if (!STAGED) f = make_float2(s_g[P] * f.x, s_g[P] * f.y);
            const float2 c = cmulf(cmulf(w2, f), e);
            const float2 cb[4] = {c, cmulf(c, make_float2(s1.z, s1.w)), cmulf(c, make_float2(s2.x, s2.y)),
                                  cmulf(c, make_float2(s2.z, s2.w))};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                gt[4 * b] += cb[b].x;
                gt[4 * b + 1] = fmaf(cb[b].x, s0.x, fmaf(-cb[b].y, s0.y, gt[4 * b + 1]));
                gt[4 * b + 2] = fmaf(cb[b].x, s0.z, fmaf(-cb[b].y, s0.w, gt[4 * b + 2]));
                gt[4 * b + 3] = fmaf(cb[b].x, s1.x, fmaf(-cb[b].y, s1.y, gt[4 * b + 3]));
            }
        }
        const float X = v.fx * C.L, Y = v.fy * C.L;
        const int ix = min((int)X, C.L - 1), iy = min((int)Y, C.L - 1);
        const float ax = X - ix, ay = Y - iy;
        const float wc[4] = {(1.f - ax) * (1.f - ay), ax * (1.f - ay), (1.f - ax) * ay, ax * ay};
        float* at = table_grad + (((size_t)v.k * L1 + iy) * L1 + ix) * 16;
#pragma unroll
        for (int cidx = 0; cidx < 4; ++cidx) {
            float* to = at + ((cidx >> 1) * L1 + (cidx & 1)) * 16;
#pragma unroll
            for (int q = 0; q < 16; q += 4)
                add4(to + q, make_float4(wc[cidx] * gt[q], wc[cidx] * gt[q + 1], wc[cidx] * gt[q + 2], wc[cidx] * gt[q + 3]),
                     aligned16);
        }
    }
}

}  // namespace

// ============================================================================

struct rick_learn {
    rick_config cfg;
    int L = 0;
    int64_t n_in = 0;
    int nvis = 0;       // placed visibilities
    double wsum = 0.0;
    std::vector<double> taper;
    LearnVis* d_vis = nullptr;
    float2* d_wv = nullptr;
    unsigned char* d_field = nullptr;  // a field's constants: sources, probes, plane phasors
    float* d_idft = nullptr;  // [2 * kMaxProbes]
    double* d_sums = nullptr; // [2 * kMaxProbes], the same before rounding
    float* d_ge = nullptr;
    KbTaps kb4;  // fitted support-4 Kaiser-Bessel taps the correction adds to
};

namespace {

void learn_free(rick_learn* Lr) {
    cudaFree(Lr->d_vis);
    cudaFree(Lr->d_wv);
    cudaFree(Lr->d_field);
    cudaFree(Lr->d_idft);
    cudaFree(Lr->d_sums);
    cudaFree(Lr->d_ge);
}

rick_status lfail(rick_status s, const char* m) {
    set_error_message(m);
    return s;
}

// A field's constants in one block (one copy to the device): kMaxSources sources,
// kMaxProbes probes, Nw x kMaxProbes phasors
size_t field_bytes(int Nw) {
    return sizeof(float4) * kMaxSources + sizeof(Probe) * kMaxProbes + sizeof(float2) * (size_t)Nw * kMaxProbes;
}

double host_i0(double x) {
    const double y = 0.25 * x * x;
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 400 && term > 1e-17 * sum; ++k) {
        term *= y / ((double)k * k);
        sum += term;
    }
    return sum;
}

}  // namespace

extern "C" {

rick_status rick_learn_create(const rick_config* cfg, int32_t lattice, const double* uvw,
                              const float* weight, int64_t nvis, rick_learn** out) {
    if (!cfg || !out || !uvw || !weight) return lfail(RICK_ERR_INVALID_ARG, "invalid argument: learn inputs");
    *out = nullptr;
    const rick_config& c = *cfg;
    if (c.kernel_kind != RICK_KERNEL_TABLE || c.support != kLearnS || c.n_channels != 1 ||
        c.N < 64 || (c.N & (c.N - 1)) || c.n_wplanes < 1 || !(c.fov_rad > 0 && c.fov_rad < 1) ||
        (c.n_wplanes > 1 && !(c.w_max > c.w_min)) || lattice < 1 || lattice > 64 || nvis < 1 ||
        nvis > (1ll << 30) || c.hermitian_fold != 0 || c.w_support >= 2 ||
        c.weighting != RICK_WEIGHT_NATURAL || (c.grid_size != 0 && c.grid_size != c.N))
        return lfail(RICK_ERR_INVALID_ARG,
                     "invalid argument: learning needs a table kernel of support 4, one channel, "
                     "no Hermitian fold, no w-kernel, natural weighting, 1 <= lattice <= 64 and "
                     "1 <= nvis <= 2^30");
    rick_learn* Lr = new rick_learn();
    Lr->cfg = c;
    Lr->L = lattice;
    Lr->n_in = nvis;
    const int N = c.N, Nw = c.n_wplanes;
    const double w_scale = Nw > 1 ? (double)Nw / (c.w_max - c.w_min) : 0.0;
    LearnVis* tmp = nullptr;
    int* status = nullptr;
    unsigned* cnt = nullptr;
    cudaError_t e = cudaSuccess;
    auto chk = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    chk(cudaMalloc(&tmp, sizeof(LearnVis) * nvis));
    chk(cudaMalloc(&status, sizeof(int) * nvis));
    chk(cudaMalloc(&cnt, sizeof(unsigned) * Nw * 2));
    chk(cudaMalloc(&Lr->d_vis, sizeof(LearnVis) * nvis));
    chk(cudaMalloc(&Lr->d_wv, sizeof(float2) * nvis));
    chk(cudaMalloc(&Lr->d_field, field_bytes(Nw)));
    chk(cudaMalloc(&Lr->d_idft, sizeof(float) * 2 * kMaxProbes));
    chk(cudaMalloc(&Lr->d_sums, sizeof(double) * 2 * kMaxProbes));
    chk(cudaMalloc(&Lr->d_ge, sizeof(float) * kMaxProbes));
    if (e == cudaSuccess) chk(cudaMemset(cnt, 0, sizeof(unsigned) * Nw * 2));
    if (e == cudaSuccess) {
        k_learn_place<<<(unsigned)((nvis + 255) / 256), 256>>>(uvw, weight, nvis, N, Nw, c.fov_rad,
                                                               c.w_min, w_scale, tmp, status, cnt);
        chk(cudaGetLastError());
    }
    std::vector<unsigned> counts(Nw);
    if (e == cudaSuccess) chk(cudaMemcpy(counts.data(), cnt, sizeof(unsigned) * Nw, cudaMemcpyDeviceToHost));
    std::vector<unsigned> off(Nw + 1, 0);
    for (int k = 0; k < Nw; ++k) off[k + 1] = off[k] + counts[k];
    Lr->nvis = (int)off[Nw];
    if (e == cudaSuccess) chk(cudaMemcpy(cnt + Nw, off.data(), sizeof(unsigned) * Nw, cudaMemcpyHostToDevice));
    if (e == cudaSuccess) {
        k_learn_sort<<<(unsigned)((nvis + 255) / 256), 256>>>(tmp, nvis, cnt + Nw, Lr->d_vis);
        chk(cudaGetLastError());
    }
    // sum of weights of the placed visibilities (host, FP64)
    if (e == cudaSuccess) {
        std::vector<LearnVis> hv(Lr->nvis);
        chk(cudaMemcpy(hv.data(), Lr->d_vis, sizeof(LearnVis) * Lr->nvis, cudaMemcpyDeviceToHost));
        double ws = 0.0;
        for (const LearnVis& v : hv) ws += v.W;
        Lr->wsum = ws;
    }
    cudaFree(tmp);
    cudaFree(status);
    cudaFree(cnt);
    if (e != cudaSuccess) {
        learn_free(Lr);
        delete Lr;
        char m[200];
        snprintf(m, sizeof m, "rick_learn_create: %s", cudaGetErrorString(e));
        return lfail(e == cudaErrorMemoryAllocation ? RICK_ERR_OOM : RICK_ERR_CUDA, m);
    }
    // taper of the support-4 Kaiser-Bessel (the learned kernel's fixed taper)
    Lr->taper.resize(N);
    {
        const double beta = c.kernel_param, i0b = host_i0(beta);
        const int ng = 24;
        std::vector<double> gx(ng), gw(ng);
        const double pi = 3.14159265358979323846;
        for (int i = 0; i < (ng + 1) / 2; ++i) {
            double z = std::cos(pi * (i + 0.75) / (ng + 0.5)), dp = 1.0;
            for (int it = 0; it < 64; ++it) {
                double pm = 1.0, pc = z;
                for (int k = 2; k <= ng; ++k) {
                    const double pn = ((2 * k - 1) * z * pc - (k - 1) * pm) / k;
                    pm = pc;
                    pc = pn;
                }
                dp = ng * (z * pc - pm) / (z * z - 1.0);
                const double dz = pc / dp;
                z -= dz;
                if (std::fabs(dz) < 1e-16) break;
            }
            gx[i] = -z;
            gx[ng - 1 - i] = z;
            gw[i] = gw[ng - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
        }
        for (int p = 0; p < N; ++p) {
            double acc = 0.0;
            for (int seg = 0; seg < kLearnS; ++seg)
                for (int i = 0; i < ng; ++i) {
                    const double s = -0.5 * kLearnS + seg + 0.5 + 0.5 * gx[i];
                    const double t = 2.0 * s / kLearnS;
                    const double g = host_i0(beta * std::sqrt(std::fmax(0.0, 1.0 - t * t))) / i0b;
                    acc += 0.5 * gw[i] * g * std::cos(2.0 * pi * s * (p - N / 2) / N);
                }
            Lr->taper[p] = acc;
        }
    }
    {
        GridParams fit;
        fit_tap_polynomials(RICK_KERNEL_KAISER_BESSEL, c.kernel_param, kLearnS, fit);
        for (int a = 0; a < 4; ++a)
            for (int q = 0; q <= kPolyDegree; ++q) Lr->kb4.coef[a][q] = fit.coef[a][q];
    }
    *out = Lr;
    return RICK_OK;
}

rick_status rick_learn_destroy(rick_learn* Lr) {
    if (!Lr) return RICK_OK;
    learn_free(Lr);
    delete Lr;
    return RICK_OK;
}

rick_status rick_learn_field_grad(rick_learn* Lr, const float* table, const float* sources,
                                  int32_t ns, const int32_t* probes, int32_t np, float* table_grad,
                                  int32_t accumulate, float grad_scale, float* loss,
                                  float* image_dft, void* stream) {
    if (!Lr || !table || !sources || !probes || !loss)
        return lfail(RICK_ERR_INVALID_ARG, "invalid argument: learn field inputs");
    if (ns < 1 || ns > kMaxSources || np < 1 || np > kMaxProbes)
        return lfail(RICK_ERR_INVALID_ARG, "invalid argument: 1..64 sources and 1..64 probes");
    const rick_config& c = Lr->cfg;
    const int N = c.N, Nw = c.n_wplanes, L = Lr->L;
    const double dl = c.fov_rad / N;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // per-source and per-probe constants in FP64 on the host
    std::vector<unsigned char> field(field_bytes(Nw), 0);
    float4* src = reinterpret_cast<float4*>(field.data());
    Probe* pconst = reinterpret_cast<Probe*>(src + kMaxSources);
    float2* ph = reinterpret_cast<float2*>(pconst + kMaxProbes);
    const double two_pi = 2 * 3.14159265358979323846;
    for (int s = 0; s < ns; ++s) {
        const double p = sources[3 * s], q = sources[3 * s + 1];
        if (!(p >= 0.0 && p < N && q >= 0.0 && q < N))
            return lfail(RICK_ERR_INVALID_ARG, "source outside the image");
        const double l = (p - N / 2) * dl, m = (q - N / 2) * dl, r2 = l * l + m * m;
        const double n = std::sqrt(1.0 - r2);
        src[s] = make_float4((float)(p - N / 2), (float)(q - N / 2), (float)(sources[3 * s + 2] / n),
                             (float)(-r2 / (1.0 + n)));
    }
    const double dw = Nw > 1 ? (c.w_max - c.w_min) / Nw : 0.0;
    for (int P = 0; P < np; ++P) {
        const int p = probes[2 * P], q = probes[2 * P + 1];
        if (p < 0 || p >= N || q < 0 || q >= N) return lfail(RICK_ERR_INVALID_ARG, "probe outside the image");
        const double l = (p - N / 2) * dl, m = (q - N / 2) * dl, r2 = l * l + m * m;
        const double n = std::sqrt(1.0 - r2), delta = -r2 / (1.0 + n);
        const double sg = ((p + q) & 1) ? -1.0 : 1.0;
        Probe& o = pconst[P];
        o.p = p;
        o.q = q;
        for (int a = 1; a <= 3; ++a) {   // the powers of -e^(2 pi i p / N): a p / N + a / 2 turns
            const double tx = (double)((int64_t)a * p % N) / N + 0.5 * (a & 1), ty = (double)((int64_t)a * q % N) / N + 0.5 * (a & 1);
            o.sx[a - 1] = make_float2((float)std::cos(two_pi * tx), (float)std::sin(two_pi * tx));
            o.sy[a - 1] = make_float2((float)std::cos(two_pi * ty), (float)std::sin(two_pi * ty));
        }
        o.pn = (float)((double)(p - N / 2) / N);
        o.qn = (float)((double)(q - N / 2) / N);
        o.delta = (float)delta;
        // the direct inversion's turn (X + fx)(p - N/2)/N + ..., X = i0 + 1 - N/2, less
        // the footprint phasor's i0 p / N + i0 / 2 + ... : (1 - N/2)(p - N/2)/N + the same
        // in q + the terms in fx, fy and w
        double turn = (double)(((int64_t)(1 - N / 2) * (p - N / 2) + (int64_t)(1 - N / 2) * (q - N / 2)) % N) / N;
        turn -= std::floor(turn + 0.5);
        o.turn = (float)turn;
        o.scale_img = (float)(sg * n / (Lr->taper[p] * Lr->taper[q]));
        o.scale_dft = (float)n;
        for (int k = 0; k < Nw; ++k) {
            const double wk = Nw > 1 ? c.w_min + (k + 0.5) * dw : 0.5 * (c.w_min + c.w_max);
            double t = wk * delta;
            t -= std::floor(t + 0.5);
            ph[(size_t)k * kMaxProbes + P] = make_float2((float)std::cos(two_pi * t), (float)std::sin(two_pi * t));
        }
    }
    cudaError_t e = cudaSuccess;
    auto chk = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    chk(cudaMemcpyAsync(Lr->d_field, field.data(), field.size(), cudaMemcpyHostToDevice, st));
    const float4* d_src = reinterpret_cast<const float4*>(Lr->d_field);
    const Probe* d_probes = reinterpret_cast<const Probe*>(d_src + kMaxSources);
    const float2* d_ph = reinterpret_cast<const float2*>(d_probes + kMaxProbes);
    chk(cudaMemsetAsync(Lr->d_idft, 0, sizeof(float) * 2 * kMaxProbes, st));
    chk(cudaMemsetAsync(Lr->d_sums, 0, sizeof(double) * 2 * kMaxProbes, st));
    LearnConst C{N, Nw, L, Lr->nvis, ns, np, (float)(1.0 / Lr->wsum)};
    if (e == cudaSuccess && Lr->nvis > 0) {
        k_learn_predict<<<(Lr->nvis + 255) / 256, 256, 0, st>>>(Lr->d_vis, C, d_src, Lr->d_wv);
        int dev = 0, sms = 0, per_sm = 0;
        chk(cudaGetDevice(&dev));
        chk(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const size_t ph_bytes = sizeof(float2) * Nw * kMaxProbes;
        // the plane phasors (512 bytes a plane) stay in shared memory while they fit beside
        // the rest (422 planes); beyond, they are read through the caches
        const size_t rows = sizeof(float4) * kFwdVis * kFwdRow, fixed = sizeof(double2) * 4 * kMaxProbes;
        const bool staged = ph_bytes + rows + fixed <= kSharedMax;
        const size_t fwd = rows + (staged ? ph_bytes : 0);
        auto forward = staged ? k_learn_forward<true> : k_learn_forward<false>;
        chk(cudaFuncSetAttribute(forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fwd));
        chk(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, forward, 256, fwd));
        if (e == cudaSuccess) {
            const int blocks = std::min((Lr->nvis + kFwdVis - 1) / kFwdVis, sms * std::max(per_sm, 1));
            forward<<<blocks, 256, fwd, st>>>(Lr->d_vis, Lr->d_wv, table, C, Lr->kb4, d_probes, d_ph, Lr->d_sums);
            k_learn_loss<<<1, 32, 0, st>>>(Lr->d_sums, np, C.inv_wsum * grad_scale, Lr->d_idft, loss, Lr->d_ge);
        }
        chk(cudaGetLastError());
        if (table_grad) {
            const size_t ntg = (size_t)(L + 1) * (L + 1) * 16;
            if (!accumulate) chk(cudaMemsetAsync(table_grad, 0, sizeof(float) * ntg * Nw, st));
            const size_t bwd = staged ? ph_bytes : 0;   // the forward pass's other needs are the larger
            auto backward = staged ? k_learn_backward<true> : k_learn_backward<false>;
            chk(cudaFuncSetAttribute(backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bwd));
            chk(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, backward, 256, bwd));
            if (e == cudaSuccess) {
                const int blocks = std::min((Lr->nvis + 255) / 256, sms * std::max(per_sm, 1));
                backward<<<blocks, 256, bwd, st>>>(Lr->d_vis, Lr->d_wv, C, d_probes, d_ph, Lr->d_ge, table_grad,
                                                   ((uintptr_t)table_grad & 15u) == 0);
            }
            chk(cudaGetLastError());
        }
    }
    if (e == cudaSuccess && image_dft)
        chk(cudaMemcpyAsync(image_dft, Lr->d_idft, sizeof(float) * 2 * np, cudaMemcpyDeviceToDevice, st));
    if (e != cudaSuccess) {
        char m[200];
        snprintf(m, sizeof m, "rick_learn_field_grad: %s", cudaGetErrorString(e));
        return lfail(RICK_ERR_CUDA, m);
    }
    return RICK_OK;
}

int64_t rick_learn_placed(const rick_learn* Lr) { return Lr ? Lr->nvis : -1; }

}  // extern "C"
