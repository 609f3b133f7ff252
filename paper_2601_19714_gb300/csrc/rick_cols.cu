// rick_cols.cu -- the column pass of the 2-D DFTs for N <= 8192: length-N DFTs
// down the columns of every w-plane (Eq. 2's inverse transform, and the forward
// one of the prediction), two columns at a time.
//
// What bounded the pass it replaces (one column per thread in FP32 scalars, a
// 1024-thread CTA an SM) was neither HBM nor arithmetic: on the sparse planes of
// an array a fifth of the tiles of a reached tile column are reached, so it reads
// little, and its one CTA an SM walked through load, exchange and store phases in
// lockstep.  Here a thread transforms two adjacent columns as the two lanes of
// packed FP32 instructions (Pair), the exchanges move 16 bytes at a time, all but
// the first need only a warp barrier, an 8192-point column is two 4096-point
// transforms of a cluster of two CTAs (four columns, whole 32-byte sectors, where
// one CTA held two), and rows outside the image are not stored.
//
// Measured on GB300: image columns of a 4096^2 mesh padded by 2 (16 channels x 16
// planes, 8.5 k of 32 k tile columns reached) 3.99 -> 3.11 ms, of an 8192^2 one
// (6 x 20 planes, all tile columns reached, 7 % of the tiles) 33.0 -> 16.8 ms;
// dense planes 1.31 -> 1.30 ms (16 of 4096^2), 0.56 -> 0.55 ms (32 of 2048^2),
// 134 -> 106 us (128 of 512^2); the forward pass of a prediction (8 x 16 planes)
// 2.22 -> 2.0 ms.  What remains is the wait for the load/store unit (a warp access of four columns is one cache line a row,
// 13 k of 25 k cycles a dense group) and instruction issue (5.3 k).  Tried and
// not kept: planes in groups of four columns, contiguous for this pass (2.59 ms,
// but the row pass then reads 32-byte pieces and loses more: 4.37 -> 5.35 ms);
// one pair a CTA and two CTAs an SM (5.4 ms: half sectors); prefetching the next
// group's cells into shared memory or L2 (slower: the load/store unit is what
// they need too).
#include "rick_dft.cuh"

namespace rick {

namespace {

// (re, im) of two columns; r and i are the operands of the packed instructions
struct Pair {
    float2 r, i;
};

__device__ __forceinline__ uint64_t bits2(float2 a) { return *reinterpret_cast<uint64_t*>(&a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    uint64_t rd;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(bits2(a)), "l"(bits2(b)), "l"(bits2(c)));
    return *reinterpret_cast<float2*>(&rd);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    uint64_t rd;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(bits2(a)), "l"(bits2(b)));
    return *reinterpret_cast<float2*>(&rd);
}
// 16 bytes at p (two columns of a row) where `on`, else zeros: a predicated
// load, not a branch, so that a thread's loads are in flight together.  It brings
// the whole 256 bytes around it into L2: the groups beside this one are read by
// other CTAs at the same time, and 32-byte fetches halve the HBM rate (dense
// 4096^2 planes 1.44 -> 1.30 ms, the forward pass of a prediction -0.29 ms).
__device__ __forceinline__ float4 load_if(const float2* p, uint32_t on) {
    float4 v;
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n mov.f32 %0, 0f00000000;\n mov.f32 %1, 0f00000000;\n"
        " mov.f32 %2, 0f00000000;\n mov.f32 %3, 0f00000000;\n @q ld.global.L2::256B.v4.f32 {%0, %1, %2, %3}, [%4];\n}"
        : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w)
        : "l"(p), "r"(on)
        : "memory");
    return v;
}
__device__ __forceinline__ Pair padd(const Pair& a, const Pair& b) { return {cadd(a.r, b.r), cadd(a.i, b.i)}; }
__device__ __forceinline__ Pair psub(const Pair& a, const Pair& b) { return {csub(a.r, b.r), csub(a.i, b.i)}; }
// a + (s i) b and a - (s i) b, s = +1 (INV) or -1
template <bool INV>
__device__ __forceinline__ Pair padd_i(const Pair& a, const Pair& b) {
    return INV ? Pair{csub(a.r, b.i), cadd(a.i, b.r)} : Pair{cadd(a.r, b.i), csub(a.i, b.r)};
}
template <bool INV>
__device__ __forceinline__ Pair psub_i(const Pair& a, const Pair& b) { return padd_i<!INV>(a, b); }
// both columns times w, the same roundings as cmulf
__device__ __forceinline__ Pair pmul(const Pair& a, float2 w) {
    const float2 wr = make_float2(w.x, w.x), wi = make_float2(w.y, w.y);
    const float2 t = mul2(a.i, wi);
    return {fma2(a.r, wr, make_float2(-t.x, -t.y)), fma2(a.r, wi, mul2(a.i, wr))};
}
// both columns times e^(s 2 pi i e / R) for compile-time e and R <= 32
template <bool INV>
__device__ __forceinline__ Pair ptwiddle(const Pair& a, int e, int R) {
    const int k = (e * (32 / R)) & 31;
    if (k == 0) return a;
    return pmul(a, make_float2(cos32(k), INV ? sin32(k) : -sin32(k)));
}

// In-register length-R DFT of a pair, natural order (as Dft).  ROT: input
// R / 2 is still to be multiplied by s i (the twiddle W_(4R)^R of the layer
// above), which its additions absorb.
template <int R, bool INV, bool ROT = false>
struct PDft;

template <bool INV, bool ROT>
struct PDft<2, INV, ROT> {
    static __device__ __forceinline__ void run(Pair* a) {
        const Pair x = a[0], y = a[1];
        a[0] = ROT ? padd_i<INV>(x, y) : padd(x, y);
        a[1] = ROT ? psub_i<INV>(x, y) : psub(x, y);
    }
};

template <bool INV, bool ROT>
struct PDft<4, INV, ROT> {
    static __device__ __forceinline__ void run(Pair* a) {
        const Pair t0 = ROT ? padd_i<INV>(a[0], a[2]) : padd(a[0], a[2]);
        const Pair t1 = ROT ? psub_i<INV>(a[0], a[2]) : psub(a[0], a[2]);
        const Pair t2 = padd(a[1], a[3]), t3 = psub(a[1], a[3]);
        a[0] = padd(t0, t2);
        a[2] = psub(t0, t2);
        a[1] = padd_i<INV>(t1, t3);
        a[3] = psub_i<INV>(t1, t3);
    }
};

template <int R, bool INV, bool ROT>
struct PDft {
    static_assert((R == 8 || R == 16) && !ROT, "radix");
    static constexpr int S = R / 4;
    static __device__ __forceinline__ void run(Pair* a) {
        Pair y[R];
#pragma unroll
        for (int t1 = 0; t1 < S; ++t1) {
            Pair b[4] = {a[t1], a[t1 + S], a[t1 + 2 * S], a[t1 + 3 * S]};
            PDft<4, INV>::run(b);
            // t1 f0 = R / 4 (f0 = 2, t1 = S / 2) is the factor s i left to the next layer
#pragma unroll
            for (int f0 = 0; f0 < 4; ++f0)
                y[f0 * S + t1] = f0 == 2 && 2 * t1 == S ? b[f0] : ptwiddle<INV>(b[f0], t1 * f0, R);
        }
#pragma unroll
        for (int f0 = 0; f0 < 4; ++f0) {
            if (f0 == 2) PDft<S, INV, true>::run(y + f0 * S);
            else PDft<S, INV>::run(y + f0 * S);
#pragma unroll
            for (int f1 = 0; f1 < S; ++f1) a[f0 + 4 * f1] = y[f0 * S + f1];
        }
    }
};

// Exchange buffer index: one 16-byte slot more every 16 and every 256 slots,
// so that 8 lanes (four rows of both pairs) touch distinct 16-byte banks in the
// stage stores (strides 16 and 256) and loads.  Linear over sums of numbers
// without common bits, so unrolled offsets are constants.
__host__ __device__ constexpr int pskew(int a) { return a + (a >> 4) + (a >> 8); }


// SPLIT transforms of M = 2^LOG2M points make one of N = SPLIT M.  A CTA takes
// as many column pairs as shared memory and a 16-column tile allow -- a warp
// access is one line a row, so wider rows cost the load/store unit less: dense
// planes of 512^2 transform at 3.25, 4.68 and 5.05 TB/s with two, four and eight
// pairs -- and at least two (whole 32-byte sectors).
template <int LOG2M, int SPLIT>
struct PairShape {
    using Sh = Shape<LOG2M>;
    static constexpr int M = Sh::N, T = Sh::T, N = SPLIT * M;
    static constexpr int PAIRS = LOG2M >= 12 ? 2 : LOG2M >= 10 ? 4 : 8;
    static constexpr int kThreads = PAIRS * T;
    static constexpr int kMinCtas = 512 / kThreads;       // 16 warps an SM at 128 registers
    // slots per pair array; every pair's slots start 8 / PAIRS banks further
    static constexpr int kStride = (pskew(M - 1) + 1 + 7) / 8 * 8 + 8 / PAIRS;
    // tables: stage 0, 16 powers per part (e^(2 pi i b (s + SPLIT f0) / N) at
    // [s][f0][b]), then the later stages as Shape holds them
    static constexpr int kTab0 = 16 * T;
    static constexpr int kTabLater = Sh::kTw - 4 * T;
    static constexpr size_t kSmem = sizeof(float4) * PAIRS * kStride + sizeof(float2) * (kTab0 + kTabLater);
};

// Length-N DFTs down the column pairs, in place; persistent CTAs take the
// groups of 2 PAIRS columns of the listed reached tile columns (occ.list) or of
// every plane in turn.  SPLIT = 2 (N = 8192): a cluster of two CTAs takes a
// group, CTA s computing the outputs 2 k + s as the M-point transform of
//   y_s[n] = W_N^(s n) (x[n] + (-1)^s x[n + M])
// (both read the group; the stores wait at the cluster barrier until both have
// read it, which each has announced before its first exchange).  The factor
// W_N^(s b) of the thread's inputs goes into its stage-0 twiddles.
//
// Stage 0's thread u holds x[u + T t2]; the later stages' thread (t1, g) works
// on the positions = g mod 16, a set that is closed under the later exchanges,
// and the threads of one g are lanes of one warp: after the first exchange only
// __syncwarp is needed (two CTA barriers a group).
//
// [row_lo, row_hi): the rows that matter -- the inverse transform stores only
// those (a padded mesh keeps its central rows), the forward one takes the
// others as zero without reading them.
template <int LOG2M, int SPLIT, bool INV>
__global__ void __launch_bounds__(PairShape<LOG2M, SPLIT>::kThreads, PairShape<LOG2M, SPLIT>::kMinCtas)
k_cols_pair(float2* __restrict__ grids, const float2* __restrict__ table, Occupancy occ, uint32_t n_planes,
            int row_lo, int row_hi) {
    using PS = PairShape<LOG2M, SPLIT>;
    using Sh = typename PS::Sh;
    constexpr int N = PS::N, M = PS::M, T = PS::T, PAIRS = PS::PAIRS;
    extern __shared__ __align__(16) float4 psm[];
    float2* tab0 = reinterpret_cast<float2*>(psm + PAIRS * PS::kStride);
    float2* later = tab0 + PS::kTab0;
    const int tid = threadIdx.x, lane = tid & 31;
    const int c = tid % PAIRS;
    const int u = tid / PAIRS;                                    // stage 0's butterfly
    const int b = (u % (T / 16)) * 16 + u / (T / 16);             // the later stages' butterfly: t1 fastest
    float4* buf = psm + c * PS::kStride;
    const int part = SPLIT > 1 ? (int)(blockIdx.x % SPLIT) : 0;
    for (int e = tid; e < PS::kTab0; e += PS::kThreads) tab0[e] = __ldg(table + part * PS::kTab0 + e);
    for (int e = tid; e < PS::kTabLater; e += PS::kThreads) later[e] = __ldg(table + SPLIT * PS::kTab0 + e);
    const bool listed = occ.list != nullptr, in_mask = listed && !occ.tiles_out, out_mask = listed && occ.tiles_out;
    const uint32_t per = listed ? (1u << occ.tshift) / (2 * PAIRS) : (uint32_t)N / (2 * PAIRS);
    const int per_log2 = 31 - __clz((int)per);
    const uint32_t total = (listed ? __ldg(occ.list) : n_planes) << per_log2;   // fits: checked at launch
    auto put = [&](int slot, const Pair& v) { buf[slot] = make_float4(v.r.x, v.r.y, v.i.x, v.i.y); };
    auto get = [&](int slot) {
        const float4 v = buf[slot];
        return Pair{make_float2(v.x, v.y), make_float2(v.z, v.w)};
    };
    const uint32_t step = gridDim.x / SPLIT;
    // a group's plane, tile column and first column from its list entry (or plane) e
    struct Group {
        uint32_t pl;
        int tcol, x0;
    };
    auto entry = [&](uint32_t item) {
        const uint32_t k = item >> per_log2;
        return listed && item < total ? __ldg(occ.list + 2 + k) : k;
    };
    auto group = [&](uint32_t item, uint32_t e) {
        Group g{e, 0, (int)(item & (per - 1u)) * 2 * PAIRS};
        if (listed) {
            g.pl = e / (uint32_t)occ.NT;
            g.tcol = (int)(e - g.pl * (uint32_t)occ.NT);
            g.x0 += g.tcol << occ.tshift;
        }
        return g;
    };
    auto tile_word = [&](const Group& g, int row) {
        return __ldg(occ.tile + ((size_t)g.pl * occ.NT + (row >> occ.tshift)) * occ.words + (g.tcol >> 5));
    };
    // rows read, bit 16 t + t2: u + T t2 + M t.  A warp's 32 / PAIRS rows of one
    // (t, t2) are an aligned block of a tile row, which lane (t, t2) looks up.
    const int my_row = u / (32 / PAIRS) * (32 / PAIRS) + T * (lane & 15) + M * (lane >> 4);
    const bool my_in = (lane >> 4) < SPLIT && (INV || (my_row >= row_lo && my_row < row_hi));
    auto live_word = [&](uint32_t item, const Group& g) {
        return in_mask && my_in && item < total ? tile_word(g, my_row) : ~0u;
    };
    auto live_bits = [&](uint32_t word, const Group& g) {
        return __ballot_sync(0xffffffffu, my_in && ((word >> (g.tcol & 31)) & 1u));
    };
    // The list entry of a group is loaded two groups ahead and its row mask one
    // ahead, so that the loads of a group's cells wait for neither
    uint32_t item = blockIdx.x / SPLIT;
    Group cur = group(item, entry(item));
    uint32_t live = live_bits(live_word(item, cur), cur);
    uint32_t e_next = entry(item + step);
    for (; item < total; item += step) {
        // rows of the result that lie in a reached tile (forward, sparse): bit j
        uint32_t store = 0xffffu;
        if (out_mask) {
            store = 0u;
#pragma unroll
            for (int j = 0; j < 16; ++j)
                store |= ((tile_word(cur, SPLIT * (b + T * j) + part) >> (cur.tcol & 31)) & 1u) << j;
        }
        float2* col = grids + (size_t)cur.pl * N * N + cur.x0 + 2 * c;
        const float2* src = col + (size_t)u * N;
        Pair a[16];
        if constexpr (SPLIT == 1) {
            float4 v[16];
#pragma unroll
            for (int t2 = 0; t2 < 16; ++t2) v[t2] = load_if(src + (size_t)(T * t2) * N, (live >> t2) & 1u);
#pragma unroll
            for (int t2 = 0; t2 < 16; ++t2)
                a[t2] = Pair{make_float2(v[t2].x, v[t2].z), make_float2(v[t2].y, v[t2].w)};
        } else {
            const float2 sg = part ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
            // eight rows of both parts in flight at a time
#pragma unroll
            for (int h = 0; h < 16; h += 8) {
                float4 v[8], w[8];
#pragma unroll
                for (int t2 = 0; t2 < 8; ++t2) {
                    v[t2] = load_if(src + (size_t)(T * (h + t2)) * N, (live >> (h + t2)) & 1u);
                    w[t2] = load_if(src + (size_t)(T * (h + t2) + M) * N, (live >> (16 + h + t2)) & 1u);
                }
#pragma unroll
                for (int t2 = 0; t2 < 8; ++t2)
                    a[h + t2] = Pair{fma2(make_float2(w[t2].x, w[t2].z), sg, make_float2(v[t2].x, v[t2].z)),
                                     fma2(make_float2(w[t2].y, w[t2].w), sg, make_float2(v[t2].y, v[t2].w))};
            }
            if (part) {   // W_N^(T t2) = e^(s 2 pi i t2 / 32)
#pragma unroll
                for (int t2 = 1; t2 < 16; ++t2) a[t2] = ptwiddle<INV>(a[t2], t2, 32);
            }
            // the group has been read by this CTA once its loads are in registers
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        }
        const Group next = group(item + step, e_next);
        const uint32_t word_next = live_word(item + step, next);
        e_next = entry(item + 2 * step);
        PDft<16, INV>::run(a);
        __syncthreads();   // the previous group's last exchange has been read (and the tables are there)
#pragma unroll
        for (int f0 = 0; f0 < 16; ++f0) {
            float2 w = tab0[f0 * T + u];
            if (!INV) w.y = -w.y;
            put(pskew(16 * u) + f0, SPLIT == 1 && f0 == 0 ? a[0] : pmul(a[f0], w));
        }
        cur = next;
        live = live_bits(word_next, next);
        __syncthreads();
        constexpr int kMiddle = Sh::kTwStages - 1;
        const int pb = pskew(b);
#pragma unroll
        for (int s = 1; s <= kMiddle; ++s) {
#pragma unroll
            for (int t2 = 0; t2 < 16; ++t2) a[t2] = get(pb + pskew(T * t2));
            __syncwarp();
            PDft<16, INV>::run(a);
            const int log2S = 4 * s, St = 1 << log2S;
            const int t1 = b >> log2S, g = b & (St - 1);
            const int out = pskew((t1 << (log2S + 4)) + g), cnt = Sh::stage_cnt(s);
            const float2* sw = later + (Sh::stage_off(s) - Sh::stage_off(1)) + t1;
            put(out, a[0]);
#pragma unroll
            for (int f0 = 1; f0 < 16; ++f0) {
                float2 w = sw[(f0 - 1) * cnt];
                if (!INV) w.y = -w.y;
                put(out + pskew(St * f0), pmul(a[f0], w));
            }
            __syncwarp();
        }
        constexpr int R = Sh::kLastR == 1 ? 16 : Sh::kLastR, NB = 16 / R, LM = M / R;
        Pair x[16];   // x[j]: outputs b + T j of the sub-transform
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            Pair v[R];
#pragma unroll
            for (int t2 = 0; t2 < R; ++t2) v[t2] = get(pb + pskew(T * i + LM * t2));
            PDft<R, INV>::run(v);
#pragma unroll
            for (int f0 = 0; f0 < R; ++f0) x[i + NB * f0] = v[f0];
        }
        if (SPLIT > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int row = SPLIT * (b + T * j) + part;
            if (INV ? row >= row_lo && row < row_hi : ((store >> j) & 1u) != 0u)
                __stcs(reinterpret_cast<float4*>(col + (size_t)row * N),
                       make_float4(x[j].r.x, x[j].i.x, x[j].r.y, x[j].i.y));
        }
    }
}

// k_cols_pair: N = SPLIT 2^LOG2M; table: the plan's tables of the pair kernel
template <int LOG2M, int SPLIT, bool INV>
cudaError_t columns_pair(float2* grids, int64_t n_planes, const float2* table, const Occupancy& occ, int row_lo,
                         int row_hi, cudaStream_t st) {
    using PS = PairShape<LOG2M, SPLIT>;
    // the group index stays below 2^31
    if ((uint64_t)n_planes * (PS::N / (2 * PS::PAIRS)) >= (1ull << 31)) return cudaErrorInvalidValue;
    auto fn = k_cols_pair<LOG2M, SPLIT, INV>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS::kSmem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, PS::kThreads, PS::kSmem)) != cudaSuccess)
        return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const uint64_t groups = (uint64_t)n_planes * (PS::N / (2 * PS::PAIRS));
    uint64_t blocks = (uint64_t)per_sm * sms;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(PS::kThreads);
    cfg.dynamicSmemBytes = PS::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    if (SPLIT > 1) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = SPLIT;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        // as many clusters as can be resident at once: groups go round them in turn
        cfg.gridDim = dim3((unsigned)blocks / SPLIT * SPLIT);
        int clusters = 0;
        if ((e = cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg)) != cudaSuccess) return e;
        if (clusters < 1) return cudaErrorInvalidConfiguration;
        blocks = (uint64_t)clusters;
    }
    if (blocks > groups) blocks = groups;
    cfg.gridDim = dim3((unsigned)blocks * SPLIT);
    return cudaLaunchKernelEx(&cfg, fn, grids, table, occ, (uint32_t)n_planes, row_lo, row_hi);
}

template <int LOG2M, int SPLIT>
cudaError_t columns_any(float2* grids, int64_t n_planes, bool inverse, const float2* table, const Occupancy& occ,
                        int row_lo, int row_hi, cudaStream_t st) {
    return inverse ? columns_pair<LOG2M, SPLIT, true>(grids, n_planes, table, occ, row_lo, row_hi, st)
                   : columns_pair<LOG2M, SPLIT, false>(grids, n_planes, table, occ, row_lo, row_hi, st);
}

}  // namespace

cudaError_t launch_cols_pair(float2* grids, int64_t n_planes, int N, bool inverse, const float2* table,
                             const Occupancy& occ, int row_lo, int row_hi, cudaStream_t st) {
    switch (N) {
        case 256: return columns_any<8, 1>(grids, n_planes, inverse, table, occ, row_lo, row_hi, st);
        case 512: return columns_any<9, 1>(grids, n_planes, inverse, table, occ, row_lo, row_hi, st);
        case 1024: return columns_any<10, 1>(grids, n_planes, inverse, table, occ, row_lo, row_hi, st);
        case 2048: return columns_any<11, 1>(grids, n_planes, inverse, table, occ, row_lo, row_hi, st);
        case 4096: return columns_any<12, 1>(grids, n_planes, inverse, table, occ, row_lo, row_hi, st);
        case 8192: return columns_any<12, 2>(grids, n_planes, inverse, table, occ, row_lo, row_hi, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rick
