// rick_degrid.cu -- prediction (degridding): transformed w-planes -> visibilities.
//
// The adjoint direction of Eq. 3: for every visibility binned for prediction,
//   V = sum_{a,b} g(i0 + a - x) g(j0 + b - y) (-1)^(i+j) F_k(i0 + a, j0 + b),
// where F_k is the forward transform of the model planes built by
// k_model_planes (so that (-1)^(i+j) F_k is the plane of the w-stacking
// prediction), times the record's plane weight and conjugated for records
// that the Hermitian fold mapped onto the mirrored plane.  Without a w-kernel
// a visibility has one record and its prediction is stored; with one
// (improved w-stacking) its Sw records each add their plane's part.
//
// A scheduling pass lists the tiles that hold records, a tile of many in runs of
// kRun records, so that no warp scans empty tiles and a dense tile is shared.  One
// warp per entry copies the tile's (T + S - 1)^2 region of the plane (rows and
// columns taken mod N, which only the fold's footprints ending on cell N use) into
// its shared buffer with asynchronous copies, all in flight together, and predicts
// the records one per lane: 2S tap polynomials (the tap index is the same in all
// lanes, so the coefficients are constant-bank operands), then one chain of fused
// multiply-adds along every footprint row and one over the rows.
//
// The chains are kept for their rounding: on planes amplified by 1/taper the
// neighbouring terms of a row cancel, and one rounding a cell at the running sum is
// all that the FP32 result then carries.  Spreading a footprint over the lanes
// (products rounded one by one, then a butterfly of adds) reads shared memory
// without bank conflicts, but its sum is 2.1, 1.8, 1.6, 1.4 and 1.3 times as far from
// 64 bits at supports 8 to 4 (both orders restated in FP32, bare mesh of 1024^2; 1.2 to
// 1.4 times on the GPU at 256^2), and it was not faster:
//
// Measured on GB300, 15.3 M records on 8 x 16 planes of 4096^2 (S = 8): 0.78 ms
// here, 0.94 ms spread over the lanes, 2.01 ms one record a lane with every tile
// visited in turn from an atomic queue and its region copied through registers.  The
// random row starts of the 32 records cost bank conflicts: at 958 k records, 27 a
// reached tile, 17.6 shared-memory wavefronts a record (7.4 of them conflicts) and 38
// warp instructions.  The row pitch (T + S - 1 plus 1, 2 or 3) does not matter.
#include <algorithm>

#include "rick_internal.cuh"

namespace rick {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRun = 1024;       // records of one entry at most

// g(a + 1 - S/2 - f) for footprint tap a (warp-uniform), by Horner in t = 2 f - 1.
__device__ __forceinline__ float tap_poly_uniform(const GridParams& G, int a, float t) {
    float acc = G.coef[a][kPolyDegree];
#pragma unroll
    for (int k = kPolyDegree - 1; k >= 0; --k) acc = fmaf(acc, t, G.coef[a][k]);
    return acc;
}

__host__ __device__ constexpr int region_pitch(int T, int S) { return T + S; }   // cells

// x v + c on both words, one packed instruction (the roundings of two fmaf)
__device__ __forceinline__ float2 fma_both(float x, float2 v, float2 c) {
    const float2 xx = make_float2(x, x);
    uint64_t rd;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(rd)
        : "l"(*reinterpret_cast<const uint64_t*>(&xx)), "l"(*reinterpret_cast<const uint64_t*>(&v)),
          "l"(*reinterpret_cast<const uint64_t*>(&c)));
    return *reinterpret_cast<float2*>(&rd);
}

// First and last record of tile `item`'s own bins.
__device__ __forceinline__ uint2 own_records(const GridParams& G, const uint32_t* __restrict__ offsets, uint32_t item) {
    const uint32_t tiles = (uint32_t)G.NT * G.NT, plane = item / tiles, tile = item - plane * tiles;
    const int kk = (int)(plane % G.nk), cc = (int)(plane / G.nk);
    const uint64_t key = ((uint64_t)(G.c0 + cc) * G.Nw + (G.k0 + kk)) * tiles + tile;
    return make_uint2(__ldg(offsets + 4 * key), __ldg(offsets + 4 * key + 4));
}

// counts[0] += entries: one per run of kRun records of every tile that has any.
__global__ void __launch_bounds__(256)
k_degrid_list(GridParams G, const uint32_t* __restrict__ offsets, uint32_t* __restrict__ counts) {
    const int lane = threadIdx.x & 31;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < G.n_items; base += stride) {
        const uint32_t item = base + lane;
        uint2 own = make_uint2(0u, 0u);
        if (item < G.n_items) own = own_records(G, offsets, item);
        const uint32_t runs = (own.y - own.x + kRun - 1) / kRun;
        uint32_t sum = runs;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(kFull, sum, o);
            if (lane >= o) sum += up;
        }
        const uint32_t total = __shfl_sync(kFull, sum, 31);
        if (total == 0u) continue;
        uint32_t at = 0u;
        if (lane == 31) at = atomicAdd(counts, total);
        at = __shfl_sync(kFull, at, 31) + sum - runs;
        for (uint32_t q = 0; q < runs; ++q)
            if (at + q < G.entry_cap) G.entries[at + q] = make_uint2(item, own.x + q * kRun);
    }
}

__device__ __forceinline__ void store_prediction(const GridParams& G, float2* __restrict__ vis_out, uint32_t index,
                                                 float weight, float2 v) {
    // the plane weight, its sign bit: conjugate
    const float gw = fabsf(weight);
    const float2 out = make_float2(gw * v.x, signbit(weight) ? -gw * v.y : gw * v.y);
    if (G.w_support >= 2) atomicAdd(vis_out + index, out);
    else vis_out[index] = out;
}

template <int SS>
__global__ void k_degrid(GridParams G, const uint32_t* __restrict__ offsets,
                         const VisRecord* __restrict__ records, const float2* __restrict__ grids,
                         float2* __restrict__ vis_out, uint32_t* __restrict__ work_counter) {
    extern __shared__ __align__(16) float smem[];
    constexpr int kS = SS > 0 ? SS : kMaxSupport;
    const int S = SS > 0 ? SS : G.S;
    const int T = G.T, N = G.N, NT = G.NT;
    const int R = T + S - 1, RP = region_pitch(T, S);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2* region = reinterpret_cast<float2*>(smem) + (size_t)warp * R * RP;
    const uint32_t tiles = (uint32_t)NT * NT, n_entries = min(__ldg(work_counter + 1), G.entry_cap);
    constexpr float kInvFrac = 1.0f / 16777216.0f;

    uint32_t entry = 0;
    if (lane == 0) entry = atomicAdd(work_counter, 1u);
    for (;;) {
        entry = __shfl_sync(kFull, entry, 0);
        if (entry >= n_entries) break;
        const uint2 e = G.entries[entry];
        if (lane == 0) entry = atomicAdd(work_counter, 1u);   // the next one, taken while this one is predicted
        const uint32_t item = e.x, plane = item / tiles, tile = item - plane * tiles;
        const int ty = (int)(tile / NT), tx = (int)(tile - (uint32_t)ty * NT);
        // the tile's region of the plane: T columns, then the S - 1 beyond, rows and
        // columns mod N
        const float2* src = grids + (size_t)plane * N * N;
        auto copy = [&](int rr, int col) {
            const int gy = (ty * T + rr) & (N - 1), gx = (tx * T + col) & (N - 1);
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(region + rr * RP + col);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src + (size_t)gy * N + gx) : "memory");
        };
        for (int x = 0; x < T; x += 32)
            if (x + lane < T)
                for (int rr = 0; rr < R; ++rr) copy(rr, x + lane);
        if (S > 1)
            for (int q = lane; q < R * (S - 1); q += 32) copy(q / (S - 1), T + q % (S - 1));
        const uint32_t re = min(e.y + (uint32_t)kRun, own_records(G, offsets, item).y);
        VisRecord rec = {};
        if (e.y + lane < re) rec = records[e.y + lane];
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        for (uint32_t r = e.y + lane; r < re; r += 32u) {
            const VisRecord cur = rec;
            if (r + 32u < re) rec = records[r + 32u];   // the lane's next record, in flight meanwhile
            const int il = (int)(cur.px >> kFracBits), jl = (int)(cur.py >> kFracBits);
            const float tx2 = fmaf(2.0f, (float)(cur.px & kFracMask) * kInvFrac, -1.0f);
            const float ty2 = fmaf(2.0f, (float)(cur.py & kFracMask) * kInvFrac, -1.0f);
            // (-1)^(i0 + j0) of the footprint's first cell (T is even)
            const float s0 = ((il + jl) & 1) ? -1.f : 1.f;
            // 1-D taps with the checkerboard folded in: (-1)^a, (-1)^b
            float gx[kS], gy[kS];
#pragma unroll
            for (int a = 0; a < kS; ++a) {
                if (a < S) {
                    const float sa = (a & 1) ? -1.f : 1.f;
                    gx[a] = s0 * sa * tap_poly_uniform(G, a, tx2);
                    gy[a] = sa * tap_poly_uniform(G, a, ty2);
                }
            }
            float2 acc = make_float2(0.f, 0.f);
            const float2* row = region + jl * RP + il;
#pragma unroll
            for (int b = 0; b < kS; ++b) {
                if (b < S) {
                    float2 rs = make_float2(0.f, 0.f);
#pragma unroll
                    for (int a = 0; a < kS; ++a)
                        if (a < S) rs = fma_both(gx[a], row[b * RP + a], rs);
                    acc = fma_both(gy[b], rs, acc);
                }
            }
            store_prediction(G, vis_out, __float_as_uint(cur.wv_re), cur.wv_im, acc);
        }
        __syncwarp();  // the region is rewritten for the next entry
    }
}

template <int SS>
cudaError_t launch_degrid_one(const GridParams& G, const uint32_t* offsets, const VisRecord* records,
                              const float2* grids, float2* vis_out, uint32_t* counter, int threads,
                              int num_sms, cudaStream_t stream) {
    const int R = G.T + G.S - 1;
    const size_t smem = (size_t)(threads / 32) * R * region_pitch(G.T, G.S) * sizeof(float2);
    auto fn = k_degrid<SS>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    uint64_t blocks = (uint64_t)per_sm * num_sms;
    const uint64_t need = ((uint64_t)G.n_items + G.entry_cap) / (threads / 32) + 1;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    fn<<<(unsigned)blocks, threads, smem, stream>>>(G, offsets, records, grids, vis_out, counter);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_degrid(const GridParams& G, const uint32_t* offsets, const VisRecord* records,
                          const float2* grids, float2* vis_out, uint32_t* work_counter, int threads,
                          int num_sms, cudaStream_t stream, int* launches) {
    if (G.n_items == 0) return cudaSuccess;
    if (G.kind == RICK_KERNEL_TABLE) return cudaErrorInvalidValue;
    const unsigned list_blocks = (unsigned)std::min<uint64_t>(((uint64_t)G.n_items + 255) / 256, (uint64_t)num_sms * 8);
    k_degrid_list<<<list_blocks, 256, 0, stream>>>(G, offsets, work_counter + 1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ++*launches;
    switch (G.S) {
        case 4: e = launch_degrid_one<4>(G, offsets, records, grids, vis_out, work_counter, threads, num_sms, stream); break;
        case 5: e = launch_degrid_one<5>(G, offsets, records, grids, vis_out, work_counter, threads, num_sms, stream); break;
        case 6: e = launch_degrid_one<6>(G, offsets, records, grids, vis_out, work_counter, threads, num_sms, stream); break;
        case 7: e = launch_degrid_one<7>(G, offsets, records, grids, vis_out, work_counter, threads, num_sms, stream); break;
        case 8: e = launch_degrid_one<8>(G, offsets, records, grids, vis_out, work_counter, threads, num_sms, stream); break;
        default: e = launch_degrid_one<0>(G, offsets, records, grids, vis_out, work_counter, threads, num_sms, stream); break;
    }
    if (e == cudaSuccess) ++*launches;
    return e;
}

}  // namespace rick
