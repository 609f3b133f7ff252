// rick_grid.cu -- convolutional gridding onto w-planes (Eq. 3), the "a1" step.
//
// Design (one GB300, HBM-bound): the unit of work is one T x T tile of one
// (channel, w-plane).  A persistent CTA takes tiles from a global counter in
// chunks ("grabs"), loads the bin offsets of the whole chunk at once, and for
// each tile
//   * accumulates every visibility that touches the tile into a shared-memory
//     tile of interleaved complex cells (row pitch T + 8 cells, so that the
//     re and im words of 8 consecutive cells of two rows hit 32 distinct
//     banks), with the checkerboard sign (-1)^(i+j) folded into the weight;
//   * hands the finished rows to the bulk-copy engine (cp.async.bulk, shared
//     -> global, one 8T-byte copy per row) and moves on: the threads never
//     hold the tile's output in registers and HBM writes overlap the next
//     tile's work;
//   * for a tile no visibility touches, copies one shared zero row T times
//     (or, with skip_empty, writes nothing: the library's pruned transforms
//     never read such a tile).
// So every grid cell is written exactly once (the zero fill is fused into
// the gridder) and no global atomics are needed: a tile is owned by one CTA,
// and the halo of neighbouring tiles is read, not written -- the binning
// stores each visibility once with its halo class.
//
// Records of the tile's own bins and of the three neighbour bins that spill
// into it form one index range.  A warp is the only writer of its tile buffer,
// so accumulation is plain FP32 load-add-store in a fixed order (no
// shared-memory atomics, which for FP32 are compare-and-swap loops, and a result
// that does not depend on scheduling).  A warp takes 32 records at once, one per
// lane, each lane prepares its record, and the warp adds them one by one
// (accumulate_slots, accumulate_slots4; accumulate_range for other supports).
// The learned support-4 kernel adds a non-separable correction interpolated from
// a per-plane lattice table.
#include <algorithm>
#include <cmath>

#include "rick_internal.cuh"

namespace rick {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxWarpGrab = 8;  // tiles a warp takes from the queue at once

// g(a + 1 - S/2 - f) for footprint tap a, by Horner in t = 2 f - 1, from the
// tap's coefficients held in registers (a lane evaluates the same tap a for
// the whole kernel, so its coefficients are loaded once: indexing the kernel
// parameter by a lane-dependent a would serialise the constant-bank reads).
__device__ __forceinline__ float tap_poly(const float (&cf)[kPolyDegree + 1], float t) {
    float acc = cf[kPolyDegree];
#pragma unroll
    for (int k = kPolyDegree - 1; k >= 0; --k) acc = fmaf(acc, t, cf[k]);
    return acc;
}

// Learned correction of a warp's 32 records: bilinear interpolation of the plane's
// (L+1)^2 x 16 lattice table, four lanes a record and 16 bytes a lane, so that a
// warp access takes eight 64-byte rows (a lane gathering its own record's rows took
// 32 lines an access, three times the load/store cycles of adding the record).
// Lane r passes record r's lattice row `at` and offsets; the 16 taps of record r go
// to slots[r stride ..].
__device__ __forceinline__ void table_taps(const GridParams& G, int at, float ax, float ay, float* slots, int stride) {
    const int lane = threadIdx.x & 31, quad = lane & 3;
    const size_t row = (size_t)(G.lattice + 1) * 4;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int r = 8 * h + (lane >> 2);
        const float x = __shfl_sync(kFull, ax, r), y = __shfl_sync(kFull, ay, r);
        const float4* t = reinterpret_cast<const float4*>(G.table) + (size_t)__shfl_sync(kFull, at, r) * 4 + quad;
        const float4 a = __ldg(t), b = __ldg(t + 4), c = __ldg(t + row), d = __ldg(t + row + 4);
        const float w00 = (1.f - x) * (1.f - y), w10 = x * (1.f - y), w01 = (1.f - x) * y, w11 = x * y;
        *reinterpret_cast<float4*>(slots + r * stride + 4 * quad) =
            make_float4(w00 * a.x + w10 * b.x + w01 * c.x + w11 * d.x, w00 * a.y + w10 * b.y + w01 * c.y + w11 * d.y,
                        w00 * a.z + w10 * b.z + w01 * c.z + w11 * d.z, w00 * a.w + w10 * b.w + w01 * c.w + w11 * d.w);
    }
}

// --- bulk copies shared -> global (sm_90+ PTX) ------------------------------

__device__ __forceinline__ void bulk_row_store(void* gdst, const void* ssrc, uint32_t bytes) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(ssrc);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n"
                 :: "l"(gdst), "r"(s), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// the shared sources of every committed group have been read
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
// every committed group has completed
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
// order this thread's generic-proxy shared writes before later async-proxy reads
__device__ __forceinline__ void fence_async_shared() {
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

// Bin bound q (0..7) of tile `item`: own bins [0,1) all classes, left
// neighbour [2,3) classes 2-3, upper [4,5) classes 1-2, upper-left [6,7)
// class 2.  Neighbours wrap around the mesh: only the Hermitian fold puts
// records in the spill classes of the last tile row or column (footprints
// ending on cell N = cell 0); without it those bins are empty.
__device__ __forceinline__ uint32_t tile_bound(const GridParams& G, const uint32_t* __restrict__ offsets,
                                               uint32_t item, uint32_t q) {
    const int NT = G.NT;
    const uint32_t tiles = (uint32_t)NT * NT;
    const uint32_t plane = item / tiles, tile = item - plane * tiles;
    const int kk = (int)(plane % G.nk), cc = (int)(plane / G.nk);
    const uint64_t kplane = ((uint64_t)(G.c0 + cc) * G.Nw + (G.k0 + kk)) * NT;
    const int ty = (int)(tile / NT), tx = (int)(tile - (uint32_t)ty * NT);
    const int txl = tx > 0 ? tx - 1 : NT - 1, tyu = ty > 0 ? ty - 1 : NT - 1;
    uint64_t key;
    int cls;
    if (q < 2) {
        key = ((kplane + ty) * NT + tx) * 4u;
        cls = q == 0 ? 0 : 4;
    } else if (q < 4) {
        key = ((kplane + ty) * NT + txl) * 4u;
        cls = q == 2 ? 2 : 4;
    } else if (q < 6) {
        key = ((kplane + tyu) * NT + tx) * 4u;
        cls = q == 4 ? 1 : 3;
    } else {
        key = ((kplane + tyu) * NT + txl) * 4u;
        cls = q == 6 ? 2 : 3;
    }
    return __ldg(offsets + key + cls);
}

// Scheduling pass: the record count of every tile, and the tiles with at
// least 64T, 16T, 4T records appended to the three lists (warp-aggregated
// atomics on the list lengths counts[0..2]); with G.light, every other tile
// with a record to the light list (length counts[4]); with G.huge, the chunks of the
// tiles to split (number counts[5]).
__global__ void k_schedule(GridParams G, const uint32_t* __restrict__ offsets,
                           uint32_t* __restrict__ counts) {
    const int lane = threadIdx.x & 31;
    const uint32_t th3 = 4u * G.T, th2 = 16u * G.T, th1 = 64u * G.T;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < G.n_items;
         base += stride) {
        const uint32_t item = base + lane;
        int level = 4;   // no list: an empty tile, or beyond the launch's last one
        if (item < G.n_items) {
            uint32_t b[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) b[q] = tile_bound(G, offsets, item, q);
            const uint32_t R = (b[1] - b[0]) + (b[3] - b[2]) + (b[5] - b[4]) + (b[7] - b[6]);
            level = R >= th1 ? 0 : R >= th2 ? 1 : R >= th3 ? 2 : R > 0 ? 3 : 4;
            if (G.huge != nullptr && R >= 2u * huge_chunk(G.T)) {
                const uint32_t n = min((R + huge_chunk(G.T) - 1u) / huge_chunk(G.T), kHugeChunks);
                const uint32_t at = atomicAdd(&counts[5], n);
                if (at <= G.huge_cap && n <= G.huge_cap - at) {
                    G.huge_done[at] = 0u;
                    for (uint32_t q = 0; q < n; ++q) G.huge[at + q] = make_uint4(item, q, n, at);
                }
            }
        }
#pragma unroll
        for (int lv = 0; lv < 4; ++lv) {
            if (lv == 3 && G.light == nullptr) break;
            const unsigned m = __ballot_sync(kFull, level == lv);
            if (m == 0u) continue;
            const int leader = __ffs(m) - 1;
            uint32_t* cnt = lv < 3 ? &counts[lv] : &counts[4];
            uint32_t at = 0;
            if (lane == leader) at = atomicAdd(cnt, (uint32_t)__popc(m));
            at = __shfl_sync(kFull, at, leader);
            if (level == lv) {
                const uint32_t pos = at + (uint32_t)__popc(m & ((1u << lane) - 1u));
                if (lv < 3) {
                    if (pos < G.list_cap) G.lists[(size_t)lv * G.list_cap + pos] = item;
                } else if (pos < G.light_cap) {
                    G.light[pos] = item;
                }
            }
        }
    }
}

// Row pitch (in cells) of a warp's tile buffer: a pass covers 16 footprint
// cells, i.e. 16 / S rows of S cells, each cell as an even/odd lane pair
// (re, im); the pitch puts those rows on disjoint bank ranges (S = 8: two
// rows 16 banks apart; S = 4: four rows 8 banks apart).
__host__ __device__ constexpr int tile_pitch(int T, int S) { return S == 4 ? T + 4 : T + 8; }

// Record g of a tile's range (own bins, then the left, upper and upper-left
// neighbours' spilling classes), its footprint starting at (i0, j0) of the tile.
__device__ __forceinline__ VisRecord tile_record(const GridParams& G, const VisRecord* __restrict__ records,
                                                 const uint32_t (&rng)[8], uint32_t g, int& i0, int& j0) {
    const uint32_t n0 = rng[1] - rng[0], n1 = rng[3] - rng[2], n2 = rng[5] - rng[4];
    const int T = G.T;
    uint32_t src;
    int dx = 0, dy = 0;
    if (g < n0) {
        src = rng[0] + g;
    } else if (g < n0 + n1) {
        src = rng[2] + (g - n0);
        dx = -T;
    } else if (g < n0 + n1 + n2) {
        src = rng[4] + (g - n0 - n1);
        dy = -T;
    } else {
        src = rng[6] + (g - n0 - n1 - n2);
        dx = -T;
        dy = -T;
    }
    VisRecord rec = records[src];
    // RICK_DEBUG: the first footprint cell lies in the record's own tile (a corrupt
    // record is dropped; the masks and clips below keep every access inside the
    // tile in any build)
    if (!RICK_DCHECK((int)(rec.px >> kFracBits) < T && (int)(rec.py >> kFracBits) < T, kCheckRecordCell, G.status)) {
        rec.wv_re = rec.wv_im = 0.f;
        rec.px = rec.py = 0;
    }
    i0 = (int)(rec.px >> kFracBits) + dx;
    j0 = (int)(rec.py >> kFracBits) + dy;
    return rec;
}

constexpr int kCellBias = 1024; // offset of a footprint's first cell, which may lie before the tile

// The columns (bits 0..7) and rows (8..15) of a footprint of support S starting at
// (i0, j0) that lie inside the tile, and the offset of its first cell (biased, 16
// bits); 0 if it does not reach the tile.
template <int S>
__device__ __forceinline__ uint32_t footprint_word(int T, int P, int i0, int j0) {
    auto inside = [&](int first) {
        const int lo = first < 0 ? min(-first, S) : 0, hi = min(S, max(T - first, 0));
        return ((1u << hi) - 1u) & ~((1u << lo) - 1u);
    };
    const uint32_t cols = inside(i0), rows = inside(j0);
    return cols != 0u && rows != 0u ? cols | (rows << 8) | ((uint32_t)(j0 * P + i0 + kCellBias) << 16) : 0u;
}

// The other supports (1 to 3, 9 to 16): accumulate records [beg, end) of one tile's
// record range into buf (interleaved re/im floats, row pitch P cells), by one warp
// that is the only writer of buf: plain FP32 load-add-store in bin order, so no
// atomics and a fixed order of additions.  rng: the tile's bin bounds -- own [0,1)
// all classes, left [2,3), up [4,5), up-left [6,7); a neighbour's records are
// relative to its origin.  The warp stages 32 records at a time in shared memory
// (fractions, W V, footprint start) and walks them: lanes 0..S-1 / S..2S-1 of a tap
// group evaluate the 2S 1-D taps, and the footprint is covered 16 cells per
// instruction, an even/odd lane pair holding the re/im words of one cell.
__device__ __forceinline__ void accumulate_range(const GridParams& G, const VisRecord* __restrict__ records,
                                                 const uint32_t (&rng)[8], uint32_t beg, uint32_t end, float* buf,
                                                 int P, const float (&cf)[kPolyDegree + 1], float4* stg4, int* stg_ij) {
    const int S = G.S, T = G.T;
    constexpr float kInvFrac = 1.0f / 16777216.0f;
    const int lane = threadIdx.x & 31;
    const int comp = lane & 1, cl = lane >> 1;       // cell slot 0..15 of a pass
    // tap groups: 32 / 2S records share one tap evaluation; lane (m, q)
    const int S2 = 2 * S, RG = 32 / S2;
    const int m = lane / S2, q = lane - m * S2;
    for (uint32_t base = beg; base < end; base += 32u) {
        const uint32_t g = base + lane;
        if (g < end) {
            int i0, j0;
            const VisRecord rec = tile_record(G, records, rng, g, i0, j0);
            stg4[lane] = make_float4((float)(rec.px & kFracMask) * kInvFrac,
                                     (float)(rec.py & kFracMask) * kInvFrac, rec.wv_re, rec.wv_im);
            stg_ij[lane] = (i0 + 256) | ((j0 + 256) << 16);
        }
        __syncwarp();
        const int cnt = (int)min(32u, end - base);
        // 1-D taps of records r0 .. r0 + RG - 1 in one go: lane (m, q) holds
        // tap q of record r0 + m (x taps q < S, y taps q - S).  The taps of
        // the next group are evaluated while the current group is
        // accumulated, so the Horner chain's latency overlaps that work.
        auto group_taps = [&](int r0) {
            float t = 0.f;
            if (m < RG && r0 + m < cnt) {
                const float4 fm = stg4[r0 + m];
                t = tap_poly(cf, fmaf(2.0f, q < S ? fm.x : fm.y, -1.0f));
            }
            return t;
        };
        float tap_next = group_taps(0);
        for (int r0 = 0; r0 < cnt; r0 += RG) {
            const float tap = tap_next;
            if (r0 + RG < cnt) tap_next = group_taps(r0 + RG);
            const int nr = min(RG, cnt - r0);
            for (int mm = 0; mm < nr; ++mm) {
                const int r = r0 + mm, tb = mm * S2;
                const float4 f = stg4[r];
                const int ij = stg_ij[r];
                const int i0 = (ij & 0xffff) - 256, j0 = (ij >> 16) - 256;
                const float wv = comp ? f.w : f.z;
                const int n16 = (S * S + 15) & ~15;
                for (int c = cl; c < n16; c += 16) {
                    const int a = c % S, b = min(c / S, S - 1);
                    const float ga = __shfl_sync(kFull, tap, tb + a);
                    const float gb = __shfl_sync(kFull, tap, tb + S + b);
                    const int i = i0 + a, j = j0 + c / S;
                    if (c < S * S && (unsigned)i < (unsigned)T && (unsigned)j < (unsigned)T) {
                        float* cell = buf + 2 * (j * P + i) + comp;
                        *cell = fmaf(((i + j) & 1) ? -wv : wv, ga * gb, *cell);
                    }
                }
                __syncwarp();
            }
        }
    }
}

// Supports 5 to 8 (separable kernels; 4 below): what a record needs is prepared once by
// one lane and read by the 32 that add it.  Lane r of a batch of 32 records
// evaluates all 2S taps of record r -- the tap index is a compile-time constant,
// so the coefficients are constant-bank operands -- multiplies the x taps by W V,
// folds the checkerboard sign (-1)^(i+j) into both, and writes a slot of kSlot
// floats: 8 products (re, im), then the y taps as the pairs (b, b + 4).  The
// position, the columns and the rows of the footprint that lie inside the tile
// travel in one word through a shuffle.  A lane then owns the cells (a, rl) and
// (a, rl + 4) of every footprint: per record it makes three shared or shuffle
// reads, two mask tests and two read-modify-writes.
//
// Against lanes that evaluate two records' taps at a time and fetch each by
// shuffle (81 instructions per record and tile visited): 512 tiles of 60 records,
// S = 7 (which took the general path, a division per cell), 203 -> 14 us; 16384^2,
// S = 7, 11.7 M visibilities 6.5 -> 1.0 ms; 4096^2, S = 8, 30.6 M 3.95 -> 2.2 ms;
// with a w-kernel, 15.3 M records, 1.98 -> 1.25 ms.  Now the load/store unit binds
// it: some 12 shared-memory wavefronts a record.
constexpr int kSlot = 28;       // 112 bytes: 16-byte stores of 8 lanes fall on distinct banks

__device__ __forceinline__ float tap_uniform(const GridParams& G, int a, float t) {
    float acc = G.coef[a][kPolyDegree];
#pragma unroll
    for (int k = kPolyDegree - 1; k >= 0; --k) acc = fmaf(acc, t, G.coef[a][k]);
    return acc;
}

template <int SS>
__device__ __forceinline__ void accumulate_slots(const GridParams& G, const VisRecord* __restrict__ records,
                                                 const uint32_t (&rng)[8], uint32_t beg, uint32_t end, float* buf,
                                                 float* slots) {
    static_assert(SS >= 5 && SS <= 8, "support");
    const int T = G.T;
    constexpr float kInvFrac = 1.0f / 16777216.0f;
    const int lane = threadIdx.x & 31;
    const int P = tile_pitch(T, SS);
    const int a = lane & 7, rl = lane >> 3;
    // this lane's bits of a record's word: column a and row rl, or row rl + 4
    const uint32_t need0 = (1u << a) | (256u << rl), need1 = (1u << a) | (4096u << rl);
    float2* cell0 = reinterpret_cast<float2*>(buf) + rl * P + a - kCellBias;
    float* mine = slots + lane * kSlot;
    const float2* xs = reinterpret_cast<const float2*>(slots) + a;
    const float2* ys = reinterpret_cast<const float2*>(slots + 16) + rl;
    for (uint32_t base = beg; base < end; base += 32u) {
        const uint32_t g = base + lane;
        uint32_t word = 0u;
        if (g < end) {
            int i0, j0;
            const VisRecord rec = tile_record(G, records, rng, g, i0, j0);
            word = footprint_word<SS>(T, P, i0, j0);
            const float tx = fmaf(2.0f, (float)(rec.px & kFracMask) * kInvFrac, -1.0f);
            const float ty = fmaf(2.0f, (float)(rec.py & kFracMask) * kInvFrac, -1.0f);
            const float sg = ((i0 + j0) & 1) ? -1.f : 1.f;
            const float re = sg * rec.wv_re, im = sg * rec.wv_im;
            float x[16], y[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float gx = t < SS ? tap_uniform(G, t, tx) : 0.f, gy = t < SS ? tap_uniform(G, t, ty) : 0.f;
                x[2 * t] = (t & 1 ? -re : re) * gx;
                x[2 * t + 1] = (t & 1 ? -im : im) * gx;
                y[t] = t & 1 ? -gy : gy;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                *reinterpret_cast<float4*>(mine + 4 * t) = make_float4(x[4 * t], x[4 * t + 1], x[4 * t + 2], x[4 * t + 3]);
            *reinterpret_cast<float4*>(mine + 16) = make_float4(y[0], y[4], y[1], y[5]);
            *reinterpret_cast<float4*>(mine + 20) = make_float4(y[2], y[6], y[3], y[7]);
        }
        __syncwarp();
        const int cnt = (int)min(32u, end - base);
        auto add = [&](uint32_t w, float2 x, float2 y) {
            float2* c = cell0 + (w >> 16);
            if ((w & need0) == need0) {
                float2 v = *c;
                v.x = fmaf(x.x, y.x, v.x);
                v.y = fmaf(x.y, y.x, v.y);
                *c = v;
            }
            if ((w & need1) == need1) {
                float2 v = c[4 * P];
                v.x = fmaf(x.x, y.y, v.x);
                v.y = fmaf(x.y, y.y, v.y);
                c[4 * P] = v;
            }
            __syncwarp();   // the next record's cells may be these
        };
        int r = 0;
        for (; r + 4 <= cnt; r += 4) {
            float2 x[4], y[4];
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                w[q] = __shfl_sync(kFull, word, r + q);
                x[q] = xs[(r + q) * (kSlot / 2)];
                y[q] = ys[(r + q) * (kSlot / 2)];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) add(w[q], x[q], y[q]);
        }
        for (; r < cnt; ++r)
            add(__shfl_sync(kFull, word, r), xs[r * (kSlot / 2)], ys[r * (kSlot / 2)]);
    }
}

// Support 4, separable or with the learned correction: the same split, with the 16
// signed taps of a record (the separable ones plus the learned correction) and
// its W V in the slot; lane (c, comp) owns one word of cell c = 4b + a, so all 32
// lanes work on every record.  2 M visibilities on 16 planes of 2048^2 (GB300, whole
// planes written): learned 315 -> 194 us, separable 198 -> 157 us.
constexpr int kSlot4 = 20;      // 80 bytes: 16-byte stores of 8 lanes fall on distinct banks

template <bool TABLE>
__device__ __forceinline__ void accumulate_slots4(const GridParams& G, const VisRecord* __restrict__ records,
                                                  const uint32_t (&rng)[8], uint32_t beg, uint32_t end, int k,
                                                  float* buf, float* slots) {
    const int T = G.T;
    constexpr float kInvFrac = 1.0f / 16777216.0f;
    const int lane = threadIdx.x & 31;
    const int P = tile_pitch(T, 4);
    const int c = lane >> 1, comp = lane & 1, a = c & 3, b = c >> 2;
    const uint32_t need = (1u << a) | (256u << b);
    float* cell0 = buf + 2 * (b * P + a - kCellBias) + comp;
    float* mine = slots + lane * kSlot4;
    for (uint32_t base = beg; base < end; base += 32u) {
        const uint32_t g = base + lane;
        uint32_t word = 0u;
        VisRecord rec = {};
        int i0 = 0, j0 = 0;
        if (g < end) rec = tile_record(G, records, rng, g, i0, j0);
        const float fx = (float)(rec.px & kFracMask) * kInvFrac, fy = (float)(rec.py & kFracMask) * kInvFrac;
        if (TABLE) {
            const int L = G.lattice;
            const float X = fx * L, Y = fy * L;
            const int ix = min((int)X, L - 1), iy = min((int)Y, L - 1);
            table_taps(G, (k * (L + 1) + iy) * (L + 1) + ix, X - ix, Y - iy, slots, kSlot4);
            __syncwarp();
        }
        if (g < end) {
            word = footprint_word<4>(T, P, i0, j0);
            const float tx = fmaf(2.0f, fx, -1.0f), ty = fmaf(2.0f, fy, -1.0f);
            float tap[16];
            if (TABLE) {
#pragma unroll
                for (int t = 0; t < 16; t += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(mine + t);
                    tap[t] = v.x;
                    tap[t + 1] = v.y;
                    tap[t + 2] = v.z;
                    tap[t + 3] = v.w;
                }
            }
            float gx[4], gy[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                gx[t] = tap_uniform(G, t, tx);
                gy[t] = tap_uniform(G, t, ty);
            }
            const bool odd = ((i0 + j0) & 1) != 0;
#pragma unroll
            for (int t = 0; t < 16; ++t) {
                float v = gx[t & 3] * gy[t >> 2];
                if (TABLE) v += tap[t];
                tap[t] = ((t ^ (t >> 2)) & 1 ? !odd : odd) ? -v : v;
            }
#pragma unroll
            for (int t = 0; t < 16; t += 4)
                *reinterpret_cast<float4*>(mine + t) = make_float4(tap[t], tap[t + 1], tap[t + 2], tap[t + 3]);
            *reinterpret_cast<float2*>(mine + 16) = make_float2(rec.wv_re, rec.wv_im);
        }
        __syncwarp();
        const int cnt = (int)min(32u, end - base);
        auto add = [&](uint32_t w, float t, float wv) {
            if ((w & need) == need) {
                float* at = cell0 + 2 * (w >> 16);
                *at = fmaf(wv, t, *at);
            }
            __syncwarp();   // the next record's cells may be these
        };
        int r = 0;
        for (; r + 4 <= cnt; r += 4) {
            float t[4], wv[4];
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                w[q] = __shfl_sync(kFull, word, r + q);
                t[q] = slots[(r + q) * kSlot4 + c];
                wv[q] = slots[(r + q) * kSlot4 + 16 + comp];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) add(w[q], t[q], wv[q]);
        }
        for (; r < cnt; ++r)
            add(__shfl_sync(kFull, word, r), slots[r * kSlot4 + c], slots[r * kSlot4 + 16 + comp]);
    }
}

// Shared memory of a gridder CTA of nw warps (bytes): one zero row, one
// T x P complex tile per warp, per-warp record staging and chunk bounds.
__host__ __device__ constexpr bool uses_slots(int SS) { return SS >= 4 && SS <= 8; }
// staging bytes of a warp's 32 records: slots, or (fractions, W V) and the cell
__host__ __device__ constexpr int staging_bytes(int SS) { 
    return 32 * (SS == 4 ? kSlot4 * 4 : uses_slots(SS) ? kSlot * 4 : (int)(sizeof(float4) + sizeof(int)));
}

__host__ __device__ inline size_t grid_smem_bytes(int T, int P, int nw, int grab_max, int SS) {
    return sizeof(float) * (2 * (size_t)T + (size_t)nw * 2 * T * P) +
           (size_t)nw * staging_bytes(SS) +
           sizeof(uint32_t) * (size_t)nw * 9 * grab_max;
}

// The gridder.  work_counter: [0] dense-tile queue, [1..3] list lengths,
// [4] tile queue, [5] light list length, [6] chunks of split tiles.
//  Phase 1 -- first the chunks of the tiles with thousands of records (an array's core
//  on a small mesh: one CTA a tile made a serial chain of 28 ms out of 6 M
//  visibilities on 512^2), whose partial tiles the last CTA of a tile adds up; then
//  dense tiles (the first two longest-first lists, >= 16T records), one per CTA: the tile's records are split evenly over the warps,
//  each accumulates its share into its own tile buffer, the buffers are summed
//  in warp order (a fixed order), and the CTA hands the rows to the bulk-copy
//  engine.
//  Phase 2 -- every other tile, one warp per tile: a warp takes `grab` queue
//  positions (the third list, then all tiles in natural order, skipping those
//  already done), accumulates into its own buffer, hands the rows to the
//  bulk-copy engine, waits until the engine has read them and clears the
//  buffer; tiles without records are written from a shared zero row.  No
//  CTA-wide barrier in this phase, so a tile delays only its own warp.
template <bool TABLE, int SS>
__global__ void k_grid(GridParams G, const uint32_t* __restrict__ offsets,
                       const VisRecord* __restrict__ records, float2* __restrict__ grids,
                       uint32_t* __restrict__ work_counter) {
    extern __shared__ __align__(128) float smem[];
    __shared__ uint32_t s_heavy;
    __shared__ uint32_t s_hrng[8];
    const int T = G.T, P = tile_pitch(G.T, SS > 0 ? SS : G.S), N = G.N, NT = G.NT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t tile_f = 2 * (size_t)T * P;                       // floats per warp tile
    float2* zrow = reinterpret_cast<float2*>(smem);                 // T zero cells
    float* bufs = smem + 2 * T;
    float* buf = bufs + warp * tile_f;                              // this warp's tile
    // staging: slots, or per warp 32 float4 and (after all of those) 32 ints
    float* stg_all = bufs + nw * tile_f;
    float* slots = stg_all + warp * (staging_bytes(SS) / 4);
    float4* stg4 = reinterpret_cast<float4*>(stg_all) + warp * 32;
    int* stg_ij = reinterpret_cast<int*>(reinterpret_cast<float4*>(stg_all) + nw * 32) + warp * 32;
    uint32_t* rng_all = reinterpret_cast<uint32_t*>(stg_all + (size_t)nw * staging_bytes(SS) / 4) +
                        warp * 9 * kMaxWarpGrab;
    uint32_t* items = rng_all + 8 * kMaxWarpGrab;
    const uint32_t tiles = (uint32_t)NT * NT;
    const uint32_t row_bytes = (uint32_t)T * sizeof(float2);
    // records [beg, end) of a tile's range into this warp's tile
    auto accumulate = [&](const uint32_t (&rng)[8], uint32_t beg, uint32_t end, int k, const float (&cf)[kPolyDegree + 1]) {
        if constexpr (SS == 4)
            accumulate_slots4<TABLE>(G, records, rng, beg, end, k, buf, slots);
        else if constexpr (uses_slots(SS))
            accumulate_slots<SS>(G, records, rng, beg, end, buf, slots);
        else
            accumulate_range(G, records, rng, beg, end, buf, P, cf, stg4, stg_ij);
    };
    // this lane's tap polynomial: lane (m, q) of a tap group of 2S lanes
    // evaluates tap q mod S (x taps q < S, y taps q >= S); zero beyond the groups
    float cf[kPolyDegree + 1] = {};
    if (!uses_slots(SS)) {
        const int S = SS > 0 ? SS : G.S;
        const int S2 = 2 * S, m = lane / S2, ta = (lane - m * S2) % S;
#pragma unroll
        for (int q = 0; q <= kPolyDegree; ++q) cf[q] = m < 32 / S2 ? G.coef[ta][q] : 0.0f;
    }
    for (int e = threadIdx.x; e < 2 * T; e += blockDim.x) smem[e] = 0.f;
    {
        float4* b4 = reinterpret_cast<float4*>(buf);
        for (int e = lane; e < (int)(tile_f / 4); e += 32) b4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    fence_async_shared();
    __syncthreads();

    // longest-first lists (if any): their lengths, capped; an overflow (which
    // the capacity bound excludes) falls back to natural order for all tiles
    uint32_t n1 = 0, n2 = 0, n3 = 0, th3 = 0xffffffffu;
    uint32_t n_light = 0, n_huge = 0;
    bool light = false;   // phase 2 visits the lists only (sparse mode)
    if (G.lists) {
        n1 = __ldg(work_counter + 1);
        n2 = __ldg(work_counter + 2);
        n3 = __ldg(work_counter + 3);
        if (n1 > G.list_cap || n2 > G.list_cap || n3 > G.list_cap) {
            n1 = n2 = n3 = 0;
        } else {
            th3 = 4u * T;
            if (G.huge != nullptr) {
                n_huge = __ldg(work_counter + 6);
                if (n_huge > G.huge_cap) n_huge = 0;
            }
            if (G.light != nullptr && G.skip_empty) {
                n_light = __ldg(work_counter + 5);
                light = n_light <= G.light_cap;
            }
        }
    }

    // ---- phase 1: dense tiles, one per CTA --------------------------------
    const uint32_t nH = n1 + n2;
    auto dense_tiles = [&]() {
    for (;;) {
        if (threadIdx.x == 0) s_heavy = atomicAdd(work_counter, 1u);
        __syncthreads();
        const uint32_t hh = s_heavy;
        if (hh >= n_huge + nH) break;
        // the chunks of the split tiles first, then the dense tiles
        const uint32_t h = hh - n_huge;
        uint4 part = make_uint4(0u, 0u, 1u, 0u);
        if (hh < n_huge) part = G.huge[hh];
        const uint32_t item = hh < n_huge ? part.x : h < n1 ? G.lists[h] : G.lists[G.list_cap + (h - n1)];
        if (!RICK_DCHECK(item < G.n_items, kCheckGridItem, G.status)) {   // uniform over the CTA
            __syncthreads();   // everyone has read s_heavy before thread 0 rewrites it
            continue;
        }
        if (threadIdx.x < 8) s_hrng[threadIdx.x] = tile_bound(G, offsets, item, threadIdx.x);
        __syncthreads();
        uint32_t rng[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) rng[q] = s_hrng[q];
        const uint32_t R = (rng[1] - rng[0]) + (rng[3] - rng[2]) + (rng[5] - rng[4]) + (rng[7] - rng[6]);
        if (hh >= n_huge && n_huge != 0u && R >= 2u * huge_chunk(T)) {   // split (uniform over the CTA)
            __syncthreads();   // s_heavy and s_hrng have been read
            continue;
        }
        const uint32_t share = part.y * nw + warp, shares = part.z * nw;
        const uint32_t beg = (uint32_t)((uint64_t)R * share / shares);
        const uint32_t end = (uint32_t)((uint64_t)R * (share + 1) / shares);
        const uint32_t plane = item / tiles, tile = item - plane * tiles;
        const int kk = (int)(plane % G.nk);
        const int ty = (int)(tile / NT), tx = (int)(tile - (uint32_t)ty * NT);
        float2* out = grids + ((uint64_t)plane * N + (uint64_t)ty * T) * N + (uint64_t)tx * T;
        accumulate(rng, beg, end, G.k0 + kk, cf);
        __syncthreads();
        // sum the warps' tiles into warp 0's in warp order, clearing the others
        {
            float4* t0 = reinterpret_cast<float4*>(bufs);
            for (int e = threadIdx.x; e < (int)(tile_f / 4); e += blockDim.x) {
                float4 acc = t0[e];
                for (int w = 1; w < nw; ++w) {
                    float4* tw = reinterpret_cast<float4*>(bufs + w * tile_f) + e;
                    const float4 v = *tw;
                    acc.x += v.x;
                    acc.y += v.y;
                    acc.z += v.z;
                    acc.w += v.w;
                    *tw = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                t0[e] = acc;
            }
        }
        if (part.z > 1u) {
            // a chunk of a split tile: its partial tile to memory; the CTA that
            // finishes the tile's last chunk adds the partial tiles in chunk order
            __syncthreads();
            const int cells2 = T * T / 2, half = T / 2;   // cells two by two
            float4* mine = G.huge_part + (size_t)(part.w + part.y) * cells2;
            for (int e = threadIdx.x; e < cells2; e += blockDim.x) {
                float4* c = reinterpret_cast<float4*>(bufs + 2 * ((e / half) * P + 2 * (e % half)));
                mine[e] = *c;
                *c = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) s_heavy = atomicAdd(G.huge_done + part.w, 1u) + 1u;
            __syncthreads();
            const bool last = s_heavy == part.z;
            __syncthreads();   // s_heavy has been read
            if (!last) continue;
            __threadfence();
            for (int e = threadIdx.x; e < cells2; e += blockDim.x) {
                const float4* from = G.huge_part + (size_t)part.w * cells2 + e;
                float4 acc = __ldcg(from);
                for (uint32_t q = 1; q < part.z; ++q) {
                    const float4 v = __ldcg(from + (size_t)q * cells2);
                    acc.x += v.x;
                    acc.y += v.y;
                    acc.z += v.z;
                    acc.w += v.w;
                }
                *reinterpret_cast<float4*>(bufs + 2 * ((e / half) * P + 2 * (e % half))) = acc;
            }
        }
        fence_async_shared();
        __syncthreads();
        for (int r = threadIdx.x; r < T; r += blockDim.x)
            bulk_row_store(out + (size_t)r * N, bufs + 2 * r * P, row_bytes);
        bulk_commit();
        bulk_wait_read();
        __syncthreads();
        {
            float4* t0 = reinterpret_cast<float4*>(bufs);
            for (int e = threadIdx.x; e < (int)(tile_f / 4); e += blockDim.x) t0[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
    }
    };

    // ---- phase 2: every other tile, one warp per tile ---------------------
    const uint32_t n_pos = n3 + (light ? n_light : G.n_items);
    auto other_tiles = [&]() {
    for (;;) {
        uint32_t first = 0;
        if (lane == 0) first = atomicAdd(work_counter + 4, G.grab);
        first = __shfl_sync(kFull, first, 0);
        if (first >= n_pos) break;
        const uint32_t n = min(G.grab, n_pos - first);
        // queue positions -> tiles: the third list, then the light list (sparse
        // mode) or every tile in natural order
        if (lane < (int)n) {
            const uint32_t pos = first + lane;
            items[lane] = pos < n3 ? G.lists[2 * (size_t)G.list_cap + pos]
                          : light  ? G.light[pos - n3]
                                   : pos - n3;
        }
        __syncwarp();
        for (uint32_t e = lane; e < 8 * n; e += 32) rng_all[e] = tile_bound(G, offsets, items[e >> 3], e & 7);
        __syncwarp();
        for (uint32_t t = 0; t < n; ++t) {
            const uint32_t item = items[t];
            const uint32_t plane = item / tiles, tile = item - plane * tiles;
            const int kk = (int)(plane % G.nk);
            const int ty = (int)(tile / NT), tx = (int)(tile - (uint32_t)ty * NT);
            float2* out = grids + ((uint64_t)plane * N + (uint64_t)ty * T) * N + (uint64_t)tx * T;
            uint32_t rng[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) rng[q] = rng_all[8 * t + q];
            const uint32_t total = (rng[1] - rng[0]) + (rng[3] - rng[2]) + (rng[5] - rng[4]) +
                                   (rng[7] - rng[6]);
            if (!light && first + t >= n3 && total >= th3) continue;  // taken from a list earlier
            if (total == 0) {
                if (!G.skip_empty) {
                    for (int r = lane; r < T; r += 32) bulk_row_store(out + (size_t)r * N, zrow, row_bytes);
                    bulk_commit();
                }
                continue;
            }
            accumulate(rng, 0u, total, G.k0 + kk, cf);
            fence_async_shared();
            __syncwarp();
            for (int r = lane; r < T; r += 32)
                bulk_row_store(out + (size_t)r * N, buf + 2 * r * P, row_bytes);
            bulk_commit();
            bulk_wait_read();
            __syncwarp();
            // clear the tile for the next one (its rows have been read)
            float4* b4 = reinterpret_cast<float4*>(buf);
            for (int e = lane; e < (int)(tile_f / 4); e += 32) b4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncwarp();
        }
        __syncwarp();  // rng_all and items are rewritten by the next chunk
    }
    };

    // Half of the CTAs start on the dense tiles and half on the others, so
    // that compute-heavy and store-heavy tiles overlap; each half then helps
    // with the other queue.  Every tile is taken exactly once either way.
    if (blockIdx.x & 1) {
        other_tiles();
        __syncthreads();
        dense_tiles();
    } else {
        dense_tiles();
        other_tiles();
    }
    bulk_wait_all();
}

template <bool TABLE, int SS>
cudaError_t launch_one(const GridParams& G, const uint32_t* offsets, const VisRecord* records,
                       float2* grids, uint32_t* counter, int threads, int num_sms,
                       cudaStream_t stream) {
    const int P = tile_pitch(G.T, SS > 0 ? SS : G.S);
    const int nw = threads / 32;
    const size_t smem = grid_smem_bytes(G.T, P, nw, kMaxWarpGrab, SS);
    auto fn = k_grid<TABLE, SS>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    uint64_t blocks = (uint64_t)per_sm * num_sms;
    // fewer tiles than resident warps x grab: one tile a warp at a time, so that
    // tiles run side by side (512 tiles of 60 records: 4 in turn took 4 times as long)
    GridParams g = G;
    while (g.grab > 1 && (uint64_t)g.n_items < blocks * nw * g.grab) g.grab >>= 1;
    const uint64_t need = (2ull * g.n_items + (uint64_t)g.grab * nw - 1) / ((uint64_t)g.grab * nw);
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    fn<<<(unsigned)blocks, threads, smem, stream>>>(g, offsets, records, grids, counter);
    return cudaGetLastError();
}

}  // namespace

double fit_tap_polynomials(int kind, double param, int S, GridParams& G) {
    // g(s) for the separable kernels (FP64)
    auto i0 = [](double x) {
        const double y = 0.25 * x * x;
        double term = 1.0, sum = 1.0;
        for (int k = 1; k < 400 && term > 1e-17 * sum; ++k) {
            term *= y / ((double)k * k);
            sum += term;
        }
        return sum;
    };
    const double inv_i0b = kind == RICK_KERNEL_KAISER_BESSEL ? 1.0 / i0(param) : 0.0;
    auto g = [&](double s) {
        if (std::fabs(s) > 0.5 * S) return 0.0;
        if (kind == RICK_KERNEL_GAUSS) return std::exp(-0.5 * s * s / (param * param));
        const double t = 2.0 * s / S;
        return i0(param * std::sqrt(std::fmax(0.0, 1.0 - t * t))) * inv_i0b;
    };
    const double pi = 3.14159265358979323846;
    const int n = kPolyDegree + 1;
    double worst = 0.0;
    for (int a = 0; a < kMaxSupport; ++a)
        for (int k = 0; k <= kPolyDegree; ++k) G.coef[a][k] = 0.0f;
    for (int a = 0; a < S; ++a) {
        // h(t) = g(a + 1 - S/2 - (t + 1)/2), t in [-1, 1]: Chebyshev interpolation at
        // the n Chebyshev points, then conversion to the monomial basis in t.
        auto h = [&](double t) { return g(a + 1 - 0.5 * S - 0.5 * (t + 1.0)); };
        double c[kPolyDegree + 1];
        for (int k = 0; k < n; ++k) {
            double acc = 0.0;
            for (int j = 0; j < n; ++j) {
                const double th = pi * (j + 0.5) / n;
                acc += h(std::cos(th)) * std::cos(k * th);
            }
            c[k] = (k == 0 ? 1.0 : 2.0) * acc / n;
        }
        double mono[kPolyDegree + 1] = {0.0}, tkm1[kPolyDegree + 2] = {0.0},
               tk[kPolyDegree + 2] = {0.0}, tkp1[kPolyDegree + 2];
        tkm1[0] = 1.0;  // T0
        tk[1] = 1.0;    // T1
        mono[0] += c[0];
        if (n > 1) mono[1] += c[1];
        for (int k = 2; k < n; ++k) {
            for (int i = 0; i <= kPolyDegree + 1; ++i) tkp1[i] = -tkm1[i] + (i > 0 ? 2.0 * tk[i - 1] : 0.0);
            for (int i = 0; i <= kPolyDegree; ++i) mono[i] += c[k] * tkp1[i];
            for (int i = 0; i <= kPolyDegree + 1; ++i) {
                tkm1[i] = tk[i];
                tk[i] = tkp1[i];
            }
        }
        for (int k = 0; k <= kPolyDegree; ++k) G.coef[a][k] = (float)mono[k];
        for (int q = 0; q <= 2000; ++q) {
            const float t = (float)(-1.0 + q / 1000.0);
            float acc = G.coef[a][kPolyDegree];
            for (int k = kPolyDegree - 1; k >= 0; --k) acc = std::fmaf(acc, t, G.coef[a][k]);
            worst = std::fmax(worst, std::fabs((double)acc - h((double)t)));
        }
    }
    return worst;
}

cudaError_t launch_grid(const GridParams& G, const uint32_t* offsets, const VisRecord* records,
                        float2* grids, uint32_t* work_counter, int threads, int num_sms,
                        cudaStream_t stream, int* launches) {
    if (G.n_items == 0) return cudaSuccess;
    if (G.grab < 1 || G.grab > (uint32_t)kMaxWarpGrab) return cudaErrorInvalidValue;
    cudaError_t e;
    if (G.lists) {
        const unsigned blocks = (unsigned)std::min<uint64_t>((G.n_items + 255) / 256, (uint64_t)num_sms * 8);
        k_schedule<<<blocks, 256, 0, stream>>>(G, offsets, work_counter + 1);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    if (G.kind == RICK_KERNEL_TABLE) {
        e = launch_one<true, 4>(G, offsets, records, grids, work_counter, threads, num_sms, stream);
    } else {
        switch (G.S) {
            case 4: e = launch_one<false, 4>(G, offsets, records, grids, work_counter, threads, num_sms, stream); break;
            case 5: e = launch_one<false, 5>(G, offsets, records, grids, work_counter, threads, num_sms, stream); break;
            case 6: e = launch_one<false, 6>(G, offsets, records, grids, work_counter, threads, num_sms, stream); break;
            case 7: e = launch_one<false, 7>(G, offsets, records, grids, work_counter, threads, num_sms, stream); break;
            case 8: e = launch_one<false, 8>(G, offsets, records, grids, work_counter, threads, num_sms, stream); break;
            default: e = launch_one<false, 0>(G, offsets, records, grids, work_counter, threads, num_sms, stream); break;
        }
    }
    if (e == cudaSuccess) ++*launches;
    return e;
}

}  // namespace rick
