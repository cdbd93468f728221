// First key pass on the tensor cores (bf16 or fp16 keys, d = 64 or 128, window W = 64, blocks of 128 keys or more).
//
// What the pass computes (Sections 2.1-2.3): 1/||k_i||, the sums of normalised keys of every episodic
// block, and the current-memory anomaly a_c(i) = -cos(k_hat_i, mu_c(i)) with its per-head min/max, where
// mu_c(i) is the mean of the last W normalised keys.  With S_i the sum of that window,
//     k_hat_i . S_i = sum_{j in window(i)} g_ij          g_ij = k_hat_i . k_hat_j
//     ||S_i||^2     = sum_{j, l in window(i)} g_jl
// so both are sums over a band of the Gram matrix of the keys.  The raw Gram entries G_ij = k_i . k_j are
// products of 16-bit numbers summed in fp32, which is what tcgen05.mma does, so the band comes out of the
// tensor cores at no cost in instruction issue: g_ij = w_i w_j G_ij with w_i = 1/||k_i||.
//
// Work is dealt out in episodic blocks: a CTA takes a contiguous share of the call's blocks and walks it in
// spans (blocks of one head) of 128-key tiles.  A span that starts inside a head starts 64 keys early, as if the
// head began there: after those 64 keys the window sums are complete, so only their outputs are dropped.  Every SM
// gets the same share whatever the number of heads, and no block sum is split between CTAs.
//
// Keys are staged by TMA (128-byte swizzle, 64-column halves) in a ring of 128-row stages; the 64 rows in front of
// stage 0 hold a second copy of the last stage's second half, so the 64 rows before a tile always lie in front of
// it.  For tile n the MMA warp forms D = K[tile] x K[64 rows before the tile .. tile]^T (128 x 192, fp32 in tensor
// memory, double buffered, one N = 192 product per 16-wide K step).  The diagonal of D holds ||k||^2 of the
// tile's rows, so the norms cost no pass over the key values.  Row r of D holds the 64 entries of the backward band
// ending at its diagonal.  Their row sums give
//     c_r = sum of g over the 64 columns ending at the diagonal       (= k_hat . S)
// and, G being symmetric, their column sums give the forward band
//     f_j = sum of g over the rows j .. j + 63 of column j            (complete one tile later at most)
// and ||S_i||^2 follows from T_i = T_{i-1} + (2 c_i - g_ii) - (2 f_{i-W} - g_{i-W,i-W}), a prefix sum over
// the tile that restarts every tile from an exact value (the sum of the 64 x 64 Gram block that ends at
// the previous tile's last row, which is in that tile's D).  f is read with a lag of 64 rows, when every row of its
// column has been seen.  The block sums of normalised keys are a second product, K[tile]^T x (1/||k|| split three ways into
// bf16), with the tile as the transposed A operand; fp16 keys form them on the FMA pipes (kFmaSums).
//
// The CTA is a pipeline of warp groups:
//     producer (1 thread)    TMA loads of the stages
//     mma      (1 warp)      issues the Gram rectangle of the tile
//     band     (2 x 4 warps) the two groups take alternate tiles: norms from the diagonal, then row and column
//                            sums of the band and the row's part of the next exact restart value
//     sums     (4 warps)     issue the product behind the block sums, add it up over the block (fp16: 8 warps, on FMA pipes)
//     scan     (2 warps)     alternate tiles: prefix sum, a_c, outputs, min/max
// Groups hand work to each other through mbarriers; every wait is bounded and a group that gives up
// records where and leaves, which makes the others give up in turn.
//
// Bound, by clocks read in the roles.  d = 128: the warp that issues the Gram products, 1340 to 1490 cycles a tile.  It is hardly ever
// idle: 550 for the products, 180 for the commit, 300 to 500 for looks at barriers whose phase is complete (keys were there at every
// look, so memory is not waited for); the band groups are busy for 2550 of the 2900 cycles that each has for a tile.
// At 1965 MHz that would be the copy rate, but the SMs do not keep that clock under the load of this pass: clock and time
// counters over the same tiles give 1650 to 1710 MHz in a call of 110 us and 1460 to 1480 in one of 2 ms.  36 x 8 heads of 8192 x
// 128 bf16 keys with the anchors' means 130 us (93 at the copy rate), 144 x 8 x 32768 x 128 2.04 ms (1.48).  d = 64: the band
// groups, 2400 of 2530 cycles; 16 x 8 x 32768 x 64 179 us (82), at 1735 to 1785 MHz.
// What moved it last: with the block sums on the FMA pipes 128 keys took 4960 warp instructions, a third of
// them for these; on the tensor cores 3265, and the 16 warps left have 128 registers each, with which a band warp
// takes the whole band out of tensor memory before it works on it: 155 -> 132 us and 222 -> 183.
#include <type_traits>

#include "nkv_sm100.cuh"

namespace nkv {

namespace {

using namespace sm100;

constexpr int kTile = 128;                    // keys per tile (rows of D)
constexpr int kHalo = 64;                     // keys in front of a tile (W = 64)
constexpr int kStageHalfBytes = kTile * 128;  // one 64-column half of a stage
constexpr int kHaloHalfBytes = kHalo * 128;
constexpr int kBandGroup = 128;
constexpr int kSumsWarp0 = 8;
constexpr int kWRing = 8;                     // tiles whose per-row scalars (1/||k||, g_ii) are kept
constexpr int kCfRing = 4;                    // band -> scan hand-over buffers
constexpr int kSumsRing = 4;                  // tiles whose block sums may be under way
constexpr uint32_t kTmemCols = 512;           // two Gram accumulators of 192 columns, two of block sums of 64
constexpr uint32_t kGramCols = kTile + kHalo, kSumsAt = 2 * kGramCols, kSumsCols = 64;
constexpr int kBarSums = 1;                   // named barrier
constexpr int kBandCols = 96;                 // columns a quarter of the tile's rows can reach

// The warps of a CTA.  kFma: block sums on the FMA pipes (eight warps) instead of the tensor cores (four).
template <bool kFma>
struct Warps {
    static constexpr int kSums = kFma ? 8 : 4, kSumsThreads = kSums * 32;
    static constexpr int kScan0 = kSumsWarp0 + kSums, kProducer = kScan0 + 2, kMma = kScan0 + 3;
    static constexpr int kThreads = (kMma + 1) * 32;
};

template <int D>
struct Cfg {
    static constexpr int kHalves = D / 64;
    static constexpr int kStages = D == 128 ? 5 : 7;
    static constexpr int kHalfBytes = kHaloHalfBytes + kStages * kStageHalfBytes;   // halo copy, then all stages of one half
    static constexpr int kRingBytes = kHalves * kHalfBytes;
    static constexpr int kLanes = D / 8;                   // lanes per row in the FMA sums group (8 columns each)
    static constexpr int kGroups = Warps<true>::kSumsThreads / kLanes;   // row groups of that group
    static constexpr int kRowsPerGroup = kTile / kGroups;
    // Norms as the right-hand side of the block sums' product: 16 rows of kRhsKeys keys.  With d = 64 the upper half of the
    // product's rows takes the upper half of the tile's keys, for which rows 8 .. 15 hold the norms.
    // One right-hand side goes with every stage.
    static constexpr int kRhsKeys = D, kRhsBytes = 16 * kRhsKeys * 2;
};
constexpr int kMaxStages = 7;

template <int D, bool kFma>
struct Smem {
    float red[2][kFma ? 8 : 1][kFma ? D : 64];   // block sums by warp (d = 64: of the upper rows), at the end of a block
    float w[kWRing][kTile];      // 1/||k|| by row (0 outside the head)
    float g[kWRing][kTile];      // g_ii by row
    float zero[kHalo];           // the weights of the rows before a span
    float c[kCfRing][kTile];     // backward band sums of a tile
    float f[kCfRing][4][kBandCols];   // column sums of the tile's band by row quarter (columns 32 q .. 32 q + 95 of D)
    float bp[kCfRing][kTile];    // row's share of the Gram block of the tile's last 64 rows
    uint64_t full[kMaxStages];   // stage landed
    uint64_t sfree[kMaxStages];  // stage no longer needed (the tile's block sums, and the product of the next tile)
    uint64_t tfull[2];           // accumulator written
    uint64_t tempty[2];          // accumulator read (one arrival per warp of the band group)
    uint64_t wready[kWRing];     // 1/||k|| of a tile written (one arrival per warp)
    uint64_t cready[kCfRing];    // band sums of a tile written (one arrival per warp)
    uint64_t cfree[kCfRing];     // band sums of a tile consumed (by the scans of the tile and of the next)
    uint64_t rready[kMaxStages]; // split norms of a tile written (one arrival per warp)
    uint64_t sdone[kSumsRing];   // block sums of a tile formed
    uint64_t sempty[2];          // accumulator of block sums read (one arrival per warp)
    uint64_t drain[5];           // products issued before a give-up have completed, by issuing warp
    uint32_t tmem_base;
};
static_assert(kMaxStages < kWRing, "a tile's 1/||k|| has to outlive its stage");
template <int D, bool kFma>
constexpr size_t smem_bytes() { return 1024 + (size_t)Cfg<D>::kRingBytes + (kFma ? 0 : Cfg<D>::kStages * Cfg<D>::kRhsBytes) + sizeof(Smem<D, kFma>); }
static_assert(smem_bytes<128, false>() <= 232448 && smem_bytes<64, false>() <= 232448 && smem_bytes<128, true>() <= 232448 &&
                  smem_bytes<64, true>() <= 232448,
              "more shared memory than an SM has");

// The spans of a CTA: blocks [first, last) of the call (head-major), cut at head boundaries.
struct Walk {
    long long at, last;
    int nb;
};
struct Span {
    int u, blk;      // head, first block
    int row0, row1;  // the rows the span outputs
    int base;        // first row of the first tile
    int tiles;
};
__device__ __forceinline__ Walk my_walk(int units, int nblocks) {
    const long long total = (long long)units * nblocks;
    Walk w;
    w.nb = nblocks;
    w.at = total * blockIdx.x / gridDim.x;
    w.last = total * (blockIdx.x + 1) / gridDim.x;
    return w;
}
__device__ __forceinline__ bool next_span(Walk& w, int block, int N, Span& s) {
    if (w.at >= w.last) return false;
    s.u = (int)(w.at / w.nb);
    s.blk = (int)(w.at - (long long)s.u * w.nb);
    const int cnt = (int)min((long long)(w.nb - s.blk), w.last - w.at);
    w.at += cnt;
    s.row0 = s.blk * block;
    s.row1 = min(N, s.row0 + cnt * block);
    s.base = s.blk ? s.row0 - kHalo : 0;
    s.tiles = (s.row1 - s.base + kTile - 1) / kTile;
    return true;
}

// 1/sqrt(x) with one Newton step behind the approximation (rounding error only)
__device__ __forceinline__ float inv_sqrt(float x) {
    const float y = rsqrtf(x);
    return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
}

// a / sqrt(T) by Newton's method: the root and the quotient each corrected once by their residual, so that a == sqrt(T)
// gives 1 (a head of equal keys has to have equal scores).  No branches: 167 us against 174 us with the IEEE root and
// division at 36 x 8 heads of 8192 x 128 keys.
__device__ __forceinline__ float quotient_by_root(float a, float T) {
    const float y = inv_sqrt(T), r0 = T * y, q0 = a * y;
    const float r = fmaf(0.5f * y, fmaf(-r0, r0, T), r0);
    return fmaf(y, fmaf(-q0, r, a), q0);
}

// Transposed reduction of V per-lane partial values over a group of L lanes (L, V powers of two, V <= L):
// afterwards lane l holds in v[0] the complete sum of value l / (L/V).
template <int V, int L>
__device__ __forceinline__ void treduce(float* v, int l) {
    int n = V;
#pragma unroll
    for (int o = L / 2; o >= 1; o >>= 1) {
        if (n > 1) {
            const int half = n / 2;
            const bool up = (l & o) != 0;
#pragma unroll
            for (int j = 0; j < V / 2; ++j) {
                if (j < half) {
                    const float send = up ? v[j] : v[j + half];
                    const float keep = up ? v[j + half] : v[j];
                    v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            n = half;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
}

// ---------------------------------------------------------------------------- producer and MMA
// TMA producer (one thread): the tiles of every span, in order.  Rows behind the head arrive as zeros.
template <int D, bool kFma>
__device__ void producer_role(const CUtensorMap* tmap, unsigned char* ring, Smem<D, kFma>* s, Walk walk, int block, int N, int H,
                              bool keep_in_l2, int* status) {
    using C = Cfg<D>;
    uint32_t n = 0;
    const uint64_t policy = keep_in_l2 ? l2_evict_normal_policy() : l2_evict_first_policy();
    Span sp;
#pragma unroll 1
    while (next_span(walk, block, N, sp)) {
        const int g = sp.u / H, h = sp.u - g * H;
#pragma unroll 1
        for (int tau = 0; tau < sp.tiles; ++tau, ++n) {
            const int st = (int)(n % C::kStages);
            const uint32_t use = n / C::kStages;
            if (use > 0 && !mbar_wait(&s->sfree[st], (use - 1) & 1u, status, 701)) {
                // giving up: the copies already armed still land in this CTA's shared memory, so stay (bounded)
                // until the last ring of them has
#pragma unroll 1
                for (uint32_t m = n - C::kStages; m < n; ++m)
#pragma unroll 1
                    for (uint32_t spin = 0; spin < (1u << 16) && !mbar_try_wait(&s->full[m % C::kStages], (m / C::kStages) & 1u);
                         ++spin)
                        __nanosleep(256);
                return;
            }
            const bool mirror = st == C::kStages - 1;   // its second half also goes in front of stage 0
            mbar_expect_tx(&s->full[st], C::kHalves * (kStageHalfBytes + (mirror ? kHaloHalfBytes : 0)));
            const int row = sp.base + kTile * tau;
#pragma unroll
            for (int half = 0; half < C::kHalves; ++half) {
                unsigned char* hb = ring + half * C::kHalfBytes;
                unsigned char* dst = hb + kHaloHalfBytes + st * kStageHalfBytes;
                tma_load_4d(dst, tmap, 64 * half, row, h, g, &s->full[st], policy);
                tma_load_4d(dst + kHaloHalfBytes, tmap, 64 * half, row + kHalo, h, g, &s->full[st], policy);
                if (mirror) tma_load_4d(hb, tmap, 64 * half, row + kHalo, h, g, &s->full[st], policy);
            }
        }
    }
}

// MMA issuer (one warp).  A = the tile's 128 rows, B = those rows and the 64 in front of them.
__device__ __forceinline__ uint32_t count_tiles(Walk walk, int block, int N) {
    uint32_t tiles = 0;
    Span sp;
#pragma unroll 1
    while (next_span(walk, block, N, sp)) tiles += (uint32_t)sp.tiles;
    return tiles;
}
template <typename T, int D, bool kFma>
__device__ void mma_role(unsigned char* ring, Smem<D, kFma>* s, uint32_t tmem_base, Walk walk, int block, int N, int* status) {
    using C = Cfg<D>;
    constexpr uint32_t idesc = umma_idesc<T>(kTile, kTile + kHalo);
    const uint32_t ring_addr = smem_addr(ring), tiles = count_tiles(walk, block, N);
    int st = 0;
    uint32_t round = 0;
#pragma unroll 1
    for (uint32_t n = 0; n < tiles; ++n) {
        const uint32_t acc = n & 1u;
        if (!warp_wait2(&s->full[st], round, &s->tempty[acc], ((n >> 1) & 1u) ^ 1u, status, 702)) return umma_drain(&s->drain[0]);
        tc_fence_after();
        // the address field of a descriptor counts 16-byte units: a K step moves it by a constant
        const uint64_t bdesc = umma_desc_sw128(ring_addr + (uint32_t)st * kStageHalfBytes);
        const uint64_t adesc = umma_desc_sw128(ring_addr + (uint32_t)st * kStageHalfBytes + kHaloHalfBytes);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
            const uint64_t koff = (uint64_t)((uint32_t)(kk >> 2) * (uint32_t)(C::kHalfBytes >> 4) + (uint32_t)(kk & 3) * 2u);
            umma_f16(tmem_base + acc * kGramCols, adesc + koff, bdesc + koff, idesc, kk > 0);
        }
        umma_commit(&s->tfull[acc]);   // (a commit takes 170 cycles to issue: whoever waits for this one frees the stage, too)
        if (++st == C::kStages) {
            st = 0;
            round ^= 1u;
        }
    }
}

// ---------------------------------------------------------------------------- sums group
// Sums of normalised keys per episodic block.  Lane group grp (8 columns per lane) takes rows
// [grp * R, grp * R + R) of every tile and keeps its running sum in registers until the block ends; then the groups'
// parts are added up over the warp and in shared memory.
template <typename T, int D>
__device__ void sums_role(const unsigned char* ring, Smem<D, true>* s, Walk walk, int block, int N, float* __restrict__ block_sums,
                          int* status) {
    using C = Cfg<D>;
    constexpr int kSumsThreads = Warps<true>::kSumsThreads;
    constexpr int R = C::kRowsPerGroup;
    const int t = threadIdx.x - kSumsWarp0 * 32, lane = t & 31;
    const int grp = t / C::kLanes, l = t % C::kLanes, r0 = grp * R;
    const unsigned char* mine = ring + (size_t)(l >> 3) * C::kHalfBytes + kHaloHalfBytes + r0 * 128;
    uint32_t n = 0, flushes = 0;
    F2 acc[4];
    Span sp;
#pragma unroll 1
    while (next_span(walk, block, N, sp)) {
        int blk = sp.blk, end = min(sp.row0 + block, N);   // the open block and the row it ends before
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p] = pack2(0.f, 0.f);
#pragma unroll 1
        for (int tau = 0; tau < sp.tiles; ++tau, ++n) {
            const int st = (int)(n % C::kStages), slot = (int)(n & (kWRing - 1));
            bool ok = warp_wait(&s->wready[slot], (n / kWRing) & 1u, status, 704);
            ok = ok && warp_wait(&s->full[st], (n / C::kStages) & 1u, status, 705);   // complete long ago: makes the copies visible
            if (!ok) {
                bar_or(kBarSums, kSumsThreads, true);
                return;
            }
            float w[R];
#pragma unroll
            for (int i = 0; i < R; i += 4) {
                const float4 q = *reinterpret_cast<const float4*>(&s->w[slot][r0 + i]);
                w[i] = q.x, w[i + 1] = q.y, w[i + 2] = q.z, w[i + 3] = q.w;
            }
            const unsigned char* rows = mine + (size_t)st * kStageHalfBytes;
            const int R0 = sp.base + kTile * tau;
            int lo = max(sp.row0 - R0, 0);                  // tile rows [lo, cut) belong to the open block
            const int hi = min(sp.row1 - R0, kTile);
#pragma unroll 1
            while (true) {
                const int cut = min(end - R0, hi);
                const int a = lo - r0, b = cut - r0;        // the same in rows of this group
                if (a < R && b > 0) {
                    float v[R];
#pragma unroll
                    for (int i = 0; i < R; ++i) v[i] = w[i];
                    if (a > 0 || b < R) {
#pragma unroll
                        for (int i = 0; i < R; ++i) v[i] = (i >= a && i < b) ? v[i] : 0.f;
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const uint4 q = *reinterpret_cast<const uint4*>(rows + i * 128 + (((l & 7) ^ ((r0 + i) & 7)) << 4));
                        F2 x[4];
                        unpack8<T>(q, x);
                        const F2 v2 = pack2(v[i], v[i]);
#pragma unroll
                        for (int p = 0; p < 4; ++p) acc[p] = fma2(x[p], v2, acc[p]);
                    }
                }
                if (end - R0 > kTile) break;
                // the block ends in this tile
                float o[8];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    unpack2(acc[p], o[2 * p], o[2 * p + 1]);
                    acc[p] = pack2(0.f, 0.f);
                }
#pragma unroll
                for (int m = C::kLanes; m < 32; m <<= 1)   // the row groups of the warp
#pragma unroll
                    for (int p = 0; p < 8; ++p) o[p] += __shfl_xor_sync(0xffffffffu, o[p], m);
                if (lane < C::kLanes) {
                    float* dst = &s->red[flushes & 1][t >> 5][l * 8];
                    *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
                    *reinterpret_cast<float4*>(dst + 4) = make_float4(o[4], o[5], o[6], o[7]);
                }
                if (bar_or(kBarSums, kSumsThreads, false)) return;
                if (t < D) {
                    float sum = 0.f;
#pragma unroll
                    for (int q = 0; q < kSumsThreads / 32; ++q) sum += s->red[flushes & 1][q][t];
                    block_sums[((int64_t)sp.u * walk.nb + blk) * D + t] = sum;
                }
                ++flushes;   // the other buffer next: the barrier of its use orders these reads before the next writes here
                if (end >= sp.row1) break;
                lo = cut;
                ++blk;
                end = min(end + block, N);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&s->sfree[st]);
        }
    }
}

// The same from the tensor cores: row c of a tile's accumulator is channel c (d = 64: rows c and 64 + c, of the lower and of
// the upper 64 keys), its columns are the products with the three parts of the norms of the block that is open where the
// tile starts and of the next one, in sums over 32 keys each.  These are added up in fp32.  Relative error of a sum of 256
// keys, root mean square against 64 bits: 4.0e-8, as in the FMA form (4.1e-8); with all keys of a tile added in tensor
// memory, which truncates, 1.1e-7.
// The four warps read the accumulator and take turns at issuing the products, a tile ahead: one warp for these and the Gram
// products needed 1900 cycles per tile, each step of it being a wait or an issue of 150 to 550.
template <typename T, int D>
__device__ void tensor_sums_role(unsigned char* ring, const unsigned char* rhs, Smem<D, false>* s, uint32_t tmem_base, Walk walk, int block,
                                 int N, float* __restrict__ block_sums, int* status) {
    using C = Cfg<D>;
    constexpr int kSumsThreads = Warps<false>::kSumsThreads, kParts = C::kRhsKeys / 32;
    const int t = threadIdx.x - kSumsWarp0 * 32, lane = t & 31, q = t >> 5;
    const bool upper = D == 64 && q >= 2;
    const uint32_t at = tmem_base + ((uint32_t)(32 * q) << 16) + kSumsAt + (upper ? 8u : 0u);
    const uint32_t ring_addr = smem_addr(ring), rhs_addr = smem_addr(rhs), tiles = count_tiles(walk, block, N);
    auto issue = [&](uint32_t m) {   // A = the tile's keys with the channels as rows, B = its split norms
        constexpr uint32_t idesc = umma_idesc<T>(kTile, 16) | kTransposeA;
        const uint32_t st = m % C::kStages, buf = m & 1u;
        if (!warp_wait2(&s->rready[st], (m / C::kStages) & 1u, &s->sempty[buf], ((m >> 1) & 1u) ^ 1u, status, 717)) return false;
        tc_fence_after();
        // the channels' second 64 rows: the other half of the stage (d = 128), or the upper 64 keys (d = 64)
        const uint64_t adesc = umma_desc_sw128_mn(ring_addr + st * kStageHalfBytes + kHaloHalfBytes,
                                                  D == 128 ? (uint32_t)C::kHalfBytes : (uint32_t)kHaloHalfBytes);
        const uint64_t bdesc = umma_desc_sw128(rhs_addr + st * C::kRhsBytes);
#pragma unroll
        for (int kk = 0; kk < C::kRhsKeys / 16; ++kk)   // 32 keys per sum in tensor memory
            umma_f16(tmem_base + kSumsAt + buf * kSumsCols + (uint32_t)(kk >> 1) * 16u, adesc + (uint64_t)(kk * 2048 >> 4),
                     bdesc + (uint64_t)((kk >> 2) * 2048 + (kk & 3) * 32 >> 4), idesc, kk & 1);
        umma_commit(&s->sdone[m & (kSumsRing - 1)]);
        return true;
    };
    auto give_up = [&] {
        umma_drain(&s->drain[1 + q]);
        if (D == 64) bar_or(kBarSums, kSumsThreads, true);
    };
    uint32_t n = 0, flushes = 0;
    Span sp;
    if (q == 0 && tiles > 0 && !issue(0)) return give_up();
#pragma unroll 1
    while (next_span(walk, block, N, sp)) {
        int blk = sp.blk, end = min(sp.row0 + block, N);   // the open block and the row it ends before
        float acc = 0.f;
#pragma unroll 1
        for (int tau = 0; tau < sp.tiles; ++tau, ++n) {
            const int rs = (int)(n & (kSumsRing - 1)), buf = (int)(n & 1);
            if (((n + 1) & 3u) == (uint32_t)q && n + 1 < tiles && !issue(n + 1)) return give_up();
            if (!warp_wait(&s->sdone[rs], (n / kSumsRing) & 1u, status, 719)) return give_up();
            if (t == 0) mbar_arrive(&s->sfree[n % C::kStages]);
            tc_fence_after();
            float v[kParts][8];
            tmem_ld8<kParts, 16>(at + (uint32_t)buf * kSumsCols, v);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s->sempty[buf]);
            float part[6];
#pragma unroll
            for (int p = 0; p < 6; ++p) {
                if constexpr (kParts == 4) part[p] = (v[0][p] + v[1][p]) + (v[2][p] + v[3][p]);
                else part[p] = v[0][p] + v[1][p];
            }
            acc += part[0] + (part[1] + part[2]);
            const int stop = min(sp.base + kTile * (tau + 1), sp.row1);
            float next = part[3] + (part[4] + part[5]);
#pragma unroll 1
            while (end <= stop) {   // the block ends in this tile
                if constexpr (D == 64) {
                    if (upper) s->red[flushes & 1][0][t - 64] = acc;
                    if (bar_or(kBarSums, kSumsThreads, false)) return umma_drain(&s->drain[1 + q]);
                    if (!upper) acc += s->red[flushes & 1][0][t];
                    ++flushes;   // the other buffer next: the barrier of its use orders these reads before the next writes here
                }
                if (!upper) block_sums[((int64_t)sp.u * walk.nb + blk) * D + t] = acc;
                if (end >= sp.row1) break;
                acc = next;
                next = 0.f;
                ++blk;
                end = min(end + block, N);
            }
        }
    }
}

// ---------------------------------------------------------------------------- band groups
// A warp takes the 32 rows of one lane quarter q of D.  Row lr of the quarter has its diagonal at column
// 64 + 32 q + lr; the band is the 64 columns that end there.  They live in three 32-column chunks X, Y, Z starting at
// column 32 q, of which the first and the last are cut by the diagonal: column o of X counts when o > lr, column o
// of Z when o <= lr.
//
// The accumulator is read in the fragment layout (tmem_ld_frag32): a thread holds columns 8 k + b0 + e
// (b0 = 2 (t % 4), k = 0..3, e = 0, 1) of the four rows 8 J + t / 4 (J = 2 half + j, value 4 k + 2 j + e of that
// half).  With r0 = t / 4 + 1 the cut 8 k + b0 + e >= 8 J + r0 is decided by k alone unless k == J
// (0 <= b0 + e <= 7, 1 <= r0 <= 8): columns with k > J lie past the cut, columns with k < J before it, and the pair
// k == J is tested against r0.  Every entry is used twice from registers: times its column's 1/||k|| for the row sum,
// times its row's for the column sum.
enum { kChunkX, kChunkY, kChunkZ };

template <int kChunk>
__device__ __forceinline__ void chunk_sums(const float (*v)[16], const float* wcol, const float* wrow, bool p0, bool p1, F2* row,
                                           F2* col) {
    F2 w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 f = *reinterpret_cast<const float2*>(wcol + 8 * k);
        w[k] = pack2(f.x, f.y);
        col[k] = pack2(0.f, 0.f);
    }
#pragma unroll
    for (int J = 0; J < 4; ++J) {
        const F2 wr = pack2(wrow[J], wrow[J]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if ((kChunk == kChunkX && k < J) || (kChunk == kChunkZ && k > J)) continue;
            float v0 = v[J >> 1][4 * k + 2 * (J & 1)], v1 = v[J >> 1][4 * k + 2 * (J & 1) + 1];
            if (kChunk != kChunkY && k == J) {
                v0 = p0 == (kChunk == kChunkX) ? v0 : 0.f;
                v1 = p1 == (kChunk == kChunkX) ? v1 : 0.f;
            }
            const F2 x = pack2(v0, v1);
            row[J] = fma2(x, w[k], row[J]);
            col[k] = fma2(x, wr, col[k]);
        }
    }
}

// Norms of the quarter's rows, one per lane: lane t has row lr = 8 (t % 4) + t / 4.  The diagonal entries of rows t / 4 + 8 J,
// in columns 8 J + b0 + e with e = (t / 4) % 2, are held by lane t / 8 of the four lanes that share these rows.
__device__ __forceinline__ float own_diagonal(const float (*z)[16], int t) {
    float G = 0.f;
#pragma unroll
    for (int J = 0; J < 4; ++J) {
        const float* c = z[J >> 1] + 4 * J + 2 * (J & 1);
        const float d = __shfl_sync(0xffffffffu, (t & 4) ? c[1] : c[0], (t & 28) | (t >> 3));
        if ((t & 3) == J) G = d;
    }
    return G;
}
// A row's norm in three bf16 parts (24 mantissa bits), as column `row` of the right-hand side of the block sums' product: in
// rows 0 .. 2 for a key of the block that is open where the tile starts, 3 .. 5 for one of the next; zeros otherwise.
template <int D>
__device__ __forceinline__ void split_norm(unsigned char* rhs, int row, float w, bool first, bool second) {
    const int kk = row & 63;
    unsigned char* at = rhs + (row >> 6) * (D == 128 ? 2048 : 1024) + (kk & 7) * 2;
    const __nv_bfloat16 hi = __float2bfloat16_rn(w);
    const float r1 = w - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1), lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
    const uint16_t part[3] = {__bfloat16_as_ushort(hi), __bfloat16_as_ushort(mid), __bfloat16_as_ushort(lo)};
#pragma unroll
    for (int line = 0; line < 6; ++line)
        *reinterpret_cast<uint16_t*>(at + line * 128 + (((kk >> 3) ^ line) << 4)) = (line < 3 ? first : second) ? part[line % 3] : (uint16_t)0;
}

// kSums: the norms go to the tensor cores as well.  kEarly (128 registers per thread): the whole band is loaded at once, and
// the next product into this accumulator is not held up by the arithmetic.
template <int D, bool kFma, bool kGiven, bool kSums>
__device__ void band_role(unsigned char* rhs, Smem<D, kFma>* s, uint32_t tmem_base, Walk walk, int block, int N,
                          const float* __restrict__ given, int64_t inv_row, int* status) {
    constexpr bool kEarly = !kFma;
    const int warp = threadIdx.x >> 5, t = threadIdx.x & 31;
    const int q = warp & 3, which = warp >> 2;   // lane quarter; the group takes tiles n with n % 2 == which
    const int b0 = 2 * (t & 3), r0 = (t >> 2) + 1;
    const bool p0 = b0 >= r0, p1 = b0 + 1 >= r0;
    const int own = 32 * q + 8 * (t & 3) + (t >> 2);   // the lane's own row where every lane has one
    const uint32_t tq = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)which * kGramCols + (uint32_t)(32 * q);
    // Columns 0 .. 63 of a span's first tile are products with whatever the ring holds, keys of another head among it.  They
    // are dropped and not only weighed with 0, which an infinity or a NaN among them would survive.
    auto drop = [](float(&v)[2][16]) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i >> 4][i & 15] = 0.f;
    };
    uint32_t n = 0;
    int st = 0, last = 0;   // stages of the tile and of the one before
    auto step = [&] {
        ++n;
        last = st;
        st = st + 1 == Cfg<D>::kStages ? 0 : st + 1;
    };
    Span sp;
#pragma unroll 1
    while (next_span(walk, block, N, sp)) {
        int end = sp.row0 + block;   // of the block that is open where the tile starts
#pragma unroll 1
        for (int tau = 0; tau < sp.tiles; ++tau, step()) {
            const int R0 = sp.base + kTile * tau;
            if (kSums && end <= R0) end += block;   // (a block has at least a tile's keys)
            if ((int)(n & 1) != which) continue;
            const int slot = (int)(n & (kWRing - 1)), prev = (int)((n - 1) & (kWRing - 1)), cb = (int)(n & (kCfRing - 1));
            const int i = R0 + own;
            const float have = kGiven && i < N ? given[sp.u * inv_row + i] : 0.f;
            if (!warp_wait(&s->tfull[which], (n >> 1) & 1u, status, 706)) return;
            if (q == 0 && t == 0 && n > 0) mbar_arrive(&s->sfree[last]);   // read as the rows in front of this tile
            tc_fence_after();
            float z[2][16], y[2][16], x_early[2][16];
            float(&x)[2][16] = *(kEarly ? &x_early : &z);
            tmem_ld_frag32(tq + 64, z[0]);
            tmem_ld_frag32(tq + 64 + (16u << 16), z[1]);
            tmem_wait_ld(z[0], z[1]);
            tmem_ld_frag32(tq + 32, y[0]);
            tmem_ld_frag32(tq + 32 + (16u << 16), y[1]);
            if constexpr (kEarly) {
                tmem_ld_frag32(tq, x[0]);
                tmem_ld_frag32(tq + (16u << 16), x[1]);
            }
            const float G = own_diagonal(z, t);
            const float wi = kGiven ? have : i < N ? inv_sqrt(fmaxf(G, kEps * kEps)) : 0.f;   // 1 / max(||k||, eps)
            s->w[slot][own] = wi;
            s->g[slot][own] = wi * wi * G;
            __syncwarp();
            if (t == 0) mbar_arrive(&s->wready[slot]);
            if constexpr (kEarly) {
                tmem_wait_ld(y[0], y[1]);
                tmem_wait_ld(x[0], x[1]);
                tc_fence_before();
                __syncwarp();
                if (t == 0) mbar_arrive(&s->tempty[which]);
            }
            if constexpr (kSums) {   // (the stage's earlier right-hand side was used up before the stage was filled again)
                split_norm<D>(rhs + st * Cfg<D>::kRhsBytes, own, wi, i >= sp.row0 && i < end && i < sp.row1, i >= end && i < sp.row1);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads these writes
                __syncwarp();
                if (t == 0) mbar_arrive(&s->rready[st]);
            }
            float wrow[4];
#pragma unroll
            for (int J = 0; J < 4; ++J) wrow[J] = s->w[slot][32 * q + 8 * J + (t >> 2)];
            F2 row[4], cx[4], cy[4], cz[4], part[4];
#pragma unroll
            for (int J = 0; J < 4; ++J) row[J] = pack2(0.f, 0.f);
            chunk_sums<kChunkZ>(z, &s->w[slot][32 * q + b0], wrow, p0, p1, row, cz);
#pragma unroll
            for (int J = 0; J < 4; ++J) part[J] = row[J];
            // the other columns belong to rows of the other warps and of the tile before
            {
                const bool both = q < 2 && tau > 0;
                if (!warp_wait2(&s->wready[slot], (n / kWRing) & 1u, &s->wready[both ? prev : slot], ((both ? n - 1 : n) / kWRing) & 1u,
                                status, 707))
                    return;
            }
            const float* before = tau > 0 ? &s->w[prev][kTile - kHalo] : s->zero;   // columns 0 .. 63
            const float* wy = q >= 1 ? &s->w[slot][32 * q - 32] : before + 32;
            const float* wx = q >= 2 ? &s->w[slot][32 * q - 64] : before + 32 * q;
            if constexpr (!kEarly) {
                tmem_wait_ld(y[0], y[1]);
                tmem_ld_frag32(tq, x[0]);
                tmem_ld_frag32(tq + (16u << 16), x[1]);
            }
            if (tau == 0 && q == 0) drop(y);
            chunk_sums<kChunkY>(y, wy + b0, wrow, p0, p1, row, cy);
            if (q == 3) {
#pragma unroll
                for (int J = 0; J < 4; ++J) part[J] = row[J];
            }
            if constexpr (!kEarly) {
                tmem_wait_ld(x[0], x[1]);
                tc_fence_before();
                __syncwarp();
                if (t == 0) mbar_arrive(&s->tempty[which]);
            }
            if (tau == 0 && q < 2) drop(x);
            chunk_sums<kChunkX>(x, wx + b0, wrow, p0, p1, row, cx);

            // row sums over the four lanes of a row; afterwards lane t holds row 8 (t % 4) + t / 4 of the quarter
            float tot[4];
#pragma unroll
            for (int J = 0; J < 4; ++J) tot[J] = hsum2(row[J]);
            treduce<4, 4>(tot, t & 3);
            // column sums over the eight row groups: value 3 m + chunk with m = 2 k + e; afterwards lane t holds
            // m = t / 4 of the three chunks
            float cs[24];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                unpack2(cx[k], cs[6 * k], cs[6 * k + 3]);
                unpack2(cy[k], cs[6 * k + 1], cs[6 * k + 4]);
                unpack2(cz[k], cs[6 * k + 2], cs[6 * k + 5]);
            }
#pragma unroll
            for (int lev = 0; lev < 3; ++lev) {
                const int half = 12 >> lev, o = 16 >> lev;
                const bool up = (t & o) != 0;
#pragma unroll
                for (int j = 0; j < 12; ++j)
                    if (j < half) {
                        const float send = up ? cs[j] : cs[j + half], keep = up ? cs[j + half] : cs[j];
                        cs[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
            }
            if (!warp_wait(&s->cfree[cb], ((n / kCfRing) & 1u) ^ 1u, status, 709)) return;
            s->c[cb][own] = wi * tot[0];
            // Gram block of the tile's last 64 rows: columns 128 .. diagonal of rows 64 .. 127
            if (q >= 2) {
                float pt[4];
#pragma unroll
                for (int J = 0; J < 4; ++J) pt[J] = hsum2(part[J]);
                treduce<4, 4>(pt, t & 3);
                s->bp[cb][own] = wi * pt[0];
            }
            const int m = t >> 2, lc = 8 * (m >> 1) + b0 + (m & 1);
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) s->f[cb][q][32 * ch + lc] = cs[ch];
            __syncwarp();
            if (t == 0) mbar_arrive(&s->cready[cb]);
        }
    }
}

// ---------------------------------------------------------------------------- scan warps
// Lane l owns rows 4 l .. 4 l + 3 of the tile: T_i = anchor + prefix of (2 c_i - g_ii) - (2 f_{i-64} - g_{i-64,i-64}).
// Row i - 64 is column r = i - R0 of the tile's D: its forward band is the sum of the column parts of this tile's row
// quarters that reach column r and, for r < 64, of those of the tile before (where it was column r + 128).  The
// anchor is the sum of the Gram block of the 64 rows before the tile.  Nothing is handed from tile to tile, so two
// warps take alternate tiles.
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x, a.y += b.y, a.z += b.z, a.w += b.w; }

// (Out of line: five roles share the instruction caches, and with this one inlined the pass took 158 instead of 154 us at
// 36 x 8 heads of 8192 x 128 keys.)
template <int D, bool kFma, bool kGiven>
__device__ __noinline__ void scan_role(Smem<D, kFma>* s, Walk walk, int block, int N, float* __restrict__ inv_norm, int64_t inv_row,
                          float* __restrict__ a_raw, int64_t raw_row, uint32_t* __restrict__ mm, int* status) {
    const int which = (threadIdx.x >> 5) - Warps<kFma>::kScan0, l = threadIdx.x & 31;
    const int r = 4 * l, q = l >> 3, c = r - 32 * q;
    uint32_t n = 0;
    Span sp;
#pragma unroll 1
    while (next_span(walk, block, N, sp)) {
        float lo = INFINITY, hi = -INFINITY;
#pragma unroll 1
        for (int tau = 0; tau < sp.tiles; ++tau, ++n) {
            if ((int)(n & 1) != which) continue;
            const int cb = (int)(n & (kCfRing - 1)), pb = (int)((n - 1) & (kCfRing - 1));
            const int slot = (int)(n & (kWRing - 1)), prev = (int)((n - 1) & (kWRing - 1));
            if (!warp_wait2(&s->cready[cb], (n / kCfRing) & 1u, &s->cready[tau > 0 ? pb : cb], ((tau > 0 ? n - 1 : n) / kCfRing) & 1u, status, 710))
                return;
            const float4 ci = ld4(&s->c[cb][r]), gi = ld4(&s->g[slot][r]), wi = ld4(&s->w[slot][r]);
            float4 F = ld4(&s->f[cb][q][c]);
            if (q >= 1) add4(F, ld4(&s->f[cb][q - 1][c + 32]));
            if (q >= 2) add4(F, ld4(&s->f[cb][q - 2][c + 64]));
            float x[4] = {2.f * ci.x - gi.x, 2.f * ci.y - gi.y, 2.f * ci.z - gi.z, 2.f * ci.w - gi.w};
            float anchor = 0.f;
            if (tau > 0 && l >= 16) {
                const float4 b = ld4(&s->bp[pb][r]), g = ld4(&s->g[prev][r]);
                anchor = ((2.f * b.x - g.x) + (2.f * b.y - g.y)) + ((2.f * b.z - g.z) + (2.f * b.w - g.w));
            }
            if (l >= 16 || tau > 0) {
                if (l < 16) {
                    add4(F, ld4(&s->f[pb][3][r + 32]));
                    if (l < 8) add4(F, ld4(&s->f[pb][2][r + 64]));
                }
                const float4 wj = l >= 16 ? ld4(&s->w[slot][r - 64]) : ld4(&s->w[prev][r + 64]);
                const float4 gj = l >= 16 ? ld4(&s->g[slot][r - 64]) : ld4(&s->g[prev][r + 64]);
                x[0] -= 2.f * (wj.x * F.x) - gj.x;
                x[1] -= 2.f * (wj.y * F.y) - gj.y;
                x[2] -= 2.f * (wj.z * F.z) - gj.z;
                x[3] -= 2.f * (wj.w * F.w) - gj.w;
            }
            __syncwarp();
            if (l == 0) {   // everything of this tile and the tile before has been read
                mbar_arrive(&s->cfree[cb]);
                if (n > 0) mbar_arrive(&s->cfree[pb]);
            }
#pragma unroll
            for (int e = 1; e < 4; ++e) x[e] += x[e - 1];
            float incl = x[3];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float y = __shfl_up_sync(0xffffffffu, incl, o);
                if (l >= o) incl += y;
            }
            const float base = warp_sum(anchor) + (incl - x[3]);
            const float cc[4] = {ci.x, ci.y, ci.z, ci.w}, ww[4] = {wi.x, wi.y, wi.z, wi.w};
            float ac[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) ac[e] = quotient_by_root(-cc[e], fmaxf(base + x[e], kEps * kEps)) + 0.f;
            const int i = sp.base + kTile * tau + r;
            float* out_a = a_raw + ((int64_t)sp.u * 3 + 2) * raw_row + i;
            float* out_w = kGiven ? out_a : inv_norm + sp.u * inv_row + i;
            if (i >= sp.row0 && i + 4 <= sp.row1 && ((reinterpret_cast<uintptr_t>(out_a) | reinterpret_cast<uintptr_t>(out_w)) & 15) == 0) {
                *reinterpret_cast<float4*>(out_a) = make_float4(ac[0], ac[1], ac[2], ac[3]);
                if (!kGiven) *reinterpret_cast<float4*>(out_w) = wi;
#pragma unroll
                for (int e = 0; e < 4; ++e) lo = fminf(lo, ac[e]), hi = fmaxf(hi, ac[e]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (i + e >= sp.row0 && i + e < sp.row1) {
                        out_a[e] = ac[e];
                        if (!kGiven) out_w[e] = ww[e];
                        lo = fminf(lo, ac[e]), hi = fmaxf(hi, ac[e]);
                    }
            }
        }
        // ---- min/max of a_c over the warp's tiles of the span
        lo = warp_min(lo);
        hi = warp_max(hi);
        if (l == 0 && lo <= hi) {
            atomicMax(&mm[(int64_t)sp.u * 6 + 4], ~ord_key(lo));
            atomicMax(&mm[(int64_t)sp.u * 6 + 5], ord_key(hi));
        }
    }
}

// Block sums of bf16 keys come from the tensor cores.  fp16 keys would need their norms as fp16 numbers, whose range is short
// of what norms span, so theirs stay on the FMA pipes.
template <typename T, bool kGiven> constexpr bool kFmaSums = !kGiven && std::is_same<T, __half>::value;

template <typename T, int D, bool kGiven>
__global__ void __launch_bounds__(Warps<kFmaSums<T, kGiven>>::kThreads, 1)
gram_pass_kernel(const __grid_constant__ CUtensorMap tmap, int block, int nblocks, int units, int H, int N, bool keep_in_l2,
                 const float* __restrict__ given, float* __restrict__ block_sums, float* __restrict__ inv_norm, int64_t inv_row, float* __restrict__ a_raw,
                 int64_t raw_row, uint32_t* __restrict__ mm, int* status) {
    using C = Cfg<D>;
    constexpr bool kFma = kFmaSums<T, kGiven>, kSums = !kFma && !kGiven;
    using W = Warps<kFma>;
    extern __shared__ unsigned char smem_raw[];
    // the swizzle atoms (8 rows x 128 bytes) must start on 1024-byte boundaries
    unsigned char* ring = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    unsigned char* rhs = ring + C::kRingBytes;
    Smem<D, kFma>* s = reinterpret_cast<Smem<D, kFma>*>(rhs + (kFma ? 0 : C::kStages * C::kRhsBytes));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < C::kStages; ++i) {
            mbar_init(&s->full[i], 1);
            mbar_init(&s->sfree[i], kFma ? W::kSums + 1 : kSums ? 2 : 1);
            mbar_init(&s->rready[i], kBandGroup / 32);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&s->tfull[i], 1);
            mbar_init(&s->tempty[i], kBandGroup / 32);
        }
        for (int i = 0; i < 5; ++i) mbar_init(&s->drain[i], 1);
        for (int i = 0; i < kWRing; ++i) mbar_init(&s->wready[i], kBandGroup / 32);
        for (int i = 0; i < kCfRing; ++i) {
            mbar_init(&s->cready[i], kBandGroup / 32);
            mbar_init(&s->cfree[i], 2);
        }
        for (int i = 0; i < kSumsRing; ++i) mbar_init(&s->sdone[i], 1);
        for (int i = 0; i < 2; ++i) mbar_init(&s->sempty[i], W::kSums);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < kHalo) s->zero[tid] = 0.f;
    // (the rows in front of the first tile, which count for nothing)
    for (int half = 0; half < C::kHalves; ++half)
        for (int i = tid; i < kHaloHalfBytes / 16; i += W::kThreads)
            reinterpret_cast<uint4*>(ring + half * C::kHalfBytes)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (kSums)
        for (int i = tid; i < C::kStages * C::kRhsBytes / 16; i += W::kThreads) reinterpret_cast<uint4*>(rhs)[i] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == W::kMma) tmem_alloc(&s->tmem_base, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s->tmem_base;
    pdl_wait();
    const Walk walk = my_walk(units, nblocks);

    if (warp == W::kProducer) {
        if (lane == 0) producer_role<D, kFma>(&tmap, ring, s, walk, block, N, H, keep_in_l2, status);
        __syncwarp();
    } else if (warp == W::kMma) {
        mma_role<T, D, kFma>(ring, s, tmem_base, walk, block, N, status);
        __syncwarp();
    } else if (warp >= W::kScan0) {
        scan_role<D, kFma, kGiven>(s, walk, block, N, inv_norm, inv_row, a_raw, raw_row, mm, status);
    } else if (warp >= kSumsWarp0) {
        if constexpr (kFma) sums_role<T, D>(ring, s, walk, block, N, block_sums, status);
        else if constexpr (kSums) tensor_sums_role<T, D>(ring, rhs, s, tmem_base, walk, block, N, block_sums, status);
    } else {
        band_role<D, kFma, kGiven, kSums>(rhs, s, tmem_base, walk, block, N, given, inv_row, status);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == W::kMma) tmem_dealloc(tmem_base, kTmemCols);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once (the library does not link against the driver).
EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

template <typename T, int D>
cudaError_t launch_typed(const CUtensorMap& tmap, const TensorView& K, int units, const ScoreParams& sp, bool keep_in_l2,
                         const float* given, float* block_sums, float* inv_norm, float* a_raw, uint32_t* mm, int* status, int sm_count,
                         cudaStream_t stream) {
    const long long total = (long long)units * sp.nblocks;
    const unsigned grid = (unsigned)(total < sm_count ? total : sm_count);
    auto launch = [&](auto kernel, int threads, size_t smem) {
        return launch_chained(kernel, grid, (unsigned)threads, smem, stream, 1, tmap, sp.block, sp.nblocks, units, K.H, K.N, keep_in_l2, given,
                              block_sums, inv_norm, sp.inv_row, a_raw, sp.raw_row, mm, status);
    };
    if (given) return launch(gram_pass_kernel<T, D, true>, Warps<false>::kThreads, smem_bytes<D, false>());
    constexpr bool kFma = kFmaSums<T, false>;
    return launch(gram_pass_kernel<T, D, false>, Warps<kFma>::kThreads, smem_bytes<D, kFma>());
}

}  // namespace

// Tensor map of 16-bit keys [G][H][N][d] for boxes of 64 columns x box_rows rows, 128-byte swizzle.
cudaError_t encode_key_map(const TensorView& K, int dtype, int G, int box_rows, CUtensorMap* out) {
    EncodeTiledFn encode = tensor_map_encoder();
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t dims[4] = {(cuuint64_t)K.d, (cuuint64_t)K.N, (cuuint64_t)K.H, (cuuint64_t)G};
    const cuuint64_t strides[3] = {(cuuint64_t)K.d * 2, (cuuint64_t)K.stride_h * 2, (cuuint64_t)K.stride_g * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    if (encode(out, dtype == NKV_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
               const_cast<void*>(K.ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

cudaError_t configure_gram_kernels() {
    cudaError_t e;
#define NKV_SET(T, D)                                                                                                    \
    if ((e = cudaFuncSetAttribute(gram_pass_kernel<T, D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,            \
                                  (int)smem_bytes<D, kFmaSums<T, false>>())) != cudaSuccess ||                           \
        (e = cudaFuncSetAttribute(gram_pass_kernel<T, D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,             \
                                  (int)smem_bytes<D, false>())) != cudaSuccess)                                          \
        return e
    NKV_SET(__nv_bfloat16, 64);
    NKV_SET(__nv_bfloat16, 128);
    NKV_SET(__half, 64);
    NKV_SET(__half, 128);
#undef NKV_SET
    return cudaSuccess;
}

// 16-bit keys of 64 or 128 columns, the paper's window of 64, blocks of at least a tile (a tile then meets at most one
// block end besides the head's), and strides a tensor map accepts (multiples of 16 bytes, base 16-byte aligned).
bool gram_pass_supported(const TensorView& K, int dtype, const ScoreParams& sp) {
    if ((dtype != NKV_BF16 && dtype != NKV_F16) || (K.d != 64 && K.d != 128) || sp.window != 64 || sp.block < kTile) return false;
    if (reinterpret_cast<uintptr_t>(K.ptr) % 16 != 0) return false;
    if (K.stride_h % 8 != 0 || K.stride_g % 8 != 0) return false;
    if (K.stride_h < (int64_t)K.N * K.d || K.stride_g < (int64_t)K.N * K.d) return false;
    CUtensorMap probe;   // the driver has the last word on what a tensor map can describe
    return encode_key_map(K, dtype, 1, kHalo, &probe) == cudaSuccess;
}

// With `given` the norms are the caller's (rows of sp.inv_row) and only a_c and its extremes are written: block_sums and
// inv_norm are null.
cudaError_t launch_gram_pass(const TensorView& K, int dtype, int G, const ScoreParams& sp, const float* given,
                             float* block_sums, float* inv_norm, float* a_raw, uint32_t* mm, int* status, int sm_count, cudaStream_t stream,
                             int64_t* launches) {
    const int units = G * K.H;
    CUtensorMap tmap;
    cudaError_t e = encode_key_map(K, dtype, G, kHalo, &tmap);
    if (e != cudaSuccess) return e;
    // keys that fit L2 (126 MB) beside the scores stay there for the second pass
    const bool keep = (int64_t)units * K.N * K.d * 2 <= ((int64_t)48 << 20);
#define NKV_ARGS tmap, K, units, sp, keep, given, block_sums, inv_norm, a_raw, mm, status, sm_count, stream
    if (dtype == NKV_BF16) e = K.d == 128 ? launch_typed<__nv_bfloat16, 128>(NKV_ARGS) : launch_typed<__nv_bfloat16, 64>(NKV_ARGS);
    else e = K.d == 128 ? launch_typed<__half, 128>(NKV_ARGS) : launch_typed<__half, 64>(NKV_ARGS);
#undef NKV_ARGS
    ++*launches;
    return e;
}

}  // namespace nkv
