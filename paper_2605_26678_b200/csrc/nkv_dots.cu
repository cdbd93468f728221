// Second key pass on the tensor cores (bf16 or fp16 keys, d = 64 or 128): a_s(i) = -cos(k_hat_i, mu_s) and
// a_e(i) = -cos(k_hat_i, mu_e(block of i)) with their per-head min/max (Section 2.3).
//
// The dots of 128 keys with the anchors are one skinny product [128 x d] x [d x 16] per tile.  The fp32
// anchors enter as three columns of the keys' type each (hi + mid + lo carries all 24 mantissa bits; products of
// 16-bit numbers are exact in fp32 and tcgen05.mma accumulates in fp32; for fp16 every anchor is scaled by the power
// of two that brings its norm to 2^9 .. 2^10, whatever it was, which puts lo's quantum at 2^-34 of the norm or below), so a
// tile's right-hand side is
//     columns 0..2  mu_s        3..5  mu_e of the block the tile starts in        6..8  mu_e of the next block
// (a tile of 128 keys touches at most two blocks because a block has at least 128 keys).  Key tiles are staged by TMA
// (128-byte swizzle); the tensor core reads them from shared memory directly.  Warp roles: TMA producer, MMA issuer, four
// warps that build the right-hand sides, four warps that turn the accumulator into scores.  Every wait is bounded.
//
// Bound: the read of the keys; no role may then need more than the 1300 cycles in which a tile of 32 KB arrives.  What
// that took: places in the tensors are counted, not divided out (per tile), right-hand sides are built per block and not
// per tile, the rows' norms and the anchors come by asynchronous copies several tiles ahead, and the products are issued
// by a warp in step (umma_f16; one thread by itself needed 1050 cycles per tile of 128 columns, 790 per tile of 64).
// 96 KB of keys in flight per SM: a bare read of 604 MB in 32 KB pieces takes 101 us with 96, 107 with 160 or 192, and this
// pass 105, 107 and 112 us with 96, 128 and 160 KB; 64 KB is too little (119).
// 16 x 8 heads of 32768 x 64 bf16 keys: 141 -> 95 us (and 141 in the FMA form of nkv_stream.cu); 36 x 8 x 8192 x 128:
// 109 -> 105; 36 x 8 x 131072 x 128: 1900 -> 1470 (6.7 TB/s).
#include "nkv_sm100.cuh"

namespace nkv {

namespace {

using namespace sm100;

constexpr int kTile = 128;                        // keys per tile
constexpr int kTileHalfBytes = kTile * 128;       // one 64-column half of a tile
constexpr int kRhsHalfBytes = 16 * 128;           // 16 right-hand-side rows of 64 columns
constexpr int kStages = 4;                        // accumulators of 32 columns (16 used)
constexpr uint32_t kTmemCols = 128;
constexpr int kPrepWarp0 = 0, kEpiWarp0 = 4, kProducerWarp = 8, kMmaWarp = 9;
constexpr int kThreads = 10 * 32;
constexpr int kMaxSlots = 8;
constexpr int kRhs = 4;                           // right-hand sides kept at once
constexpr int kAhead = 8;                         // tiles (blocks) whose per-row inputs (anchors) are on their way

// Sizes for head dimension D (64 or 128): a key row is D / 64 swizzled halves of 128 bytes.
template <int D>
struct Cfg {
    static constexpr int kHalves = D / 64;
    static constexpr int kSlots = 384 / D;                       // key tiles staged at once (96 KB)
    static constexpr int kTileBytes = kHalves * kTileHalfBytes;
    static constexpr int kRhsBytes = kHalves * kRhsHalfBytes;
    static constexpr int kPrepWarps = D / 32;                    // one thread per column
    static constexpr size_t kRhsAt = (size_t)kSlots * kTileBytes;             // offsets of the parts behind the tiles
    static constexpr size_t kRowsAt = kRhsAt + (size_t)kRhs * kRhsBytes;      // [kAhead][2][kTile] floats
    static constexpr size_t kMuAt = kRowsAt + (size_t)kAhead * 2 * kTile * 4; // [kAhead][D] floats
    static constexpr size_t kInvAt = kMuAt + (size_t)kAhead * D * 4;          // [kAhead][D] floats (fp16: 1/||mu_e||)
    static constexpr size_t kSmemAt = kInvAt + (size_t)kAhead * D * 4;
    static_assert(kSlots <= kMaxSlots, "barrier arrays too small");
};

struct Smem {
    uint64_t full[kMaxSlots];   // key tile landed
    uint64_t kfree[kMaxSlots];  // tile consumed by the MMAs
    uint64_t rready[kRhs];      // right-hand side written (one arrival per building warp)
    uint64_t rfree[kRhs];       // consumed by the MMAs of all its tiles
    uint64_t tfull[kStages];    // accumulator written
    uint64_t tempty[kStages];   // accumulator read (one arrival per reading warp)
    uint64_t drain;             // products issued before a give-up have completed
    uint32_t tmem_base;
};
template <int D>
constexpr size_t smem_bytes() {
    return 1024 + Cfg<D>::kSmemAt + sizeof(Smem);
}

// A CTA's tiles: `count` of them from tile `first` on, counted through the heads.
struct TileRange {
    long long first;
    int count, tiles_per_unit;
};
__device__ __forceinline__ TileRange my_tiles(int units, int N) {
    TileRange r;
    r.tiles_per_unit = (N + kTile - 1) / kTile;
    const long long total = (long long)units * r.tiles_per_unit;
    r.first = total * blockIdx.x / gridDim.x;
    r.count = (int)(total * (blockIdx.x + 1) / gridDim.x - r.first);
    return r;
}
// Where a role is: head, first key of the tile, the block it lies in and that block's end.  Every role steps through the
// tiles on its own; the steps are additions (a division per tile and role cost as much as the rest of its work).
struct Place {
    int u, i0, blk, blk_end;
    __device__ __forceinline__ Place(TileRange tr, int block) {
        u = (int)(tr.first / tr.tiles_per_unit);
        i0 = (int)(tr.first - (long long)u * tr.tiles_per_unit) * kTile;
        blk = i0 / block;
        blk_end = (blk + 1) * block;
    }
    __device__ __forceinline__ bool next(int N, int block) {   // true: another head or block
        i0 += kTile;
        if (i0 >= N) {
            ++u;
            i0 = blk = 0;
            blk_end = block;
            return true;
        }
        if (i0 < blk_end) return false;   // a block has at least kTile keys, so it is the next one otherwise
        ++blk;
        blk_end += block;
        return true;
    }
};
// Position in a ring and the parity of the round.
template <int kSize>
struct Ring {
    int at = 0;
    uint32_t round = 0;
    __device__ __forceinline__ void next() {
        if (++at == kSize) {
            at = 0;
            round ^= 1u;
        }
    }
};

// Four bytes into shared memory behind the thread's back.  (Loads into registers that are due several tiles later share a
// handful of scoreboards with newer ones and get waited for too early: 12 tiles ahead was slower than one.)
__device__ __forceinline__ void copy4(float* dst_smem, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

// ---------------------------------------------------------------------------- roles
template <int D>
__device__ void dots_producer(const CUtensorMap* tmap, unsigned char* tiles, Smem* s, TileRange tr, int H, int N, int* status) {
    using C = Cfg<D>;
    const uint64_t policy = l2_evict_first_policy();   // keys are read once per pass
    Ring<C::kSlots> slot;
    int u = (int)(tr.first / tr.tiles_per_unit), i0 = (int)(tr.first - (long long)u * tr.tiles_per_unit) * kTile;
    int g = u / H, h = u - g * H;
    for (int n = 0; n < tr.count; ++n, slot.next()) {
        if (n >= C::kSlots && !mbar_wait(&s->kfree[slot.at], slot.round ^ 1u, status, 711)) {
            // giving up: the copies already armed still land in this CTA's shared memory, so stay (bounded)
            // until they have
            for (int m = n - C::kSlots; m < n; ++m)
                for (uint32_t spin = 0; spin < (1u << 16) && !mbar_try_wait(&s->full[m % C::kSlots], (uint32_t)((m / C::kSlots) & 1)); ++spin)
                    __nanosleep(256);
            return;
        }
        unsigned char* dst = tiles + (size_t)slot.at * C::kTileBytes;
        mbar_expect_tx(&s->full[slot.at], C::kTileBytes);
#pragma unroll
        for (int half = 0; half < C::kHalves; ++half)
            tma_load_4d(dst + half * kTileHalfBytes, tmap, 64 * half, i0, h, g, &s->full[slot.at], policy);
        i0 += kTile;
        if (i0 >= N) {
            i0 = 0;
            if (++h == H) {
                h = 0;
                ++g;
            }
        }
    }
}

template <typename T, int D>
__device__ void dots_mma(unsigned char* tiles, unsigned char* rhs, Smem* s, uint32_t tmem_base, TileRange tr, int N, int block,
                         int* status) {
    using C = Cfg<D>;
    constexpr uint32_t idesc = umma_idesc<T>(kTile, 16);
    const uint64_t tiles_desc = umma_desc_sw128(smem_addr(tiles)), rhs_desc = umma_desc_sw128(smem_addr(rhs));
    Ring<C::kSlots> slot;
    Ring<kStages> stage;
    Ring<kRhs> r;
    Place at(tr, block);
    bool fresh = true;   // another right-hand side
    for (int n = 0; n < tr.count; ++n, slot.next(), stage.next()) {
        if ((fresh && !warp_wait(&s->rready[r.at], r.round, status, 713)) ||
            !warp_wait(&s->tempty[stage.at], stage.round ^ 1u, status, 714) || !warp_wait(&s->full[slot.at], slot.round, status, 712))
            return umma_drain(&s->drain);
        tc_fence_after();
        const uint64_t a = tiles_desc + (uint32_t)(slot.at * C::kTileBytes >> 4), b = rhs_desc + (uint32_t)(r.at * C::kRhsBytes >> 4);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
            umma_f16(tmem_base + (uint32_t)stage.at * 32u, a + (uint32_t)((kk >> 2) * kTileHalfBytes + (kk & 3) * 32 >> 4),
                     b + (uint32_t)((kk >> 2) * kRhsHalfBytes + (kk & 3) * 32 >> 4), idesc, kk > 0);
        umma_commit(&s->tfull[stage.at]);
        umma_commit(&s->kfree[slot.at]);
        fresh = at.next(N, block);
        if (fresh && n + 1 < tr.count) {
            umma_commit(&s->rfree[r.at]);
            r.next();
        }
    }
}

// Thread k writes column k of the nine right-hand-side rows of every block (rows 9..15 stay zero).
// fp16 has five exponent bits: an anchor of norm 1 / inv enters times the power of two below inv, times 2^10, and inv's
// mantissa is left for the epilogue (both exact).
template <typename T> constexpr bool kScaled = false;
template <> constexpr bool kScaled<__half> = true;
constexpr float kAnchorScale = 1024.f;
__device__ __forceinline__ float scale_of(float inv) { return __uint_as_float(__float_as_uint(inv) & 0x7f800000u) * kAnchorScale; }
template <typename T>
__device__ __forceinline__ float rest_of(float inv) {   // 1 / ||mu|| over the scale that the dots carry
    return kScaled<T> ? __uint_as_float((__float_as_uint(inv) & 0x007fffffu) | 0x3f800000u) * (1.f / kAnchorScale) : inv;
}
template <typename T> __device__ __forceinline__ T narrow(float v);
template <> __device__ __forceinline__ __nv_bfloat16 narrow<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ __half narrow<__half>(float v) { return __float2half_rn(v); }
template <typename T> __device__ __forceinline__ float widen(T v) { return (float)v; }

template <typename T, int D>
__device__ void dots_prep(unsigned char* rhs, float* mu, float* inv, Smem* s, ScoreParams sp, TileRange tr, int units, int N,
                          const float* __restrict__ mu_s, const float* __restrict__ mu_e, const float* __restrict__ inv_s,
                          const float* __restrict__ inv_e, int* status) {
    using C = Cfg<D>;
    const int k = threadIdx.x - kPrepWarp0 * 32, lane = k & 31;
    if (k >= D) return;   // d = 64 needs two of the four warps
    const int half = k >> 6, kk = k & 63;
    Place at(tr, sp.block);
    // The anchors of a head's blocks follow one another, and the next head's come behind them: element k of row j of that
    // sequence waits in mu[j % kAhead][k], fetched kAhead - 1 rows ahead.  A thread reads what it has copied itself.
    const int64_t rows = (int64_t)units * sp.nblocks;
    int64_t row = (int64_t)at.u * sp.nblocks + at.blk, fetched = row;
    auto fetch_to = [&](int64_t end) {
        for (; fetched < end; ++fetched) {
            if (fetched < rows) copy4(mu + (int)(fetched % kAhead) * D + k, mu_e + fetched * D + k);
            if (kScaled<T> && fetched < rows) copy4(inv + (int)(fetched % kAhead) * D + k, inv_e + fetched);
            copies_commit();
        }
    };
    int cur_u = -1;
    float v[3] = {0.f, 0.f, 0.f}, s_next = mu_s[(int64_t)at.u * D + k];
    float i_next = kScaled<T> ? inv_s[at.u] : 0.f;
    Ring<kRhs> r;
    bool fresh = true, wrapped = false;
    for (int n = 0; n < tr.count; ++n, fresh = at.next(N, sp.block)) {
        if (!fresh) continue;
        row = (int64_t)at.u * sp.nblocks + at.blk;
        fetch_to(row + kAhead);
        copies_wait<kAhead - 2>();   // rows `row` and `row` + 1 are here
        if (at.u != cur_u) {
            cur_u = at.u;
            v[0] = kScaled<T> ? s_next * scale_of(i_next) : s_next;
            if (cur_u + 1 < units) {
                s_next = mu_s[(int64_t)(cur_u + 1) * D + k];
                if (kScaled<T>) i_next = inv_s[cur_u + 1];
            }
        }
        const int here = (int)(row % kAhead) * D + k, after = (int)((row + 1) % kAhead) * D + k;
        v[1] = mu[here];
        v[2] = at.blk + 1 < sp.nblocks ? mu[after] : 0.f;
        if (kScaled<T>) {
            v[1] *= scale_of(inv[here]);
            if (at.blk + 1 < sp.nblocks) v[2] *= scale_of(inv[after]);
        }
        if (wrapped && !mbar_wait(&s->rfree[r.at], r.round ^ 1u, status, 715)) break;
        unsigned char* base = rhs + (size_t)r.at * C::kRhsBytes + (size_t)half * kRhsHalfBytes + (kk & 7) * 2;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const T hi = narrow<T>(v[a]);
            const float r1 = v[a] - widen(hi);
            const T mid = narrow<T>(r1);
            const T lo = narrow<T>(r1 - widen(mid));
            const T part[3] = {hi, mid, lo};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int line = 3 * a + j;   // row of the right-hand side, 8-row groups 1024 bytes apart
                *reinterpret_cast<T*>(base + (line >> 3) * 1024 + (line & 7) * 128 + ((((kk >> 3) ^ (line & 7))) << 4)) = part[j];
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads these writes
        __syncwarp();
        if (lane == 0) mbar_arrive(&s->rready[r.at]);
        r.next();
        wrapped = wrapped || r.at == 0;
    }
    copies_wait<0>();
}

// Thread r reads row r of the accumulator: the key's dots with mu_s and with the two candidate mu_e.
template <typename T>
__device__ void dots_epilogue(Smem* s, float* rows, uint32_t tmem_base, ScoreParams sp, TileRange tr, int units, int N,
                              const float* __restrict__ inv_norm, const float* __restrict__ inv_s,
                              const float* __restrict__ inv_e, float* __restrict__ a_raw, uint32_t* __restrict__ mm,
                              int* status) {
    const int r = threadIdx.x - kEpiWarp0 * 32, q = r >> 5, lane = r & 31;
    int cur_u = -1;
    float rs = 0.f;
    float lo_s = INFINITY, hi_s = -INFINITY, lo_e = INFINITY, hi_e = -INFINITY;
    auto flush = [&]() {   // the warp's min/max of the head it has been working on
        if (cur_u < 0) return;
        lo_s = warp_min(lo_s);
        hi_s = warp_max(hi_s);
        lo_e = warp_min(lo_e);
        hi_e = warp_max(hi_e);
        if (lane == 0 && lo_s <= hi_s) {
            atomicMax(&mm[(int64_t)cur_u * 6 + 0], ~ord_key(lo_s));
            atomicMax(&mm[(int64_t)cur_u * 6 + 1], ord_key(hi_s));
            atomicMax(&mm[(int64_t)cur_u * 6 + 2], ~ord_key(lo_e));
            atomicMax(&mm[(int64_t)cur_u * 6 + 3], ord_key(hi_e));
        }
        lo_s = lo_e = INFINITY;
        hi_s = hi_e = -INFINITY;
    };
    // 1 / ||k|| and 1 / ||mu_e|| of this thread's row, copied kAhead tiles ahead: with the key copies of a whole ring queued
    // in front of them such loads take microseconds
    Place to(tr, sp.block), at = to;
    auto fetch = [&](int n) {
        if (n < tr.count) {
            float* dst = rows + (n % kAhead) * 2 * kTile + r;
            const int i = min(to.i0 + r, N - 1);
            copy4(dst, inv_norm + to.u * sp.inv_row + i);
            copy4(dst + kTile, inv_e + (int64_t)to.u * sp.nblocks + to.blk + (i >= to.blk_end ? 1 : 0));
            to.next(N, sp.block);
        }
        copies_commit();
    };
    for (int k = 0; k < kAhead; ++k) fetch(k);
    Ring<kStages> stage;
    float rs_next = tr.count > 0 ? inv_s[at.u] : 0.f;
    for (int n = 0; n < tr.count; ++n, stage.next(), at.next(N, sp.block)) {
        if (at.u != cur_u) {
            flush();
            cur_u = at.u;
            rs = rest_of<T>(rs_next);
            if (cur_u + 1 < units) rs_next = inv_s[cur_u + 1];
        }
        copies_wait<kAhead - 1>();
        const float inv_i = rows[(n % kAhead) * 2 * kTile + r], re = rest_of<T>(rows[((n % kAhead) * 2 + 1) * kTile + r]);
        fetch(n + kAhead);
        const int i = at.i0 + r;
        const bool second = i >= at.blk_end;   // the key lies in the block after the tile's first
        if (!mbar_wait(&s->tfull[stage.at], stage.round, status, 716)) break;
        tc_fence_after();
        float d[16];
        tmem_ld16(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)stage.at * 32u, d);
        tmem_wait_ld(d);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&s->tempty[stage.at]);
        const float ds = d[0] + d[1] + d[2];
        const float de = second ? d[6] + d[7] + d[8] : d[3] + d[4] + d[5];
        const float a_s = -(ds * inv_i) * rs + 0.f;
        const float a_e = -(de * inv_i) * re + 0.f;
        if (i < N) {
            float* out = a_raw + (int64_t)cur_u * 3 * sp.raw_row + i;
            out[0] = a_s;
            out[sp.raw_row] = a_e;
            lo_s = fminf(lo_s, a_s);
            hi_s = fmaxf(hi_s, a_s);
            lo_e = fminf(lo_e, a_e);
            hi_e = fmaxf(hi_e, a_e);
        }
    }
    copies_wait<0>();
    flush();
}

template <typename T, int D>
__global__ void __launch_bounds__(kThreads, 1)
anchor_dots_kernel(const __grid_constant__ CUtensorMap tmap, ScoreParams sp, int units, int H, int N,
                   const float* __restrict__ mu_s, const float* __restrict__ mu_e, const float* __restrict__ inv_norm,
                   const float* __restrict__ inv_s, const float* __restrict__ inv_e, float* __restrict__ a_raw,
                   uint32_t* __restrict__ mm, int* status) {
    using C = Cfg<D>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* tiles = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    unsigned char* rhs = tiles + C::kRhsAt;
    float* rows = reinterpret_cast<float*>(tiles + C::kRowsAt);
    float* mu = reinterpret_cast<float*>(tiles + C::kMuAt);
    float* inv = reinterpret_cast<float*>(tiles + C::kInvAt);
    Smem* s = reinterpret_cast<Smem*>(tiles + C::kSmemAt);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const TileRange tr = my_tiles(units, N);

    if (tid == 0) {
        for (int i = 0; i < C::kSlots; ++i) {
            mbar_init(&s->full[i], 1);
            mbar_init(&s->kfree[i], 1);
        }
        for (int i = 0; i < kRhs; ++i) {
            mbar_init(&s->rready[i], C::kPrepWarps);
            mbar_init(&s->rfree[i], 1);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&s->tfull[i], 1);
            mbar_init(&s->tempty[i], 4);
        }
        mbar_init(&s->drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < kRhs * C::kRhsBytes / 16; i += kThreads) reinterpret_cast<uint4*>(rhs)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == kMmaWarp) tmem_alloc(&s->tmem_base, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s->tmem_base;
    pdl_wait();

    if (warp == kProducerWarp) {
        if (lane == 0) dots_producer<D>(&tmap, tiles, s, tr, H, N, status);
        __syncwarp();
    } else if (warp == kMmaWarp) {
        dots_mma<T, D>(tiles, rhs, s, tmem_base, tr, N, sp.block, status);
        __syncwarp();
    } else if (warp >= kEpiWarp0) {
        dots_epilogue<T>(s, rows, tmem_base, sp, tr, units, N, inv_norm, inv_s, inv_e, a_raw, mm, status);
    } else {
        dots_prep<T, D>(rhs, mu, inv, s, sp, tr, units, N, mu_s, mu_e, inv_s, inv_e, status);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem_base, kTmemCols);
}

}  // namespace

cudaError_t configure_dots_kernels() {
    cudaError_t e;
#define NKV_SET(T, D)                                                                                                    \
    if ((e = cudaFuncSetAttribute(anchor_dots_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,                 \
                                  (int)smem_bytes<D>())) != cudaSuccess)                                                  \
        return e
    NKV_SET(__nv_bfloat16, 64);
    NKV_SET(__nv_bfloat16, 128);
    NKV_SET(__half, 64);
    NKV_SET(__half, 128);
#undef NKV_SET
    return cudaSuccess;
}

// 16-bit keys of 64 or 128 columns, strides a tensor map accepts, and blocks of at least 128 keys (a tile
// of 128 keys then touches at most two blocks).
bool anchor_dots_supported(const TensorView& K, int dtype, const ScoreParams& sp) {
    if ((dtype != NKV_BF16 && dtype != NKV_F16) || (K.d != 64 && K.d != 128) || sp.block < kTile) return false;
    if (reinterpret_cast<uintptr_t>(K.ptr) % 16 != 0) return false;
    if (K.stride_h % 8 != 0 || K.stride_g % 8 != 0) return false;
    if (K.stride_h < (int64_t)K.N * K.d || K.stride_g < (int64_t)K.N * K.d) return false;
    CUtensorMap probe;   // the driver has the last word on what a tensor map can describe
    return encode_key_map(K, dtype, 1, kTile, &probe) == cudaSuccess;
}

cudaError_t launch_anchor_dots(const TensorView& K, int dtype, int G, const ScoreParams& sp, const float* mu_s,
                               const float* mu_e, const float* inv_norm, const float* inv_s, const float* inv_e,
                               float* a_raw, uint32_t* mm, int* status, int sm_count, cudaStream_t stream,
                               int64_t* launches) {
    CUtensorMap tmap;
    cudaError_t e = encode_key_map(K, dtype, G, kTile, &tmap);
    if (e != cudaSuccess) return e;
    const int units = G * K.H;
    const long long total = (long long)units * ((K.N + kTile - 1) / kTile);
    const unsigned grid = (unsigned)(total < sm_count ? total : sm_count);
#define NKV_DOTS(T, D)                                                                                                    \
    e = launch_chained(anchor_dots_kernel<T, D>, grid, kThreads, smem_bytes<D>(), stream, 1, tmap, sp, units, K.H, K.N,  \
                       mu_s, mu_e, inv_norm, inv_s, inv_e, a_raw, mm, status)
    if (dtype == NKV_BF16) {
        if (K.d == 128) NKV_DOTS(__nv_bfloat16, 128);
        else NKV_DOTS(__nv_bfloat16, 64);
    } else {
        if (K.d == 128) NKV_DOTS(__half, 128);
        else NKV_DOTS(__half, 64);
    }
#undef NKV_DOTS
    ++*launches;
    return e;
}

}  // namespace nkv
