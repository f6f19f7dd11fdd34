// Device-wide scan and stable LSD radix sort.
//
// Radix sort: 8-bit digits, tiles of 2048 items, the whole sort in one launch (k_sort).
// Scan: reduce-then-scan over 4096-element blocks, recursing on the partials.
#include "cr_device.cuh"
#include "cr_internal.cuh"

namespace {

constexpr int kSortBlock = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortBlock * kSortItems;  // 2048 items per tile
constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanBlock * kScanItems;  // 4096 elements per block

// ---------------------------------------------------------------- scan ----
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v)
{
    const uint32_t lane = cr_lane();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (uint32_t)o) v += u;
    }
    return v;
}

// Exclusive scan of one value per thread across a 1024-thread block; returns
// the exclusive prefix and writes the block total to *total.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T *total)
{
    __shared__ T warp_sums[32];
    const uint32_t lane = cr_lane(), warp = threadIdx.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T s = warp_sums[lane];  // 1024 threads: 32 warps, every lane has a warp sum
        T si = warp_incl_scan(s);
        warp_sums[lane] = si - s;
        if (lane == 31) *total = si;
    }
    __syncthreads();
    T r = warp_sums[warp] + inc - v;
    __syncthreads();
    return r;
}

template <typename T>
__global__ void __launch_bounds__(kScanBlock) k_scan_reduce(const T *__restrict__ in, uint64_t n,
                                                            T *__restrict__ partial)
{
    __shared__ T tot;
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
    T s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        uint64_t i = base + (uint64_t)j * kScanBlock + threadIdx.x;
        if (i < n) s += in[i];
    }
    block_excl_scan<T>(s, &tot);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

// Scan one 4096-element block (blocked arrangement: thread t owns 4 consecutive
// elements), adding the block's offset from `partial` (exclusive) if given.
template <typename T>
__global__ void __launch_bounds__(kScanBlock) k_scan_block(const T *__restrict__ in, T *__restrict__ out,
                                                           uint64_t n, const T *__restrict__ partial,
                                                           int inclusive, T *__restrict__ total_out)
{
    __shared__ T tot;
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    T x[kScanItems];
    T s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        x[j] = (base + j < n) ? in[base + j] : (T)0;
        s += x[j];
    }
    T pre = block_excl_scan<T>(s, &tot);
    if (partial) pre += partial[blockIdx.x];
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        T nx = pre + x[j];
        if (base + j < n) out[base + j] = inclusive ? nx : pre;
        pre = nx;
    }
    if (total_out && threadIdx.x == kScanBlock - 1 && blockIdx.x == gridDim.x - 1) *total_out = pre;
}

// Eight consecutive elements, in 16-byte accesses where all of them are there (`in` on a
// 16-byte boundary, i a multiple of 8).
template <typename T>
__device__ __forceinline__ void load8(T (&x)[8], const T *__restrict__ in, uint64_t i, uint64_t n)
{
    if (i + 8 <= n) {
        constexpr int kQuads = (int)(8 * sizeof(T) / sizeof(uint4));
        union {
            uint4 q[kQuads];
            T t[8];
        } u;
#pragma unroll
        for (int j = 0; j < kQuads; ++j) u.q[j] = reinterpret_cast<const uint4 *>(in + i)[j];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = u.t[j];
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = i + j < n ? in[i + j] : (T)0;
    }
}
template <typename T>
__device__ __forceinline__ void store8(const T (&x)[8], T *__restrict__ out, uint64_t i, uint64_t n)
{
    if (i + 8 <= n) {
        constexpr int kQuads = (int)(8 * sizeof(T) / sizeof(uint4));
        union {
            uint4 q[kQuads];
            T t[8];
        } u;
#pragma unroll
        for (int j = 0; j < 8; ++j) u.t[j] = x[j];
#pragma unroll
        for (int j = 0; j < kQuads; ++j) reinterpret_cast<uint4 *>(out + i)[j] = u.q[j];
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (i + j < n) out[i + j] = x[j];
    }
}

// Scan of up to kScanOne elements (arrays on 16-byte boundaries) by one CTA, eight consecutive
// elements per thread and round, the next round's loads in flight: one launch instead of three.
constexpr uint32_t kScanOne = 32768;
template <typename T>
__global__ void __launch_bounds__(kScanBlock) k_scan_one(const T *in, T *out, uint64_t n, int inclusive,
                                                         T *__restrict__ total_out)
{
    __shared__ T tot;
    T carry = 0, x[8];
    const uint64_t i0 = (uint64_t)threadIdx.x * 8;
    load8(x, in, i0, n);
    for (uint64_t t0 = 0; t0 < n; t0 += 8ull * kScanBlock) {
        const uint64_t i = t0 + i0;
        T y[8], s = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            y[j] = x[j];
            s += x[j];
        }
        load8(x, in, i + 8ull * kScanBlock, n);  // (elements that this round does not write)
        T pre = carry + block_excl_scan<T>(s, &tot);
        carry += tot;
        __syncthreads();  // (tot is written again)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const T nx = pre + y[j];
            y[j] = inclusive ? nx : pre;
            pre = nx;
        }
        store8(y, out, i, n);
    }
    if (total_out && threadIdx.x == 0) *total_out = carry;
}

// Elements of partial sums needed below a scan of n elements (all levels).
static uint64_t scan_partials_size(uint64_t n)
{
    uint64_t total = 0;
    uint64_t m = (n + kScanTile - 1) / kScanTile;
    while (m > 1) {
        total += m + 32;
        m = (m + kScanTile - 1) / kScanTile;
    }
    return total;
}

template <typename T>
int scan_rec(cr_ctx *ctx, const T *in, T *out, uint64_t n, int inclusive, T *d_total, T *partials)
{
    uint64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 1) {
        CR_LAUNCH(ctx, k_scan_block<T>, 1, kScanBlock, 0, in, out, n, (const T *)nullptr, inclusive, d_total);
        return CR_OK;
    }
    if (n <= kScanOne && (((uintptr_t)in | (uintptr_t)out) & 15u) == 0) {
        CR_LAUNCH(ctx, k_scan_one<T>, 1, kScanBlock, 0, in, out, n, inclusive, d_total);
        return CR_OK;
    }
    T *partial = partials;
    CR_LAUNCH(ctx, k_scan_reduce<T>, (unsigned int)nb, kScanBlock, 0, in, n, partial);
    CR_TRY(scan_rec<T>(ctx, partial, partial, nb, 0, (T *)nullptr, partials + nb + 32));
    CR_LAUNCH(ctx, k_scan_block<T>, (unsigned int)nb, kScanBlock, 0, in, out, n, (const T *)partial, inclusive,
              d_total);
    return CR_OK;
}

template <typename T>
int scan_impl(cr_ctx *ctx, const T *in, T *out, uint64_t n, int inclusive, T *d_total)
{
    if (n == 0) return CR_OK;
    void *p = nullptr;
    CR_TRY(cr_scratch(ctx, SCR_SCAN, (size_t)(scan_partials_size(n) + 32) * sizeof(T), &p));
    return scan_rec<T>(ctx, in, out, n, inclusive, d_total, reinterpret_cast<T *>(p));
}

// ---------------------------------------------------------- radix sort ----
// The whole sort is one launch.  Its work is a sequence of phases of `tiles` items each: the
// digit counts of every pass (an LSD sort only reorders the items), a phase per 8-bit digit,
// and for a plan the histogram's arrays and a second sort by count.  Blocks take items in
// order by a ticket and wait, before an item, until the phase before is done, so what a
// block waits for is always held by a block that is running, however few of them are.
constexpr uint32_t kSortPasses = 12;           // 8 of a 64-bit key, up to 4 of a 32-bit one
constexpr uint32_t kSortPhases = kSortPasses + 2;
constexpr uint32_t kSortSpin = 1u << 20;       // looks at a word that does not come, ~0.5 s

// Counters of a sort, zero before it.
struct sort_counters {
    uint32_t digits[kSortPasses][256];  // items of each digit value, per pass
    uint32_t done[kSortPhases];         // items finished, per phase
    uint32_t ticket, gave_up;
    uint32_t pad[48];
};
static_assert(sizeof(sort_counters) % 256 == 0, "the tile states start aligned");

struct sort_job {
    const unsigned long long *k_in;  // the keys, and their values (NULL: the positions)
    const uint32_t *v_in;
    unsigned long long *k[2];        // pass p of the keys writes k[p & 1], v[p & 1]
    uint32_t *v[2];
    // a plan's histogram (order NULL: keys only): outputs, sort keys, positions
    cr_plan_info_dev *info;
    unsigned long long *ukey, *ucnt;
    uint32_t *s[2], *o[2], *order;
    uint32_t passes2;                // of the sort keys n_sum - count
    unsigned long long n_sum;
    unsigned long long n, skip_le;   // items (n_dev: at most), and the count up to which nothing is done
    const unsigned long long *n_dev;
    sort_counters *C;
    unsigned long long *states[2];   // [tiles][256] of the even and the odd passes
    uint32_t *status;
};

inline uint64_t sort_tiles(uint64_t n) { return (n + kSortTile - 1) / kSortTile; }

// A tile's state of one digit: how far it is in the top two bits, a count below.
constexpr unsigned long long kTileCount = 1ull << 62, kTilePrefix = 2ull << 62, kTileValue = kTileCount - 1ull;
constexpr uint32_t kLookBack = 8;  // predecessors read at once

struct sort_smem {
    uint32_t wcnt[kSortBlock / 32][256];  // digit counts per warp (or per pass, in the counting phases)
    uint32_t base[256], wsum[kSortBlock / 32];
    uint32_t ticket, ok;
};

// One tile of a pass: the block ranks its 2048 items stably (warp w owns 256 consecutive
// items, in rounds of 32), and thread d finds how many items of digit d the tiles before hold
// by looking back over their states, eight at a time: a tile first publishes its own count,
// without waiting, then the total through it.  What other blocks wrote is read past the L1.
template <typename K>
__device__ __forceinline__ void sort_tile(sort_smem &S, uint32_t tile, const K *kin, const uint32_t *vin, K *kout,
                                          uint32_t *vout, uint64_t n, int shift, const uint32_t *counts,
                                          unsigned long long *states, unsigned long long *next_states,
                                          sort_counters *C, uint32_t *status)
{
    constexpr int kWarps = kSortBlock / 32;
    const uint32_t tid = threadIdx.x, lane = cr_lane(), warp = tid >> 5, lt = (1u << lane) - 1u;
    const uint64_t i0 = (uint64_t)tile * kSortTile + warp * 256u + lane;
    K key[kSortItems];
    uint32_t rank[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) key[j] = i0 + 32u * j < n ? __ldcg(kin + i0 + 32u * j) : (K)0;
    const uint32_t total = __ldcg(counts + tid);
    next_states[(uint64_t)tile * 256 + tid] = 0;  // of the pass before: no longer read
#pragma unroll
    for (int w = 0; w < kWarps; ++w) S.wcnt[w][tid] = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const uint32_t d = (uint32_t)(key[j] >> shift) & 0xffu;
        const bool in = i0 + 32u * j < n;
        uint32_t peers = __ballot_sync(0xffffffffu, in);  // valid lanes of the round with this digit
#pragma unroll
        for (int bt = 0; bt < 8; ++bt) {
            const uint32_t B = __ballot_sync(0xffffffffu, (d >> bt) & 1u);
            peers &= ((d >> bt) & 1u) ? B : ~B;
        }
        const uint32_t before = S.wcnt[warp][d];
        __syncwarp();
        rank[j] = before + (uint32_t)__popc(peers & lt);
        if (in && (peers & lt) == 0) S.wcnt[warp][d] = before + (uint32_t)__popc(peers);
        __syncwarp();
    }
    // items of the smaller digits: exclusive scan of the pass's 256 counts
    uint32_t incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) S.wsum[warp] = incl;
    __syncthreads();
    uint32_t smaller = incl - total;
    for (uint32_t w = 0; w < warp; ++w) smaller += S.wsum[w];
    // thread d: digit d's items in the warps before, and in the tile
    uint32_t mine = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = S.wcnt[w][tid];
        S.wcnt[w][tid] = mine;
        mine += c;
    }
    volatile unsigned long long *st = states + tid;
    unsigned long long before = 0;
    if (tile) {
        st[(uint64_t)tile * 256] = kTileCount | mine;
        uint32_t t = tile, spin = 0;  // tiles t .. tile - 1 are counted
        for (bool more = true; more;) {
            unsigned long long s[kLookBack];
#pragma unroll
            for (uint32_t x = 0; x < kLookBack; ++x) {  // (tile 0's state is its prefix: none before it is needed)
                s[x] = kTilePrefix;
                if (x < t) s[x] = st[(uint64_t)(t - 1u - x) * 256];
            }
#pragma unroll
            for (uint32_t x = 0; x < kLookBack; ++x) {
                if (!more || !(s[x] >> 62)) break;  // (not there yet)
                before += s[x] & kTileValue;
                --t;
                more = !(s[x] & kTilePrefix);
            }
            if (more && ++spin >= kSortSpin) {  // never: the items then go too low, not out of range
                C->gave_up = 1;
                atomicOr(status, CR_FLAG_TIMEOUT);
                break;
            }
        }
    }
    st[(uint64_t)tile * 256] = kTilePrefix | (before + mine);
    S.base[tid] = smaller + (uint32_t)before;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const uint64_t i = i0 + 32u * j;
        if (i >= n) continue;
        const uint32_t d = (uint32_t)(key[j] >> shift) & 0xffu, pos = S.base[d] + S.wcnt[warp][d] + rank[j];
        kout[pos] = key[j];
        vout[pos] = vin ? __ldcg(vin + i) : (uint32_t)i;
    }
}

// Bound: the chain of phases (the wait for the one before, a tile's loads, its look-back), 5-7
// us each.  Builds of one plan from 500,000 requests, C = 16,384, this sort in them: 500,000 keys
// 282 us (304 with a launch per pass, 486 with three: tile counts, scan, scatter); 145 keys,
// which it leaves alone, 82 us (142, 315: launches that find nothing to do are not free).
__global__ void __launch_bounds__(kSortBlock, 3) k_sort(const __grid_constant__ sort_job J)
{
    uint64_t n = J.n;
    if (J.n_dev) {
        const uint64_t u = *J.n_dev;
        if (u <= J.skip_le) return;
        n = u < n ? u : n;
    }
    __shared__ sort_smem S;
    uint32_t *cnt = &S.wcnt[0][0];  // [8 * 256]
    sort_counters *C = J.C;
    const uint32_t tid = threadIdx.x, lt = (1u << cr_lane()) - 1u;
    const uint32_t tiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
    const uint32_t phases = J.order ? 10u + J.passes2 : 9u;
    for (;;) {
        __syncthreads();  // (the shared memory of the item before)
        if (tid == 0) {
            const uint32_t t = atomicAdd(&C->ticket, 1u), phase = t / tiles;
            S.ticket = t;
            S.ok = 1;
            if (phase > 0 && phase < phases) {
                const volatile uint32_t *done = &C->done[phase - 1u];
                uint32_t spin = 0;
                while (*done < tiles && ++spin < kSortSpin) {}
                if (*done < tiles) {  // never
                    S.ok = 0;
                    C->gave_up = 1;
                    atomicOr(J.status, CR_FLAG_TIMEOUT);
                }
                __threadfence();
            }
        }
        __syncthreads();
        const uint32_t phase = S.ticket / tiles, tile = S.ticket - phase * tiles;
        if (phase >= phases || !S.ok) return;
        const uint64_t i0 = (uint64_t)tile * kSortTile + tid;
        if (phase == 0) {
            for (uint32_t x = tid; x < 8u * 256u; x += kSortBlock) cnt[x] = 0;
            J.states[0][(uint64_t)tile * 256 + tid] = 0;
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kSortItems; ++j) {
                const uint64_t i = i0 + (uint64_t)j * kSortBlock;
                if (i >= n) break;
                const unsigned long long key = J.k_in[i];
#pragma unroll
                for (int p = 0; p < 8; ++p) atomicAdd(&cnt[256 * p + ((uint32_t)(key >> (8 * p)) & 0xffu)], 1u);
            }
            __syncthreads();
            for (uint32_t x = tid; x < 8u * 256u; x += kSortBlock)
                if (cnt[x]) atomicAdd(&C->digits[0][0] + x, cnt[x]);
        } else if (phase <= 8) {
            const uint32_t p = phase - 1u, w = p & 1u;
            sort_tile<unsigned long long>(S, tile, p ? J.k[w ^ 1u] : J.k_in, p ? J.v[w ^ 1u] : J.v_in, J.k[w], J.v[w], n,
                                          (int)(8u * p), C->digits[p], J.states[w], J.states[w ^ 1u], C, J.status);
        } else if (phase == 9) {
            // the sorted pairs as the plan's histogram, the second sort's keys and their digits
            for (uint32_t x = tid; x < 4u * 256u; x += kSortBlock) cnt[x] = 0;
            __syncthreads();
#pragma unroll
            for (int j = 0; j < kSortItems; ++j) {
                const uint64_t u = i0 + (uint64_t)j * kSortBlock;
                const bool in = u < n;
                uint32_t key = 0;
                if (in) {
                    const uint32_t c = __ldcg(J.v[1] + u);
                    J.ukey[u] = __ldcg(J.k[1] + u);
                    J.ucnt[u] = c;
                    J.s[1][u] = key = (uint32_t)(J.n_sum - c);
                }
                // most counts are equal: one atomic per distinct sort key of the warp
                const uint32_t peers = __match_any_sync(0xffffffffu, key) & __ballot_sync(0xffffffffu, in);
                if (in && (peers & lt) == 0)
                    for (uint32_t p = 0; p < J.passes2; ++p)
                        atomicAdd(&cnt[256u * p + ((key >> (8u * p)) & 0xffu)], (uint32_t)__popc(peers));
            }
            __syncthreads();
            for (uint32_t x = tid; x < 256u * J.passes2; x += kSortBlock)
                if (cnt[x]) atomicAdd(&C->digits[8][0] + x, cnt[x]);
        } else {
            const uint32_t p = phase - 10u, w = p & 1u;
            sort_tile<uint32_t>(S, tile, J.s[w ^ 1u], p ? J.o[w ^ 1u] : nullptr, J.s[w],
                                p + 1u == J.passes2 ? J.order : J.o[w], n, (int)(8u * p), C->digits[8u + p], J.states[w],
                                J.states[w ^ 1u], C, J.status);
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            const uint32_t d = atomicAdd(&C->done[phase], 1u) + 1u;
            // the order is whole (S stays 0 if a wait gave up: nothing is admitted then)
            if (J.order && phase + 1u == phases && d == tiles && !*(volatile uint32_t *)&C->gave_up) J.info->S = n;
        }
    }
}

int sort_launch(cr_ctx *ctx, sort_job &J, bool zero)
{
    uint4 *p;
    uint32_t quads;
    CR_TRY(cr_sort_counters(ctx, J.n, &p, &quads));
    J.C = (sort_counters *)p;
    J.states[0] = (unsigned long long *)(J.C + 1);
    J.states[1] = J.states[0] + sort_tiles(J.n) * 256;
    J.status = ctx->d_status;
    if (zero) CR_CUDA(ctx, cudaMemsetAsync(J.C, 0, sizeof(sort_counters), ctx->stream));
    CR_LAUNCH(ctx, k_sort, cr_blocks(sort_tiles(J.n), 1, (unsigned int)ctx->num_sms * 3u), kSortBlock, 0, J);
    return CR_OK;
}

}  // namespace

int cr_scan_u32(cr_ctx *ctx, const uint32_t *in, uint32_t *out, uint64_t n, uint32_t *d_total)
{
    return scan_impl<uint32_t>(ctx, in, out, n, 0, d_total);
}

int cr_scan_u64_inclusive(cr_ctx *ctx, const unsigned long long *in, unsigned long long *out, uint64_t n)
{
    return scan_impl<unsigned long long>(ctx, in, out, n, 1, (unsigned long long *)nullptr);
}

int cr_sort_counters(cr_ctx *ctx, uint64_t n, uint4 **counters, uint32_t *quads)
{
    if (n >= (1ull << 32)) return cr_fail(ctx, CR_EINVAL, "radix sort: n >= 2^32");
    void *p;
    CR_TRY(cr_scratch(ctx, SCR_SORT_HIST, sizeof(sort_counters) + 2 * sort_tiles(n) * 256 * sizeof(unsigned long long), &p));
    *counters = (uint4 *)p;
    *quads = (uint32_t)(sizeof(sort_counters) / sizeof(uint4));
    return CR_OK;
}

int cr_radix_sort_u64(cr_ctx *ctx, const unsigned long long *k_in, uint64_t n, const unsigned long long **k_out,
                      const uint32_t **pos_out)
{
    *k_out = k_in;
    *pos_out = nullptr;
    if (n == 0) return CR_OK;
    sort_job J = {};
    J.k_in = k_in;
    J.n = n;
    for (int x = 0; x < 2; ++x) {
        void *k, *v;
        CR_TRY(cr_scratch(ctx, x ? SCR_SORT_K1 : SCR_SORT_K0, n * sizeof(unsigned long long), &k));
        CR_TRY(cr_scratch(ctx, x ? SCR_SORT_V1 : SCR_SORT_V0, n * sizeof(uint32_t), &v));
        J.k[x] = (unsigned long long *)k;
        J.v[x] = (uint32_t *)v;
    }
    CR_TRY(sort_launch(ctx, J, true));
    *k_out = J.k[1];  // eight passes: the last one writes buffers 1
    *pos_out = J.v[1];
    return CR_OK;
}

int cr_plan_sort_histogram(cr_ctx *ctx, cr_plan_info_dev *info, uint64_t n, unsigned long long skip_le,
                           unsigned long long *k0, uint32_t *v0, unsigned long long *k1, uint32_t *v1,
                           unsigned long long *ukey, unsigned long long *ucnt, uint32_t *sA, uint32_t *sB,
                           uint32_t *oB, uint32_t *order)
{
    sort_job J = {};
    J.k_in = k0;
    J.v_in = v0;
    J.k[0] = k1;
    J.v[0] = v1;
    J.k[1] = k0;
    J.v[1] = v0;
    J.info = info;
    J.ukey = ukey;
    J.ucnt = ucnt;
    J.s[0] = sB;  // pass p of the second sort reads s[p & 1 ^ 1]: sA first
    J.s[1] = sA;
    J.o[0] = oB;
    J.o[1] = v0;  // (the counts have been copied out by then)
    J.order = order;
    J.passes2 = 1;
    while (J.passes2 < 4 && (n >> (8 * J.passes2))) ++J.passes2;  // n - count < 2^(8 passes)
    J.n_sum = J.n = n;
    J.n_dev = &info->U;
    J.skip_le = skip_le;
    return sort_launch(ctx, J, false);
}
