// a8, a9: shadow replay (cr_shadow_replay).
//
//   partition  one stable counting sort per replica by destination: each
//              (replica, destination) stream's request indices in arrival
//              order; the replay gathers each request's (key, prefix, suffix)
//              record, packed once per call, through them
//   replay     one warp per (stream, chunk); the stream's recent keys live in
//              shared memory by access time, with a bitmap of last accesses and a
//              hash index from key to time, and 32 requests are simulated per
//              step, one per lane.  A request's depth (its LRU stack distance) decides the
//              hit at every smaller capacity at once, because LRU caches are
//              nested (Mattson et al. 1970): the cache of capacity c is the c
//              most recent entries of any larger one.
//   state      kept between calls as keys in recency order (most recent first).
//   tokens     the byte-aware variant (cr_replay_create_tokens): capacities in
//              prefix tokens, the same window with each time's tokens (k_lru_tokens).
#include <stdlib.h>
#include <string.h>

#include "cr_device.cuh"
#include "cr_internal.cuh"

namespace {

struct replay_caps {
    uint32_t n_caps;
    uint32_t cap[CR_MAX_CAPS];
};

struct rec16 {
    unsigned long long key;
    uint32_t P, S;
};

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (uint32_t)o) v += y;
    }
    return v;
}

// ---- partition: one stable counting sort per replica, by destination --------
// Tiles of 8192 requests.  k_part_count writes each tile's destination counts
// at [(replica * R + r) * ntiles + tile]; one exclusive scan of that array
// gives every (stream, tile) its output base, in stream-major order.
// k_part_scatter ranks each tile's requests stably (warp-private counters),
// stages their request indices in shared memory in (destination, arrival)
// order, and writes them out so that consecutive threads write consecutive
// positions of a destination's run.  The replay reads each request's
// (key, prefix, suffix) record, packed once per call by k_part_records,
// through these indices.
constexpr int kPartBlock = 256;
constexpr int kPartWarps = kPartBlock / 32;
constexpr int kPartPer = 32;                      // requests per thread
constexpr int kPartTile = kPartBlock * kPartPer;  // 8192
constexpr uint32_t kNoDest = 0xffffu;

// Counts of one tile in u32 bins [R], one shared-memory atomic add per item.  A warp's
// lanes take consecutive items, 16 loads of two bytes in flight each: a replica's row may
// start on any even address (n is often odd), and round-robin destinations, consecutive in
// memory, fall into different banks.  51 M destinations, R = 1024, n odd: 144 -> 53 us
// against 32 consecutive items per lane.
// One more row of blocks packs a (key, prefix, suffix) record per request, read by the
// replay through the indices.
__global__ void __launch_bounds__(kPartBlock) k_part_count(const uint16_t *__restrict__ dest, unsigned long long n,
                                                           uint32_t R, uint32_t ntiles, uint32_t n_rep,
                                                           uint32_t *__restrict__ cnt,
                                                           const unsigned long long *__restrict__ keys,
                                                           const uint32_t *__restrict__ plen,
                                                           const uint32_t *__restrict__ slen,
                                                           rec16 *__restrict__ recs, uint32_t *status)
{
    extern __shared__ uint32_t pcb[];  // [R]
    const uint32_t rep = blockIdx.y, tile = blockIdx.x, lane = cr_lane();
    if (rep == n_rep) {
        const unsigned long long i0 = (unsigned long long)tile * kPartTile;
        for (unsigned long long i = i0 + threadIdx.x; i < n && i < i0 + kPartTile; i += kPartBlock) {
            rec16 r;
            r.key = keys[i];
            r.P = plen[i];
            r.S = slen[i];
            recs[i] = r;
        }
        return;
    }
    for (uint32_t r = threadIdx.x; r < R; r += kPartBlock) pcb[r] = 0;
    __syncthreads();
    const uint16_t *D = dest + (unsigned long long)rep * n;
    const unsigned long long base = (unsigned long long)tile * kPartTile;
    const uint32_t cnt_t = (uint32_t)min((unsigned long long)kPartTile, n - base);
    bool bad = false;
    constexpr uint32_t kInFlight = 16;
    for (uint32_t i0 = threadIdx.x; i0 < cnt_t; i0 += kPartBlock * kInFlight) {
        uint32_t d[kInFlight];
#pragma unroll
        for (uint32_t x = 0; x < kInFlight; ++x) {
            const uint32_t i = i0 + x * kPartBlock;
            d[x] = i < cnt_t ? D[base + i] : 0x10000u;
        }
#pragma unroll
        for (uint32_t x = 0; x < kInFlight; ++x) {
            if (d[x] < R)
                atomicAdd(&pcb[d[x]], 1u);
            else if (d[x] != 0x10000u)
                bad = true;  // skipped: reported through the status word
        }
    }
    __syncthreads();
    for (uint32_t r = threadIdx.x; r < R; r += kPartBlock) cnt[((unsigned long long)rep * R + r) * ntiles + tile] = pcb[r];
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, CR_FLAG_BADDEST);
}

// start[s] = first record of stream s = (replica, r); start[ns] = number of records.
__global__ void k_part_starts(const uint32_t *__restrict__ off, uint32_t ns, uint32_t ntiles,
                              const uint32_t *__restrict__ total, uint32_t *__restrict__ start, uint32_t *next)
{
    if (blockIdx.x == 0 && threadIdx.x < 3) next[threadIdx.x] = 0;  // the work items' counters
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s <= ns; s += gridDim.x * blockDim.x)
        start[s] = s < ns ? off[(unsigned long long)s * ntiles] : *total;
}

// Shared memory of k_part_scatter: per-warp counters wc[8][R] (u16), the tile's
// destination offsets toff[R] (u32), and the tile's items in (destination, arrival) order
// (u32: destination << 16 | item number).
__host__ __device__ inline size_t part_scatter_smem(uint32_t R)
{
    return (size_t)R * kPartWarps * 2 + (size_t)R * 4 + (size_t)kPartTile * 4;
}

// From this R on, a round's equal destinations are found by writing lane numbers to the
// counters (BALLOTS false): few of 32 requests then share one.  Below, one ballot per bit
// of the destination.
constexpr uint32_t kPartSparse = 192;

// Bound: instructions (ranking about half).  51 M destinations, R = 1024: 345 -> 239 us;
// ranks are kept in registers instead of shared memory (a pass less; 80 registers and 32
// bytes of spills, three blocks per SM: four with 64 registers spill more and take 315 us), and the lane numbers take about 20
// instructions per 32 requests where a ballot per destination bit takes 50.
template <bool BALLOTS>
__global__ void __launch_bounds__(kPartBlock, 3) k_part_scatter(const uint16_t *__restrict__ dest, unsigned long long n,
                                                                uint32_t R, uint32_t ntiles,
                                                                const uint32_t *__restrict__ off,
                                                                uint32_t *__restrict__ out, unsigned long long m)
{
    extern __shared__ uint4 psm[];
    uint16_t *wc = reinterpret_cast<uint16_t *>(psm);                            // [8][R]
    uint32_t *toff = reinterpret_cast<uint32_t *>(wc + (size_t)R * kPartWarps);  // [R]
    uint32_t *sitem = toff + R;                                                  // [kPartTile]
    __shared__ uint32_t part[kPartBlock];
    __shared__ uint32_t s_valid;
    const uint32_t rep = blockIdx.y, tile = blockIdx.x, lane = cr_lane(), warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    uint4 *wc4 = reinterpret_cast<uint4 *>(wc);
    for (uint32_t r = threadIdx.x; r < R; r += kPartBlock) wc4[r] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    const uint16_t *D = dest + (unsigned long long)rep * n;
    const unsigned long long base = (unsigned long long)tile * kPartTile;
    const uint32_t cnt = (uint32_t)min((unsigned long long)kPartTile, n - base);
    // ranks: warp w takes items [1024 w, 1024 w + 1024) of the tile, 32 at a time
    // (lane order is arrival order); all 32 rounds' destinations are read up front.
    constexpr uint32_t kPerWarp = kPartTile / kPartWarps;
    const uint32_t nb = 32u - (uint32_t)__clz(R);
    volatile uint16_t *wcw = wc + (size_t)warp * R;
    uint32_t dv[kPartPer / 2];  // two rounds' destinations per word (kNoDest: no item)
    uint32_t rk[kPartPer / 2];  // and ranks among the warp's items of the destination
#pragma unroll
    for (int x = 0; x < kPartPer / 2; ++x) {
        const uint32_t i0 = warp * kPerWarp + (2u * x) * 32u + lane, i1 = i0 + 32u;
        const uint32_t a = i0 < cnt ? D[base + i0] : kNoDest, c = i1 < cnt ? D[base + i1] : kNoDest;
        dv[x] = (a < R ? a : kNoDest) | ((c < R ? c : kNoDest) << 16);
        rk[x] = 0;
    }
#pragma unroll
    for (uint32_t j = 0; j < (uint32_t)kPartPer; ++j) {
        const uint32_t d = (dv[j >> 1] >> (16 * (j & 1))) & 0xffffu;
        const bool in = d != kNoDest;
        const uint32_t before = in ? wcw[d] : 0u;
        uint32_t peers = 1u << lane;  // the round's lanes with this destination
        if (BALLOTS) {
            // one ballot per bit of the destination (R stands for "no item")
            const uint32_t dd = in ? d : R;
            peers = 0xffffffffu;
            for (uint32_t bt = 0; bt < nb; ++bt) {
                const uint32_t bit = (dd >> bt) & 1u;
                const uint32_t B = __ballot_sync(0xffffffffu, bit);
                peers &= bit ? B : ~B;
            }
            __syncwarp();
        } else {
            // every lane writes its number to its counter: a lane that does not read it back
            // shares its destination, and those lanes' destinations are settled one by one
            __syncwarp();
            if (in) wcw[d] = (uint16_t)lane;
            __syncwarp();
            uint32_t lost = __ballot_sync(0xffffffffu, in && wcw[d] != lane);
            while (lost) {  // uniform; every pass settles at least one lane
                const uint32_t dl = __shfl_sync(0xffffffffu, d, __ffs(lost) - 1);
                const uint32_t same = __ballot_sync(0xffffffffu, d == dl);
                if (d == dl) peers = same;
                lost &= ~same;
            }
            __syncwarp();
        }
        rk[j >> 1] |= (before + (uint32_t)__popc(peers & lt)) << (16 * (j & 1));
        if (in && (peers & lt) == 0) wcw[d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // per destination: exclusive prefix over the 8 warps and its total; then the
    // tile's destination offsets by a block scan over thread-contiguous ranges of R
    const uint32_t per = (R + kPartBlock - 1) / kPartBlock, r0 = threadIdx.x * per;
    uint32_t run = 0;
    for (uint32_t r = r0; r < r0 + per && r < R; ++r) {
        uint16_t acc = 0;
#pragma unroll
        for (int w = 0; w < kPartWarps; ++w) {
            const uint16_t x = wc[(size_t)w * R + r];
            wc[(size_t)w * R + r] = acc;
            acc = (uint16_t)(acc + x);
        }
        toff[r] = acc;  // the destination's total until the scan below
        run += acc;
    }
    part[threadIdx.x] = run;
    __syncthreads();
    if (threadIdx.x < 32) {  // exclusive scan of the 256 partials by one warp
        constexpr int kPer = kPartBlock / 32;
        uint32_t x[kPer], sum = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            x[k] = part[threadIdx.x * kPer + k];
            sum += x[k];
        }
        const uint32_t incl = warp_incl_scan(sum, lane);
        uint32_t ex = incl - sum;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            part[threadIdx.x * kPer + k] = ex;
            ex += x[k];
        }
        if (threadIdx.x == 31) s_valid = incl;
    }
    __syncthreads();
    run = part[threadIdx.x];
    for (uint32_t r = r0; r < r0 + per && r < R; ++r) {
        const uint32_t t = toff[r];
        toff[r] = run;
        run += t;
    }
    __syncthreads();
    // staging: every valid item at its place in (destination, arrival) order
#pragma unroll
    for (uint32_t j = 0; j < (uint32_t)kPartPer; ++j) {
        const uint32_t d = (dv[j >> 1] >> (16 * (j & 1))) & 0xffffu;
        if (d == kNoDest) continue;
        const uint32_t pos = toff[d] + wc[(size_t)warp * R + d] + ((rk[j >> 1] >> (16 * (j & 1))) & 0xffffu);
        sitem[pos] = (d << 16) | (warp * kPerWarp + j * 32u + lane);
    }
    // each destination's output position minus its staging position (mod 2^32), in
    // the counters' space, which the staging no longer needs
    uint32_t *gb = reinterpret_cast<uint32_t *>(wc);  // [R]
    const uint32_t *O = off + (unsigned long long)rep * R * ntiles;
    __syncthreads();
    for (uint32_t r = threadIdx.x; r < R; r += kPartBlock) gb[r] = O[(unsigned long long)r * ntiles + tile] - toff[r];
    __syncthreads();
    // output: consecutive threads write consecutive positions of each destination's run
    const uint32_t valid = s_valid;
    for (uint32_t j = threadIdx.x; j < valid; j += kPartBlock) {
        const uint32_t it = sitem[j], d = it >> 16;
        if (d >= R) continue;  // never: every staged item is valid (guards the writes)
        const uint32_t o = gb[d] + j;
        if (o < m) out[o] = (uint32_t)base + (it & 0xffffu);
    }
}

// Work items: every stream's chunks (an empty stream gets one that carries its state
// over); all but a stream's last have CL requests.  Items longer than `longer` requests come
// first, so that the launch does not end with a few SMs on a hot key's stream (sticky-hash
// replicas have streams 13 times the mean: SMs were busy 78% of the launch; 48 replicas x
// 1,066,667 requests, 2.23 -> 1.90 ms a call).
__device__ __forceinline__ uint32_t long_chunks(uint32_t len, uint32_t nch, uint32_t CL, uint32_t longer)
{
    return (CL > longer ? nch - 1u : 0u) + (len - (nch - 1u) * CL > longer ? 1u : 0u);
}

// nch[s] = chunks of stream s; next[2] += the long ones.
__global__ void k_chunk_counts(const uint32_t *__restrict__ start, uint32_t ns, uint32_t CL, uint32_t longer,
                               uint32_t *__restrict__ nch, uint32_t *next)
{
    uint32_t nf = 0;
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < ns; s += gridDim.x * blockDim.x) {
        const uint32_t len = start[s + 1] - start[s];
        const uint32_t c = len ? (len + CL - 1) / CL : 1u;
        nch[s] = c;
        nf += long_chunks(len, c, CL, longer);
    }
    nf = __reduce_add_sync(0xffffffffu, nf);
    if ((threadIdx.x & 31u) == 0 && nf) atomicAdd(&next[2], nf);
}

// map[x] and map[items_max + x]: item x's stream and chunk.  f / b: places of the stream's long
// / other chunks.
struct item_map {
    uint32_t *__restrict__ map;
    uint64_t items_max;
    uint32_t CL, longer;
    __device__ __forceinline__ void put(uint32_t s, uint32_t len, uint32_t n, uint32_t f, uint32_t b, uint32_t c) const
    {
        const bool full = CL > longer;  // all chunks but the last have CL requests
        uint32_t x = (full ? f : b) + c;
        if (c + 1u == n) x = len - c * CL > longer ? f + (full ? c : 0u) : b + (full ? 0u : c);
        if (x < items_max) {
            map[x] = s;
            map[items_max + x] = c;
        }
    }
};

// coff[s]: chunks of the streams before s; next[0], next[1]: long and other items placed so far.
__global__ void k_item_map(const uint32_t *__restrict__ start, const uint32_t *__restrict__ coff, uint32_t ns,
                           uint32_t CL, uint32_t longer, uint32_t *next, uint32_t *__restrict__ map,
                           uint64_t items_max)
{
    const uint32_t lane = threadIdx.x & 31u, first = next[2];
    for (uint32_t s0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; s0 < ns; s0 += gridDim.x * blockDim.x) {
        const uint32_t s = s0 + lane;
        const bool in = s < ns;
        const uint32_t len = in ? start[s + 1] - start[s] : 0u, nch = in ? coff[s + 1] - coff[s] : 0u;
        const uint32_t nf = nch ? long_chunks(len, nch, CL, longer) : 0u;
        const uint32_t fi = warp_incl_scan(nf, lane), bi = warp_incl_scan(nch - nf, lane);
        uint32_t f0 = 0, b0 = 0;
        if (lane == 31) {
            if (fi) f0 = atomicAdd(&next[0], fi);
            if (bi) b0 = atomicAdd(&next[1], bi);
        }
        f0 = __shfl_sync(0xffffffffu, f0, 31) + fi - nf;
        b0 = __shfl_sync(0xffffffffu, b0, 31) + first + bi - (nch - nf);
        const item_map M = {map, items_max, CL, longer};
        for (uint32_t c = 0; c < nch; ++c) M.put(s, len, nch, f0, b0, c);
    }
}

// The same for up to kItemsCta streams by one CTA, stream starts included: one launch in
// place of k_part_starts, k_chunk_counts, a scan and k_item_map.  A warp takes 32 consecutive
// streams at a time; the chunks of a stream with more than a few are left for a warp of their
// own (one lane took 120 us over the 3,907 chunks of a call on one stream).  30 replicas x
// 133,333 requests, 64 destinations, with the records packed in the count launch: 212 -> 192 us
// a call; one interval of 20,000 requests, two replicas 154 -> 142 us.  8,000 / 12,288 / 20,480
// / 30,720 streams of a few requests, partition: 38 / 46 / 58 / 70 us, in four launches 38 (from
// 8,193) / 46 / 50 / 50.
constexpr uint32_t kItemsCta = 8192, kItemsMany = 512;
__global__ void __launch_bounds__(1024) k_items_cta(const uint32_t *__restrict__ off, uint32_t ns, uint32_t ntiles,
                                                    const uint32_t *__restrict__ total_in, uint32_t *start, uint32_t CL,
                                                    uint32_t longer, uint32_t *__restrict__ total,
                                                    uint32_t *__restrict__ map, uint64_t items_max)
{
    extern __shared__ uint32_t st[];  // [ns + 1] the starts again
    __shared__ uint32_t s_long, s_other, n_long;  // places given out, long items
    __shared__ uint3 many[kItemsMany];            // streams of many chunks: stream, f, b
    __shared__ uint32_t n_many;
    const uint32_t lane = threadIdx.x & 31u;
    if (threadIdx.x == 0) s_long = s_other = n_long = n_many = 0;
#pragma unroll 4
    for (uint32_t s = threadIdx.x; s <= ns; s += 1024u)
        start[s] = st[s] = s < ns ? off[(unsigned long long)s * ntiles] : *total_in;
    __syncthreads();
    auto chunks = [&](uint32_t s, uint32_t &len, uint32_t &nch, uint32_t &nf) {
        const bool in = s < ns;
        len = in ? st[s + 1] - st[s] : 0u;
        nch = in ? (len ? (len + CL - 1u) / CL : 1u) : 0u;
        nf = nch ? long_chunks(len, nch, CL, longer) : 0u;
    };
    const item_map M = {map, items_max, CL, longer};
    uint32_t len, nch, nf, sum = 0;
    for (uint32_t s0 = threadIdx.x & ~31u; s0 < ns; s0 += 1024u) {
        chunks(s0 + lane, len, nch, nf);
        sum += nf;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0 && sum) atomicAdd(&n_long, sum);
    __syncthreads();
    for (uint32_t s0 = threadIdx.x & ~31u; s0 < ns; s0 += 1024u) {
        chunks(s0 + lane, len, nch, nf);
        const uint32_t fi = warp_incl_scan(nf, lane), bi = warp_incl_scan(nch - nf, lane);
        uint32_t f0 = 0, b0 = 0;
        if (lane == 31) {
            if (fi) f0 = atomicAdd(&s_long, fi);
            if (bi) b0 = atomicAdd(&s_other, bi);
        }
        f0 = __shfl_sync(0xffffffffu, f0, 31) + fi - nf;
        b0 = __shfl_sync(0xffffffffu, b0, 31) + n_long + bi - (nch - nf);
        if (nch > 4u) {
            const uint32_t i = atomicAdd(&n_many, 1u);
            if (i < kItemsMany) {
                many[i] = make_uint3(s0 + lane, f0, b0);
                nch = 0;
            }
        }
        for (uint32_t c = 0; c < nch; ++c) M.put(s0 + lane, len, nch, f0, b0, c);
    }
    __syncthreads();
    if (threadIdx.x == 0) *total = n_long + s_other;
    for (uint32_t i = threadIdx.x >> 5; i < min(n_many, kItemsMany); i += 32u) {
        const uint3 e = many[i];
        chunks(e.x, len, nch, nf);
        for (uint32_t c = lane; c < nch; c += 32u) M.put(e.x, len, nch, e.y, e.z, c);
    }
}

// State before and after a call: [stream][cmax] (token capacities: [stream][kTokMax]), most
// recent first.
struct replay_state {
    const unsigned long long *keys_in;
    const uint32_t *cum_in;  // token capacities: tokens of entries 0 .. j
    const uint32_t *fill_in;
    unsigned long long *keys_out;
    uint32_t *cum_out;
    uint32_t *fill_out;
};

inline replay_state state_of(const cr_replay *rp)
{
    return {rp->d_keys[rp->cur],     rp->d_size[rp->cur],     rp->d_fill[rp->cur],
            rp->d_keys[rp->cur ^ 1], rp->d_size[rp->cur ^ 1], rp->d_fill[rp->cur ^ 1]};
}

__device__ __forceinline__ uint32_t sat_add(uint32_t a, uint32_t b)
{
    const uint32_t v = a + b;
    return v < a ? 0xffffffffu : v;
}

// ---- replay of calls whose streams are mostly empty or a few requests long ----------
// One warp per item, the list in registers (lane j holds entry j), one request at a time: items
// whose carried-in keys and requests are at most 32 together; empty streams carry their state
// over whatever its size; the others are left in rest[1 ..], their number in rest[0].  Nothing
// in shared memory, so that the chain of dependent reads (item, stream, state, indices,
// records) overlaps over three to five times the warps that the windows below leave room for,
// which an item of two requests pays for without using them.  Simulation alone, 24 replicas x
// 1,000 requests over 8,192 destinations, 24,576 tokens 289 -> 53 us, capacity 128 107 -> 55;
// 48 x 4,096 over 1,024, 24,576 tokens 125 -> 37 (prefixes of 175 tokens on average, lists of
// 140: 216 -> 212).
template <bool TOKENS>
__global__ void __launch_bounds__(256) k_replay_short(const __grid_constant__ replay_caps caps, uint32_t lim, uint32_t stride,
                                                      uint32_t R, uint32_t ns, const uint32_t *__restrict__ start,
                                                      const uint32_t *__restrict__ map, uint32_t items_max,
                                                      const uint32_t *__restrict__ total, const uint32_t *__restrict__ idx,
                                                      const rec16 *__restrict__ recs, uint32_t nrec, const replay_state st,
                                                      unsigned long long *__restrict__ ctr, uint32_t *rest, uint32_t *status)
{
    __shared__ uint32_t s_rest, s_at;
    const uint32_t lane = cr_lane(), w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (threadIdx.x == 0) s_rest = 0;
    __syncthreads();
    const bool mine = w < *total;
    uint32_t s = 0, ci = 0, b = 0, e = 0, fin = 0;
    if (mine) {
        s = min(map[w], ns - 1u);
        ci = map[items_max + w];
        b = start[s];
        e = start[s + 1];
        fin = min(st.fill_in[s], stride);
    }
    const uint32_t n = e - b;
    const bool few = mine && n && ci == 0 && n <= 32u && fin <= 32u - n;
    uint32_t at = 0;
    if (mine && n && !few && lane == 0) at = atomicAdd(&s_rest, 1u);
    __syncthreads();
    if (threadIdx.x == 0 && s_rest) s_at = atomicAdd(rest, s_rest);
    __syncthreads();
    if (mine && n && !few && lane == 0) rest[1u + s_at + at] = w;
    const unsigned long long *kin = st.keys_in + (size_t)s * stride;
    unsigned long long *kout = st.keys_out + (size_t)s * stride;
    const uint32_t *cin = TOKENS ? st.cum_in + (size_t)s * stride : nullptr;
    uint32_t *cout = TOKENS ? st.cum_out + (size_t)s * stride : nullptr;
    if (mine && n == 0) {
        for (uint32_t j = lane; j < fin; j += 32) {
            kout[j] = kin[j];
            if (TOKENS) cout[j] = cin[j];
        }
        if (lane == 0) st.fill_out[s] = fin;
    }
    if (!few) return;  // (whole warps: no barrier follows)
    const uint32_t mycap = lane < caps.n_caps ? caps.cap[lane] : 0u;
    rec16 r = {0ull, 0u, 0u};
    if (lane < n) r = recs[min(idx[b + lane], nrec - 1u)];
    unsigned long long kr = lane < fin ? kin[lane] : 0ull;
    uint32_t cr = TOKENS && lane < fin ? cin[lane] : 0u, f = fin;  // tokens through the entry; entries
    uint32_t hits = 0;
    unsigned long long hit_tok = 0;
    for (uint32_t q = 0; q < n; ++q) {  // uniform
        const unsigned long long x = __shfl_sync(0xffffffffu, r.key, q);
        const uint32_t P = __shfl_sync(0xffffffffu, r.P, q);
        const uint32_t match = __ballot_sync(0xffffffffu, lane < f && kr == x);
        const bool found = match != 0;
        const uint32_t pos = found ? (uint32_t)__ffs(match) - 1u : f;  // f <= 31 when it is not found
        uint32_t depth = pos + 1u;
        if (TOKENS) {
            depth = __shfl_sync(0xffffffffu, cr, pos);
            const uint32_t before = __shfl_sync(0xffffffffu, cr, pos ? pos - 1u : 0u);
            if (found && depth - (pos ? before : 0u) != P && lane == 0) atomicOr(status, CR_FLAG_BADSIZE);
        }
        if (found && depth <= mycap) {  // lane c: capacity c
            ++hits;
            hit_tok += P;
        }
        // entries [0, pos) move down one place and now follow x
        const unsigned long long ku = __shfl_up_sync(0xffffffffu, kr, 1);
        const uint32_t cu = TOKENS ? __shfl_up_sync(0xffffffffu, cr, 1) : 0u;
        if (lane <= pos) {
            kr = lane ? ku : x;
            cr = TOKENS ? (lane ? sat_add(cu, P) : P) : 0u;
        }
        f += found ? 0u : 1u;
        if (TOKENS) {
            const uint32_t over = __ballot_sync(0xffffffffu, lane < f && cr > lim);
            if (over) f = (uint32_t)__ffs(over) - 1u;
        } else {
            f = min(f, lim);
        }
    }
    if (lane < f) {
        kout[lane] = kr;
        if (TOKENS) cout[lane] = cr;
    }
    if (lane == 0) st.fill_out[s] = f;
    const unsigned long long prompt = cr_warp_sum_u64(lane < n ? (unsigned long long)r.P + r.S : 0ull);
    if (lane < caps.n_caps) {
        unsigned long long *C = ctr + (((unsigned long long)(s / R) * caps.n_caps + lane) * R + s % R) * CR_CTR_FIELDS;
        atomicAdd(&C[0], (unsigned long long)n);
        if (hits) atomicAdd(&C[1], (unsigned long long)hits);
        if (hit_tok) atomicAdd(&C[2], hit_tok);
        atomicAdd(&C[3], prompt);
        atomicAdd(&C[4], prompt - hit_tok);
    }
}

// Which calls start with it (*rest != NULL then): streams of up to two requests on average, or,
// for token capacities whose lists seldom pass 32 prefixes, of up to eight.  Once lists are
// longer its launch is lost: ten replicas x 3,000 requests over 1,000 destinations, capacity
// 128, lists full 19 -> 29 us; four x 60,000 over 8,192 54 -> 89.
template <bool TOKENS>
int launch_short(cr_ctx *ctx, const cr_replay *rp, const replay_caps &caps, uint32_t lim, const uint32_t *start,
                 const uint32_t *map, uint32_t items_max, const uint32_t *total, uint64_t m, uint64_t items,
                 const uint32_t *idx, const rec16 *recs, uint64_t *d_ctr, uint32_t **rest)
{
    *rest = nullptr;
    if (m > (TOKENS && lim <= (1u << 16) ? 8u : 2u) * rp->n_streams) return CR_OK;
    void *p;
    CR_TRY(cr_scratch(ctx, SCR_REPLAY_REST, (items + 1) * sizeof(uint32_t), &p));
    *rest = (uint32_t *)p;
    CR_CUDA(ctx, cudaMemsetAsync(p, 0, sizeof(uint32_t), ctx->stream));
    CR_LAUNCH(ctx, k_replay_short<TOKENS>, (unsigned int)((items + 7) / 8), 256, 0, caps, lim, rp->cmax, rp->R,
              (uint32_t)rp->n_streams, start, map, items_max, total, idx, recs, (uint32_t)(m / rp->n_rep), state_of(rp),
              (unsigned long long *)d_ctr, *rest, ctx->d_status);
    return CR_OK;
}

// ---- replay: batched stack distances over access times -------------------------
// One warp per (stream, chunk) holds the LRU stack in shared memory, indexed by
// TIME.  Times 0 .. 32 nw - 1 form a window: the carried-in keys take the first
// ones in recency order, then every step of 32 requests takes one 32-bit word of
// times (the request on lane l of the step at word w has time 32 w + l).  KT holds
// the key accessed at each time, a bitmap marks the times that are some key's
// LAST access, and an index maps each key of the window to that time.  The recency
// position of a key (0 = most recent) is the number of live bits above its time,
// which one warp-wide scan of the words' popcounts gives for every lane of a step
// at once.  An access clears the key's old bit, sets its bit in the new word and
// writes the new time into its index entry; nothing else moves.  A key that falls
// below the largest capacity is left where it is: its position is past every
// capacity, so it counts as a miss, and it goes when the window is used up and the
// cmax most recent keys are renumbered 0 .. fill-1 (compaction).
//
// Bound: the latency of a step's dependence chain (match, index probe, popcount scan,
// insert) at the warps per SM that the window allows (14 at cmax 1024), 15.3 warp
// instructions per (request, replica) pair.  Keys indexed by slot, with an eviction per
// new key (search for the oldest live bits, index erase, slot hand-over), took 16.6 and a
// chain about a third longer: 48 replicas x 1,066,667 requests over 1,024 destinations
// at capacities 64 / 256 / 1024, partition included, 2.78 -> 2.23 ms (1.72 with the item
// order and the partition below); 30 replicas x 133,333 over 64 destinations at capacity
// 128, 270 -> 237 us (207).  Indexing only the
// requests' keys and streaming the carried-in ones past them fits 24 warps, but costs 18
// instructions per pair and measured 2.88 ms.
//
// A step is 32 consecutive requests of the stream, one per lane.  The depth of
// request i (its LRU stack distance, Mattson et al. 1970) follows from the
// state before the step and the step itself:
//   - key seen earlier in the step, last at lane j: 1 + the number of distinct
//     keys among lanes (j, i), at most 31;
//   - first time in the step, at recency position d0 before it: d0 + 1 + the
//     number of distinct keys among lanes < i that were deeper than d0 or
//     absent;
//   - absent before the step: a miss at every capacity.
// A request hits capacity c iff its depth <= c.
constexpr uint32_t kNone = 0xffffffffu;
constexpr uint32_t kStash = 32;              // index entries that found both buckets full
constexpr uint32_t kDegraded = 0x80000000u;  // stash overflowed: lookups scan the window

// Index: buckets of four 16-bit entries (tag above, time in the low `tb` bits; 0 =
// empty, so a tag is never 0), two candidate buckets per key.  A new key goes into
// the emptier one (the first when equal); a key whose buckets are both full goes to
// a small stash; if even the stash is full the index is marked degraded and lookups
// scan the window.  An entry stays where it is until the next compaction.
struct window_lru {
    unsigned long long *KT;   // [32 nw] key accessed at each time
    unsigned long long *bkt;  // [nb] index buckets
    uint16_t *E;              // the buckets as entries [4 nb], then the stash [kStash]
    uint32_t *BM;             // [nw] bit t of word w: time 32 w + t is a key's last access
    uint32_t *stash_n;        // stash entries claimed (| kDegraded once it overflowed)
    uint16_t *PX;             // [nw] compaction: live bits below each word
    uint32_t nw, nb, tmask;   // words, buckets, (1 << tb) - 1
    // token capacities only
    uint32_t *TK;             // [32 nw] prefix tokens of the request at each time
    uint32_t *SL, *SH;        // [nw] a word's live tokens: sum of their low 16 bits, sum of the rest
    uint2 *OP;                // [32] the step's requests: order of their keys at its start, tokens
};

__host__ __device__ inline size_t window_lru_bytes(uint32_t nw, uint32_t nb, bool tokens = false)
{
    const size_t base = (size_t)nw * 256 + (size_t)nb * 8 + kStash * 2 + (size_t)(nw + 1) * 4 + (size_t)(nw + 1) / 2 * 4;
    return (base + (tokens ? (size_t)nw * 136 + 32 * 8 + 8 : 0) + 15) & ~(size_t)15;
}

__device__ __forceinline__ window_lru window_lru_at(unsigned char *base, uint32_t nw, uint32_t nb)
{
    window_lru X;
    X.KT = reinterpret_cast<unsigned long long *>(base);
    X.bkt = X.KT + (size_t)nw * 32;
    X.E = reinterpret_cast<uint16_t *>(X.bkt);
    X.BM = reinterpret_cast<uint32_t *>(X.E + (size_t)nb * 4 + kStash);
    X.stash_n = X.BM + nw;
    X.PX = reinterpret_cast<uint16_t *>(X.stash_n + 1);
    X.nw = nw;
    X.nb = nb;
    X.tmask = (1u << (32 - __clz(32u * nw - 1u))) - 1u;
    X.TK = reinterpret_cast<uint32_t *>(X.PX + (nw + 1u) / 2u * 2u);
    X.SL = X.TK + (size_t)nw * 32;
    X.SH = X.SL + nw;
    X.OP = reinterpret_cast<uint2 *>((reinterpret_cast<uintptr_t>(X.SH + nw) + 7u) & ~(uintptr_t)7u);
    return X;
}

struct key_hash {
    uint32_t b1, b2, tag;  // buckets; tag in place, i.e. above the time bits
};

__device__ __forceinline__ key_hash sl_hash(const window_lru &X, unsigned long long key)
{
    const unsigned long long h = key * 0x9e3779b97f4a7c15ull;  // an odd multiplier spreads every key bit upwards
    key_hash r;
    r.b1 = __umulhi((uint32_t)(h >> 32), X.nb);
    r.b2 = __umulhi((uint32_t)(h >> 22), X.nb);
    r.tag = max((uint32_t)(h >> 28) & (0xffffu & ~X.tmask), X.tmask + 1u);
    return r;
}

// Is `key` in the index?  `time` receives its last access, `loc` its entry (kNone when
// a degraded index does not hold it).  The eight entries' tags are compared as
// halfwords, four words at once; only tag matches read their key.
__device__ __forceinline__ bool sl_lookup(const window_lru &X, const key_hash &H, unsigned long long key,
                                          uint32_t wnow, uint32_t &time, uint32_t &loc)
{
    const uint32_t T2 = H.tag * 0x10001u, lm = (0x7fffu & ~X.tmask) * 0x10001u;
    auto match = [&](uint32_t x) {  // bit 15 / 31: that half's tag equals the key's
        const uint32_t y = x ^ T2;
        return ~(((y & lm) + lm) | y) & 0x80008000u;
    };
    const unsigned long long v1 = X.bkt[H.b1], v2 = X.bkt[H.b2];
    // bits 12 .. 15: low halves of words 0 .. 3, bits 28 .. 31: their high halves
    uint32_t M = (match((uint32_t)v1) >> 3) | (match((uint32_t)(v1 >> 32)) >> 2) | (match((uint32_t)v2) >> 1) |
                 match((uint32_t)(v2 >> 32));
    time = 0;
    loc = kNone;
    while (M) {
        const uint32_t p = (uint32_t)__ffs(M) - 1u;
        M &= M - 1u;
        const uint32_t at = ((p & 2u) ? H.b2 : H.b1) * 4u + ((p & 1u) << 1) + (p >> 4);
        const uint32_t t = X.E[at] & X.tmask;
        if (X.KT[t] == key) {
            time = t;
            loc = at;
            return true;
        }
    }
    const uint32_t sn = *X.stash_n;
    if (sn) {
        for (uint32_t i = 0; i < (sn & ~kDegraded) && i < kStash; ++i) {
            const uint32_t e = X.E[4u * X.nb + i];
            if (e != 0 && X.KT[e & X.tmask] == key) {
                time = e & X.tmask;
                loc = 4u * X.nb + i;
                return true;
            }
        }
        if (sn & kDegraded)
            for (uint32_t t = 0; t < 32u * wnow; ++t)
                if (((X.BM[t >> 5] >> (t & 31u)) & 1u) && X.KT[t] == key) {
                    time = t;
                    return true;
                }
    }
    return false;
}

// Index an absent key last accessed at `time`.  A lost compare-and-swap means another
// lane changed the bucket, so the next look sees it; the bound only guards the loop.
__device__ __forceinline__ void sl_insert(const window_lru &X, const key_hash &H, uint32_t time)
{
    const unsigned long long ent = H.tag | time;
    auto empty = [](uint32_t x) { return ~(((x & 0x7fff7fffu) + 0x7fff7fffu) | x | 0x7fff7fffu); };
    for (int it = 0; it < 64; ++it) {
        const unsigned long long v1 = X.bkt[H.b1], v2 = X.bkt[H.b2];
        // bits 14, 30, 15, 31: entries 0 .. 3 are empty
        const uint32_t z1 = (empty((uint32_t)v1) >> 1) | empty((uint32_t)(v1 >> 32));
        const uint32_t z2 = (empty((uint32_t)v2) >> 1) | empty((uint32_t)(v2 >> 32));
        if (!(z1 | z2)) break;  // both buckets full
        const bool one = __popc(z1) >= __popc(z2);
        const uint32_t b = one ? H.b1 : H.b2, p = (uint32_t)__ffs(one ? z1 : z2) - 1u;
        const unsigned long long v = one ? v1 : v2;
        if (atomicCAS(&X.bkt[b], v, v | (ent << (((p & 1u) << 5) | (p & 16u)))) == v) return;
    }
    const uint32_t i = atomicAdd(X.stash_n, 1u) & ~kDegraded;
    if (i < kStash)
        X.E[4u * X.nb + i] = (uint16_t)ent;
    else
        atomicOr(X.stash_n, kDegraded);
}

// An empty index (warp-cooperative).
__device__ __forceinline__ void sl_clear_index(const window_lru &X, uint32_t lane)
{
    for (uint32_t x = lane; x < X.nb; x += 32) X.bkt[x] = 0;
    X.E[4u * X.nb + lane] = 0;
    if (lane == 0) *X.stash_n = 0;
    __syncwarp();
}

// Live times [a, a + fill); the next step takes the first word above them.
__device__ __forceinline__ void sl_live_range(const window_lru &X, uint32_t a, uint32_t fill, uint32_t lane)
{
    for (uint32_t w = lane; w < X.nw; w += 32) {
        const uint32_t lo = max(32u * w, a), hi = min(32u * w + 32u, a + fill);
        X.BM[w] = lo < hi ? (0xffffffffu >> (32u - (hi - lo))) << (lo & 31u) : 0u;
    }
}

// Live times below any time of the window: lane l keeps word 32 g + l of every
// group g of 32 words and the number of live bits in the words before it.
template <int NG>
struct live_prefix {
    uint32_t w[NG], ex[NG];
    __device__ __forceinline__ void load(const uint32_t *BM, uint32_t nw, uint32_t lane)
    {
        // both groups' popcounts in one scan: group g in bits 16 g .. 16 g + 15
        // (a group holds at most 1024 live bits, so the halves never carry)
        uint32_t pc = 0;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const uint32_t wi = 32u * g + lane;
            w[g] = wi < nw ? BM[wi] : 0u;
            pc |= (uint32_t)__popc(w[g]) << (16 * g);
        }
        const uint32_t incl = warp_incl_scan(pc, lane);
        const uint32_t ex2 = incl - pc;
        ex[0] = ex2 & 0xffffu;
        if (NG > 1) ex[NG - 1] = (ex2 >> 16) + (__shfl_sync(0xffffffffu, incl, 31) & 0xffffu);
    }
    // live times < s; every lane of the warp must call it
    __device__ __forceinline__ uint32_t below(uint32_t s) const
    {
        const uint32_t src = (s >> 5) & 31u, g = s >> 10;
        uint32_t e = 0, b = 0;
#pragma unroll
        for (int gg = 0; gg < NG; ++gg) {
            const uint32_t ee = __shfl_sync(0xffffffffu, ex[gg], src), bb = __shfl_sync(0xffffffffu, w[gg], src);
            if (g == (uint32_t)gg) {
                e = ee;
                b = bb;
            }
        }
        return e + (uint32_t)__popc(b & ((1u << (s & 31u)) - 1u));
    }
};

// Keep the `fill` most recent of the window's `live` keys, renumbered 0 .. fill-1 in
// order: every index entry takes its new time (or is emptied), then the keys move down.
template <int NG, bool TOKENS = false>
__device__ __forceinline__ void sl_compact(const window_lru &X, uint32_t live, uint32_t fill, uint32_t lane)
{
    live_prefix<NG> LP;
    LP.load(X.BM, X.nw, lane);
#pragma unroll
    for (int g = 0; g < NG; ++g)
        if (32u * g + lane < X.nw) X.PX[32u * g + lane] = (uint16_t)LP.ex[g];
    __syncwarp();
    const uint32_t drop = live - fill;
    const bool rebuild = *X.stash_n != 0;  // a stash in use: index the kept keys afresh below
    for (uint32_t b = lane; b < X.nb && !rebuild; b += 32) {
        const unsigned long long v = X.bkt[b];
        unsigned long long nv = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const uint32_t e = (uint32_t)(v >> (16 * p)) & 0xffffu;
            const uint32_t t = e & X.tmask, wd = t >> 5;
            const uint32_t rank = X.PX[wd] + (uint32_t)__popc(X.BM[wd] & ((1u << (t & 31u)) - 1u));
            if (e != 0 && rank >= drop) nv |= (unsigned long long)((e - t) | (rank - drop)) << (16 * p);
        }
        X.bkt[b] = nv;
    }
    // keys move to lower times, words in order: a word is read whole before anything above
    // its first live key's new time is written
    for (uint32_t w = 0; w < X.nw; ++w) {
        const uint32_t bits = X.BM[w], rank = X.PX[w] + (uint32_t)__popc(bits & ((1u << lane) - 1u));
        const unsigned long long k = X.KT[32u * w + lane];
        const uint32_t tk = TOKENS ? X.TK[32u * w + lane] : 0u;
        __syncwarp();
        if (((bits >> lane) & 1u) && rank >= drop) {
            X.KT[rank - drop] = k;
            if (TOKENS) X.TK[rank - drop] = tk;
        }
        __syncwarp();
    }
    sl_live_range(X, 0, fill, lane);
    __syncwarp();
    if (rebuild) {
        sl_clear_index(X, lane);
        for (uint32_t t = lane; t < fill; t += 32) sl_insert(X, sl_hash(X, X.KT[t]), t);
        __syncwarp();
    }
}

// One work item.
template <int NC, int NG, bool SMALL>
__device__ __forceinline__ void lru_item(uint32_t w, const replay_caps &caps, uint32_t cmax, uint32_t nw, uint32_t nb,
                                         uint32_t R, uint32_t ns, uint32_t CL, const uint32_t *__restrict__ start,
                                         const uint32_t *__restrict__ map, uint32_t items_max,
                                         const uint32_t *__restrict__ idx, const rec16 *__restrict__ recs,
                                         uint32_t nrec, const replay_state &st, unsigned long long *__restrict__ ctr,
                                         uint32_t *status)
{
    extern __shared__ uint4 smb[];
    const uint32_t lane = cr_lane(), warp = threadIdx.x >> 5;
    const window_lru X =
        window_lru_at(reinterpret_cast<unsigned char *>(smb) + window_lru_bytes(nw, nb) * warp, nw, nb);

    const uint32_t s = min(map[w], ns - 1u), ci = map[items_max + w];  // the item's stream and chunk
    const uint32_t b = start[s], e = start[s + 1];
    const uint32_t p0 = b + ci * CL;
    const uint32_t p1 = (e - p0) < CL ? e : p0 + CL;
    const uint32_t rep = s / R, r = s % R;
    const uint32_t fill_in = min(st.fill_in[s], cmax);
    const unsigned long long *kin = st.keys_in + (unsigned long long)s * cmax;
    const uint32_t lt = (1u << lane) - 1u, gt = ~(lt | (1u << lane));

    if (b == e) {  // nothing routed here: carry the state over unchanged
        unsigned long long *kout = st.keys_out + (unsigned long long)s * cmax;
        for (uint32_t q = lane; q < fill_in; q += 32) kout[q] = kin[q];
        if (lane == 0) st.fill_out[s] = fill_in;
        return;
    }

    // ---- state at p0: the most recent keys at the highest times below `top` ----------
    uint32_t live = 0, top = cmax;  // live keys of the window
    sl_clear_index(X, lane);
    if (ci == 0) {
        // the carried-in keys, eight loads in flight per lane
        top = live = fill_in;
        for (uint32_t q0 = 0; q0 < fill_in; q0 += 256) {
            unsigned long long kk[8];
#pragma unroll
            for (uint32_t x = 0; x < 8; ++x) {
                const uint32_t q = q0 + 32u * x + lane;
                kk[x] = q < fill_in ? kin[q] : 0ull;
            }
#pragma unroll
            for (uint32_t x = 0; x < 8; ++x) {
                const uint32_t q = q0 + 32u * x + lane;
                if (q < fill_in) {
                    X.KT[top - 1u - q] = kk[x];
                    sl_insert(X, sl_hash(X, kk[x]), top - 1u - q);
                }
            }
        }
    } else {
        // walk backwards collecting distinct keys, most recent first; keys are loaded two
        // steps early, through request indices read four steps early (in a hot key's stream
        // the walk is long, and nothing else hides the two dependent loads)
        for (uint32_t x = lane; x < nw; x += 32) X.BM[x] = 0;
        __syncwarp();
        const uint32_t back = p0 - b;
        const uint32_t vtot = back + fill_in;
        auto index_at = [&](uint32_t v) { return v < back ? min(idx[p0 - 1u - v], nrec - 1u) : 0u; };
        auto key_at = [&](uint32_t v, uint32_t ix) {
            return v < back ? recs[ix].key : (v < vtot ? kin[v - back] : 0ull);
        };
        uint32_t ix2 = index_at(lane + 64u), ix3 = index_at(lane + 96u);
        unsigned long long k0 = key_at(lane, index_at(lane)), k1 = key_at(lane + 32u, index_at(lane + 32u));
        for (uint32_t v0 = 0; v0 < vtot && live < cmax; v0 += 32) {
            const uint32_t v = v0 + lane;
            const bool valid = v < vtot;
            const unsigned long long key = k0;
            k0 = k1;
            k1 = key_at(v + 64u, ix2);
            ix2 = ix3;
            ix3 = index_at(v + 128u);
            const uint32_t vm = __ballot_sync(0xffffffffu, valid);
            const uint32_t peers = __match_any_sync(0xffffffffu, key) & vm;
            const key_hash H = sl_hash(X, key);
            uint32_t at, loc;
            const bool fresh = valid && (peers & lt) == 0 && !sl_lookup(X, H, key, (cmax + 31u) / 32u, at, loc);
            const uint32_t bal = __ballot_sync(0xffffffffu, fresh);
            const uint32_t pos = live + __popc(bal & lt);
            __syncwarp();
            if (fresh && pos < cmax) {
                const uint32_t t = top - 1u - pos;
                X.KT[t] = key;
                atomicOr(&X.BM[t >> 5], 1u << (t & 31u));  // (a degraded index is searched through the bitmap)
                sl_insert(X, H, t);
            }
            live = min(cmax, live + (uint32_t)__popc(bal));
            __syncwarp();
        }
    }
    sl_live_range(X, top - live, live, lane);
    uint32_t wnow = (top + 31u) / 32u;
    __syncwarp();

    unsigned long long my_prompt = 0, my_tok[NC];
    uint32_t my_hit[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) my_hit[c] = 0, my_tok[c] = 0;

    // the next step's records are gathered one step early, through request
    // indices read two steps early
    rec16 ahead = {0ull, 0u, 0u};
    if (p0 + lane < p1) {
        const uint32_t ix = idx[p0 + lane];
        (void)CR_DCHECK(ix < nrec, status);
        ahead = recs[min(ix, nrec - 1u)];  // (the bound guards the gather)
    }
    uint32_t ix_next = p0 + 32u + lane < p1 ? idx[p0 + 32u + lane] : 0u;
    for (uint32_t t0 = p0; t0 < p1; t0 += 32) {
        if (wnow == nw) {
            const uint32_t keep = min(live, cmax);
            sl_compact<NG>(X, live, keep, lane);
            live = keep;
            wnow = (live + 31u) / 32u;
        }
        const uint32_t cnt = (p1 - t0) < 32u ? (p1 - t0) : 32u;
        const bool valid = lane < cnt;
        const rec16 mine = ahead;
        if (t0 + 32u + lane < p1) {
            (void)CR_DCHECK(ix_next < nrec, status);
            ahead = recs[min(ix_next, nrec - 1u)];
        }
        ix_next = t0 + 64u + lane < p1 ? idx[t0 + 64u + lane] : 0u;
        if (valid) my_prompt += (unsigned long long)mine.P + mine.S;
        const uint32_t now = 32u * wnow + lane;
        X.KT[now] = mine.key;
        const uint32_t vm = cnt == 32 ? 0xffffffffu : (1u << cnt) - 1u;
        const uint32_t grp = __match_any_sync(0xffffffffu, mine.key) & vm;
        const uint32_t below = grp & lt, above = grp & gt;
        const bool first = valid && below == 0;
        const bool last = valid && above == 0;
        const key_hash H = sl_hash(X, mine.key);
        uint32_t s_old = 0, loc = kNone;
        const bool found = valid && sl_lookup(X, H, mine.key, wnow, s_old, loc);
        const bool res = first && found;  // first occurrence of a key of the window
        (void)CR_DCHECK(s_old < 32u * wnow + 32u, status);

        // recency position at the step's start: live times above the key's
        live_prefix<NG> LP;
        LP.load(X.BM, nw, lane);
        const uint32_t D = live - 1u - LP.below(s_old);
        // a first occurrence at old position D is pushed deeper by the step's earlier
        // first occurrences that were deeper or absent: between the absent ones
        // (jlo) and all of them (jhi).  Where that range straddles a capacity the
        // exact count decides the hit: those lanes (a few per step) are counted one
        // at a time against every lane; any count in the range decides the others.
        const uint32_t firstm = __ballot_sync(0xffffffffu, first);
        const uint32_t absm = __ballot_sync(0xffffffffu, first && !found);
        const uint32_t jlo = (uint32_t)__popc(absm & lt), jhi = (uint32_t)__popc(firstm & lt);
        bool amb = false;
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < (int)caps.n_caps && D + 1u + jlo <= caps.cap[c] && caps.cap[c] < D + 1u + jhi) amb = true;
        uint32_t jx = jhi;
        for (uint32_t am = __ballot_sync(0xffffffffu, res && amb); am; am &= am - 1u) {  // uniform
            const uint32_t a = (uint32_t)__ffs(am) - 1u;
            const uint32_t Da = __shfl_sync(0xffffffffu, D, a);
            const uint32_t deeper = __ballot_sync(0xffffffffu, first && (!found || D > Da));
            if (lane == a) jx = (uint32_t)__popc(deeper & lt);
        }
        uint32_t dep_rep = 1u;
        if (SMALL) {
            // a repeat of lane j: 1 + the distinct keys of lanes (j, i), i.e. the lanes
            // there whose key does not recur before i (next occurrence lane > i);
            // compared bit-sliced over the 6-bit next-occurrence lane; only needed
            // below capacity 32 (a repeat's depth is at most 31)
            const uint32_t next = above ? (uint32_t)__ffs(above) - 1u : 32u;
            uint32_t gN = 0, eN = 0xffffffffu;
#pragma unroll
            for (int bt = 5; bt >= 0; --bt) {
                const uint32_t BN = __ballot_sync(0xffffffffu, (next >> bt) & 1u);
                const uint32_t MN = 0u - ((lane >> bt) & 1u);
                gN |= eN & BN & ~MN;
                eN &= ~(BN ^ MN);
            }
            const uint32_t win = lt & ~((2u << (31u - (uint32_t)__clz(below | 1u))) - 1u);
            dep_rep = 1u + (uint32_t)__popc(gN & win);
        }
        const uint32_t depth = res ? D + 1u + jx : (valid && !first ? dep_rep : kNone);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (c < (int)caps.n_caps && depth <= caps.cap[c]) {
                my_hit[c] += 1;
                my_tok[c] += mine.P;
            }
        }

        // ---- state after the step: every key of the step takes its last access's time ----
        __syncwarp();  // (the bitmap and the index have been read)
        if (res) atomicAnd(&X.BM[s_old >> 5], ~(1u << (s_old & 31u)));
        if (last && loc != kNone) X.E[loc] = (uint16_t)(H.tag | now);
        const uint32_t lastm = __ballot_sync(0xffffffffu, last);
        __syncwarp();
        if (last && !found) sl_insert(X, H, now);
        if (lane == 0) X.BM[wnow] = lastm;
        live += (uint32_t)__popc(absm);
        ++wnow;
        __syncwarp();
    }

    // ---- counters -------------------------------------------------------------
    my_prompt = cr_warp_sum_u64(my_prompt);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        if (c < (int)caps.n_caps) {
            const unsigned long long h = cr_warp_sum_u64(my_hit[c]);
            const unsigned long long tk = cr_warp_sum_u64(my_tok[c]);
            if (lane == 0) {
                unsigned long long *C = ctr + (((unsigned long long)rep * caps.n_caps + c) * R + r) * CR_CTR_FIELDS;
                atomicAdd(&C[0], (unsigned long long)(p1 - p0));
                if (h) atomicAdd(&C[1], h);
                if (tk) atomicAdd(&C[2], tk);
                atomicAdd(&C[3], my_prompt);
                atomicAdd(&C[4], my_prompt - tk);
            }
        }
    }
    // ---- the stream's last chunk hands the state to the next call, most recent first
    if (p1 == e) {
        unsigned long long *kout = st.keys_out + (unsigned long long)s * cmax;
        const uint32_t keep = min(live, cmax);
        uint32_t above = live;  // live keys from word x on
        for (uint32_t x = 0; x < wnow; ++x) {
            const uint32_t bits = X.BM[x];
            const uint32_t q = above - 1u - (uint32_t)__popc(bits & lt);
            if (((bits >> lane) & 1u) && q < keep) kout[q] = X.KT[32u * x + lane];
            above -= (uint32_t)__popc(bits);
        }
        if (lane == 0) st.fill_out[s] = keep;
    }
}

// The items 0 .. *total - 1, or those that `list` names (k_replay_short's leftovers, whose
// number the host does not know: the grid then is what the GPU holds at once).
template <int NC, int NG, bool SMALL>
__global__ void __launch_bounds__(128, 5)
k_lru_stamp(const __grid_constant__ replay_caps caps, uint32_t cmax, uint32_t nw, uint32_t nb, uint32_t R,
             uint32_t ns, uint32_t CL, const uint32_t *__restrict__ start, const uint32_t *__restrict__ map, uint32_t items_max,
             const uint32_t *__restrict__ total, const uint32_t *__restrict__ list, const uint32_t *__restrict__ idx,
             const rec16 *__restrict__ recs, uint32_t nrec, const replay_state st, unsigned long long *__restrict__ ctr,
             uint32_t *status)
{
    const uint32_t wpb = blockDim.x >> 5, n = *total;
    for (uint32_t w = blockIdx.x * wpb + (threadIdx.x >> 5); w < n; w += gridDim.x * wpb) {
        lru_item<NC, NG, SMALL>(list ? list[w] : w, caps, cmax, nw, nb, R, ns, CL, start, map, items_max, idx, recs, nrec,
                                st, ctr, status);
        __syncwarp();
    }
}

// Words of the window: the cmax keys that a compaction leaves plus twelve steps before the
// next one.  More steps cost warps per SM, fewer cost compactions: at cmax 1024, 4 / 8 / 12 / 17 /
// 20 / 32 steps measured 1.80 / 1.73 / 1.73 / 1.83 / 1.80 / 2.02 ms, at cmax 128 223 / 217 / 215 /
// 215 / 219 / 254 us (the shapes above).
inline uint32_t window_words(uint32_t cmax)
{
    return (cmax + 31) / 32 + 12;
}

// The same for token capacities, whose lists may hold 1024 prefixes but, up to 65,536 tokens,
// seldom hold a hundred: four steps then cost few compactions and leave room for 12 warps per
// SM instead of 10 (24,576 tokens: 331 -> 261 us).
inline uint32_t token_words(uint32_t capmax)
{
    return capmax <= (1u << 16) ? CR_MAX_CAP / 32u + 4u : window_words(CR_MAX_CAP);
}

// Index buckets of a window: 1.5 entries per time, so that two full buckets are rare even
// when every request of the window has a key of its own.
inline uint32_t window_buckets(uint32_t nw) { return 12u * nw; }

// Registers and shared memory decide the warps per block (the most warps per SM; at most
// 32 blocks and 64 warps per SM).
uint32_t window_warps(size_t per_warp, uint32_t regs, uint32_t *per_sm)
{
    const uint32_t warps_regs = 65536u / (((regs * 32u + 255u) / 256u) * 256u);
    uint32_t best = 0, wpb = 1;
    for (uint32_t x = 4; x >= 1; --x) {
        uint32_t nb = (uint32_t)((size_t)(227 * 1024) / (per_warp * x + 1024));
        nb = nb < 32u ? nb : 32u;
        nb = nb < warps_regs / x ? nb : warps_regs / x;
        const uint32_t wps = nb * x < 64u ? nb * x : 64u;
        if (wps > best) {
            best = wps;
            wpb = x;
        }
    }
    *per_sm = best;
    return wpb;
}

// Blocks of a replay launch: one warp per item, or for leftovers what the GPU holds at once.
inline unsigned int item_grid(const cr_ctx *ctx, uint64_t items, uint32_t wpb, uint32_t per_sm, const uint32_t *rest)
{
    const uint64_t all = (items + wpb - 1) / wpb, held = (uint64_t)ctx->num_sms * (per_sm / wpb);
    return (unsigned int)(rest && held < all ? held : all);
}

template <int NC, int NG, bool SMALL>
int launch_stamp(cr_ctx *ctx, cr_replay *rp, const replay_caps &caps, uint32_t CL, const uint32_t *start,
                  const uint32_t *map, uint32_t items_max, const uint32_t *total, uint64_t m, const uint32_t *idx,
                  const rec16 *recs, uint64_t *d_ctr)
{
    const uint32_t cmax = rp->cmax, nw = window_words(cmax), nb = window_buckets(nw);
    cudaFuncAttributes fa;
    uint32_t regs = 64, per_sm = 0;
    if (cudaFuncGetAttributes(&fa, k_lru_stamp<NC, NG, SMALL>) == cudaSuccess && fa.numRegs > 0)
        regs = (uint32_t)fa.numRegs;
    else
        cudaGetLastError();
    const size_t per_warp = window_lru_bytes(nw, nb);
    const uint32_t wpb = window_warps(per_warp, regs, &per_sm);
    const size_t smem = per_warp * wpb;
    if (smem > kDefaultSmem)
        CR_CUDA(ctx, cudaFuncSetAttribute(k_lru_stamp<NC, NG, SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)smem));
    const uint32_t ns = rp->n_rep * rp->R;
    const uint64_t items = (uint64_t)ns + (m + CL - 1) / CL;  // upper bound on work items
    const int pr = cr_prof_begin(ctx, ctx->stream, CR_PROF_REPLAY);
    uint32_t *rest;
    CR_TRY(launch_short<false>(ctx, rp, caps, cmax, start, map, items_max, total, m, items, idx, recs, d_ctr, &rest));
    CR_LAUNCH(ctx, (k_lru_stamp<NC, NG, SMALL>), item_grid(ctx, items, wpb, per_sm, rest), wpb * 32, smem, caps, cmax, nw,
              nb, rp->R, ns, CL, start, map, items_max, rest ? rest : total, rest ? rest + 1 : nullptr, idx, recs,
              (uint32_t)(m / rp->n_rep), state_of(rp), (unsigned long long *)d_ctr, ctx->d_status);
    cr_prof_end(ctx, ctx->stream, pr);
    rp->cur ^= 1;
    return CR_OK;
}

template <int NC>
int launch_stamp_nc(cr_ctx *ctx, cr_replay *rp, const replay_caps &caps, uint32_t CL, const uint32_t *start,
                    const uint32_t *map, uint32_t items_max, const uint32_t *total, uint64_t m, const uint32_t *idx,
                 const rec16 *recs, uint64_t *d_ctr)
{
    uint32_t cmin = 0xffffffffu;
    for (uint32_t c = 0; c < caps.n_caps; ++c) cmin = caps.cap[c] < cmin ? caps.cap[c] : cmin;
    const bool small = cmin < 32;  // a repeat within a step can miss only below capacity 32
    if (window_words(rp->cmax) <= 32)
        return small ? launch_stamp<NC, 1, true>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr)
                     : launch_stamp<NC, 1, false>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr);
    return small ? launch_stamp<NC, 2, true>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr)
                 : launch_stamp<NC, 2, false>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr);
}

int launch_batch(cr_ctx *ctx, cr_replay *rp, const replay_caps &caps, uint32_t CL, const uint32_t *start,
                 const uint32_t *map, uint32_t items_max, const uint32_t *total, uint64_t m, const uint32_t *idx,
                 const rec16 *recs, uint64_t *d_ctr)
{
    if (caps.n_caps == 1) return launch_stamp_nc<1>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr);
    if (caps.n_caps <= 3) return launch_stamp_nc<3>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr);
    return launch_stamp_nc<CR_MAX_CAPS>(ctx, rp, caps, CL, start, map, items_max, total, m, idx, recs, d_ctr);
}

// ---- token-weighted variant ---------------------------------------------------
// Capacities count prefix tokens.  With one prefix length per key, the cache of capacity
// c holds the longest run of most recent prefixes whose tokens fit in c (evictions always
// take the least recent), so a request hits at c iff its key is among the kTokMax most
// recent and the tokens of the keys from the most recent through it are <= c.  The same
// window as above (times, bitmap of last accesses, index), with the tokens of every time
// and each word's live tokens: a step takes 32 requests of the stream, one per lane.
// The tokens above a key at the step's start are those of the words above its own (one
// warp scan) plus the live times above it in its word, added one by one; a word whose
// words above already exceed the largest capacity is not looked into.  The step's own
// requests count for request i when they are the last of their key before i and, for a
// first occurrence, their key was deeper than i's or absent (for a repeat, when they
// follow its previous occurrence): one pass over the 32 lanes.  Sums saturate at
// 2^32 - 1, above every capacity (<= 2^31).
//
// One request at a time over a list in recency order took 84 warp instructions per
// (request, replica) pair.  20 replicas x 166,667 requests over 30 destinations, 24,576
// tokens, partition included: 594 -> 265 us.  Bound, as above: the latency of a step's
// dependence chain at 12 warps per SM.
constexpr uint32_t kTokMax = CR_MAX_CAP;  // prefixes per list
// Below this largest capacity a step's sums of prefixes cut to it cannot pass 2^32.
constexpr uint32_t kTokNarrow = 1u << 26;

// Inclusive sum over the lanes from this one up.
__device__ __forceinline__ uint32_t warp_sat_suffix(uint32_t v, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(0xffffffffu, v, o);
        if (lane + (uint32_t)o < 32u) v = sat_add(v, y);
    }
    return v;
}

// Each word's live tokens from the bitmap and the times' tokens (words below `wend`;
// cleared above).
__device__ __forceinline__ void tk_word_sums(const window_lru &X, uint32_t wend, uint32_t lane)
{
    for (uint32_t w = wend + lane; w < X.nw; w += 32) X.SL[w] = X.SH[w] = 0;
    for (uint32_t w = 0; w < wend; ++w) {
        const uint32_t bits = X.BM[w];
        const uint32_t v = ((bits >> lane) & 1u) ? X.TK[32u * w + lane] : 0u;
        const uint32_t l = __reduce_add_sync(0xffffffffu, v & 0xffffu), h = __reduce_add_sync(0xffffffffu, v >> 16);
        if (lane == 0) {
            X.SL[w] = l;
            X.SH[w] = h;
        }
    }
    __syncwarp();
}

// The cached list from the most recent key down, each(position, time, tokens through it):
// the live keys of the words below wend whose tokens fit in capmax, at most kTokMax.
// Returns their count.
template <typename Each>
__device__ __forceinline__ uint32_t tk_list(const window_lru &X, uint32_t wend, uint32_t capmax, uint32_t lane, Each each)
{
    uint32_t n = 0, cum = 0;
    for (uint32_t w = wend; w-- > 0;) {
        const uint32_t bits = X.BM[w];
        if (!bits) continue;
        const bool live = (bits >> lane) & 1u;
        const uint32_t c = sat_add(cum, warp_sat_suffix(live ? X.TK[32u * w + lane] : 0u, lane));
        const uint32_t q = n + (uint32_t)__popc(bits & ~((2u << lane) - 1u));
        const bool fits = live && c <= capmax && q < kTokMax;
        const uint32_t fm = __ballot_sync(0xffffffffu, fits);
        if (fits) each(q, 32u * w + lane, c);
        n += (uint32_t)__popc(fm);
        if (fm != bits) break;  // everything older is further down the list
        cum = __shfl_sync(0xffffffffu, c, 0);
    }
    return n;
}

// One work item.
template <int NC>
__device__ __forceinline__ void token_item(uint32_t w, const replay_caps &caps, uint32_t capmax, uint32_t nw, uint32_t nb,
                                           uint32_t R, uint32_t ns, uint32_t CL, const uint32_t *__restrict__ start,
                                           const uint32_t *__restrict__ map, uint32_t items_max,
                                           const uint32_t *__restrict__ idx, const rec16 *__restrict__ recs,
                                           uint32_t nrec, const replay_state &st, unsigned long long *__restrict__ ctr,
                                           uint32_t *status)
{
    extern __shared__ uint4 smb[];
    const uint32_t lane = cr_lane(), warp = threadIdx.x >> 5;
    const window_lru X =
        window_lru_at(reinterpret_cast<unsigned char *>(smb) + window_lru_bytes(nw, nb, true) * warp, nw, nb);
    const uint32_t s = min(map[w], ns - 1u), ci = map[items_max + w];  // the item's stream and chunk
    const uint32_t b = start[s], e = start[s + 1];
    const uint32_t p0 = b + ci * CL;
    const uint32_t p1 = (e - p0) < CL ? e : p0 + CL;
    const uint32_t rep = s / R, r = s % R;
    const uint32_t fin = min(st.fill_in[s], kTokMax);
    const unsigned long long *kin = st.keys_in + (size_t)s * kTokMax;
    const uint32_t *cin = st.cum_in + (size_t)s * kTokMax;
    const uint32_t lt = (1u << lane) - 1u, gt = ~(lt | (1u << lane));
    if (b == e) {  // nothing routed here: carry the state over unchanged
        for (uint32_t j = lane; j < fin; j += 32) {
            st.keys_out[(size_t)s * kTokMax + j] = kin[j];
            st.cum_out[(size_t)s * kTokMax + j] = cin[j];
        }
        if (lane == 0) st.fill_out[s] = fin;
        return;
    }

    // ---- state at p0: the cached keys at the highest times below `top` ----------------
    uint32_t live = 0, top = kTokMax;
    sl_clear_index(X, lane);
    for (uint32_t x = lane; x < nw; x += 32) X.BM[x] = 0;
    __syncwarp();
    if (ci == 0) {
        top = live = fin;
        for (uint32_t q = lane; q < fin; q += 32) {
            const unsigned long long key = kin[q];
            const key_hash H = sl_hash(X, key);
            X.KT[top - 1u - q] = key;
            X.TK[top - 1u - q] = cin[q] - (q ? cin[q - 1u] : 0u);
            sl_insert(X, H, top - 1u - q);
        }
    } else {
        // the state at p0 is the longest run of most recent distinct prefixes that fits:
        // walk back over the stream, then over the carried-in list, keeping each key's most
        // recent access; the first distinct prefix that does not fit ends the run
        const uint32_t back = p0 - b, vtot = back + fin;
        uint32_t cum = 0;
        bool stop = false;
        auto index_at = [&](uint32_t v) { return v < back ? min(idx[p0 - 1u - v], nrec - 1u) : 0u; };
        auto load = [&](uint32_t v, uint32_t ix, unsigned long long &key, uint32_t &P) {
            key = 0;
            P = 0;
            if (v < back) {
                const rec16 x = recs[ix];
                key = x.key;
                P = x.P;
            } else if (v < vtot) {
                const uint32_t j = v - back;
                key = kin[j];
                P = cin[j] - (j ? cin[j - 1u] : 0u);
            }
        };
        unsigned long long kn;
        uint32_t Pn, ixn = index_at(lane + 32u);
        load(lane, index_at(lane), kn, Pn);
        for (uint32_t v0 = 0; v0 < vtot && live < kTokMax && !stop; v0 += 32) {
            const bool valid = v0 + lane < vtot;
            const unsigned long long key = kn;
            const uint32_t P = Pn;
            load(v0 + 32u + lane, ixn, kn, Pn);
            ixn = index_at(v0 + 64u + lane);
            const uint32_t vm = __ballot_sync(0xffffffffu, valid);
            const uint32_t peers = __match_any_sync(0xffffffffu, key) & vm;
            const key_hash H = sl_hash(X, key);
            uint32_t at, loc;
            const bool fresh = valid && (peers & lt) == 0 && !sl_lookup(X, H, key, (kTokMax + 31u) / 32u, at, loc);
            const uint32_t bal = __ballot_sync(0xffffffffu, fresh);
            const uint32_t pos = live + (uint32_t)__popc(bal & lt);
            uint32_t c = fresh ? P : 0u;  // tokens through this lane
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, c, o);
                if (lane >= (uint32_t)o) c = sat_add(c, y);
            }
            c = sat_add(c, cum);
            const uint32_t over = __ballot_sync(0xffffffffu, fresh && (c > capmax || pos >= kTokMax));
            const uint32_t take = over ? bal & ((1u << (__ffs(over) - 1)) - 1u) : bal;
            __syncwarp();
            if ((take >> lane) & 1u) {
                const uint32_t t = top - 1u - pos;
                X.KT[t] = key;
                X.TK[t] = P;
                atomicOr(&X.BM[t >> 5], 1u << (t & 31u));  // (a degraded index is searched through the bitmap)
                sl_insert(X, H, t);
            }
            live += (uint32_t)__popc(take);
            cum = __shfl_sync(0xffffffffu, c, 31);
            stop = over != 0;
            __syncwarp();
        }
    }
    sl_live_range(X, top - live, live, lane);
    uint32_t wnow = (top + 31u) / 32u;
    __syncwarp();
    tk_word_sums(X, wnow, lane);

    unsigned long long my_prompt = 0, my_tok[NC];
    uint32_t my_hit[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) my_hit[c] = 0, my_tok[c] = 0;

    const bool wide = capmax >= kTokNarrow;
    // records are gathered one step early, through request indices read two steps early
    rec16 ahead = {0ull, 0u, 0u};
    if (p0 + lane < p1) ahead = recs[min(idx[p0 + lane], nrec - 1u)];  // (the bound guards the gather)
    uint32_t ix_next = p0 + 32u + lane < p1 ? idx[p0 + 32u + lane] : 0u;
    for (uint32_t t0 = p0; t0 < p1; t0 += 32) {
        if (wnow == nw) {
            const uint32_t keep = tk_list(X, wnow, capmax, lane, [](uint32_t, uint32_t, uint32_t) {});
            sl_compact<2, true>(X, live, keep, lane);
            live = keep;
            wnow = (live + 31u) / 32u;
            tk_word_sums(X, wnow, lane);
        }
        const uint32_t cnt = (p1 - t0) < 32u ? (p1 - t0) : 32u;
        const bool valid = lane < cnt;
        const rec16 mine = ahead;
        if (t0 + 32u + lane < p1) {
            (void)CR_DCHECK(ix_next < nrec, status);
            ahead = recs[min(ix_next, nrec - 1u)];
        }
        ix_next = t0 + 64u + lane < p1 ? idx[t0 + 64u + lane] : 0u;
        if (valid) my_prompt += (unsigned long long)mine.P + mine.S;
        const uint32_t now = 32u * wnow + lane;
        X.KT[now] = mine.key;
        X.TK[now] = mine.P;
        const uint32_t vm = cnt == 32 ? 0xffffffffu : (1u << cnt) - 1u;
        const uint32_t grp = __match_any_sync(0xffffffffu, mine.key) & vm;
        const uint32_t below = grp & lt, above = grp & gt;
        const bool first = valid && below == 0;
        const bool last = valid && above == 0;
        const key_hash H = sl_hash(X, mine.key);
        uint32_t s_old = 0, loc = kNone;
        const bool found = valid && sl_lookup(X, H, mine.key, wnow, s_old, loc);
        const bool res = first && found;

        // tokens of the words above each word (group g: words 32 g .. 32 g + 31)
        uint32_t ab[2], sum1 = 0;
#pragma unroll
        for (int g = 1; g >= 0; --g) {
            const uint32_t wi = 32u * g + lane;
            const unsigned long long v = wi < nw ? X.SL[wi] + ((unsigned long long)X.SH[wi] << 16) : 0ull;
            const uint32_t incl = warp_sat_suffix(v > 0xffffffffull ? 0xffffffffu : (uint32_t)v, lane);
            const uint32_t y = __shfl_down_sync(0xffffffffu, incl, 1);
            ab[g] = sat_add(lane < 31u ? y : 0u, sum1);
            sum1 = __shfl_sync(0xffffffffu, incl, 0);
        }
        const uint32_t a0 = __shfl_sync(0xffffffffu, ab[0], (s_old >> 5) & 31u),
                       a1 = __shfl_sync(0xffffffffu, ab[1], (s_old >> 5) & 31u);
        uint32_t cum = s_old < 1024u ? a0 : a1;  // first occurrence: tokens through its key, at the step's start
        uint32_t own = 0;                        // its key's tokens at its last access
        if (res) {
            own = X.TK[s_old];
            cum = sat_add(cum, own);
            uint32_t bits = X.BM[s_old >> 5] & ~((2u << (s_old & 31u)) - 1u);
            for (; bits && cum <= capmax; bits &= bits - 1u)
                cum = sat_add(cum, X.TK[(s_old & ~31u) + (uint32_t)__ffs(bits) - 1u]);
        }
        // its position, where the list is long enough for the limit on prefixes to matter
        uint32_t pos = 0;
        if (live + 32u > kTokMax) {  // uniform
            live_prefix<2> LP;
            LP.load(X.BM, nw, lane);
            const uint32_t bl = LP.below(s_old);
            pos = live - 1u - bl;
        }
        // a repeat: the step's requests since the previous occurrence
        const uint32_t prev = below ? 31u - (uint32_t)__clz(below) : 0u;
        const uint32_t P_prev = __shfl_sync(0xffffffffu, mine.P, prev);
        if (valid && !first) {
            own = P_prev;
            cum = P_prev;
            pos = 0;
        }
        // request j counts for request i when it is the last of its key before i (its next
        // occurrence after lane i: M, compared bit-sliced) and its key was deeper or absent
        // (order below i's) or, for a repeat i, j follows the previous occurrence
        const uint32_t order = found ? s_old + 1u : 0u;
        X.OP[lane] = make_uint2(order, wide ? mine.P : min(mine.P, kTokNarrow));
        const bool open = valid && (first ? found : true) && cum <= capmax;  // not decided yet
        __syncwarp();
        if (__any_sync(0xffffffffu, open)) {
            const uint32_t next = above ? (uint32_t)__ffs(above) - 1u : 32u;
            uint32_t gN = 0, eN = 0xffffffffu;
#pragma unroll
            for (int bt = 5; bt >= 0; --bt) {
                const uint32_t BN = __ballot_sync(0xffffffffu, (next >> bt) & 1u);
                const uint32_t MN = 0u - ((lane >> bt) & 1u);
                gN |= eN & BN & ~MN;
                eN &= ~(BN ^ MN);
            }
            const uint32_t M = gN & lt & (first ? 0xffffffffu : ~((2u << prev) - 1u));
            const uint32_t my_order = first ? order : 0xffffffffu;
            uint32_t n_in = 0;
            if (!wide) {
#pragma unroll
                for (uint32_t j = 0; j < 31; ++j) {
                    const uint2 o = X.OP[j];
                    const bool counts = ((M >> j) & 1u) && o.x < my_order;
                    if (counts) cum += o.y;
                    if (counts) ++n_in;
                }
            } else {
                for (uint32_t j = 0; j < 31; ++j) {
                    const uint2 o = X.OP[j];
                    const bool counts = ((M >> j) & 1u) && o.x < my_order;
                    cum = sat_add(cum, counts ? o.y : 0u);
                    n_in += counts ? 1u : 0u;
                }
            }
            pos += n_in;
        }
        const bool listed = open && cum <= capmax && pos < kTokMax;
        if (listed && own != mine.P) atomicOr(status, CR_FLAG_BADSIZE);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (c < (int)caps.n_caps && listed && cum <= caps.cap[c]) {
                my_hit[c] += 1;
                my_tok[c] += mine.P;
            }
        }

        // ---- state after the step: every key of the step takes its last access's time ----
        const uint32_t absm = __ballot_sync(0xffffffffu, first && !found);
        const uint32_t old = res ? X.TK[s_old] : 0u;
        __syncwarp();  // (the bitmap, the sums and the index have been read)
        if (res) {
            atomicAnd(&X.BM[s_old >> 5], ~(1u << (s_old & 31u)));
            atomicSub(&X.SL[s_old >> 5], old & 0xffffu);
            atomicSub(&X.SH[s_old >> 5], old >> 16);
        }
        if (last && loc != kNone) X.E[loc] = (uint16_t)(H.tag | now);
        const uint32_t lastm = __ballot_sync(0xffffffffu, last);
        const uint32_t sl = __reduce_add_sync(0xffffffffu, last ? mine.P & 0xffffu : 0u),
                       sh = __reduce_add_sync(0xffffffffu, last ? mine.P >> 16 : 0u);
        __syncwarp();
        if (last && !found) sl_insert(X, H, now);
        if (lane == 0) {
            X.BM[wnow] = lastm;
            X.SL[wnow] = sl;
            X.SH[wnow] = sh;
        }
        live += (uint32_t)__popc(absm);
        ++wnow;
        __syncwarp();
    }

    // ---- counters -------------------------------------------------------------
    my_prompt = cr_warp_sum_u64(my_prompt);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        if (c < (int)caps.n_caps) {
            const unsigned long long h = cr_warp_sum_u64(my_hit[c]);
            const unsigned long long tk = cr_warp_sum_u64(my_tok[c]);
            if (lane == 0) {
                unsigned long long *C = ctr + (((unsigned long long)rep * caps.n_caps + c) * R + r) * CR_CTR_FIELDS;
                atomicAdd(&C[0], (unsigned long long)(p1 - p0));
                if (h) atomicAdd(&C[1], h);
                if (tk) atomicAdd(&C[2], tk);
                atomicAdd(&C[3], my_prompt);
                atomicAdd(&C[4], my_prompt - tk);
            }
        }
    }
    if (p1 == e) {  // the stream's last chunk hands the state to the next call
        unsigned long long *kout = st.keys_out + (size_t)s * kTokMax;
        uint32_t *cout = st.cum_out + (size_t)s * kTokMax;
        const uint32_t n = tk_list(X, wnow, capmax, lane, [&](uint32_t q, uint32_t t, uint32_t c) {
            kout[q] = X.KT[t];
            cout[q] = c;
        });
        if (lane == 0) st.fill_out[s] = n;
    }
}

template <int NC>
__global__ void __launch_bounds__(128, 4)
k_lru_tokens(const __grid_constant__ replay_caps caps, uint32_t capmax, uint32_t nw, uint32_t nb, uint32_t R,
             uint32_t ns, uint32_t CL, const uint32_t *__restrict__ start, const uint32_t *__restrict__ map,
             uint32_t items_max, const uint32_t *__restrict__ total, const uint32_t *__restrict__ list,
             const uint32_t *__restrict__ idx, const rec16 *__restrict__ recs, uint32_t nrec, const replay_state st,
             unsigned long long *__restrict__ ctr, uint32_t *status)
{
    const uint32_t wpb = blockDim.x >> 5, n = *total;
    for (uint32_t w = blockIdx.x * wpb + (threadIdx.x >> 5); w < n; w += gridDim.x * wpb) {
        token_item<NC>(list ? list[w] : w, caps, capmax, nw, nb, R, ns, CL, start, map, items_max, idx, recs, nrec, st, ctr,
                       status);
        __syncwarp();
    }
}

template <int NC>
int launch_tokens(cr_ctx *ctx, cr_replay *rp, const replay_caps &caps, uint32_t CL, const uint32_t *start,
                  const uint32_t *map, uint32_t items_max, const uint32_t *total, uint64_t m, const uint32_t *idx,
                  const rec16 *recs, uint64_t *d_ctr)
{
    uint32_t capmax = 0;
    for (uint32_t c = 0; c < caps.n_caps; ++c) capmax = caps.cap[c] > capmax ? caps.cap[c] : capmax;
    const uint32_t nw = token_words(capmax), nb = window_buckets(nw);
    cudaFuncAttributes fa;
    uint32_t regs = 96, per_sm = 0;
    if (cudaFuncGetAttributes(&fa, k_lru_tokens<NC>) == cudaSuccess && fa.numRegs > 0)
        regs = (uint32_t)fa.numRegs;
    else
        cudaGetLastError();
    const size_t per_warp = window_lru_bytes(nw, nb, true);
    const uint32_t wpb = window_warps(per_warp, regs, &per_sm);
    const size_t smem = per_warp * wpb;
    if (smem > kDefaultSmem)
        CR_CUDA(ctx, cudaFuncSetAttribute(k_lru_tokens<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const uint32_t ns = rp->n_rep * rp->R;
    const uint64_t items = (uint64_t)ns + (m + CL - 1) / CL;  // upper bound on work items
    const int pt = cr_prof_begin(ctx, ctx->stream, CR_PROF_REPLAY);
    uint32_t *rest;
    CR_TRY(launch_short<true>(ctx, rp, caps, capmax, start, map, items_max, total, m, items, idx, recs, d_ctr, &rest));
    CR_LAUNCH(ctx, (k_lru_tokens<NC>), item_grid(ctx, items, wpb, per_sm, rest), wpb * 32, smem, caps, capmax, nw, nb, rp->R,
              ns, CL, start, map, items_max, rest ? rest : total, rest ? rest + 1 : nullptr, idx, recs,
              (uint32_t)(m / rp->n_rep), state_of(rp), (unsigned long long *)d_ctr, ctx->d_status);
    cr_prof_end(ctx, ctx->stream, pt);
    rp->cur ^= 1;
    return CR_OK;
}

}  // namespace

extern "C" int cr_replay_create(cr_ctx *ctx, uint32_t n_rep, uint32_t R, const uint32_t *caps, uint32_t n_caps,
                                cr_replay **out)
{
    if (!ctx || !out || !caps) return CR_EINVAL;
    *out = nullptr;
    if (n_rep == 0 || n_rep > CR_MAX_REPLICAS) return cr_fail(ctx, CR_EINVAL, "replay: n_rep=%u", n_rep);
    if (R == 0 || R > CR_MAX_R) return cr_fail(ctx, CR_EINVAL, "replay: R=%u", R);
    if (n_caps == 0 || n_caps > CR_MAX_CAPS) return cr_fail(ctx, CR_EINVAL, "replay: n_caps=%u", n_caps);
    uint32_t cmax = 0;
    for (uint32_t c = 0; c < n_caps; ++c) {
        if (caps[c] == 0 || caps[c] > CR_MAX_CAP) return cr_fail(ctx, CR_EINVAL, "replay: cap %u", caps[c]);
        cmax = caps[c] > cmax ? caps[c] : cmax;
    }
    if ((uint64_t)n_rep * R >= (1ull << 31)) return cr_fail(ctx, CR_EINVAL, "replay: too many streams");
    cr_replay *rp = (cr_replay *)calloc(1, sizeof(cr_replay));
    if (!rp) return cr_fail(ctx, CR_ENOMEM, "replay: host allocation failed");
    rp->n_rep = n_rep;
    rp->R = R;
    rp->n_caps = n_caps;
    rp->cmax = cmax;
    memcpy(rp->caps, caps, n_caps * sizeof(uint32_t));
    rp->n_streams = (uint64_t)n_rep * R;
    for (int b = 0; b < 2; ++b) {
        if (cudaMalloc(&rp->d_keys[b], rp->n_streams * cmax * sizeof(unsigned long long)) != cudaSuccess ||
            cudaMalloc(&rp->d_fill[b], rp->n_streams * sizeof(uint32_t)) != cudaSuccess) {
            cudaGetLastError();
            for (int x = 0; x < 2; ++x) {
                if (rp->d_keys[x]) cudaFree(rp->d_keys[x]);
                if (rp->d_fill[x]) cudaFree(rp->d_fill[x]);
            }
            free(rp);
            return cr_fail(ctx, CR_ENOMEM, "replay: cannot allocate state");
        }
    }
    *out = rp;
    return cr_replay_reset(ctx, rp);
}

extern "C" int cr_replay_create_tokens(cr_ctx *ctx, uint32_t n_rep, uint32_t R, const uint32_t *token_caps,
                                       uint32_t n_caps, cr_replay **out)
{
    if (!ctx || !out || !token_caps) return CR_EINVAL;
    *out = nullptr;
    if (n_rep == 0 || n_rep > CR_MAX_REPLICAS) return cr_fail(ctx, CR_EINVAL, "replay: n_rep=%u", n_rep);
    if (R == 0 || R > CR_MAX_R) return cr_fail(ctx, CR_EINVAL, "replay: R=%u", R);
    if (n_caps == 0 || n_caps > CR_MAX_CAPS) return cr_fail(ctx, CR_EINVAL, "replay: n_caps=%u", n_caps);
    for (uint32_t c = 0; c < n_caps; ++c)
        if (token_caps[c] == 0 || token_caps[c] > (1u << 31))
            return cr_fail(ctx, CR_EINVAL, "replay: token capacity %u outside 1..2^31", token_caps[c]);
    if ((uint64_t)n_rep * R >= (1ull << 31)) return cr_fail(ctx, CR_EINVAL, "replay: too many streams");
    cr_replay *rp = (cr_replay *)calloc(1, sizeof(cr_replay));
    if (!rp) return cr_fail(ctx, CR_ENOMEM, "replay: host allocation failed");
    rp->n_rep = n_rep;
    rp->R = R;
    rp->n_caps = n_caps;
    rp->cmax = kTokMax;
    rp->tokens = 1;
    memcpy(rp->caps, token_caps, n_caps * sizeof(uint32_t));
    rp->n_streams = (uint64_t)n_rep * R;
    for (int x = 0; x < 2; ++x) {  // double-buffered: chunks of a stream read the old state
        if (cudaMalloc(&rp->d_keys[x], rp->n_streams * kTokMax * sizeof(unsigned long long)) != cudaSuccess ||
            cudaMalloc(&rp->d_size[x], rp->n_streams * kTokMax * sizeof(uint32_t)) != cudaSuccess ||
            cudaMalloc(&rp->d_fill[x], rp->n_streams * sizeof(uint32_t)) != cudaSuccess) {
            cudaGetLastError();
            cr_replay_destroy(ctx, rp);
            return cr_fail(ctx, CR_ENOMEM, "replay: cannot allocate state");
        }
    }
    *out = rp;
    return cr_replay_reset(ctx, rp);
}

extern "C" int cr_replay_reset(cr_ctx *ctx, cr_replay *rp)
{
    if (!ctx || !rp) return CR_EINVAL;
    for (int b = 0; b < 2; ++b)
        if (rp->d_fill[b])
            CR_CUDA(ctx, cudaMemsetAsync(rp->d_fill[b], 0, rp->n_streams * sizeof(uint32_t), ctx->stream));
    return CR_OK;
}

extern "C" int cr_replay_destroy(cr_ctx *ctx, cr_replay *rp)
{
    if (!rp) return CR_OK;
    if (ctx) cudaStreamSynchronize(ctx->stream);
    for (int b = 0; b < 2; ++b) {
        if (rp->d_keys[b]) cudaFree(rp->d_keys[b]);
        if (rp->d_fill[b]) cudaFree(rp->d_fill[b]);
    }
    for (int b = 0; b < 2; ++b)
        if (rp->d_size[b]) cudaFree(rp->d_size[b]);
    free(rp);
    return CR_OK;
}

// ---- a8 / a9 as separate calls --------------------------------------------------
// A partitioned input: every (replica, destination) stream's request indices in
// arrival order, the packed records, the streams' starts and their chunking.
struct cr_replay_input {
    uint32_t n_rep, R, tokens;   // shape of the replay it was built for (n_rep 0: no partition)
    uint32_t CL;                 // chunk length of the work items
    uint64_t n, m;               // requests, (request, replica) pairs
    uint32_t ns, ntiles;
    uint32_t *d_idx;             // [m]
    rec16 *d_recs;               // [n]
    uint32_t *d_cnt;             // [ns * ntiles + 2]: tile counts -> offsets, and their total
    uint32_t *d_start;           // [ns + 1]
    uint32_t *d_coff;            // [ns + 4]: work-item offsets, their total, k_item_map's counters; then its map
    uint32_t items_max;          // upper bound on the work items; the map is [2 items_max]
    uint64_t cap_m, cap_n, cap_cnt, cap_ns, cap_coff;
};

static int grow_u32(cr_ctx *ctx, uint32_t **p, uint64_t *cap, uint64_t need)
{
    if (*cap >= need && *p) return CR_OK;
    if (*p) {
        // the old buffer may still be read by work on any stream (a simulation ordered after
        // the partition by an event): wait for the whole device before freeing it
        CR_CUDA(ctx, cudaDeviceSynchronize());
        cudaFree(*p);
        *p = nullptr;
    }
    const uint64_t c = need + need / 4 + 64;
    if (cudaMalloc((void **)p, c * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        *cap = 0;
        return cr_fail(ctx, CR_ENOMEM, "replay input: cannot allocate %llu words", (unsigned long long)c);
    }
    *cap = c;
    return CR_OK;
}

extern "C" int cr_replay_input_create(cr_ctx *ctx, cr_replay_input **out)
{
    if (!ctx || !out) return CR_EINVAL;
    *out = (cr_replay_input *)calloc(1, sizeof(cr_replay_input));
    return *out ? CR_OK : cr_fail(ctx, CR_ENOMEM, "replay input: host allocation failed");
}

extern "C" int cr_replay_input_destroy(cr_ctx *ctx, cr_replay_input *in)
{
    if (!in) return CR_OK;
    if (ctx) cudaStreamSynchronize(ctx->stream);
    cudaFree(in->d_idx);
    cudaFree(in->d_recs);
    cudaFree(in->d_cnt);
    cudaFree(in->d_start);
    cudaFree(in->d_coff);
    free(in);
    return CR_OK;
}

extern "C" int cr_replay_partition(cr_ctx *ctx, const cr_replay *rp, const uint64_t *d_key, const uint32_t *d_plen,
                                   const uint32_t *d_slen, const uint16_t *d_dest, uint64_t n, cr_replay_input *in)
{
    if (!ctx || !rp || !in) return CR_EINVAL;
    cr_nvtx_range nv("cr_replay_partition");
    const uint64_t m = n * rp->n_rep;
    if (n >= (1ull << 31) || m >= 0xffffffffull)
        return cr_fail(ctx, CR_EINVAL, "cr_replay_partition: n * n_rep must be < 2^32 - 1");
    if (n && (!d_key || !d_plen || !d_slen || !d_dest))
        return cr_fail(ctx, CR_EINVAL, "cr_replay_partition: NULL pointer");
    const uint32_t R = rp->R, ns = (uint32_t)rp->n_streams;
    const uint32_t ntiles = (uint32_t)((n + kPartTile - 1) / kPartTile);
    const uint64_t ncnt = (uint64_t)ns * ntiles;
    if (ncnt >= 0xffffffffull) return cr_fail(ctx, CR_EINVAL, "cr_replay_partition: too many (stream, tile) pairs");
    in->n_rep = 0;  // holds nothing until everything below is enqueued: simulate refuses it
    in->R = R;
    in->tokens = (uint32_t)rp->tokens;
    in->n = n;
    in->m = m;
    in->ns = ns;
    in->ntiles = ntiles;
    if (rp->tokens) {
        uint32_t capmax = 0;
        for (uint32_t c = 0; c < rp->n_caps; ++c) capmax = rp->caps[c] > capmax ? rp->caps[c] : capmax;
        // about two chunks per warp that the GPU holds at once (20 replicas x 166,667 requests:
        // 512 / 768 / 1024 / 1536 requests measured 282 / 289 / 261 / 340 us), but long against
        // the rebuild walk, which reaches back until the largest capacity fills
        const uint32_t nw = token_words(capmax);
        uint32_t per_sm = 1;
        window_warps(window_lru_bytes(nw, window_buckets(nw), true), 96, &per_sm);
        const uint64_t fill = (m / (2ull * ctx->num_sms * per_sm) + 255u) & ~255ull;
        const uint32_t lo = capmax <= (1u << 16) ? 512u : (capmax <= (1u << 17) ? 1024u : 4096u);
        in->CL = fill < lo ? lo : (fill > 16u * lo ? 16u * lo : (uint32_t)fill);
    } else {
        // about one chunk per warp that the GPU holds at once, but long enough that
        // rebuilding an LRU state of cmax entries is amortised, and not so long that one hot
        // stream outlasts the rest.  Against 16 cmax whatever the call's size: 30 replicas x
        // 133,333 over 64 destinations at cmax 128 230 -> 214 us; two streams of 100,000 at cmax
        // 1024 1.7-5.3 -> 0.36 ms; 160 streams of 62,500 6.2 -> 0.91 ms
        const uint32_t nw = window_words(rp->cmax);
        uint32_t per_sm = 1;
        window_warps(window_lru_bytes(nw, window_buckets(nw)), 96, &per_sm);
        const uint64_t fill = m / ((uint64_t)ctx->num_sms * per_sm);
        const uint32_t lo = rp->cmax * 4u > 256u ? rp->cmax * 4u : 256u, hi = rp->cmax * 32u > 256u ? rp->cmax * 32u : 256u;
        in->CL = fill < lo ? lo : (fill > hi ? hi : (uint32_t)fill);
    }
    if (n == 0) {
        in->n_rep = rp->n_rep;
        return CR_OK;
    }
    CR_TRY(grow_u32(ctx, &in->d_idx, &in->cap_m, m));
    CR_TRY(grow_u32(ctx, (uint32_t **)&in->d_recs, &in->cap_n, n * (sizeof(rec16) / sizeof(uint32_t))));
    CR_TRY(grow_u32(ctx, &in->d_cnt, &in->cap_cnt, ncnt + 2));
    CR_TRY(grow_u32(ctx, &in->d_start, &in->cap_ns, (uint64_t)ns + 2));
    const uint64_t items_max = (uint64_t)ns + m / in->CL + 1;  // every stream's chunks, at least one each
    in->items_max = (uint32_t)items_max;
    CR_TRY(grow_u32(ctx, &in->d_coff, &in->cap_coff, (uint64_t)ns + 4 + 2 * items_max));
    uint32_t *cnt = in->d_cnt, *nrec = cnt + ncnt, *start = in->d_start;
    uint32_t *coff = in->d_coff, *total = coff + ns, *next = coff + ns + 1;
    const uint32_t longer = (uint32_t)(2u * (n / R + 1u));  // twice the mean stream
    const unsigned int gcap = (unsigned int)ctx->num_sms * 8u;
    const size_t csmem = (size_t)R * sizeof(uint32_t), ssmem = part_scatter_smem(R);
    if (csmem > kDefaultSmem)
        CR_CUDA(ctx, cudaFuncSetAttribute(k_part_count, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csmem));
    auto *scatter = R >= kPartSparse ? k_part_scatter<false> : k_part_scatter<true>;
    if (ssmem > kDefaultSmem)
        CR_CUDA(ctx, cudaFuncSetAttribute(scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssmem));
    const int pp = cr_prof_begin(ctx, ctx->stream, CR_PROF_PARTITION);
    CR_LAUNCH(ctx, k_part_count, dim3(ntiles, rp->n_rep + 1), kPartBlock, csmem, d_dest, (unsigned long long)n, R, ntiles,
              rp->n_rep, cnt, (const unsigned long long *)d_key, d_plen, d_slen, in->d_recs, ctx->d_status);
    CR_TRY(cr_scan_u32(ctx, cnt, cnt, ncnt, nrec));
    CR_LAUNCH(ctx, scatter, dim3(ntiles, rp->n_rep), kPartBlock, ssmem, d_dest, (unsigned long long)n, R, ntiles,
              (const uint32_t *)cnt, in->d_idx, (unsigned long long)m);
    if (ns <= kItemsCta) {
        const size_t ismem = ((size_t)ns + 1) * sizeof(uint32_t);
        if (ismem > kDefaultSmem)
            CR_CUDA(ctx, cudaFuncSetAttribute(k_items_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ismem));
        CR_LAUNCH(ctx, k_items_cta, 1, 1024, ismem, (const uint32_t *)cnt, ns, ntiles, (const uint32_t *)nrec, start, in->CL,
                  longer, total, coff + ns + 4, items_max);
    } else {
        CR_LAUNCH(ctx, k_part_starts, cr_blocks((uint64_t)ns + 1, 256, gcap), 256, 0, (const uint32_t *)cnt, ns, ntiles,
                  (const uint32_t *)nrec, start, next);
        CR_LAUNCH(ctx, k_chunk_counts, cr_blocks(ns, 256, gcap), 256, 0, (const uint32_t *)start, ns, in->CL, longer,
                  coff, next);
        CR_TRY(cr_scan_u32(ctx, coff, coff, ns, total));
        CR_LAUNCH(ctx, k_item_map, cr_blocks(ns, 256, gcap), 256, 0, (const uint32_t *)start, (const uint32_t *)coff, ns,
                  in->CL, longer, next, coff + ns + 4, items_max);
    }
    cr_prof_end(ctx, ctx->stream, pp);
    in->n_rep = rp->n_rep;
    return CR_OK;
}

extern "C" int cr_replay_simulate(cr_ctx *ctx, cr_replay *rp, const cr_replay_input *in, uint64_t *d_ctr)
{
    if (!ctx || !rp || !in) return CR_EINVAL;
    cr_nvtx_range nv("cr_replay_simulate");
    if (in->n_rep != rp->n_rep || in->R != rp->R || in->tokens != (uint32_t)rp->tokens)
        return cr_fail(ctx, CR_EINVAL, "cr_replay_simulate: the input was partitioned for another replay shape");
    if (in->n == 0) return CR_OK;
    if (!d_ctr) return cr_fail(ctx, CR_EINVAL, "cr_replay_simulate: d_ctr is NULL");
    const uint32_t ns = in->ns;
    const uint64_t m = in->m;
    const uint32_t *start = in->d_start, *map = in->d_coff + ns + 4, *total = in->d_coff + ns;
    replay_caps caps;
    caps.n_caps = rp->n_caps;
    for (uint32_t c = 0; c < CR_MAX_CAPS; ++c) caps.cap[c] = c < rp->n_caps ? rp->caps[c] : 0;
    if (rp->tokens) {
        const uint32_t *idx = in->d_idx;
        if (caps.n_caps == 1)
            return launch_tokens<1>(ctx, rp, caps, in->CL, start, map, in->items_max, total, m, idx, in->d_recs, d_ctr);
        if (caps.n_caps <= 3)
            return launch_tokens<3>(ctx, rp, caps, in->CL, start, map, in->items_max, total, m, idx, in->d_recs, d_ctr);
        return launch_tokens<CR_MAX_CAPS>(ctx, rp, caps, in->CL, start, map, in->items_max, total, m, idx, in->d_recs,
                                          d_ctr);
    }
    return launch_batch(ctx, rp, caps, in->CL, start, map, in->items_max, total, m, in->d_idx, in->d_recs, d_ctr);
}

extern "C" int cr_shadow_replay(cr_ctx *ctx, cr_replay *rp, const uint64_t *d_key, const uint32_t *d_plen,
                                const uint32_t *d_slen, const uint16_t *d_dest, uint64_t n, uint64_t *d_ctr)
{
    if (!ctx || !rp) return CR_EINVAL;
    cr_nvtx_range nv("cr_shadow_replay");
    if (n == 0) return CR_OK;
    if (!d_key || !d_plen || !d_slen || !d_dest || !d_ctr)
        return cr_fail(ctx, CR_EINVAL, "cr_shadow_replay: NULL pointer");
    if (!ctx->replay_in) CR_TRY(cr_replay_input_create(ctx, &ctx->replay_in));
    CR_TRY(cr_replay_partition(ctx, rp, d_key, d_plen, d_slen, d_dest, n, ctx->replay_in));
    return cr_replay_simulate(ctx, rp, ctx->replay_in, d_ctr);
}

extern "C" int cr_replay_export_state(cr_ctx *ctx, const cr_replay *rp, uint32_t rep, uint32_t r,
                                      uint64_t *keys_out, uint32_t *fill_out)
{
    if (!ctx || !rp || !keys_out || !fill_out) return CR_EINVAL;
    if (rep >= rp->n_rep || r >= rp->R) return cr_fail(ctx, CR_EINVAL, "export_state: bad stream");
    const uint64_t s = (uint64_t)rep * rp->R + r;
    uint32_t fill = 0;
    CR_CUDA(ctx, cudaMemcpyAsync(&fill, rp->d_fill[rp->cur] + s, sizeof(uint32_t), cudaMemcpyDeviceToHost,
                                 ctx->stream));
    CR_TRY(cr_sync(ctx));
    if (fill)
        CR_CUDA(ctx, cudaMemcpyAsync(keys_out, rp->d_keys[rp->cur] + s * rp->cmax, fill * sizeof(uint64_t),
                                     cudaMemcpyDeviceToHost, ctx->stream));
    *fill_out = fill;
    return cr_sync(ctx);
}

extern "C" int cr_replay_import_state(cr_ctx *ctx, cr_replay *rp, uint32_t rep, uint32_t r, const uint64_t *keys,
                                      uint32_t fill)
{
    if (!ctx || !rp || (fill && !keys)) return CR_EINVAL;
    if (rp->tokens) return cr_fail(ctx, CR_EINVAL, "import_state: token-weighted replays keep prefix sizes too");
    if (rep >= rp->n_rep || r >= rp->R) return cr_fail(ctx, CR_EINVAL, "import_state: bad stream");
    if (fill > rp->cmax) return cr_fail(ctx, CR_EINVAL, "import_state: %u keys exceed capacity %u", fill, rp->cmax);
    // the keys of one LRU are distinct
    uint64_t *tmp = (uint64_t *)malloc((size_t)(fill ? fill : 1) * sizeof(uint64_t));
    if (!tmp) return cr_fail(ctx, CR_ENOMEM, "import_state: host allocation failed");
    memcpy(tmp, keys, (size_t)fill * sizeof(uint64_t));
    qsort(tmp, fill, sizeof(uint64_t), [](const void *a, const void *b) {
        const uint64_t x = *(const uint64_t *)a, y = *(const uint64_t *)b;
        return x < y ? -1 : (x > y ? 1 : 0);
    });
    int dup = 0;
    for (uint32_t i = 1; i < fill; ++i) dup |= tmp[i] == tmp[i - 1];
    free(tmp);
    if (dup) return cr_fail(ctx, CR_EINVAL, "import_state: a key is listed twice");
    const uint64_t s = (uint64_t)rep * rp->R + r;
    if (fill)
        CR_CUDA(ctx, cudaMemcpyAsync(rp->d_keys[rp->cur] + s * rp->cmax, keys, (size_t)fill * sizeof(uint64_t),
                                     cudaMemcpyHostToDevice, ctx->stream));
    CR_CUDA(ctx, cudaMemcpyAsync(rp->d_fill[rp->cur] + s, &fill, sizeof(uint32_t), cudaMemcpyHostToDevice,
                                 ctx->stream));
    return cr_sync(ctx);  // blocking: the host arrays may be reused when the call returns
}
