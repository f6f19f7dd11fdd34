// a7: batched dispatch (cr_route_batch) and the ring of the bounded-load
// comparison policy (cr_ring_*).
//
// Two passes.  k_route_cand runs over every (replica, request) pair at once and
// does all the work that does not depend on the live load: the table probe,
// the Philox draws of power-of-two choices, the ring position of consistent
// hashing with bounded loads, round robin and the jump hash.  Round-robin and
// hash replicas are then finished (their loads are counted by k_route_count);
// every other replica leaves one packed candidate per request.  The
// load-dependent pass then walks each replica's requests in arrival order:
//   - batches longer than a warp: k_route_resolve, one CTA per replica that
//     holds the live load in shared memory, twice; a batch is resolved by all its
//     threads against the batch-start loads while its requests add up in the
//     other copy, and the two swap at the boundary;
//   - batches of at most 32 requests (batch_B = 1 is exact sequential
//     dispatch): k_route_resolve_warp, one CTA per replica whose first warp
//     takes S = floor(32 / B) * B requests (whole batches) per step, and whose
//     other warps compute the candidates of later steps (no candidate pass).
//     Inside a step a request's decision depends on the destinations of the
//     earlier batches of the step; the warp finds them by fixed-point
//     iteration: every lane decides from the step-start loads plus the lanes
//     of earlier batches that currently sit on each of its choices, until no
//     lane changes.  After iteration t the first t batches are final, so at
//     most S iterations are needed and typically two or three; the result is
//     the sequential one.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "cr_device.cuh"
#include "cr_internal.cuh"

namespace {

constexpr int kRouteBlock = 1024;
constexpr uint32_t kEmpty = 0xffffffffu;
constexpr size_t kSmemBudget = 200 * 1024;  // dynamic shared memory a resolve CTA may take

// 48 bytes: a replica uses either a plan (CACHEROUTE-type) or a ring (CHWBL).
struct route_desc {
    uint32_t policy;
    int32_t tbits;                    // log2 table slots (plan policies)
    unsigned long long seed;
    union {
        const cr_table_slot *table;      // plan
        const unsigned long long *rpoint;  // ring points
    };
    union {
        const uint16_t *members;         // plan: member lists
        const uint16_t *rowner;          // ring: owner of each point
    };
    union {
        const cr_plan_info_dev *info;    // plan, device: its counters
        const uint32_t *rdir;            // ring: start directory
    };
    union {
        const uint32_t *adm_k;           // plan: k_b in admission order, NULL when it has no entry kSetCap
        struct {
            uint32_t rM;                 // ring points
            int32_t rdbits;              // log2 directory entries
        };
    };
};
static_assert(sizeof(route_desc) == 48, "route_desc layout");

struct route_args {
    route_desc d[CR_MAX_REPLICAS];
    uint32_t dep[CR_MAX_REPLICAS];    // load-dependent replicas, one CTA each in the resolve pass
    uint32_t cand[CR_MAX_REPLICAS];   // candidate pass: replica order, costliest policy first
    uint32_t rr_b0[CR_MAX_REPLICAS];  // round robin: (g0 + seed) mod 2^64 mod R
    unsigned long long rr_wrap[CR_MAX_REPLICAS];  // round robin: first i where g0 + seed + i wraps (~0: never)
};

// Candidate encoding, one u32 per (replica, request):
//   kind 0 FIXED  bits 0..15  destination (RR, HASH, and keys with k_b = 1)
//   kind 1 PAIR   bits 0..12  d1, bits 13..25 d2 (power-of-two choices; R <= 8192)
//   kind 2 SET    bits 0..29  table slot of a key with k_b > 1; tables of at most 2^29 slots:
//                 bits 0..28, and bit 29 set for kLongSet members or more
//   kind 3 RING   bits 0..29  first ring index at or after the key's position
constexpr uint32_t kFixed = 0u << 30, kPair = 1u << 30, kSet = 2u << 30, kRing = 3u << 30,
                   kKindMask = 3u << 30, kLow30 = 0x3fffffffu, kLow29 = 0x1fffffffu, kLongBit = 1u << 29;
constexpr uint32_t kLongSet = 16;

__device__ __forceinline__ uint32_t set_slot(const route_desc &rd, uint32_t c) { return c & ((1u << rd.tbits) - 1u); }

__device__ __forceinline__ uint32_t p2c_pair(unsigned long long seed, uint32_t policy, unsigned long long g,
                                             uint32_t R)
{
    cr_u64x4 u = cr_philox4x64_10(g, 0ull, 0ull, 0ull, seed, (unsigned long long)policy);
    uint32_t d1 = cr_scale(u.x, R);
    uint32_t d2 = d1 + 1u + cr_scale(u.y, (unsigned long long)(R - 1));  // < 2R: one subtraction is mod R
    if (d2 >= R) d2 -= R;
    return kPair | d1 | (d2 << 13);
}

// First ring index whose point is >= h, wrapping to 0 past the last point.
__device__ __forceinline__ uint32_t ring_start(const route_desc &rd, unsigned long long h)
{
    uint32_t j = rd.rdir[h >> (64 - rd.rdbits)];
    while (j < rd.rM && rd.rpoint[j] < h) ++j;
    return j == rd.rM ? 0u : j;
}

// ceil(5 (m + 1) / (4 R)): the per-destination bound at epsilon = 1/4.
__device__ __forceinline__ unsigned long long chwbl_cap(unsigned long long m, uint32_t R)
{
    const unsigned long long den = 4ull * R;
    return (5ull * (m + 1ull) + den - 1ull) / den;
}

// Entries of a replica's row of candidates: rows start on 16-byte boundaries.
__host__ __device__ inline unsigned long long cand_row(unsigned long long n) { return (n + 3ull) & ~3ull; }

// Everything that does not depend on the live load, for every (replica, request).
// A warp takes 32 consecutive requests, reads their keys once and computes the
// candidates of the replicas of its group for them (blockIdx.y = group g of
// gridDim.y: replicas args.cand[g], args.cand[g + G], ..., so every group mixes
// costly and cheap policies; one group when the requests alone fill the GPU);
// round robin and sticky-hash replicas write their destinations directly.
// Consecutive replicas that route with the same plan (the seeds of one policy) share its
// table probe: 24 replicas on ten plans, 1,066,667 requests, the plan-and-route turn around it 2.80 -> 2.70 ms.
// Plan replicas' table misses queue per warp in shared memory, and the warp draws
// their power-of-two choices 32 at a time, so the Philox rounds run with every lane
// busy.
__global__ void __launch_bounds__(256) k_route_cand(const __grid_constant__ route_args args, uint32_t n_rep,
                                                    const unsigned long long *__restrict__ keys,
                                                    unsigned long long n, unsigned long long g0, uint32_t R,
                                                    uint32_t *__restrict__ cand, uint16_t *__restrict__ dest)
{
    __shared__ unsigned long long q_req[256 / 32][64];  // replica << 40 | request
    const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
    unsigned long long *Q = q_req[threadIdx.x >> 5];
    uint32_t qn = 0;  // queued, < 32 between rounds
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long wb = (unsigned long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); wb < n;
         wb += stride) {  // uniform over the warp
        const unsigned long long i = wb + lane;
        const bool valid = i < n;
        const unsigned long long key = valid ? keys[i] : 0ull;
        const cr_table_slot *probed = nullptr;  // the table that `c` comes from
        uint32_t c = 0xffffffffu;
        for (uint32_t x = blockIdx.y; x < n_rep; x += gridDim.y) {  // uniform
            const uint32_t rep = args.cand[x];
            const route_desc &rd = args.d[rep];
            const unsigned long long o = (unsigned long long)rep * n + i, oc = (unsigned long long)rep * cand_row(n) + i;
            switch (rd.policy) {
            case CR_POLICY_RR:
                // (g0 + i + seed) mod 2^64 mod R: before the sum wraps, (b0 + i mod R) mod R
                if (valid) {
                    uint32_t r;
                    if (i < args.rr_wrap[rep] && i < (1ull << 32)) {
                        r = args.rr_b0[rep] + (uint32_t)i % R;
                        if (r >= R) r -= R;
                    } else {
                        r = (uint32_t)((g0 + rd.seed + i) % R);
                    }
                    dest[o] = (uint16_t)r;
                }
                break;
            case CR_POLICY_HASH:
                if (valid) dest[o] = (uint16_t)cr_jump_hash(cr_fmix64(key ^ rd.seed), R);
                break;
            case CR_POLICY_P2C:
                if (valid) cand[oc] = p2c_pair(rd.seed, rd.policy, g0 + i, R);
                break;
            case CR_POLICY_CHWBL:
                if (valid) cand[oc] = kRing | ring_start(rd, cr_fmix64(key ^ rd.seed));
                break;
            default: {
                if (rd.table != probed) {  // uniform: replicas of one plan share a probe
                    probed = rd.table;
                    c = 0xffffffffu;
                    if (valid) {
                        const unsigned long long mask = (1ull << rd.tbits) - 1ull;
                        unsigned long long sl = cr_table_home(key, rd.tbits);
                        for (;;) {
                            const cr_table_slot slot = rd.table[sl];
                            if (slot.koff == kEmpty) break;
                            if (slot.key == key) {
                                c = slot.k == 1 ? (kFixed | slot.m0)
                                                : (kSet | (slot.k >= kLongSet && rd.tbits < 30 ? kLongBit : 0u) | (uint32_t)sl);
                                break;
                            }
                            sl = (sl + 1) & mask;
                        }
                    }
                }
                if (valid && c != 0xffffffffu) cand[oc] = c;
                const bool miss = valid && c == 0xffffffffu;
                const uint32_t mm = __ballot_sync(0xffffffffu, miss);
                if (miss) Q[qn + (uint32_t)__popc(mm & lt)] = ((unsigned long long)rep << 40) | i;
                qn += (uint32_t)__popc(mm);
                __syncwarp();
                if (qn >= 32u) {
                    const unsigned long long e = Q[qn - 32u + lane];
                    const uint32_t er = (uint32_t)(e >> 40);
                    const unsigned long long j = e & ((1ull << 40) - 1ull);
                    cand[(unsigned long long)er * cand_row(n) + j] = p2c_pair(args.d[er].seed, args.d[er].policy, g0 + j, R);
                    qn -= 32u;
                    __syncwarp();
                }
            }
            }
        }
    }
    if (lane < qn) {
        const unsigned long long e = Q[lane];
        const uint32_t er = (uint32_t)(e >> 40);
        const unsigned long long j = e & ((1ull << 40) - 1ull);
        cand[(unsigned long long)er * cand_row(n) + j] = p2c_pair(args.d[er].seed, args.d[er].policy, g0 + j, R);
    }
}

// Live-load counts of the load-independent replicas.
__global__ void __launch_bounds__(256) k_route_count(const uint16_t *__restrict__ dest, unsigned long long n,
                                                     uint32_t R, unsigned long long *__restrict__ load)
{
    extern __shared__ uint32_t hist[];
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) hist[r] = 0;
    __syncthreads();
    const uint16_t *D = dest + (unsigned long long)blockIdx.y * n;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x)
        atomicAdd(&hist[D[i]], 1u);
    __syncthreads();
    unsigned long long *L = load + (unsigned long long)blockIdx.y * R;
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x)
        if (hist[r]) atomicAdd(&L[r], (unsigned long long)hist[r]);
}

// Walk the ring from index j for the first owner whose load is below cap.
// The least-loaded destination always is, so the walk ends within M steps
// unless the load sum has wrapped; then the first owner is taken and the
// overflow flag raised.
template <typename LoadOf>
__device__ __forceinline__ uint32_t ring_walk(const route_desc &rd, const uint16_t *own, uint32_t j,
                                              unsigned long long cap, LoadOf load_of, uint32_t *status)
{
    const uint32_t j0 = j;
    for (uint32_t t = 0; t < rd.rM; ++t) {
        const uint32_t d = own[j];
        if (load_of(d) < cap) return d;
        j = (j + 1 == rd.rM) ? 0u : j + 1;
    }
    atomicOr(status, CR_FLAG_OVERFLOW);
    return own[j0];
}

// Least-loaded member of T(b) = mem[off .. off + k), first member m0 given;
// ties keep the earlier member.  Members are read four at a time.
template <typename LoadOf>
__device__ __forceinline__ uint32_t set_min(const uint16_t *mem, uint32_t off, uint32_t k, uint32_t m0,
                                            LoadOf load_of)
{
    uint32_t best = m0;
    unsigned long long bl = load_of(best);
    uint32_t m = 1;
    for (; m + 4 <= k; m += 4) {
        uint32_t d[4];
        unsigned long long l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) d[u] = mem[off + m + u];
#pragma unroll
        for (int u = 0; u < 4; ++u) l[u] = load_of(d[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (l[u] < bl) {
                bl = l[u];
                best = d[u];
            }
    }
    for (; m < k; ++m) {
        const uint32_t d = mem[off + m];
        const unsigned long long l = load_of(d);
        if (l < bl) {
            bl = l;
            best = d;
        }
    }
    return best;
}

// Copy a replica's u16 side array -- a plan's member lists, or a ring's
// owners -- into shared memory when it fits (cap entries); returns the array
// the decisions read.
__device__ __forceinline__ const uint16_t *stage_aux(const route_desc &rd, uint16_t *sm, unsigned long long cap)
{
    const uint16_t *src = rd.policy == CR_POLICY_CHWBL ? rd.rowner : rd.members;
    if (cap == 0 || src == nullptr) return src;
    const unsigned long long nk = rd.policy == CR_POLICY_CHWBL ? rd.rM : (rd.info ? rd.info->sum_k : cap + 1);
    if (nk > cap) return src;
    for (unsigned long long x = threadIdx.x; x < nk; x += blockDim.x) sm[x] = src[x];
    return sm;
}

// One decision against the batch-start loads.  A bounded-load replica's
// candidates are all RING; every other replica's are FIXED, PAIR or SET, so
// the two cases are compiled apart.  m: requests in the load vector the batch
// sees (the bounded-load rule's m).
// Replica classes of the resolution loop, compiled apart: a plan replica's
// candidates are FIXED, PAIR or SET, a power-of-two-choices replica's only PAIR,
// a bounded-load replica's only RING.
constexpr int kResolvePlan = 0, kResolveRing = 1, kResolvePair = 2;

template <int MODE>
__device__ __forceinline__ uint32_t resolve(uint32_t c, const route_desc &rd, const uint16_t *mem,
                                            const unsigned long long *L, unsigned long long m, uint32_t R,
                                            uint32_t *status)
{
    auto load_of = [&](uint32_t d) { return L[d]; };
    if (MODE == kResolveRing) return ring_walk(rd, mem, c & kLow30, chwbl_cap(m, R), load_of, status);
    if (MODE == kResolvePair) {
        const uint32_t d1 = c & 0x1fffu, d2 = (c >> 13) & 0x1fffu;
        return L[d1] <= L[d2] ? d1 : d2;
    }
    const uint32_t kind = c & kKindMask;
    if (kind == kFixed) return c & 0xffffu;
    if (kind == kPair) {
        const uint32_t d1 = c & 0x1fffu, d2 = (c >> 13) & 0x1fffu;
        return L[d1] <= L[d2] ? d1 : d2;
    }
    const cr_table_slot slot = rd.table[set_slot(rd, c)];
#ifdef CR_DEBUG_CHECKS
    // the member list of the slot lies inside the plan's members (sum of k_b)
    if (!CR_DCHECK(rd.info == nullptr || (unsigned long long)slot.koff + slot.k <= rd.info->sum_k, status))
        return 0;
#endif
    return set_min(mem, slot.koff, slot.k, slot.m0, load_of);
}

// Candidates are staged in shared memory a whole chunk (a multiple of the
// batch, at most kStage requests) ahead: while chunk c is resolved from one
// buffer, chunk c+1's loads are in flight into registers and land in the other.
constexpr uint32_t kStage = 16384;

// Asynchronous global -> shared copies (the next chunk lands while this one is resolved,
// without holding registers).
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Start copying chunk [c1, c1 + CH) of the candidates into buffer nb.  Rows of candidates
// start and end on 16-byte boundaries, as the buffers do: a chunk of whole quadruples is
// copied 16 bytes at a time (up to three of the row's padding entries with it).
__device__ __forceinline__ void stage_next(uint32_t *nb, const uint32_t *__restrict__ Cd, unsigned long long c1,
                                           unsigned long long n, uint32_t CH)
{
    if ((CH & 3u) == 0) {
        for (uint32_t q = threadIdx.x * 4u; q < CH && c1 + q < n; q += blockDim.x * 4u) cp_async16(&nb[q], &Cd[c1 + q]);
        return;
    }
    for (uint32_t q = threadIdx.x; q < CH && c1 + q < n; q += blockDim.x) cp_async4(&nb[q], &Cd[c1 + q]);
}

// Sum of a replica's load vector on entry (the m of the bounded-load rule).
__device__ __forceinline__ unsigned long long block_load_sum(const unsigned long long *L, uint32_t R)
{
    __shared__ unsigned long long s_tot;
    if (threadIdx.x == 0) s_tot = 0;
    __syncthreads();
    unsigned long long t = 0;
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) t += L[r];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(&s_tot, t);
    __syncthreads();
    return s_tot;
}

// The batch loop of one replica (L already holds its loads; ends with a barrier).
template <int MODE>
__device__ __forceinline__ void resolve_batches(const route_desc &rd, const uint16_t *mem, unsigned long long *L,
                                                uint32_t *delta, uint32_t *cbuf, const uint32_t *__restrict__ Cd,
                                                uint16_t *__restrict__ D, unsigned long long n, uint32_t B,
                                                uint32_t CH, uint32_t R, unsigned long long tot0, uint32_t *status)
{
    const uint32_t tid = threadIdx.x;
    if (CH == 0) {
        // batches longer than the stage: candidates straight from global memory
        for (unsigned long long b0 = 0; b0 < n; b0 += B) {
            const unsigned long long b1 = (b0 + B < n) ? b0 + B : n;
            for (unsigned long long i = b0 + tid; i < b1; i += blockDim.x) {
                const uint32_t d = resolve<MODE>(Cd[i], rd, mem, L, tot0 + b0, R, status);
                if (!CR_DCHECK(d < R, status)) continue;
                D[i] = (uint16_t)d;
                atomicAdd(&delta[d], 1u);
            }
            __syncthreads();
            for (uint32_t r = tid; r < R; r += blockDim.x) {
                L[r] += delta[r];
                delta[r] = 0;
            }
            __syncthreads();
        }
        return;
    }
    cp_async_wait_all();  // the caller has started the first chunk's copy
    __syncthreads();
    int cur = 0;
    for (unsigned long long c0 = 0; c0 < n; c0 += CH) {
        const unsigned long long c1 = (c0 + CH < n) ? c0 + CH : n;
        stage_next(cbuf + (size_t)(cur ^ 1) * CH, Cd, c1, n, CH);  // next chunk in flight
        const uint32_t *cb = cbuf + (size_t)cur * CH;
        uint16_t *Dc = D + c0;
        const uint32_t len = (uint32_t)(c1 - c0);  // chunk offsets fit 32 bits
        for (uint32_t o0 = 0; o0 < len; o0 += B) {
            const uint32_t o1 = (o0 + B < len) ? o0 + B : len;
            for (uint32_t o = o0 + tid; o < o1; o += blockDim.x) {
                const uint32_t d = resolve<MODE>(cb[o], rd, mem, L, tot0 + c0 + o0, R, status);
                if (!CR_DCHECK(d < R, status)) continue;
                Dc[o] = (uint16_t)d;
                atomicAdd(&delta[d], 1u);
            }
            __syncthreads();
            for (uint32_t r = tid; r < R; r += blockDim.x) {
                L[r] += delta[r];
                delta[r] = 0;
            }
            __syncthreads();
        }
        cp_async_wait_all();
        __syncthreads();
        cur ^= 1;
    }
}

// ---- batches on 32-bit relative loads ----------------------------------------
// The live loads are held as differences from their minimum (the caller checks that
// every load stays below 2^32 above it) in two buffers.  In batch b the decisions read
// one of them, A = the loads at the start of the batch, and every request adds itself to
// the other, W, which starts equal; when the batch's barrier is passed the two swap, and
// the new W catches up by a copy before a second barrier.  (Adding the requests of batch
// b - 1 to W again instead, without the copy and its barrier, costs a second atomic per
// request: few destinations then meet in it.)
//
// Plan replicas: inside a batch every request of a key with k_b > 1 goes to the same
// member, the least loaded of T(b) at the batch start (ties to the earlier member).  The
// CTA keeps those keys' member lists in shared memory, collected when a staged chunk is
// scanned, and the scan rewrites their candidates to the key's index.  One warp per key
// finds its member between the two barriers; warp w holds the members of key w in
// registers.  Keys past the capacity keep their
// SET candidate, and each request reads the members from the plan.
//   RING (not otherwise used by plan replicas)  index of a tracked key
// A plan with more replicated keys than can be tracked has only those of kLongSet members
// or more tracked: deciding a key costs its warp ~0.1 us a batch, and a list shorter than
// that is scanned as fast by the request itself.  R = 8192, two replicas of 100,000
// requests, 2,000 replicated keys of 2 to 145 members, batches of 1,024: 0.41 ms (whichever
// keys came first tracked, and the map left to fill up: 1.92; none tracked: 1.23).
// Bound: issue slots of the replica's SM (about 2.5 of 4 per cycle).  24 plan replicas of
// 1,066,667 requests, R = 1024, batches of 1,024: the plan-and-route turn around it 3.23 ->
// 2.80 ms against 64-bit loads with a pass over the destinations per batch and a map lookup
// per request; 20 replicas of 166,667 requests at R = 30: 158 -> 125 us.
constexpr uint32_t kSetCap = 256;      // keys with k_b > 1 tracked per replica
constexpr uint32_t kSetMapCap = 512;   // open-addressing map: table slot -> key index
constexpr uint32_t kSetPool = 4096;    // member entries of the tracked keys
constexpr uint16_t kSetNone = 0xffffu;

struct set_cache {
    uint32_t map_slot[kSetMapCap];  // table slot of each map entry, kEmpty when free
    uint16_t map_j[kSetMapCap];     // key index of each map entry, kSetNone until its list is there
    uint32_t off[kSetCap];          // first member of key j in the pool
    uint16_t k[kSetCap];            // its members (0: they did not fit)
    uint16_t res[kSetCap];          // least-loaded member of each key
    uint16_t pool[kSetPool];
    uint32_t n, used;
    uint32_t only[2];               // both kLongBit: only keys with long member lists are tracked
};

// Shared-memory layout of k_route_resolve: loads [R] u64 and counts [R] u32 (or the two
// relative load buffers), at the next 16-byte boundary two staging buffers [CH] u32, member
// lists / ring owners [MC] u16, then (plan replicas) the key cache, 16-byte aligned.
__host__ __device__ inline size_t resolve_stage_at(uint32_t R) { return ((size_t)R * 12 + 15) & ~(size_t)15; }
__host__ __device__ inline size_t resolve_cache_at(uint32_t R, uint32_t CH, unsigned long long MC)
{
    return (resolve_stage_at(R) + (size_t)CH * 8 + (size_t)MC * 2 + 15) & ~(size_t)15;
}

__device__ __forceinline__ uint32_t set_hash(uint32_t slot) { return (slot * 0x9E3779B1u) >> 23; }  // 9 bits

// Index of the key of table slot `slot` (a SET candidate), tracked from now on if it is new
// and fits; kSetNone while another thread is still adding it, or when it does not fit.
__device__ uint32_t set_index(set_cache &S, const route_desc &rd, const uint16_t *mem, uint32_t slot)
{
    uint32_t h = set_hash(slot);
    for (uint32_t it = 0; it < kSetMapCap; ++it, h = (h + 1) & (kSetMapCap - 1)) {
        uint32_t cur = *(volatile uint32_t *)&S.map_slot[h];
        if (cur == kEmpty) {
            if (*(volatile uint32_t *)&S.n >= kSetCap) return kSetNone;
            cur = atomicCAS(&S.map_slot[h], kEmpty, slot);
            if (cur == kEmpty) {
                const uint32_t j = atomicAdd(&S.n, 1u);
                if (j >= kSetCap) {
                    // threads that were here together overran the limit: free the entry again, or
                    // the map fills up and every key it does not hold walks all of it.  A key that
                    // has passed over the entry may no longer be found, and keeps its SET candidates.
                    *(volatile uint32_t *)&S.map_slot[h] = kEmpty;
                    return kSetNone;
                }
                const cr_table_slot ts = rd.table[slot];
                const uint32_t off = atomicAdd(&S.used, (uint32_t)ts.k);
                const bool fits = off + ts.k <= kSetPool;
                for (uint32_t m = 0; fits && m < ts.k; ++m) S.pool[off + m] = mem[(size_t)ts.koff + m];
                S.off[j] = off;
                S.k[j] = fits ? ts.k : (uint16_t)0;
                if (!fits) return kSetNone;
                *(volatile uint16_t *)&S.map_j[h] = (uint16_t)j;
                return j;
            }
        }
        if (cur == slot) return *(volatile uint16_t *)&S.map_j[h];
    }
    return kSetNone;
}

// The staged chunk's SET candidates to key indices, four candidates per thread at a time.
__device__ __forceinline__ void set_scan(set_cache &S, const route_desc &rd, const uint16_t *mem, uint32_t *cb,
                                         uint32_t len, uint32_t CH)
{
    const uint32_t which = kSet | (S.only[0] & S.only[1]), mask = kKindMask | which;
    for (uint32_t q = threadIdx.x * 4u; q < len; q += blockDim.x * 4u) {
        uint32_t c[4];
        if ((CH & 3u) == 0) {
            const uint4 v = *reinterpret_cast<const uint4 *>(&cb[q]);
            c[0] = v.x, c[1] = v.y, c[2] = v.z, c[3] = v.w;
        } else {
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) c[u] = q + u < len ? cb[q + u] : 0u;
        }
        // a key that stands in its first map entry needs no walk; the four looks are independent
        uint32_t sets = 0, left = 0;
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) sets |= (c[u] & mask) == which && q + u < len ? 1u << u : 0u;
        if (!sets) continue;
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            if (!((sets >> u) & 1u)) continue;
            const uint32_t slot = c[u] & kLow29, h = set_hash(slot);
            if (*(volatile uint32_t *)&S.map_slot[h] == slot) {
                const uint32_t j = *(volatile uint16_t *)&S.map_j[h];
                if (j != kSetNone) c[u] = kRing | j;
            } else {
                left |= 1u << u;
            }
        }
        if ((CH & 3u) == 0) {
            *reinterpret_cast<uint4 *>(&cb[q]) = make_uint4(c[0], c[1], c[2], c[3]);
        } else {
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
                if ((sets >> u) & 1u) cb[q + u] = c[u];
        }
        for (; left; left &= left - 1u) {
            const uint32_t u = (uint32_t)__ffs(left) - 1u;
            const uint32_t j = set_index(S, rd, mem, cb[q + u] & kLow29);
            if (j != kSetNone) cb[q + u] = kRing | j;
        }
    }
}

// res[j] of tracked keys j0, j0 + step, .. < n (one warp): the first member with the least load.
__device__ __forceinline__ void set_results(set_cache &S, const uint32_t *A, uint32_t j0, uint32_t step, uint32_t n)
{
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t j = j0; j < n; j += step) {
        const uint32_t off = S.off[j], k = S.k[j];
        if (k == 0) continue;
        uint32_t bl = 0xffffffffu, bp = 0xffffffffu;
        for (uint32_t p = lane; p < k; p += 32) {
            const uint32_t l = A[S.pool[off + p]];
            if (l < bl || bp == 0xffffffffu) {  // positions rise within a lane: the first minimum stays
                bl = l;
                bp = p;
            }
        }
        const uint32_t ml = __reduce_min_sync(0xffffffffu, bl);
        const uint32_t mp = __reduce_min_sync(0xffffffffu, bl == ml ? bp : 0xffffffffu);
        if (lane == 0) S.res[j] = S.pool[off + mp];
    }
}

// ONE: a batch has at most one request per thread, whose next candidate is read a batch
// early.  Returns the buffer that holds the loads at the end.
template <bool ONE, bool PLAN>
__device__ __forceinline__ uint32_t *resolve_relative(const route_desc &rd, const uint16_t *mem, uint32_t *A,
                                                      uint32_t *W, set_cache &S, uint32_t *cbuf,
                                                      const uint32_t *__restrict__ Cd, uint16_t *__restrict__ D,
                                                      unsigned long long n, uint32_t B, uint32_t CH, uint32_t R,
                                                      uint32_t *status)
{
    const uint32_t tid = threadIdx.x, T = blockDim.x, lane = tid & 31u, warp = tid >> 5;
    auto decide = [&](uint32_t c) -> uint32_t {
        if (!PLAN) {
            const uint32_t d1 = c & 0x1fffu, d2 = (c >> 13) & 0x1fffu;
            return A[d1] <= A[d2] ? d1 : d2;
        }
        // FIXED and PAIR without a branch: for FIXED the two fields read are the
        // destination (< R <= 8192) and 0, in range as well; others read entry 0
        const uint32_t kind = c & kKindMask;
        const bool two = kind < kSet;
        const uint32_t d1 = two ? (c & 0x1fffu) : 0u, d2 = two ? ((c >> 13) & 0x1fffu) : 0u;
        const bool p1 = A[d1] <= A[d2];
        if (two) return kind == kFixed ? (c & 0xffffu) : (p1 ? d1 : d2);
        if (kind == kRing) return S.res[c & (kSetCap - 1u)];
        const cr_table_slot slot = rd.table[c & kLow29];
        if (!CR_DCHECK(rd.info == nullptr || (unsigned long long)slot.koff + slot.k <= rd.info->sum_k, status))
            return 0u;
        auto load_of = [&](uint32_t r) { return (unsigned long long)A[r]; };
        return set_min(mem, slot.koff, slot.k, slot.m0, load_of);
    };
    if (PLAN) {
        for (uint32_t x = tid; x < kSetMapCap; x += T) {
            S.map_slot[x] = kEmpty;
            S.map_j[x] = kSetNone;
        }
        // more replicated keys than can be tracked (k_b is non-increasing in admission order): only
        // those with long member lists (two warps: the two reads are in flight together)
        if (tid == 0) {
            S.n = S.used = 0;
            S.only[0] = rd.adm_k && rd.info->n_adm > kSetCap ? kLongBit : 0u;
        }
        if (tid == 32) S.only[1] = rd.adm_k && rd.adm_k[kSetCap] > 1u ? kLongBit : 0u;
    }
    cp_async_wait_all();  // the caller has started the first chunk's copy
    __syncthreads();
    // a scan that met new keys is repeated, for the candidates whose key another thread was
    // just adding (uniform: keys are added only while scanning)
    uint32_t known = 0;
    auto scan = [&](uint32_t *buf, uint32_t len) {
        set_scan(S, rd, mem, buf, len, CH);
        __syncthreads();
        if (S.n != known) {
            known = S.n;
            set_scan(S, rd, mem, buf, len, CH);
            __syncthreads();
        }
    };
    if (PLAN) scan(cbuf, n < CH ? (uint32_t)n : CH);
    int cur = 0;
    for (unsigned long long c0 = 0; c0 < n; c0 += CH) {
        const unsigned long long c1 = (c0 + CH < n) ? c0 + CH : n;
        uint32_t *nb = cbuf + (size_t)(cur ^ 1) * CH;
        uint32_t *cb = cbuf + (size_t)cur * CH;
        uint16_t *Dc = D + c0;
        const uint32_t len = (uint32_t)(c1 - c0);
        uint32_t keys = 0;            // tracked
        uint32_t my_k = 0, my_m = 0;  // this warp's first key, when its members fit the lanes
        if (PLAN) {
            keys = min(known, kSetCap);
            if (warp < keys && S.k[warp] <= 32u) {
                my_k = S.k[warp];
                my_m = my_k ? S.pool[S.off[warp] + min(lane, my_k - 1u)] : 0u;
            }
            set_results(S, A, warp, T >> 5, keys);
            __syncthreads();
        }
        stage_next(nb, Cd, c1, n, CH);
        uint32_t cn = ONE && tid < min(B, len) ? cb[tid] : 0u;  // ONE: the next batch's candidate
        for (uint32_t o0 = 0; o0 < len; o0 += B) {
            const uint32_t o1 = (o0 + B < len) ? o0 + B : len;
            if (ONE) {
                const uint32_t o = o0 + tid, c = cn;
                cn = o1 + tid < len ? cb[o1 + tid] : 0u;
                if (o < o1) {
                    const uint32_t d = decide(c);
                    if (CR_DCHECK(d < R, status)) {
                        Dc[o] = (uint16_t)d;
                        atomicAdd(&W[d], 1u);
                    }
                }
            } else {
                // up to four requests at a time: every read before the first atomic; as many as the
                // warp has left (100,000 requests, R = 30, batches of 1,025: 112.6 us with four always,
                // 77.0 so)
                auto take = [&](auto num, uint32_t o) {
                    constexpr uint32_t N = decltype(num)::value;
                    uint32_t c[N], d[N];
#pragma unroll
                    for (uint32_t u = 0; u < N; ++u) c[u] = o + u * T < o1 ? cb[o + u * T] : 0u;  // (0: FIXED, entry 0)
#pragma unroll
                    for (uint32_t u = 0; u < N; ++u) d[u] = decide(c[u]);
#pragma unroll
                    for (uint32_t u = 0; u < N; ++u) {
                        if (o + u * T >= o1 || !CR_DCHECK(d[u] < R, status)) continue;
                        Dc[o + u * T] = (uint16_t)d[u];
                        atomicAdd(&W[d[u]], 1u);
                    }
                };
                for (uint32_t ow = o0 + (tid & ~31u); ow < o1; ow += 4u * T) {  // uniform over the warp
                    const uint32_t left = o1 - ow;
                    if (left > 2u * T)
                        take(std::integral_constant<uint32_t, 4>(), ow + lane);
                    else if (left > T)
                        take(std::integral_constant<uint32_t, 2>(), ow + lane);
                    else
                        take(std::integral_constant<uint32_t, 1>(), ow + lane);
                }
            }
            __syncthreads();
            uint32_t *t = A;
            A = W;
            W = t;
            for (uint32_t r = tid; r < R; r += T) W[r] = A[r];
            if (PLAN && keys) {
                uint32_t j0 = warp;
                if (my_k) {  // of equal loads, the lowest lane's
                    const uint32_t l = lane < my_k ? A[my_m] : 0xffffffffu;
                    const uint32_t least = __ballot_sync(0xffffffffu, l == __reduce_min_sync(0xffffffffu, l));
                    if (lane == (uint32_t)__ffs(least) - 1u) S.res[warp] = (uint16_t)my_m;
                    j0 += T >> 5;
                }
                set_results(S, A, j0, T >> 5, keys);
            }
            __syncthreads();
        }
        if (c1 == n) break;
        cp_async_wait_all();
        __syncthreads();
        if (PLAN) scan(nb, n - c1 < CH ? (uint32_t)(n - c1) : CH);
        cur ^= 1;
    }
    return A;
}

// The replica's loads as differences from their minimum in A and W (= A + R), and the
// minimum; false (neither is then meaningful) when a load could pass 2^32 - 1 above it, or
// 2^64 (loads wrap there, and are compared wrapped).
__device__ __forceinline__ bool loads_relative(const unsigned long long *Lg, uint32_t R, unsigned long long n,
                                               uint32_t *A, uint32_t *W, unsigned long long &base)
{
    __shared__ unsigned long long s_lo[32], s_hi[32];
    const uint32_t lane = threadIdx.x & 31u, warps = min((R + 31u) / 32u, blockDim.x >> 5);  // those with a load
    unsigned long long lo = ~0ull, hi = 0;
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) {
        const unsigned long long v = Lg[r];
        lo = v < lo ? v : lo;
        hi = v > hi ? v : hi;
        A[r] = (uint32_t)v;
    }
    auto reduce = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
            lo = a < lo ? a : lo;
            hi = b > hi ? b : hi;
        }
    };
    if ((threadIdx.x >> 5) < warps) {
        reduce();
        if (lane == 0) {
            s_lo[threadIdx.x >> 5] = lo;
            s_hi[threadIdx.x >> 5] = hi;
        }
    }
    __syncthreads();
    lo = lane < warps ? s_lo[lane] : ~0ull;
    hi = lane < warps ? s_hi[lane] : 0ull;
    if (warps > 1)
        reduce();
    else
        lo = s_lo[0], hi = s_hi[0];
    base = lo;
    if (n >= 0xffffffffull || hi - lo >= 0xffffffffull - n || hi > ~0ull - n) return false;
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) A[r] = W[r] = A[r] - (uint32_t)base;  // mod 2^32
    __syncthreads();
    return true;
}

__global__ void __launch_bounds__(kRouteBlock, 1) k_route_resolve(const __grid_constant__ route_args args,
                                                               const uint32_t *__restrict__ cand,
                                                               unsigned long long n, uint32_t B, uint32_t CH,
                                                               uint32_t R, unsigned long long *__restrict__ load,
                                                               uint16_t *__restrict__ dest, uint32_t *status,
                                                               unsigned long long MC, int plan_x)
{
    extern __shared__ __align__(16) unsigned long long sh[];
    unsigned char *shb = reinterpret_cast<unsigned char *>(sh);
    unsigned long long *L = sh;                              // [R] live load
    uint32_t *delta = reinterpret_cast<uint32_t *>(sh + R);  // [R] this batch
    uint32_t *cbuf = reinterpret_cast<uint32_t *>(shb + resolve_stage_at(R));  // [2][CH] staged candidates
    uint16_t *smem_aux = reinterpret_cast<uint16_t *>(cbuf + 2 * (size_t)CH);  // [MC] members or ring owners
    const uint32_t rep = args.dep[blockIdx.x];
    const route_desc rd = args.d[rep];
    unsigned long long *Lg = load + (unsigned long long)rep * R;
    const uint32_t *Cd = cand + (unsigned long long)rep * cand_row(n);
    uint16_t *D = dest + (unsigned long long)rep * n;
    const bool plan = rd.policy != CR_POLICY_CHWBL && rd.policy != CR_POLICY_P2C;
    if (CH > 0) stage_next(cbuf, Cd, 0, n, CH);
    const uint16_t *mem = stage_aux(rd, smem_aux, MC);
    if (CH > 0 && rd.policy != CR_POLICY_CHWBL && (plan_x || !plan)) {
        uint32_t *A = reinterpret_cast<uint32_t *>(sh), *W = A + R, *F;  // in place of the 64-bit loads
        set_cache &S = *reinterpret_cast<set_cache *>(shb + resolve_cache_at(R, CH, MC));
        unsigned long long base;
        if (loads_relative(Lg, R, n, A, W, base)) {  // uniform over the block
            if (plan)
                F = B <= blockDim.x ? resolve_relative<true, true>(rd, mem, A, W, S, cbuf, Cd, D, n, B, CH, R, status)
                                    : resolve_relative<false, true>(rd, mem, A, W, S, cbuf, Cd, D, n, B, CH, R, status);
            else
                F = B <= blockDim.x ? resolve_relative<true, false>(rd, mem, A, W, S, cbuf, Cd, D, n, B, CH, R, status)
                                    : resolve_relative<false, false>(rd, mem, A, W, S, cbuf, Cd, D, n, B, CH, R, status);
            for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) Lg[r] = base + F[r];
            return;
        }
    }
    // loads 2^32 - n or more apart, batches longer than the stage, bounded loads: 64-bit
    // loads and counts, every request of a key scanning its members
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) {
        L[r] = Lg[r];
        delta[r] = 0;
    }
    if (rd.policy == CR_POLICY_CHWBL) {  // uniform over the block
        const unsigned long long tot0 = block_load_sum(L, R);
        resolve_batches<kResolveRing>(rd, mem, L, delta, cbuf, Cd, D, n, B, CH, R, tot0, status);
    } else if (rd.policy == CR_POLICY_P2C) {
        __syncthreads();  // orders the copies above
        resolve_batches<kResolvePair>(rd, mem, L, delta, cbuf, Cd, D, n, B, CH, R, 0ull, status);
    } else {
        __syncthreads();
        resolve_batches<kResolvePlan>(rd, mem, L, delta, cbuf, Cd, D, n, B, CH, R, 0ull, status);
    }
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) Lg[r] = L[r];
}

// ---- batches of at most one warp: one CTA per replica ------------------------
// Warp 0 resolves; warps 1 .. kPrepWarps prepare.  A step is S = floor(32 / B) * B
// requests (whole batches), one per lane; a chunk is kPrepWarps steps.  While the
// resolver works through chunk c, preparer w computes step w of chunk c + 1 into
// the other half of a double buffer -- the candidates themselves (table probe,
// Philox draws or ring position) and everything about the step that does not
// depend on the live load -- and writes out the destinations of chunk c - 1.  The
// resolver's serial chain is then only what the loads decide, on loads held
// relative to their minimum in 32 bits:
//   - two choices d1, d2 (power-of-two choices; a key with k_b = 1 is d1 = d2, one
//     with k_b = 2 its two members, ties to the first): the preparer leaves, per
//     lane, the lanes of the step whose first / second choice is this lane's d1 /
//     d2 (four bit masks, built from one ballot per destination bit).  With S the
//     ballot of the lanes on their second choice, the earlier lanes on d1 are
//     popc(select(S, second == d1, first == d1) & earlier), so one iteration of the
//     fixed point is two selects, two popcounts, a compare and a ballot in
//     registers: no shared memory, no atomics.
//   - bounded loads, R <= 32: the preparer leaves the bound and the first eight
//     distinct owners of the walk; an iteration compares the first four at once
//     (then the next four, then the walk itself), lane r holding the mask of the
//     lanes on destination r (five ballots).
//   - bounded loads on more destinations, and steps with a key of three or more
//     members: lane masks per destination in shared memory (masked_step).
//   - loads spread over 2^30 or more, or near 2^64 (sums wrap): the same masked
//     steps on 64-bit loads.
// Bound by the latency of the resolver's chain (a ballot and the branch on it cost
// ~50 cycles, a popcount ~20, a shared-memory read ~29 on this GPU).  Measured on a
// GB300 with B = 1, R = 30, 83,333 requests, five replicas: power-of-two choices 0.83
// ms, plan replicas 0.68 ms, bounded loads 1.58 ms; all fifteen 1.42 ms, where one
// warp that did all of it (every iteration re-reading loads and masks from shared
// memory, bound computed by division inside the chain) took 3.7 ms.  256 requests,
// one plan replica at R = 64: 62 -> 15 us a call (no staging of member lists, no
// candidate launch).  Bounded loads on R > 32 cost 1.87 ms (masked_step).
constexpr int kPrepWarps = 8;
// warps 4 and 8 stay idle: the resolver has its SM sub-partition's issue slots to itself
constexpr int kWarpPathWarps = kPrepWarps + 3;
constexpr unsigned long long kNarrow = 1ull << 30;  // spread of the loads during a call, 32-bit loops
constexpr uint32_t kOwn8 = 32;                      // destinations up to which ring walks go through eight distinct owners

// Shared memory of the kernel: the double-buffered steps, then loads [R] u64 (the
// 32-bit loops use the first half) and lane masks [R] u32.
struct prep_buf {
    uint4 m[2][kPrepWarps][32];      // two choices: lanes with first == d1, second == d1, first == d2, second == d2
                                     // ring: owners, eight u8 in (x, y) for R <= 32, else four u16 in (x, y); bound lo, hi
    uint32_t d[2][kPrepWarps][32];   // two choices: d1 | d2 << 16; ring: first ring index
    uint2 set[2][kPrepWarps][32];    // keys of three or more members: member offset, members (else 0)
    uint16_t out[2][kPrepWarps][32]; // destinations decided
    uint32_t any_set[2][kPrepWarps]; // some lane of the step has such a key
};

// Table slot of a plan replica's key (koff = kEmpty: not in the table).
__device__ __forceinline__ cr_table_slot plan_probe(const route_desc &rd, unsigned long long key)
{
    const unsigned long long mask = (1ull << rd.tbits) - 1ull;
    unsigned long long sl = cr_table_home(key, rd.tbits);
    cr_table_slot slot = rd.table[sl];
    while (slot.koff != kEmpty && slot.key != key) {  // at least twice as many slots as keys: an empty one ends it
        sl = (sl + 1) & mask;
        slot = rd.table[sl];
    }
    return slot;
}

// Prepare one step (one warp): its lanes' requests into half `h`, step `w` of the buffer.
__device__ __forceinline__ void prepare_step(prep_buf &pb, uint32_t h, uint32_t w, const route_desc &rd, bool active,
                                             unsigned long long key, unsigned long long g, uint32_t R, uint32_t nb,
                                             unsigned long long seen_m)
{
    const uint32_t lane = cr_lane();
    const uint32_t am = __ballot_sync(0xffffffffu, active);
    if (rd.policy == CR_POLICY_CHWBL) {
        uint4 m = make_uint4(0, 0, 0, 0);
        uint32_t j0 = 0;
        if (active) {
            uint32_t j = j0 = ring_start(rd, cr_fmix64(key ^ rd.seed));
            const unsigned long long cap = chwbl_cap(seen_m, R);
            m.z = (uint32_t)cap;
            m.w = (uint32_t)(cap >> 32);
            if (R <= kOwn8) {
                // the first eight distinct owners, or as many as the first 16 ring points give; shorter
                // lists repeat the first one, which changes no decision (an owner met again is as
                // full as before).  The lane that looks longest holds up its warp, and with few
                // destinations the eighth owner is far or not there at all: 3 R points then (64
                // points, two replicas of 20,000 requests, B = 1: R = 2 377 -> 164 us, R = 8 421 -> 188)
                const uint32_t most = min(rd.rM, min(3u * R, 16u));
                uint32_t met = 0, k = 0, lo = 0, hi = 0, o0 = rd.rowner[j];
                for (uint32_t t = 0; t < most && k < 8u; ++t) {
                    const uint32_t o = rd.rowner[j];
                    j = j + 1 == rd.rM ? 0u : j + 1;
                    if ((met >> o) & 1u) continue;
                    met |= 1u << o;
                    if (k < 4u)
                        lo |= o << (8 * k);
                    else
                        hi |= o << (8 * (k - 4u));
                    ++k;
                }
                for (; k < 8u; ++k) {
                    if (k < 4u)
                        lo |= o0 << (8 * k);
                    else
                        hi |= o0 << (8 * (k - 4u));
                }
                m.x = lo;
                m.y = hi;
            } else {
                uint32_t o[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    o[q] = rd.rowner[j];
                    j = j + 1 == rd.rM ? 0u : j + 1;
                }
                m.x = o[0] | (o[1] << 16);
                m.y = o[2] | (o[3] << 16);
            }
        }
        pb.m[h][w][lane] = m;
        pb.d[h][w][lane] = j0;
        return;
    }
    uint32_t d1 = 0, d2 = 0;
    uint2 set = make_uint2(0, 0);
    bool draw = active;  // power-of-two choices: every request, or a plan replica's keys outside the table
    if (rd.policy != CR_POLICY_P2C) {
        cr_table_slot slot;
        slot.koff = kEmpty;
        if (active) slot = plan_probe(rd, key);
        __syncwarp();  // the draws below run once for the whole warp, not once per probe length
        if (slot.koff != kEmpty) {
            draw = false;
            d1 = d2 = slot.m0;
            if (slot.k > 1) d2 = rd.members[(size_t)slot.koff + 1];
            if (slot.k > 2) {
                set = make_uint2(slot.koff, slot.k);
                for (uint32_t q = 2; q < slot.k; q += 64)  // brings the list into this SM's L1
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(rd.members + (size_t)slot.koff + q));
            }
        }
        __syncwarp();
    }
    if (draw) {
        const uint32_t c = p2c_pair(rd.seed, rd.policy, g, R);
        d1 = c & 0x1fffu;
        d2 = (c >> 13) & 0x1fffu;
    }
    __syncwarp();
    uint32_t e11 = am, e21 = am, e12 = am, e22 = am;
#pragma unroll
    for (uint32_t b = 0; b < 13; ++b) {
        if (b < nb) {  // uniform
            const uint32_t b1 = __ballot_sync(0xffffffffu, (d1 >> b) & 1u);
            const uint32_t b2 = __ballot_sync(0xffffffffu, (d2 >> b) & 1u);
            const uint32_t x1 = 0u - ((d1 >> b) & 1u), x2 = 0u - ((d2 >> b) & 1u);
            e11 &= ~(b1 ^ x1);
            e21 &= ~(b2 ^ x1);
            e12 &= ~(b1 ^ x2);
            e22 &= ~(b2 ^ x2);
        }
    }
    const bool any = __any_sync(0xffffffffu, set.y != 0u);
    pb.m[h][w][lane] = active ? make_uint4(e11, e21, e12, e22) : make_uint4(0, 0, 0, 0);
    pb.d[h][w][lane] = d1 | (d2 << 16);
    pb.set[h][w][lane] = set;
    if (lane == 0) pb.any_set[h][w] = any;
}

// bit by bit: sel ? b : a
__device__ __forceinline__ uint32_t bit_select(uint32_t sel, uint32_t a, uint32_t b) { return (a & ~sel) | (b & sel); }

// What the resolver's steps share.
struct step_ctx {
    uint32_t lane, bit, earlier;  // earlier: lanes of the earlier batches of the step
    bool several;                 // more than one batch per step
    uint32_t max_it;
    uint32_t *status;
};

// A step decided through the lane masks in shared memory (zero between steps): `decide(earlier)`
// gives this lane's destination from the step-start loads plus the lanes of `earlier` on each
// destination.  After iteration t the first t batches of the step are final.
template <typename LT, typename Decide>
__device__ __forceinline__ uint32_t masked_step(const step_ctx &X, LT *L, uint32_t *mask, bool active, uint32_t R,
                                                Decide decide)
{
    uint32_t d = active ? decide(0u) : 0u;
    if (!CR_DCHECK(d < R, X.status)) d = 0;
    if (active) atomicOr(&mask[d], X.bit);
    __syncwarp();
    if (X.several) {
        for (uint32_t it = 0;; ++it) {
            uint32_t nd = active ? decide(X.earlier) : d;
            if (!CR_DCHECK(nd < R, X.status)) nd = 0;
            const uint32_t moved = __ballot_sync(0xffffffffu, nd != d);
            if (!moved) break;
            if (it >= X.max_it) {  // unreachable: max_it iterations always settle the step
                if (X.lane == 0) atomicOr(X.status, CR_FLAG_TIMEOUT);
                break;
            }
            if (nd != d) {
                atomicAnd(&mask[d], ~X.bit);
                atomicOr(&mask[nd], X.bit);
                d = nd;
            }
            __syncwarp();
        }
    }
    if (active) {
        const uint32_t mk = mask[d];
        if ((mk & (0u - mk)) == X.bit) L[d] += (LT)__popc(mk);  // lowest lane adds
    }
    __syncwarp();
    if (active) mask[d] = 0;
    __syncwarp();
    return d;
}

// A two-choice or set step through the masks.
template <typename LT>
__device__ __forceinline__ uint32_t set_step(const step_ctx &X, LT *L, uint32_t *mask, const route_desc &rd,
                                             bool active, uint32_t R, uint32_t d12, uint2 set)
{
    const uint32_t d1 = d12 & 0xffffu, d2 = d12 >> 16;
    return masked_step(X, L, mask, active, R, [&](uint32_t earlier) {
        auto seen = [&](uint32_t x) { return (unsigned long long)(LT)(L[x] + (LT)__popc(mask[x] & earlier)); };
        if (set.y) return set_min(rd.members, set.x, set.y, d1, seen);
        return seen(d1) <= seen(d2) ? d1 : d2;
    });
}

// A bounded-load step through the masks: the first four owners of the walk, then the walk itself.
template <typename LT>
__device__ __forceinline__ uint32_t ring_step(const step_ctx &X, LT *L, uint32_t *mask, const route_desc &rd,
                                              bool active, uint32_t R, uint4 m, uint32_t j0, unsigned long long cap)
{
    const uint32_t o[4] = {m.x & 0xffffu, m.x >> 16, m.y & 0xffffu, m.y >> 16};
    uint32_t t[4];  // free places of each owner (32: more than the step can take)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const unsigned long long l = L[o[w]];
        t[w] = l >= cap ? 0u : (cap - l < 32ull ? (uint32_t)(cap - l) : 32u);
    }
    return masked_step(X, L, mask, active, R, [&](uint32_t earlier) {
        uint32_t f[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) f[w] = (uint32_t)__popc(mask[o[w]] & earlier);
        if (f[0] < t[0]) return o[0];
        if (f[1] < t[1]) return o[1];
        if (f[2] < t[2]) return o[2];
        if (f[3] < t[3]) return o[3];
        auto seen = [&](uint32_t x) { return (unsigned long long)(LT)(L[x] + (LT)__popc(mask[x] & earlier)); };
        return ring_walk(rd, rd.rowner, j0, cap, seen, X.status);
    });
}

// One chunk of two-choice steps on 32-bit loads.
__device__ __forceinline__ void resolve_pairs(const step_ctx &X, prep_buf &pb, uint32_t h, uint32_t steps,
                                              uint32_t *L, uint32_t *mask, const route_desc &rd, uint32_t R)
{
    const uint32_t lane = X.lane, below = X.bit - 1u;
    uint4 mn = pb.m[h][0][lane];
    uint32_t dn = pb.d[h][0][lane], an = pb.any_set[h][0];
#pragma unroll 1
    for (uint32_t q = 0; q < steps; ++q) {
        const uint4 m = mn;
        const uint32_t d12 = dn, any = an;
        if (q + 1 < steps) {
            mn = pb.m[h][q + 1][lane];
            dn = pb.d[h][q + 1][lane];
            an = pb.any_set[h][q + 1];
        }
        const uint32_t d1 = d12 & 0xffffu, d2 = d12 >> 16;
        if (any) {
            const uint32_t d = set_step(X, L, mask, rd, m.x != 0u, R, d12, pb.set[h][q][lane]);
            pb.out[h][q][lane] = (uint16_t)d;
            continue;
        }
        const uint32_t a1 = m.x & X.earlier, a2 = m.y & X.earlier, b1 = m.z & X.earlier, b2 = m.w & X.earlier;
        const uint32_t l1 = L[d1], l2 = L[d2];
        const int diff = (int)(l1 - l2);
        uint32_t sel = __ballot_sync(0xffffffffu, diff > 0);
        if (X.several) {
            // the first `it` batches are final after pass `it`: at most max_it passes change anything
            auto pass = [&](uint32_t now) {
                const int x = diff + __popc(bit_select(now, a1, a2)) - __popc(bit_select(now, b1, b2));
                return __ballot_sync(0xffffffffu, x > 0);
            };
            sel = pass(sel);
            for (uint32_t it = 0; it <= X.max_it; ++it) {
                const uint32_t ns = pass(sel);
                const bool same = ns == sel;
                sel = ns;
                if (same) break;
            }
        }
        const bool second = (sel & X.bit) != 0u;
        const uint32_t mine = second ? bit_select(sel, m.z, m.w) : bit_select(sel, m.x, m.y);
        const uint32_t d = second ? d2 : d1;
        // the lowest lane of each destination adds its lanes (an inactive lane's masks are empty)
        if ((mine & (below | X.bit)) == X.bit) L[d] = (second ? l2 : l1) + (uint32_t)__popc(mine);
        pb.out[h][q][lane] = (uint16_t)d;
        __syncwarp();
    }
}

// One chunk of bounded-load steps on 32-bit loads relative to `base`, R <= 32: lane r holds the
// mask of the lanes on destination r.
__device__ __forceinline__ void resolve_ring32(const step_ctx &X, prep_buf &pb, uint32_t h, uint32_t steps,
                                               uint32_t *L, const route_desc &rd, uint32_t R, unsigned long long base)
{
    const uint32_t lane = X.lane;
    uint32_t xr[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) xr[b] = 0u - ((lane >> b) & 1u);
    uint4 mn = pb.m[h][0][lane];
#pragma unroll 1
    for (uint32_t q = 0; q < steps; ++q) {
        const uint4 m = mn;
        if (q + 1 < steps) mn = pb.m[h][q + 1][lane];
        const unsigned long long cap64 = (unsigned long long)m.z | ((unsigned long long)m.w << 32);
        const bool active = cap64 != 0ull;  // a bound is at least 1
        const uint32_t am = __ballot_sync(0xffffffffu, active);
        // the bound never is below the least load; far above every load it only has to stay there
        const int cap = cap64 - base < 0x7fffffffull ? (int)(cap64 - base) : 0x7fffffff;
        // free places of the first four owners of the walk (at most 0: none)
        uint32_t o[4];
        int t[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            o[w] = (m.x >> (8 * w)) & 0xffu;
            t[w] = cap - (int)L[o[w]];
        }
        uint32_t c = t[0] > 0 ? o[0] : (t[1] > 0 ? o[1] : (t[2] > 0 ? o[2] : o[3])), M = 0;
        for (uint32_t it = 0; it <= X.max_it + 1u; ++it) {
            uint32_t mr = am;
#pragma unroll
            for (int b = 0; b < 5; ++b) mr &= ~(__ballot_sync(0xffffffffu, (c >> b) & 1u) ^ xr[b]);
            M = mr;
            int f[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) f[w] = __popc(__shfl_sync(0xffffffffu, mr, o[w]) & X.earlier);
            uint32_t nc = f[0] < t[0] ? o[0] : (f[1] < t[1] ? o[1] : (f[2] < t[2] ? o[2] : o[3]));
            bool left = active && f[0] >= t[0] && f[1] >= t[1] && f[2] >= t[2] && f[3] >= t[3];
            if (!__any_sync(0xffffffffu, left || (active && nc != c))) break;
            if (__any_sync(0xffffffffu, left)) {  // the next four owners of the walk
                uint32_t n2 = 0xffu;
#pragma unroll
                for (int w = 3; w >= 0; --w) {
                    const uint32_t ow = (m.y >> (8 * w)) & 0xffu;
                    const int fw = __popc(__shfl_sync(0xffffffffu, mr, ow) & X.earlier);
                    n2 = fw < cap - (int)L[ow] ? ow : n2;
                }
                if (left && n2 != 0xffu) {
                    nc = n2;
                    left = false;
                }
                if (__any_sync(0xffffffffu, left)) {  // rare: the walk itself, all lanes together
                    uint32_t j = pb.d[h][q][lane];
                    const uint32_t first = left ? (uint32_t)rd.rowner[j] : 0u;
                    for (uint32_t x = 0; x < rd.rM; ++x) {
                        const uint32_t ow = left ? (uint32_t)rd.rowner[j] : 0u;
                        const uint32_t mo = __shfl_sync(0xffffffffu, mr, ow & 31u);
                        if (left && (int)L[ow & 31u] + __popc(mo & X.earlier) < cap) {
                            nc = ow;
                            left = false;
                        }
                        j = j + 1 >= rd.rM ? 0u : j + 1;
                        if (!__any_sync(0xffffffffu, left)) break;
                    }
                    if (left) {  // no destination below the bound: only when a load sum has wrapped
                        nc = first;
                        atomicOr(X.status, CR_FLAG_OVERFLOW);
                    }
                }
                if (!__any_sync(0xffffffffu, active && nc != c)) break;
            }
            if (!CR_DCHECK(!active || nc < R, X.status)) nc = 0;
            if (active) c = nc;
        }
        pb.out[h][q][lane] = (uint16_t)c;
        if (lane < R) L[lane] += (uint32_t)__popc(M);
        __syncwarp();
    }
}

__global__ void __launch_bounds__(32 * kWarpPathWarps)
k_route_resolve_warp(const __grid_constant__ route_args args, const unsigned long long *__restrict__ keys,
                     unsigned long long n, unsigned long long g0, uint32_t B, uint32_t R,
                     unsigned long long *__restrict__ load, uint16_t *__restrict__ dest, uint32_t *status)
{
    extern __shared__ uint4 sh4[];
    prep_buf &pb = *reinterpret_cast<prep_buf *>(sh4);
    unsigned long long *L64 = reinterpret_cast<unsigned long long *>(reinterpret_cast<unsigned char *>(sh4) +
                                                                     sizeof(prep_buf));
    uint32_t *L32 = reinterpret_cast<uint32_t *>(L64);
    uint32_t *mask = reinterpret_cast<uint32_t *>(L64 + R);
    __shared__ unsigned long long s_tot, s_max, s_min;
    const uint32_t rep = args.dep[blockIdx.x];
    const route_desc &rd = args.d[rep];
    unsigned long long *Lg = load + (unsigned long long)rep * R;
    uint16_t *D = dest + (unsigned long long)rep * n;
    const uint32_t lane = cr_lane(), warp = threadIdx.x >> 5;
    const bool resolver = warp == 0, preparer = (warp & 3u) != 0;
    const uint32_t pw = preparer ? warp - 1u - (warp >> 2) : 0u;  // preparer number, its step of every chunk
    const bool ring = rd.policy == CR_POLICY_CHWBL;
    if (threadIdx.x == 0) {
        s_tot = s_max = 0;
        s_min = ~0ull;
    }
    __syncthreads();
    {
        unsigned long long tot = 0, mx = 0, mi = ~0ull;
        for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) {
            const unsigned long long v = Lg[r];
            L64[r] = v;
            mask[r] = 0;
            tot += v;
            mx = v > mx ? v : mx;
            mi = v < mi ? v : mi;
        }
        // one 64-bit shared atomic (a compare-and-swap loop) per warp, not per thread: five
        // requests at R = 520 17.3 -> 9.4 us
        if ((threadIdx.x & ~31u) < R) {
            tot = cr_warp_sum_u64(tot);
            mx = ~cr_warp_min_u64(~mx);
            mi = cr_warp_min_u64(mi);
            if (lane == 0) {
                atomicAdd(&s_tot, tot);
                atomicMax(&s_max, mx);
                atomicMin(&s_min, mi);
            }
        }
    }
    __syncthreads();
    const unsigned long long tot0 = s_tot, base = s_min;
    // the 32-bit loops: the loads stay within 2^30 of the least one, and nothing wraps
    const bool narrow = s_max < (1ull << 47) && n < kNarrow && s_max - base < kNarrow - n;
    if (narrow) {  // in place: a thread's 64-bit words are read before any 32-bit word is written
        for (uint32_t r0 = 0; r0 < R; r0 += blockDim.x) {
            const uint32_t r = r0 + threadIdx.x;
            const uint32_t v = r < R ? (uint32_t)(L64[r] - base) : 0u;
            __syncthreads();
            if (r < R) L32[r] = v;
            __syncthreads();
        }
    }
    const uint32_t S = (32u / B) * B;               // requests per step: whole batches
    const uint32_t bstart = (lane / B) * B;         // first lane of this lane's batch
    step_ctx X;
    X.lane = lane;
    X.bit = 1u << lane;
    X.earlier = (1u << bstart) - 1u;
    X.several = S > B;
    X.max_it = S;
    X.status = status;
    const uint32_t nb = R > 1 ? 32u - (uint32_t)__clz(R - 1u) : 0u;  // bits of a destination, <= 13
    const unsigned long long CHR = (unsigned long long)S * kPrepWarps;  // requests per chunk
    const unsigned long long nchunks = (n + CHR - 1) / CHR;
    const bool own8 = ring && R <= kOwn8;
    // preparer pw: step pw of a chunk; the chunk after's key is in flight meanwhile
    auto index_of = [&](unsigned long long c) { return c * CHR + (unsigned long long)pw * S + lane; };
    auto key_of = [&](unsigned long long c) {
        const unsigned long long i = index_of(c);
        return (lane < S && i < n) ? keys[i] : 0ull;
    };
    auto prepare_chunk = [&](unsigned long long c, unsigned long long key) {
        const unsigned long long i = index_of(c);
        prepare_step(pb, (uint32_t)(c & 1), pw, rd, lane < S && i < n, key, g0 + i, R, nb,
                     tot0 + (i - lane) + bstart);
    };
    auto write_chunk = [&](unsigned long long c) {
        const unsigned long long i = index_of(c);
        if (lane < S && i < n) D[i] = pb.out[c & 1][pw][lane];
    };
    unsigned long long knext = 0;
    if (preparer) {
        const unsigned long long k0 = key_of(0);
        knext = key_of(1);
        prepare_chunk(0, k0);
    }
    __syncthreads();
    for (unsigned long long c = 0; c < nchunks; ++c) {
        if (preparer) {
            if (c > 0) write_chunk(c - 1);  // before its half is prepared anew
            if (c + 1 < nchunks) {
                const unsigned long long key = knext;
                knext = key_of(c + 2);
                prepare_chunk(c + 1, key);
            }
        } else if (resolver) {
            const uint32_t h = (uint32_t)(c & 1);
            const unsigned long long left = n - c * CHR;
            const uint32_t steps = left >= CHR ? (uint32_t)kPrepWarps : (uint32_t)((left + S - 1) / S);
            if (narrow && !ring) {
                resolve_pairs(X, pb, h, steps, L32, mask, rd, R);
            } else if (narrow && own8) {
                resolve_ring32(X, pb, h, steps, L32, rd, R, base);
            } else {
#pragma unroll 1
                for (uint32_t q = 0; q < steps; ++q) {
                    const uint4 m = pb.m[h][q][lane];
                    const uint32_t dj = pb.d[h][q][lane];
                    uint32_t d;
                    if (!ring) {
                        d = set_step(X, L64, mask, rd, m.x != 0u, R, dj, pb.set[h][q][lane]);
                    } else {
                        const unsigned long long cap = (unsigned long long)m.z | ((unsigned long long)m.w << 32);
                        const bool active = lane < S && (c * kPrepWarps + q) * S + lane < n;
                        uint4 ow = m;
                        if (own8) {  // the first four of the eight owners
                            ow.x = (m.x & 0xffu) | ((m.x & 0xff00u) << 8);
                            ow.y = ((m.x >> 16) & 0xffu) | ((m.x >> 24) << 16);
                        }
                        if (narrow)
                            d = ring_step(X, L32, mask, rd, active, R, ow, dj, cap - base);
                        else
                            d = ring_step(X, L64, mask, rd, active, R, ow, dj, cap);
                    }
                    pb.out[h][q][lane] = (uint16_t)d;
                }
            }
        }
        __syncthreads();
    }
    if (preparer) write_chunk(nchunks - 1);
    for (uint32_t r = threadIdx.x; r < R; r += blockDim.x) Lg[r] = narrow ? base + L32[r] : L64[r];
}

// ---- ring construction ------------------------------------------------------

__global__ void __launch_bounds__(256) k_ring_points(unsigned long long seed, unsigned long long M,
                                                     unsigned long long *__restrict__ pt)
{
    for (unsigned long long k = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; k < M;
         k += (unsigned long long)gridDim.x * blockDim.x)
        pt[k] = cr_fmix64(seed + (k + 1ull) * CR_GAMMA);  // SplitMix64 output k
}

// Sorted points (stable: equal points keep ascending owner) -> point and owner arrays.
__global__ void __launch_bounds__(256) k_ring_finish(const unsigned long long *__restrict__ ks,
                                                     const uint32_t *__restrict__ pos, unsigned long long M,
                                                     uint32_t V, unsigned long long *__restrict__ pt,
                                                     uint16_t *__restrict__ ow)
{
    for (unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; j < M;
         j += (unsigned long long)gridDim.x * blockDim.x) {
        pt[j] = ks[j];
        ow[j] = (uint16_t)(min((unsigned long long)pos[j], M - 1ull) / V);  // (a sort that gave up leaves places unset)
    }
}

// dir[t] = first ring index whose point is >= t << (64 - dbits) (M if none).
__global__ void __launch_bounds__(256) k_ring_dir(const unsigned long long *__restrict__ pt, unsigned long long M,
                                                  int dbits, uint32_t *__restrict__ dir)
{
    const unsigned long long nd = 1ull << dbits;
    for (unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; t < nd;
         t += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long h = t << (64 - dbits);
        unsigned long long lo = 0, hi = M;
        while (lo < hi) {
            const unsigned long long mid = (lo + hi) >> 1;
            if (pt[mid] < h)
                lo = mid + 1;
            else
                hi = mid;
        }
        dir[t] = (uint32_t)lo;
    }
}

}  // namespace

static int ring_fill(cr_ctx *ctx, cr_ring *g, uint64_t seed)
{
    const unsigned int gcap = (unsigned int)ctx->num_sms * 8u;
    const unsigned long long M = g->M;
    const unsigned long long *ks = nullptr;
    const uint32_t *pos = nullptr;
    CR_LAUNCH(ctx, k_ring_points, cr_blocks(M, 256, gcap), 256, 0, (unsigned long long)seed, M, g->d_point);
    CR_TRY(cr_radix_sort_u64(ctx, g->d_point, M, &ks, &pos));
    CR_LAUNCH(ctx, k_ring_finish, cr_blocks(M, 256, gcap), 256, 0, ks, pos, M, g->V, g->d_point, g->d_owner);
    CR_LAUNCH(ctx, k_ring_dir, cr_blocks(1ull << g->dbits, 256, gcap), 256, 0, (const unsigned long long *)g->d_point,
              M, (int)g->dbits, g->d_dir);
    return CR_OK;
}

extern "C" int cr_ring_create(cr_ctx *ctx, uint32_t R, uint32_t vnodes, uint64_t seed, cr_ring **out)
{
    if (!ctx || !out) return CR_EINVAL;
    *out = nullptr;
    if (R == 0 || R > CR_MAX_R) return cr_fail(ctx, CR_EINVAL, "cr_ring_create: R=%u outside 1..%u", R, CR_MAX_R);
    if (vnodes == 0 || vnodes > CR_MAX_VNODES)
        return cr_fail(ctx, CR_EINVAL, "cr_ring_create: vnodes=%u outside 1..%u", vnodes, CR_MAX_VNODES);
    const uint64_t M = (uint64_t)R * vnodes;
    int dbits = 1;
    while ((1ull << dbits) < M) ++dbits;
    cr_ring *g = (cr_ring *)calloc(1, sizeof(cr_ring));
    if (!g) return cr_fail(ctx, CR_ENOMEM, "cr_ring_create: host allocation failed");
    g->R = R;
    g->V = vnodes;
    g->M = M;
    g->dbits = (uint32_t)dbits;
    if (cudaMalloc(&g->d_point, M * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMalloc(&g->d_owner, M * sizeof(uint16_t)) != cudaSuccess ||
        cudaMalloc(&g->d_dir, (1ull << dbits) * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        cr_ring_destroy(ctx, g);
        return cr_fail(ctx, CR_ENOMEM, "cr_ring_create: device allocation of %llu points failed",
                       (unsigned long long)M);
    }
    const int st = ring_fill(ctx, g, seed);
    if (st != CR_OK) {
        cr_ring_destroy(ctx, g);
        return st;
    }
    *out = g;
    return CR_OK;
}

extern "C" int cr_ring_destroy(cr_ctx *ctx, cr_ring *g)
{
    if (!g) return CR_OK;
    if (ctx) cudaStreamSynchronize(ctx->stream);
    if (g->d_point) cudaFree(g->d_point);
    if (g->d_owner) cudaFree(g->d_owner);
    if (g->d_dir) cudaFree(g->d_dir);
    free(g);
    return CR_OK;
}

extern "C" int cr_ring_export(cr_ctx *ctx, const cr_ring *g, uint64_t *point, uint16_t *owner)
{
    if (!ctx || !g) return CR_EINVAL;
    if (point)
        CR_CUDA(ctx, cudaMemcpyAsync(point, g->d_point, g->M * sizeof(uint64_t), cudaMemcpyDeviceToHost, ctx->stream));
    if (owner)
        CR_CUDA(ctx, cudaMemcpyAsync(owner, g->d_owner, g->M * sizeof(uint16_t), cudaMemcpyDeviceToHost, ctx->stream));
    return cr_sync(ctx);
}

static int launch_resolve(cr_ctx *ctx, cudaStream_t rs, const route_args &args, const uint32_t *cand,
                          const uint64_t *d_key, uint64_t n, uint64_t g0, uint32_t batch_B, uint32_t R, uint64_t mc,
                          uint32_t n_dep, uint64_t *d_load, uint16_t *d_dest);

extern "C" int cr_route_batch(cr_ctx *ctx, const cr_plan *const *plans, const cr_replica *reps, uint32_t n_rep,
                              uint32_t R, const uint64_t *d_key, uint64_t n, uint64_t first_req_index,
                              uint32_t batch_B, uint64_t *d_load, uint16_t *d_dest)
{
    if (!ctx) return CR_EINVAL;
    cr_nvtx_range nv("cr_route_batch");
    if (R == 0 || R > CR_MAX_R) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: R=%u outside 1..%u", R, CR_MAX_R);
    if (n_rep == 0 || n_rep > CR_MAX_REPLICAS || !reps)
        return cr_fail(ctx, CR_EINVAL, "cr_route_batch: n_rep=%u outside 1..%u", n_rep, CR_MAX_REPLICAS);
    if (batch_B == 0) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: batch_B must be >= 1");
    if (n >= (1ull << 40)) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: n >= 2^40");
    if (!d_load) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: d_load is NULL");
    if (n > 0 && (!d_key || !d_dest)) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: NULL key or dest");
    route_args args;
    memset(&args, 0, sizeof(args));
    uint64_t mc = 0;  // largest u16 side array: a plan's member lists or a ring's owners
    for (uint32_t i = 0; i < n_rep; ++i) {
        route_desc &d = args.d[i];
        d.policy = reps[i].policy;
        d.seed = reps[i].seed;
        if (reps[i].policy > CR_POLICY_CHWBL || reps[i].reserved != 0)
            return cr_fail(ctx, CR_EINVAL, "cr_route_batch: replica %u has policy %u", i, reps[i].policy);
        if (reps[i].policy <= CR_POLICY_CR_NOREPL) {
            const cr_plan *p = plans ? plans[i] : nullptr;
            if (!p || !p->built)
                return cr_fail(ctx, CR_EINVAL, "cr_route_batch: replica %u needs a built plan", i);
            if (p->R != R)
                return cr_fail(ctx, CR_EINVAL, "cr_route_batch: replica %u plan has R=%u, call has R=%u", i, p->R, R);
            int bits = 0;
            while ((1ull << bits) < p->table_slots) ++bits;
            if (bits > 30) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: plan table too large");
            d.tbits = bits;
            d.table = p->d_table;
            d.members = p->d_members;
            d.info = p->d_info;
            d.adm_k = p->cap_adm > kSetCap ? p->d_adm_k : nullptr;  // (as many keys as can be tracked: all of them)
            mc = std::max<uint64_t>(mc, (uint64_t)p->R * p->W);  // sum of k_b <= C = R W
        } else if (reps[i].policy == CR_POLICY_CHWBL) {
            const cr_ring *g = reps[i].ring;
            if (!g) return cr_fail(ctx, CR_EINVAL, "cr_route_batch: replica %u needs a ring", i);
            if (g->R != R)
                return cr_fail(ctx, CR_EINVAL, "cr_route_batch: replica %u ring has R=%u, call has R=%u", i, g->R, R);
            d.rpoint = g->d_point;
            d.rowner = g->d_owner;
            d.rdir = g->d_dir;
            d.rM = (uint32_t)g->M;
            d.rdbits = (int32_t)g->dbits;
            mc = std::max<uint64_t>(mc, g->M);
        }
    }
    if (n == 0) return CR_OK;
    // replicas whose choices depend on the live load
    uint32_t n_dep = 0;
    for (uint32_t i = 0; i < n_rep; ++i)
        if (reps[i].policy != CR_POLICY_RR && reps[i].policy != CR_POLICY_HASH) args.dep[n_dep++] = i;
    // candidate rows, costliest policy first, so that the grid's last wave holds cheap rows
    // (per request: jump hash ~8 jumps, Philox ~10 rounds, plan probe + Philox for misses,
    // ring lookup, round robin)
    // (batches of at most a warp: only the load-independent replicas; k_route_resolve_warp
    // computes the others' candidates itself)
    const bool warp_path = batch_B <= 32;
    uint32_t n_cand = 0;
    {
        auto cost = [&](uint32_t p) {
            return p == CR_POLICY_HASH ? 0 : p == CR_POLICY_P2C ? 1 : p <= CR_POLICY_CR_NOREPL ? 2
                 : p == CR_POLICY_CHWBL ? 3 : 4;
        };
        for (uint32_t c = 0; c <= 4; ++c)
            for (uint32_t i = 0; i < n_rep; ++i) {
                const uint32_t p = reps[i].policy;
                if (warp_path && p != CR_POLICY_RR && p != CR_POLICY_HASH) continue;
                if ((uint32_t)cost(p) == c) args.cand[n_cand++] = i;
            }
    }
    // split routing: the candidates scratch is free once the last resolution has read it
    const cudaStream_t rs = ctx->resolve_stream ? ctx->resolve_stream : ctx->stream;
    const bool split = rs != ctx->stream;
    if (split && ctx->resolve_recorded) CR_CUDA(ctx, cudaStreamWaitEvent(ctx->stream, ctx->ev_resolve, 0));
    uint32_t *cand = nullptr;
    const uint64_t *key_dep = d_key;
    if (!warp_path) {
        void *pc;
        CR_TRY(cr_scratch(ctx, SCR_ROUTE_DESC, (size_t)cand_row(n) * n_rep * sizeof(uint32_t), &pc));
        cand = (uint32_t *)pc;
    } else if (split && n_dep) {
        // the resolution reads the keys on its own stream: from a copy, so that the caller's
        // keys are still read on the context's stream only
        void *pc;
        CR_TRY(cr_scratch(ctx, SCR_ROUTE_DESC, (size_t)n * sizeof(uint64_t), &pc));
        CR_CUDA(ctx, cudaMemcpyAsync(pc, d_key, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, ctx->stream));
        key_dep = (const uint64_t *)pc;
    }
    const int pcand = cr_prof_begin(ctx, ctx->stream, CR_PROF_ROUTE_CAND);
    for (uint32_t i = 0; i < n_rep; ++i) {
        const uint64_t base = (uint64_t)first_req_index + reps[i].seed;  // wraps mod 2^64 as the policy does
        args.rr_b0[i] = (uint32_t)(base % R);
        args.rr_wrap[i] = base ? 0ull - base : ~0ull;
    }
    // request blocks; replica groups only as many as it takes to reach ~16 blocks per SM
    const unsigned int cbx = cr_blocks(n, 256, (unsigned int)ctx->num_sms * 32u);
    const unsigned int want = (unsigned int)ctx->num_sms * 16u;
    unsigned int cgy = (want + cbx - 1) / cbx;
    cgy = cgy < 1 ? 1 : (cgy > n_cand ? n_cand : cgy);
    if (n_cand)
        CR_LAUNCH(ctx, k_route_cand, dim3(cbx, cgy), 256, 0, args, n_cand,
                  (const unsigned long long *)d_key, (unsigned long long)n, (unsigned long long)first_req_index, R,
                  cand, d_dest);
    cr_prof_end(ctx, ctx->stream, pcand);
    // load counts of RR / HASH replicas (their choices never read the load)
    for (uint32_t i = 0; i < n_rep; ++i) {
        if (reps[i].policy != CR_POLICY_RR && reps[i].policy != CR_POLICY_HASH) continue;
        uint32_t j = i;
        while (j + 1 < n_rep && (reps[j + 1].policy == CR_POLICY_RR || reps[j + 1].policy == CR_POLICY_HASH)) ++j;
        dim3 grid(cr_blocks(n, 256, 64), j - i + 1);
        CR_LAUNCH(ctx, k_route_count, grid, 256, (size_t)R * sizeof(uint32_t), d_dest + (uint64_t)i * n,
                  (unsigned long long)n, R, (unsigned long long *)d_load + (uint64_t)i * R);
        i = j;
    }
    if (split) {  // the resolution (and the caller's later readers) follow everything above
        CR_CUDA(ctx, cudaEventRecord(ctx->ev_cand, ctx->stream));
        CR_CUDA(ctx, cudaStreamWaitEvent(rs, ctx->ev_cand, 0));
    }
    if (n_dep) {
        const int pr = cr_prof_begin(ctx, rs, CR_PROF_ROUTE_RESOLVE);
        CR_TRY(launch_resolve(ctx, rs, args, cand, key_dep, n, first_req_index, batch_B, R, mc, n_dep, d_load, d_dest));
        cr_prof_end(ctx, rs, pr);
    }
    if (split) {
        CR_CUDA(ctx, cudaEventRecord(ctx->ev_resolve, rs));
        ctx->resolve_recorded = 1;
    }
    return CR_OK;
}

// The load-dependent resolution of every dependent replica, enqueued on stream rs.
static int launch_resolve(cr_ctx *ctx, cudaStream_t rs, const route_args &args, const uint32_t *cand,
                          const uint64_t *d_key, uint64_t n, uint64_t g0, uint32_t batch_B, uint32_t R, uint64_t mc,
                          uint32_t n_dep, uint64_t *d_load, uint16_t *d_dest)
{
    // member lists and ring owners go to shared memory when they fit beside the loads
    auto with_members = [&](size_t base, uint64_t *MC) {
        *MC = (mc && base + mc * sizeof(uint16_t) <= kSmemBudget) ? mc : 0;
        return base + *MC * sizeof(uint16_t);
    };
    uint64_t MC;
    if (batch_B <= 32) {
        const size_t smem = sizeof(prep_buf) + (size_t)R * (sizeof(unsigned long long) + sizeof(uint32_t));
        if (smem > kDefaultSmem)
            CR_CUDA(ctx, cudaFuncSetAttribute(k_route_resolve_warp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)smem));
        CR_LAUNCH_ON(ctx, rs, k_route_resolve_warp, n_dep, 32 * kWarpPathWarps, smem, args,
                     (const unsigned long long *)d_key, (unsigned long long)n, (unsigned long long)g0, batch_B, R,
                     (unsigned long long *)d_load, d_dest, ctx->d_status);
        return CR_OK;
    }
    // staging chunk: a whole number of batches, at most kStage requests, whole quadruples
    // (16-byte copies) where four batches fit
    uint32_t unit = batch_B;
    while ((unit & 3u) && unit <= kStage / 2u) unit *= 2u;
    if (unit & 3u) unit = batch_B;  // none fit: the largest chunk then
    uint32_t CH = unit <= kStage ? (kStage / unit) * unit : 0u;  // 0: no staging
    const size_t loads = resolve_stage_at(R);
    // plan replicas take the key cache when it fits beside a stage of at least one batch
    // (the stage shrinks by whole batches)
    bool any_plan = false;
    bool slots29 = true;  // slot numbers leave bit 29 of a candidate free
    for (uint32_t i = 0; i < n_dep; ++i)
        if (args.d[args.dep[i]].policy <= CR_POLICY_CR_NOREPL) {
            any_plan = true;
            slots29 = slots29 && args.d[args.dep[i]].tbits < 30;
        }
    const size_t px = sizeof(set_cache);
    int plan_x = 0;
    if (any_plan && slots29 && CH) {
        uint32_t ch = CH;
        while (ch >= unit && loads + (size_t)ch * 8 + 16 + px > kSmemBudget) ch -= unit;
        if (ch < unit && unit > batch_B) {
            unit = batch_B;
            ch = CH;
            while (ch >= unit && loads + (size_t)ch * 8 + 16 + px > kSmemBudget) ch -= unit;
        }
        if (ch >= unit) {
            CH = ch;
            plan_x = 1;
        }
    }
    size_t smem;
    if (plan_x) {
        const size_t fixed = loads + (size_t)CH * 8 + 16 + px;
        MC = (mc && fixed + mc * sizeof(uint16_t) <= kSmemBudget) ? mc : 0;
        smem = resolve_cache_at(R, CH, MC) + px;
    } else {
        smem = with_members(loads + 2ull * CH * sizeof(uint32_t), &MC);
    }
    if (smem > kDefaultSmem)
        CR_CUDA(ctx, cudaFuncSetAttribute(k_route_resolve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // no more threads than a batch has requests (a barrier of idle warps costs time), but
    // enough to stage candidates, and, where a plan's keys can have members by the dozen, warps
    // to decide those keys at once.  Ten replicas x 535,947 requests, R = 587, batches of 333:
    // 384 / 512 / 768 / 1,024 threads 2.55 / 2.01 / 1.66 / 1.68 ms; R = 30 without replicated
    // keys, batches of 256: 256 / 512 / 768 threads 182 / 192 / 211 us
    const uint32_t least = any_plan && R > 64 ? 768u : 256u;
    const uint32_t threads = batch_B >= (uint32_t)kRouteBlock ? (uint32_t)kRouteBlock
                                                              : std::max(least, (batch_B + 31u) / 32u * 32u);
    CR_LAUNCH_ON(ctx, rs, k_route_resolve, n_dep, threads, smem, args, (const uint32_t *)cand, (unsigned long long)n,
              batch_B, CH, R, (unsigned long long *)d_load, d_dest, ctx->d_status, (unsigned long long)MC, plan_x);
    return CR_OK;
}
