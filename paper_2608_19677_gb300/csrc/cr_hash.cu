// a1: prefix-span routing key (cr_hash_prefixes).
//
// The key is the wrapping sum of one SplitMix64-mixed term per 64-bit word
// (two int32 tokens) of the prefix plus a length term, so any partition of the
// words over lanes gives the same result.  One warp hashes one request: lanes
// stride over the span with 16-byte streaming loads (four tokens = two words
// per load, up to eight loads in flight per lane: the next group of four is
// fetched while the current one is mixed; words that straddle two vectors take
// their first token from the neighbouring lane), then the warp reduces its partial
// sums; the next request's span descriptor is fetched a request ahead.  The path is an HBM stream of 4*P bytes per request; the
// per-word mix (about two dozen integer instructions) keeps the ALU just under that stream
// rate on sm_103a.
#include "cr_device.cuh"
#include "cr_internal.cuh"

namespace {

constexpr int kHashBlock = 256;

__device__ __forceinline__ unsigned long long word_term(uint32_t lo, uint32_t hi, unsigned long long k)
{
    unsigned long long w = (unsigned long long)lo | ((unsigned long long)hi << 32);
    return cr_fmix64(w ^ k);
}

// Four rows of 32 aligned 16-byte vectors, one per lane; vectors from v1 on are not read.
template <bool FULL>
__device__ __forceinline__ void load4(int4 (&x)[4], const int4 *__restrict__ b4, uint32_t v, uint32_t v1)
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t i = v + 32u * q;
        if (FULL || i < v1)
            x[q] = __ldcs(b4 + i);
        else
            x[q] = make_int4(0, 0, 0, 0);
    }
}

// Mix one group.  k: key of the word whose tokens are (x, y) of this lane's first vector when
// the span starts on an even token of its vector, or (y, z) when it starts on an odd one.
// An odd start puts every second word across two vectors: (w of the vector before, x); the
// vector before is the previous lane's, or the previous row's last (`carry`, lane 0 only).
// Vectors in [v, v1) count; `head` marks the lane and row whose straddling word lies outside.
template <bool ODD, bool FULL>
__device__ __forceinline__ unsigned long long mix4(const int4 (&x)[4], unsigned long long k, uint32_t v, uint32_t v1,
                                                   uint32_t lane, bool head, uint32_t &carry)
{
    const unsigned long long G64 = 64ull * CR_GAMMA;
    unsigned long long acc = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned long long kq = k + (unsigned long long)q * G64;
        const bool in = FULL || v + 32u * q < v1;
        if (!ODD) {
            if (in) acc += word_term(x[q].x, x[q].y, kq) + word_term(x[q].z, x[q].w, kq + CR_GAMMA);
        } else {
            const uint32_t r = __shfl_sync(0xffffffffu, (uint32_t)x[q].w, (lane + 31u) & 31u);
            const uint32_t before = lane ? r : carry;
            carry = r;  // lane 0: this row's last w
            if (in) {
                acc += word_term(x[q].y, x[q].z, kq);
                if (q > 0 || !head) acc += word_term(before, x[q].x, kq - CR_GAMMA);
            }
        }
    }
    return acc;
}

// The words of a span that lie inside its aligned vectors [v0, v1), two groups in flight: the next
// group loads while the current one is mixed.
template <bool ODD>
__device__ __forceinline__ unsigned long long vector_words(const int4 *__restrict__ b4, uint32_t v0, uint32_t v1,
                                                           unsigned long long k, uint32_t lane)
{
    const unsigned long long G256 = 256ull * CR_GAMMA;
    unsigned long long acc = 0;
    uint32_t carry = 0;
    int4 cur[4];
    uint32_t vb = v0;  // first vector of the group (uniform over the warp)
    const uint32_t groups = (v1 - v0) >> 7;
    if (groups)
        load4<true>(cur, b4, vb + lane, v1);
    else
        load4<false>(cur, b4, vb + lane, v1);
    for (uint32_t g = 0; g < groups; ++g) {
        int4 nxt[4];
        if (g + 1 < groups)
            load4<true>(nxt, b4, vb + 128u + lane, v1);
        else
            load4<false>(nxt, b4, vb + 128u + lane, v1);
        acc += mix4<ODD, true>(cur, k, vb + lane, v1, lane, g == 0 && lane == 0, carry);
#pragma unroll
        for (int q = 0; q < 4; ++q) cur[q] = nxt[q];
        vb += 128u;
        k += G256;
    }
    if (vb < v1) acc += mix4<ODD, false>(cur, k, vb + lane, v1, lane, groups == 0 && lane == 0, carry);
    return acc;
}

// A short span word by word, a few rounds of the warp (the lane's partial sum): the vector
// path mixes four rows of 32 vectors whatever there is, and words across vectors by shuffles.
// 100,000 spans at odd starts, 16 / 64 / 128 / 192 tokens: 36.9 / 38.9 / 38.9 / 45.1 -> 24.6 /
// 24.6 / 28.7 / 36.9 us; at 200 tokens both take 45.  Not inlined: the loops for long spans
// keep their registers (inlined, spans of 1,025 and 4,097 tokens took 2-3% more).
constexpr uint32_t kShortMin = 8, kShortMax = 192;
__device__ __noinline__ unsigned long long short_words(const int32_t *__restrict__ base, uint32_t P,
                                                       unsigned long long salt, uint32_t lane)
{
    unsigned long long acc = 0;
#pragma unroll 2
    for (uint32_t w = lane; 2u * w < P; w += 32u) {
        const uint32_t lo = (uint32_t)__ldcs(base + 2u * w);
        const uint32_t hi = 2u * w + 1u < P ? (uint32_t)__ldcs(base + 2u * w + 1u) : 0u;
        acc += word_term(lo, hi, salt + (unsigned long long)(w + 1u) * CR_GAMMA);
    }
    return acc;
}

// 64 registers per thread: 32 warps per SM, which measured faster than larger
// unrolls at lower occupancy.
// A span may start on any token of a 16-byte vector (sh = start address / 4 mod 4): the
// aligned vectors that lie inside it are read whole, and the words at its ends that they
// do not hold (at most two before, three after) one per lane with scalar loads, so nothing
// outside the span is read.  5,000 spans of 1,024-4,096 tokens packed back to back (any start):
// 28 -> 18 us against 4- and 8-byte loads (16.5 with the spans in L2); aligned spans (166,667 of
// ~2,300 tokens) 286 -> 283 us.
__global__ void __launch_bounds__(kHashBlock, 4)
k_hash_prefixes(const int32_t *__restrict__ tok, const unsigned long long *__restrict__ off,
                const uint32_t *__restrict__ plen, unsigned long long n, unsigned long long salt,
                unsigned long long *__restrict__ out)
{
    const uint32_t lane = cr_lane();
    const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    unsigned long long r = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    unsigned long long o_next = 0;
    uint32_t P_next = 0;
    if (r < n) {
        o_next = off[r];
        P_next = plen[r];
    }
    for (; r < n; r += nwarps) {
        const unsigned long long o = o_next;
        const uint32_t P = P_next;
        if (r + nwarps < n) {  // the next request's span descriptor is in flight meanwhile
            o_next = off[r + nwarps];
            P_next = plen[r + nwarps];
        }
        const int32_t *base = tok + o;
        unsigned long long acc = 0;
        // vector v holds tokens 4v - sh .. 4v - sh + 3 of the span; [v0, v1) lie inside it
        const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(base) >> 2) & 3u;
        uint32_t v0 = 0, v1 = P >> 2, head = 0, rest = 0, sw = 0;
        int32_t slo = 0, shi = 0;
        if (sh | (P & 3u)) {  // uniform; whole vectors only otherwise, as records padded to 16 bytes have
            if (P - kShortMin <= kShortMax - kShortMin) {
                acc = short_words(base, P, salt, lane);
                v1 = 0;
            } else {
                const uint32_t nw = P / 2u + (P & 1u);
                uint32_t tail = nw;  // words [0, head) and [tail, nw) are left to scalar loads
                v0 = sh ? 1u : 0u;
                v1 = (uint32_t)(((unsigned long long)P + sh) >> 2);
                head = nw;
                if (v1 > v0) {
                    head = 2u * v0 - (sh >> 1);  // first word that vector v0 holds whole
                    tail = 2u * (v1 - 1u) - (sh >> 1) + ((sh & 1u) ? 1u : 2u);
                }
                // at most five, one per lane: in flight while the vectors are mixed
                rest = head + (nw - tail);
                sw = lane < head ? lane : tail + (lane - head);
                if (lane < rest) {
                    slo = __ldcs(base + 2 * sw);
                    if (2 * sw + 1 < P) shi = __ldcs(base + 2 * sw + 1);
                }
            }
        }
        if (v1 > v0) {
            const int4 *b4 = reinterpret_cast<const int4 *>(base - (int)sh);
            // key of this lane's first word: word 2 (v0 + lane) - sh / 2
            const unsigned long long k = salt + (unsigned long long)(head + 2u * lane + 1u) * CR_GAMMA;
            acc = (sh & 1u) ? vector_words<true>(b4, v0, v1, k, lane) : vector_words<false>(b4, v0, v1, k, lane);
        }
        if (lane < rest)
            acc += word_term((uint32_t)slo, (uint32_t)shi, salt + (unsigned long long)(sw + 1u) * CR_GAMMA);
        acc = cr_warp_sum_u64(acc);
        if (lane == 0) out[r] = cr_fmix64(salt ^ (unsigned long long)P) + acc;
    }
}

}  // namespace

extern "C" int cr_hash_prefixes(cr_ctx *ctx, const int32_t *d_tokens, const uint64_t *d_off,
                                const uint32_t *d_plen, uint64_t n, uint64_t salt, uint64_t *d_key_out)
{
    cr_nvtx_range nv("cr_hash_prefixes");
    if (!ctx) return CR_EINVAL;
    if (n == 0) return CR_OK;
    if (!d_tokens || !d_off || !d_plen || !d_key_out)
        return cr_fail(ctx, CR_EINVAL, "cr_hash_prefixes: NULL pointer");
    const unsigned int warps_per_block = kHashBlock / 32;
    // many more blocks than fit at once (32 per SM): blocks start as others
    // finish, which evens out the widely varying span lengths across the SMs
    unsigned int grid = cr_blocks(n, warps_per_block, (unsigned int)ctx->num_sms * 32u);
    const int pi = cr_prof_begin(ctx, ctx->stream, CR_PROF_HASH);
    CR_LAUNCH(ctx, k_hash_prefixes, grid, kHashBlock, 0, d_tokens, (const unsigned long long *)d_off,
              d_plen, (unsigned long long)n, (unsigned long long)salt, (unsigned long long *)d_key_out);
    cr_prof_end(ctx, ctx->stream, pi);
    return CR_OK;
}
