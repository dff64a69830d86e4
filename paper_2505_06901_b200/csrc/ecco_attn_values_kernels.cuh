// ecco_attn_values_kernels.cuh -- K5: attention output over a compressed V cache
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

namespace {

// ---------------------------------------------------------------------------------------------
// K5: attention output over a compressed V cache (Eq. 3: softmax(QK^T / sqrt(d_k)) V).
// out[b][hq][d] = sum_t p[b][hq][t] * V~[b][hq / q_per_kv][t][d] with p = softmax_t(scores).
// A lane owns one token (one group) as in K3, but here the sum runs over tokens, i.e. across lanes: the groups are
// decoded into tiles (decode_to_tiles), then every tile is contracted on the tensor cores:
// (V tile)^T [16 dims x 32 tokens] x P^T [32 tokens x 8 heads] with mma.m16n8k16, fp32 accumulators
// (4 registers per 16 dims, 32 for the 128 dims).  p is split into an fp16 head and an fp16 remainder
// (two MMAs) so that its rounding does not show.  The result does not depend on scheduling.
//
// The softmax is formed on the way: p is taken relative to the largest score that the warp has seen of the row, and sums
// and accumulators are rescaled when a larger one comes, so the scores are read once and no kernel has to go before this one
// (a statistics kernel in front cost 25 us on a cache of 128 rows x 8 heads x 32768 scores and 4 us on the shortest rows).
// ---------------------------------------------------------------------------------------------
constexpr uint32_t kAvSlots = 8;                                            // reduction slots: see flush

constexpr float kProbScale = 32768.0f;                                      // a power of two: exact
constexpr int kPieceFloats = kGroup * 8 + 16;              // sums of [128 dims][8 heads], 8 sums of weights, 8 maxima

// factor that takes sums relative to maximum m to maximum m_new >= m; an empty side has m = -inf and sums of zero
__device__ __forceinline__ float rescale(float m, float m_new) { return m == m_new ? 1.0f : __expf(m - m_new); }

template <int kMaxWarps, bool kGiveUp>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
ecco_attn_values_kernel(const uint8_t* __restrict__ d_meta, const uint8_t* __restrict__ d_vblocks, int heads, int seq,
                        int q_per_kv, int unit_warps, int n_teams, const float* d_scores, float* __restrict__ d_out, float* __restrict__ d_partial,
                        Ticket* d_tickets, Ticket tag)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    release_dependents();
    const DecodeTables tb = plan_decode_tables(smem_u32(smem), d_meta, false);       // one symbol per lookup: the tiles need the room
    constexpr uint32_t kFull = 0xffffffffu, kSlotFloats = kGroup * 8 + 8;       // sums, sums of weights
    // A team of nw warps takes a head at a time.  One team: all CTAs share the units, and the CTA's other warps help with the
    // reductions.  Several: every team has whole heads of its own and meets at a barrier of its own.
    const uint32_t fit = decode_warps(tb, kTiledWarpBytes), nw = min(fit, static_cast<uint32_t>(unit_warps));
    const uint32_t teams = min(static_cast<uint32_t>(n_teams), fit / nw), team = teams > 1 ? warp / nw : 0;
    const int tid = static_cast<int>(threadIdx.x - team * nw * 32u), n_threads = static_cast<int>(teams > 1 ? nw * 32u : blockDim.x);
    auto team_sync = [&]() {
        if (teams == 1) __syncthreads();
        else if (nw == 1) __syncwarp();                    // up to sixteen teams: more than there are barriers beside the CTA's
        else asm volatile("bar.sync %0, %1;" ::"r"(team + 1u), "r"(nw * 32u) : "memory");
    };
    const int kTokens = static_cast<int>(nw) * 32;         // tokens per unit: one per thread of the working warps
    const bool working = warp < (teams > 1 ? teams * nw : nw);
    // small CTA-wide words in the misc area at the start of shared memory (the barrier word is its first)
    unsigned int& ticket = *reinterpret_cast<unsigned int*>(smem + 32);
    float* max_s = reinterpret_cast<float*>(smem + 64);    // [warps][8 heads]
    static_assert(64 + kMaxWarps * 8 * 4 <= kMisc, "maxima fit the misc area");
    const uint32_t tiles = tb.warp_base + warp * kTiledWarpBytes;
    // over the team's arrays: slots of [128 dims][8 heads]
    float* out_s = reinterpret_cast<float*>(smem + (tb.warp_base - tb.base) + team * nw * kTiledWarpBytes);
    const uint32_t first_warp = team * nw;

    const int chunks = (seq + kTokens - 1) / kTokens;
    const int64_t U = static_cast<int64_t>(heads) * chunks;
    // the CTAs that share a head count each other in (ticket), so every CTA of the split must own a unit: the
    // launch may bring more CTAs than there are units (the host does not know how many warps find room)
    const int G = static_cast<int>(min(static_cast<int64_t>(gridDim.x), U)), c = blockIdx.x;
    if (teams == 1 && c >= G) return;
    const int all_teams = static_cast<int>(gridDim.x * teams), my_team = static_cast<int>(team * gridDim.x) + c;
    const UnitSplit split(teams > 1 ? heads : U, teams > 1 ? all_teams : G);                // of heads or of units
    const int me = teams > 1 ? my_team : c, scale = teams > 1 ? chunks : 1;
    const int64_t u0 = split.begin(me) * scale, u1 = split.begin(me + 1) * scale;
    // (head, first token) of a unit: advanced by one unit at a time, not divided out of its number
    int bh = static_cast<int>(divide(static_cast<uint64_t>(u0), static_cast<uint64_t>(chunks)));
    int token = static_cast<int>(u0 - static_cast<int64_t>(bh) * chunks) * kTokens;
    auto block_ptr = [&](int head, int from) { return d_vblocks + (static_cast<uint64_t>(head) * seq + min(from + tid, seq - 1)) * kBlockBytes; };
    issue_decode_tables(tb, d_meta);
    if (u0 < u1 && working) prefetch_block_l2(block_ptr(bh, token));
    if (!finish_decode_tables<kGiveUp>(tb)) {
        if (teams == 1 && tid == 0) {                      // passes the tickets of the heads it shares: at most the first and the last
            const int ends[2] = {bh, static_cast<int>(divide(static_cast<uint64_t>(u1 - 1), static_cast<uint64_t>(chunks)))};
            for (int i = 0; i < 2; ++i) {
                const int last = split.owner(static_cast<int64_t>(ends[i] + 1) * chunks - 1) - split.owner(static_cast<int64_t>(ends[i]) * chunks);
                if (last && (i == 0 || ends[1] != ends[0])) pass_ticket(d_tickets + ends[i], last, tag);
            }
        }
        return;
    }
    dependency_wait();                                     // everything but the host-written tables: after the previous kernel of the stream
    if (teams > 1 && (!working || u0 >= u1)) return;
    const float T = tb.T;
    if (teams == 1 && tid == 0) {                                        // thread 0 takes the tickets: of the heads at the ends of this CTA's units
        Ticket* const ends[2] = {d_tickets + bh, d_tickets + divide(static_cast<uint64_t>(u1 - 1), static_cast<uint64_t>(chunks))};
        const Ticket seen[2] = {look_at_ticket(ends[0]), look_at_ticket(ends[1])};
        claim_ticket(ends[0], seen[0], tag);
        if (ends[1] != ends[0]) claim_ticket(ends[1], seen[1], tag);
    }

    float acc[8][4];                                       // [16-dim chunk][mma accumulator]
    float m = -INFINITY, l = 0.0f;                         // of head lane / 4: maximum so far, this lane's part of the sum of weights
    auto clear_acc = [&]() {
        m = -INFINITY;
        l = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    };
    clear_acc();

    // scales acc and l from maximum m to maximum `to` (per head lane / 4; accumulator column j & 1 is head (lane % 4) * 2 + (j & 1))
    auto rescale_to = [&](float to) {
        const float f = rescale(m, to);
        const float f0 = __shfl_sync(kFull, f, (lane & 3u) * 8), f1 = __shfl_sync(kFull, f, (lane & 3u) * 8 + 4);
        l *= f;
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) { acc[ch][0] *= f0; acc[ch][1] *= f1; acc[ch][2] *= f0; acc[ch][3] *= f1; }
        m = to;
    };
    // All tokens of head bh seen by this CTA are in acc.  The warps agree on the maxima and reduce in a fixed order (in rounds of
    // kAvSlots warps: warp w adds its sums to slot w mod kAvSlots, the first round by plain stores; then the slots are
    // added in slot order); then either store (this CTA owns the whole head) or hand a piece to the slot-and-ticket reduction.
    auto flush = [&](int bh) {
        if (working && (lane & 3u) == 0) max_s[warp * 8 + (lane >> 2)] = m;
        team_sync();                                   // every warp is done with its tiles: the slots lie over them
        auto top_of = [&](uint32_t head) {
            float top = max_s[first_warp * 8 + head];
            for (uint32_t w = 1; w < nw; ++w) top = fmaxf(top, max_s[(first_warp + w) * 8 + head]);
            return top;
        };
        if (working) rescale_to(top_of(lane >> 2));
        for (uint32_t first = 0; first < nw; first += kAvSlots) {
            const uint32_t w = warp - first_warp;
            if (w >= first && w < first + kAvSlots && w < nw) {
                float* slot = out_s + (w - first) * kSlotFloats;
#pragma unroll
                for (int ch = 0; ch < 8; ++ch)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int dim = ch * 16 + static_cast<int>(lane >> 2) + (j >= 2 ? 8 : 0);
                        const int head = static_cast<int>(lane & 3u) * 2 + (j & 1);
                        const float v = acc[ch][j];
                        slot[dim * 8 + head] = first ? slot[dim * 8 + head] + v : v;
                    }
                float s = l + __shfl_xor_sync(kFull, l, 1);
                s += __shfl_xor_sync(kFull, s, 2);
                if ((lane & 3u) == 0) {
                    float* at = slot + kGroup * 8 + (lane >> 2);
                    *at = first ? *at + s : s;
                }
            }
            team_sync();
        }
        const uint32_t used = min(nw, kAvSlots);
        for (int i = tid; i < static_cast<int>(kSlotFloats); i += n_threads) {
            float sum = out_s[i];
            for (uint32_t sl = 1; sl < used; ++sl) sum += out_s[sl * kSlotFloats + i];
            out_s[i] = sum;
        }
        team_sync();
        const UnitSplit split(U, G);                       // again: not held in registers through the decode
        const int c_lo = teams > 1 ? 0 : split.owner(static_cast<int64_t>(bh) * chunks);
        const int c_hi = teams > 1 ? 0 : split.owner(static_cast<int64_t>(bh + 1) * chunks - 1);
        auto store = [&](int i, float v, float weights) {
            if ((i & 7) < q_per_kv) d_out[(static_cast<size_t>(bh) * q_per_kv + (i & 7)) * kGroup + (i >> 3)] = v / weights;
        };
        if (c_lo == c_hi) {
            for (int i = tid; i < kGroup * 8; i += n_threads) store(i, out_s[i], out_s[kGroup * 8 + (i & 7)]);
        } else {
            float* mine = d_partial + static_cast<size_t>(c + bh) * kPieceFloats;
            for (int i = tid; i < kPieceFloats; i += n_threads) mine[i] = i < kGroup * 8 + 8 ? out_s[i] : top_of(i & 7);
            __threadfence();
            team_sync();
            if (tid == 0) ticket = take_ticket(&d_tickets[bh]);
            team_sync();
            if (ticket == static_cast<unsigned int>(c_hi - c_lo)) {
                __threadfence();
                const float* piece = d_partial + static_cast<size_t>(c_lo + bh) * kPieceFloats;
                const int n = c_hi - c_lo + 1;             // at most 256
                // factor of every piece and head, then the heads' sums of weights: warp h does head h (a CTA has eight warps at least)
                float *fac = out_s, *weights = out_s + n * 8;
                if (warp < 8) {
                    const float* pw = piece + kGroup * 8 + warp;
                    float top = -INFINITY, sum = 0.0f;
                    for (int k = lane; k < n; k += 32) top = fmaxf(top, __ldcg(pw + 8 + static_cast<size_t>(k) * kPieceFloats));
#pragma unroll
                    for (int o = 16; o; o >>= 1) top = fmaxf(top, __shfl_xor_sync(kFull, top, o));
                    for (int k = lane; k < n; k += 32) {
                        const float f = rescale(__ldcg(pw + 8 + static_cast<size_t>(k) * kPieceFloats), top);
                        fac[k * 8 + warp] = f;
                        sum += f * __ldcg(pw + static_cast<size_t>(k) * kPieceFloats);
                    }
#pragma unroll
                    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
                    if (lane == 0) weights[warp] = sum;
                }
                team_sync();
                for (int i = tid; i < kGroup * 2; i += n_threads) {            // four heads of a dim at a time, eight loads in flight
                    const float4* from = reinterpret_cast<const float4*>(piece) + i;
                    const float4* by = reinterpret_cast<const float4*>(fac) + (i & 1);
                    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    auto add = [&](float4 f, float4 x) { v.x += f.x * x.x; v.y += f.y * x.y; v.z += f.z * x.z; v.w += f.w * x.w; };
                    int k = 0;
                    for (; k + 8 <= n; k += 8) {
                        float4 x[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = __ldcg(from + static_cast<size_t>(k + j) * (kPieceFloats / 4));
#pragma unroll
                        for (int j = 0; j < 8; ++j) add(by[(k + j) * 2], x[j]);
                    }
                    for (; k < n; ++k) add(by[k * 2], __ldcg(from + static_cast<size_t>(k) * (kPieceFloats / 4)));
                    const float vs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) store(i * 4 + j, vs[j], weights[(i & 1) * 4 + j]);
                }
                if (tid == 0) d_tickets[bh] = 0;
            }
        }
        team_sync();
    };

    for (int n = static_cast<int>(u1 - u0); n > 0; --n) {
        const int head = bh, first_token = token, tile_base = first_token + static_cast<int>(warp - first_warp) * 32;
        const bool valid = tile_base + static_cast<int>(lane) < seq;
        if ((token += kTokens) >= seq) { token = 0; ++bh; }
        if (working) {                                     // warps without room for their arrays only help with the reductions
            uint32_t p_hi[4], p_lo[4];                     // P^T fragments (B operand): head = lane / 4, tokens (lane % 4) * 2 + {0, 1} + 8 j
            {                                              // (behind the decode, not held through it: 518 -> 541 us with 19 warps, 534 -> 562 with 16)
                const int r = static_cast<int>(lane >> 2);
                const float* srow = d_scores + (static_cast<size_t>(head) * q_per_kv + min(r, q_per_kv - 1)) * seq;
                float s[8], top = m;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int tk = tile_base + static_cast<int>(lane & 3u) * 2 + 8 * (j >> 1) + (j & 1);
                    s[j] = r < q_per_kv && tk < seq ? __ldcg(srow + tk) : -INFINITY;
                    top = fmaxf(top, s[j]);
                }
                top = fmaxf(top, __shfl_xor_sync(kFull, top, 1));
                top = fmaxf(top, __shfl_xor_sync(kFull, top, 2));
                if (__any_sync(kFull, top > m)) rescale_to(top);               // rare once a few tiles have passed
                // Probabilities enter the tensor cores as fp16 pairs (value + remainder).  Taken as they are, everything
                // below 6e-5 would sit in fp16's subnormal range (one part in a thousand at p = 3e-5); scaled by 2^15 they keep
                // 22 bits down to 2e-12, and exp(s - max) <= 1 cannot overflow.  The sum of weights carries the same factor.
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // a masked score (-inf) has weight zero, also before any finite one
                    const float p0 = s[2 * j] == -INFINITY ? 0.0f : __expf(s[2 * j] - m) * kProbScale;
                    const float p1 = s[2 * j + 1] == -INFINITY ? 0.0f : __expf(s[2 * j + 1] - m) * kProbScale;
                    l += p0 + p1;
                    const __half h0 = __float2half_rn(p0), h1 = __float2half_rn(p1);
                    const __half l0 = __float2half_rn(p0 - __half2float(h0)), l1 = __float2half_rn(p1 - __half2float(h1));
                    p_hi[j] = static_cast<uint32_t>(__half_as_ushort(h0)) | (static_cast<uint32_t>(__half_as_ushort(h1)) << 16);
                    p_lo[j] = static_cast<uint32_t>(__half_as_ushort(l0)) | (static_cast<uint32_t>(__half_as_ushort(l1)) << 16);
                }
            }
            Block cur;                                     // fetched now, prefetched into L2 one unit earlier
            ldg_block(cur, block_ptr(head, first_token));
            if (n > 1) {
                prefetch_block_l2(block_ptr(bh, token));
                // the scores of this warp's tokens in the next unit, one 128-byte line per query head: into L2 now
                const int nt = token + static_cast<int>(warp - first_warp) * 32;
                if (static_cast<int>(lane) < q_per_kv && nt < seq)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(d_scores + (static_cast<size_t>(bh) * q_per_kv + lane) * seq + nt));
            }
            decode_to_tiles<false, true>(cur, tb, tiles, T, valid);             // past the end of the row: zeros
            // Per 16-dim tile: (V tile)^T x P^T on the tensor cores.  They cut their sums off instead of rounding them, so only a tile's 32
            // tokens are summed there: error of 16 x 32 x 300 tokens (three tiles to a warp) 2.5e-7 -> 1.6e-7 of the result, of 16 x 8 x
            // 32768 2.3e-6 -> 2.0e-7; [8][32][4096][128] 141.6 -> 142.6 us.
            const uint32_t a_at = tiles + tile_byte((lane >> 4) * 8 + (lane & 7u), ((lane >> 3) & 1u) * 8);
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                uint32_t a[2][4];
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) ldmatrix_x4_trans(a[ks], a_at + ch * kTileBytes + ks * 512);     // tokens + 16: the same swizzle
                float part[4];
                mma_16816_first(part, a[0], p_hi[0], p_hi[1]);
                mma_16816(part, a[0], p_lo[0], p_lo[1]);
                mma_16816(part, a[1], p_hi[2], p_hi[3]);
                mma_16816(part, a[1], p_lo[2], p_lo[3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[ch][j] += part[j];
            }
        }
        if (n == 1 || bh != head) { flush(head); clear_acc(); }                 // the head's last unit here
    }
}


}  // namespace
