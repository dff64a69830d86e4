// ecco_decode_core.cuh -- the group decoder with the value table in registers
// Part of the one translation unit ecco_kernels.cu; included from there only.
#pragma once

// What bounds the decoding kernels is the shared-memory pipe (one wavefront per clock and SM) and the integer pipe (two
// warp instructions per clock and SM), so this decoder is laid out to spend little of both:
//  * Sixteen dequantised values per lane are 32 bytes.  They stay in eight registers as two byte planes (low bytes and
//    high bytes in rank order) and eight ranks are turned into eight fp16 values by byte permutes (map_ranks): no value
//    table in shared memory, hence one wavefront per symbol and 1-2 KB per warp less than a table lookup per value.
//  * Eight symbols per step from one 64-bit window: three words per refill, four pair-table lookups, one escape branch per
//    two lookups and one end-of-stream vote per step.  The escapes are plain branches: a warp vote in front of them costs more
//    instructions per step than the branch saves (layer of 7B shape 128.5 -> 123.2 us, batch-1 products 161.7 -> 152.4 us).
//  * The sixteen values come from a table of centroids that is already in rank order for every codebook
//    (build_rank_tables, made once per CTA from the staged image): two 16-byte loads and eight packed multiplications.
// Against the decoder with the value table in shared memory and four symbols per step (16.8 instructions, 8.2 of them on the
// integer pipe, and 5.3 wavefronts per symbol of a warp on weights, ncu): ecco_decompress over a 7B-shaped layer 137.5 -> 122.3 us,
// over a [16][8][32768][128] cache 407.4 -> 351.8 us.
namespace {

// Shared memory of a CTA, from its 1 KB-aligned base: misc words (the barrier word first: images come and go, the barrier stays), patterns
// and codebook records, then the tables of the decode and the arrays of as many warps as find room behind them, and the ID_KP table as the
// last part.  The first three fill the gap in front of the pair tables, which are aligned to the widest.  The sizes come from the image's header, so the kernels are
// launched with all the shared memory an SM has and lay themselves out once they have read it.
constexpr uint32_t kMisc = 1024;
constexpr uint32_t kSmemPat = kMisc;                                 // [64][16] fp16
constexpr uint32_t kSmemRec = kSmemPat + kPatternBytes;              // [256] x 16 B codebook records, see build_rank_tables
constexpr uint32_t kSmemPairMin = kSmemRec + kCbRecBytes;            // 7168
constexpr uint32_t kCentBytes = kMaxPatterns * kCodebooks * 32;      // centroids in rank order, fp16 [256][16]
constexpr uint32_t kBitRows = 19;                                    // 16 words of a block, three rows of scratch for the outliers
constexpr uint32_t kBitBytes = kBitRows * 128;
// A lane whose stream has ended goes on reading rows after its own: the next warp's or, behind the last warp, what lies there.  What it
// decodes is cut to zero.  Whatever bytes the tables hold, an ID_KP entry moves the position by 255 bits at most, a step by 127 (the
// sum of four entries' lengths is taken modulo 128; one symbol at a time 8 x 15) and the second window of the last step lies 63 bits
// on: the third word of it is the furthest.  So the last part of a CTA's shared memory belongs to a table that is longer than that.
constexpr uint32_t kFurthestRow = (kHeaderBits + 255 + 15 * 127 + 63) / 32 + 2;
static_assert((kFurthestRow + 1 - kBitRows) * 128 <= kKpLutBytes, "a lane that runs on stays in the CTA's shared memory");

struct DecodeTables {
    uint32_t base;          // misc area (barrier word at +0)
    uint32_t pair, kp, cent, shape;
    uint32_t warp_base;     // per-warp arrays
    uint32_t shape_bytes, pair_bytes;
    bool pairs;             // two symbols per lookup
    float T;
    uint32_t hash_lo, hash_hi;
};
__device__ __forceinline__ DecodeTables plan_decode_tables(uint32_t smem_base, const uint8_t* d_meta, bool use_pairs)
{
    const DevHeader* hd = reinterpret_cast<const DevHeader*>(d_meta);
    DecodeTables tb;
    tb.base = smem_base;
    tb.shape_bytes = min(__ldg(&hd->shape_bytes), kMaxShapes * 256u) & ~255u;     // clamped: a bad header cannot overrun shared memory
    tb.pair_bytes = use_pairs ? min(__ldg(&hd->pair_bytes), kPairBudgetBytes) & ~511u : 0u;
    const uint32_t align = min(max(__ldg(&hd->pair_align), 512u), 2u << kPairMaxBits);
    tb.pair = smem_base + kSmemPairMin;
    if (tb.pair_bytes) tb.pair = (tb.pair + align - 1u) & ~(align - 1u);
    tb.kp = smem_base + kSmemCtaBytes - kKpLutBytes;      // see kFurthestRow
    tb.cent = tb.pair + tb.pair_bytes;
    tb.shape = (tb.cent + kCentBytes + 255u) & ~255u;
    tb.warp_base = (tb.shape + tb.shape_bytes + 127u) & ~127u;
    tb.pairs = tb.pair_bytes != 0;
    tb.T = __ldg(&hd->T);
    tb.hash_lo = __ldg(&hd->hash_lo);
    tb.hash_hi = __ldg(&hd->hash_hi);
    return tb;
}
// warps of this CTA that have room for warp_bytes each (the others sit the launch out)
__device__ __forceinline__ uint32_t decode_warps(const DecodeTables& tb, uint32_t warp_bytes, uint32_t tail_bytes = 0)
{
    const uint32_t used = tb.warp_base - tb.base + kKpLutBytes + tail_bytes;
    const uint32_t room = used < kSmemCtaBytes ? kSmemCtaBytes - used : 0u;
    return min(room / warp_bytes, blockDim.x >> 5);
}
// first = false re-arms a barrier that an earlier phase initialised
__device__ __forceinline__ void issue_decode_tables(const DecodeTables& tb, const uint8_t* d_meta, bool first = true)
{
    const uint32_t bar = tb.base;
    if (threadIdx.x == 0) {
        if (first) mbar_init(bar, 1);
        const DevHeader* hd = reinterpret_cast<const DevHeader*>(d_meta);
        mbar_expect_tx(bar, kFixedTableBytes + tb.shape_bytes + tb.pair_bytes);
        bulk_g2s(tb.base + kSmemPat, d_meta + kOffPattern, kPatternBytes, bar);
        bulk_g2s(tb.base + kSmemRec, d_meta + kOffCbRec, kCbRecBytes, bar);
        bulk_g2s(tb.kp, d_meta + kOffKpLut, kKpLutBytes, bar);
        bulk_g2s(tb.shape, d_meta + kOffShapeLut, tb.shape_bytes, bar);
        if (tb.pair_bytes) bulk_g2s(tb.pair, d_meta + __ldg(&hd->off_pair), tb.pair_bytes, bar);
    }
}
// From the staged patterns and records: the centroids of every codebook in rank order, and the records rewritten in place
// as what a lane needs to know when it opens a group: { blut, plut, mask, rank of the abs-max symbol } (see LaneGroup).
// The place of the abs-max symbol holds 1.0: times the group scale it gives the magnitude of the abs-max (its sign is
// put in when a group is opened).  A row of centroids is two 16-byte halves, swapped in every second block of four rows:
// lanes that read the same half of random rows then meet eight bank groups instead of four.
__device__ __forceinline__ uint32_t cent_row(const DecodeTables& tb, uint32_t cb) { return tb.cent + cb * 32u + ((cb << 2) & 16u); }
__device__ __forceinline__ void build_rank_tables(const DecodeTables& tb)
{
    for (uint32_t cb = threadIdx.x; cb < kMaxPatterns * kCodebooks; cb += blockDim.x) {
        const uint32_t rec = tb.base + kSmemRec + cb * 16;
        const uint32_t x = lds_u32(rec), nib[2] = {lds_u32(rec + 8), lds_u32(rec + 12)};     // tables; symbol -> rank
        uint32_t c[8];
        const uint32_t pat = tb.base + kSmemPat + (cb >> 2) * 32;
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]) : "r"(pat));
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7]) : "r"(pat + 16));
        c[7] = (c[7] & 0xffffu) | 0x3c000000u;
        const uint32_t row = cent_row(tb, cb);
#pragma unroll
        for (int s = 0; s < 16; ++s) sts_u16(row ^ (((nib[s >> 3] >> ((s & 7) * 4)) & 15u) * 2), s & 1 ? c[s >> 1] >> 16 : c[s >> 1] & 0xffffu);
        const uint32_t shape = (x >> 8) & 0xffu, rot = table_rotation(shape);
        sts_v4(rec, (tb.shape + shape * 256u) | rot, (tb.pair + ((x & 0xffu) << 9)) | rot, (2u << ((x >> 16) & 15u)) - 2u, nib[1] >> 28);
    }
    __syncthreads();
}
// The whole CTA waits for its tables and builds the rest; false (CTA-uniform) if the bounded wait expired.  Then it has waited for the
// previous kernel of the stream, too: see dependency_wait.
// kGiveUp (tests): every second CTA does as if it had expired; its copies have landed.
template <bool kGiveUp = false>
__device__ __forceinline__ bool finish_decode_tables(const DecodeTables& tb, uint32_t parity = 0)
{
    bool there = bounded_wait(tb.base, parity, kWaitLimit);
    if (kGiveUp && (blockIdx.x & 1u)) {
        there = false;
        if (threadIdx.x == 0) atomicExch(&g_device_status, ECCO_ERR_DEVICE_TIMEOUT);
    }
    if (!there) { dependency_wait(); return false; }
    build_rank_tables(tb);
    return true;
}

// What a lane knows about its group.
struct LaneGroup {
    uint32_t p;             // position of the next stream bit, minus one: a window that starts one bit early has the byte
                            // offset of a 2-byte table entry in its bits 1..W
    uint32_t blut;          // shared address of the shape table, OR-ed with its rotation
    uint32_t plut, mask;    // the same for the pair table; ((1 << W) - 1) << 1
    uint32_t vlo[4], vhi[4];    // the sixteen values in rank order: low bytes, high bytes
};

// Pattern retriever and mapper (Sec. 4.2): scale byte, ID_HF, Huffman-coded ID_KP from the group's first 22 stream bits
// (hdr, first bit in bit 0), then value = fp16_rn(centroid * scale).  The product of two fp16 numbers rounded once to fp16 is
// the same number whether it is formed by one fp16 multiplication or in fp32 (where it is exact), so the packed fp16
// product is used whenever the scale is an fp16 number: 448 * 2^e finite and 2^-9 * 2^e not below fp16's last place.
__device__ __forceinline__ LaneGroup open_lane_group(uint32_t hdr, uint32_t first_bit, const DecodeTables& tb, float T)
{
    LaneGroup g;
    const uint32_t kpe = lds_u16(tb.kp + ((hdr >> (kHeaderBits - 1)) & 0x1ffeu));
    g.p = first_bit + kHeaderBits - 1u + (kpe >> 8);
    const uint32_t cb = (kpe & (kMaxPatterns - 1u)) * kCodebooks + ((hdr >> 8) & 3u);
    uint32_t top;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(g.blut), "=r"(g.plut), "=r"(g.mask), "=r"(top) : "r"(tb.base + kSmemRec + cb * 16));
    uint32_t c[8];
    const uint32_t row = cent_row(tb, cb);
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]) : "r"(row));
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7]) : "r"(row ^ 16u));
    if (T >= 3.0517578125e-5f && T <= 128.0f) {            // 2^-15 .. 2^7, uniform over the tensor
        // exact: the scale's E4M3 value by the hardware's conversion (its one code that would read as NaN is 480 here) times 2^e
        const uint32_t q = hdr & 0x7fu;
        uint32_t m;
        asm("{\n\t.reg .b16 b;\n\tcvt.u16.u32 b, %1;\n\tcvt.rn.f16x2.e4m3x2 %0, b;\n\t}" : "=r"(m) : "r"(q * 0x101u));
        if (q == 0x7fu) m = 0x5f805f80u;
        const __half2 s2 = __hmul2(*reinterpret_cast<const __half2*>(&m), __float2half2_rn(T));
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const __half2 v = __hmul2(*reinterpret_cast<const __half2*>(&c[j]), s2);
            c[j] = *reinterpret_cast<const uint32_t*>(&v);
        }
    } else {
        const float s = fp8_to_float(hdr & 0x7fu) * T;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&c[j]));
            const __half2 v = __floats2half2_rn(f.x * s, f.y * s);
            c[j] = *reinterpret_cast<const uint32_t*>(&v);
        }
    }
    const uint32_t sign = (hdr & 0x80u) << ((top & 3u) * 8);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        g.vlo[j] = prmt(c[2 * j], c[2 * j + 1], 0x6420u);
        g.vhi[j] = prmt(c[2 * j], c[2 * j + 1], 0x7531u) ^ ((top >> 2) == static_cast<uint32_t>(j) ? sign : 0u);
    }
    return g;
}
// 64-byte block: its words go to the lane's column of the transposed bit-stream array (bits = address of its row 0)
__device__ __forceinline__ LaneGroup open_block(const Block& blk, uint32_t bits, const DecodeTables& tb, float T)
{
#pragma unroll
    for (int i = 0; i < 16; ++i) sts_u32(bits + i * 128, blk.w[i]);
    return open_lane_group(blk.w[0], 0u, tb, T);
}

// Eight ranks (nibbles, first symbol lowest) -> eight fp16 values, two to a word.  A byte permute selects among eight
// bytes with three bits of a nibble, so both halves of a plane are read and the ranks' top bits choose between them.
__device__ __forceinline__ void map_ranks(const LaneGroup& g, uint32_t ranks, uint32_t (&v)[4])
{
    const uint32_t sel = ranks & 0x77777777u, pick = ((ranks >> 1) & 0x44444444u) | 0x32103210u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t s = sel >> (16 * h), k = pick >> (16 * h);
        const uint32_t lo = prmt(prmt(g.vlo[0], g.vlo[1], s), prmt(g.vlo[2], g.vlo[3], s), k);
        const uint32_t hi = prmt(prmt(g.vhi[0], g.vhi[1], s), prmt(g.vhi[2], g.vhi[3], s), k);
        v[2 * h] = prmt(lo, hi, 0x5140u);
        v[2 * h + 1] = prmt(lo, hi, 0x7362u);
    }
}

// table entries: the tables are read-only while a CTA decodes, so the compiler may move these loads
__device__ __forceinline__ uint32_t lds_shape(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds_pair(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ bool warp_any(bool x) { return __any_sync(0xffffffffu, x); }

// keeps the first n_ok of eight values and zeroes the rest
__device__ __forceinline__ void cut_values(uint32_t (&v)[4], int n_ok)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t keep;                                     // shl: amounts above 31 give zero
        asm("shl.b32 %0, -1, %1;" : "=r"(keep) : "r"(max(16 * n_ok - 32 * k, 0)));
        v[k] &= ~keep;
    }
}

// decode_group (below) symbol by symbol through the shape tables, for images without pair tables and for kernels whose arrays leave no room for
// them: twice the lookups (3.4 wavefronts per symbol of a warp instead of 1.7).
struct NoRefill {};
template <uint32_t kEndBit, int kFreeSteps, class Sink, class Refill = NoRefill>
__device__ __forceinline__ uint32_t decode_group_by_one(LaneGroup& g, uint32_t bits, Sink&& sink, Refill&& refill = {})
{
    bool complete = true;
    uint32_t q = g.p + 1u;
    auto step = [&](int i, auto tested) {
        constexpr bool kTest = decltype(tested)::value;
        const uint32_t row = bits + (q >> 5) * 128;        // past its end a lane reads whatever follows: see kFurthestRow
        const uint32_t w0 = lds_u32(row), w1 = lds_u32(row + 128), w2 = lds_u32(row + 256);
        const uint32_t lo = __funnelshift_r(w0, w1, q), hi = __funnelshift_r(w1, w2, q);
        uint32_t e[8], x = lo, n = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (j == 4) { x = __funnelshift_rc(lo, hi, n); q += n; n = 0; }    // up to 32 bits
            e[j] = lds_shape(g.blut ^ ((x >> n) & 0xffu));
            n += e[j] >> 4;
        }
        // ranks are the low nibbles: even and odd symbols side by side in bytes (multiply-adds: the integer pipe is the busier one)
        const uint32_t ev = (e[6] * 256u + e[4]) * 65536u + (e[2] * 256u + e[0]), od = (e[7] * 256u + e[5]) * 65536u + (e[3] * 256u + e[1]);
        const uint32_t ranks = (ev & 0x0f0f0f0fu) | ((od * 16u) & 0xf0f0f0f0u);
        q += n;
        bool cutting = false;
        int n_ok = 8;
        if (kTest && warp_any(q > kEndBit)) {
            cutting = true;                                // some lane's stream ends in this step: how many of its codewords end by then
            uint32_t at = q;
#pragma unroll
            for (int j = 7; j >= 0; --j) {
                if (at > kEndBit) n_ok = j;                // positions only grow
                at -= e[j] >> 4;
            }
            complete = complete && n_ok == 8;
        }
        sink(i, ranks, cutting, n_ok);
        if constexpr (!cuda::std::is_same_v<cuda::std::remove_reference_t<Refill>, NoRefill>) {
            uint32_t p = q - 1u;
            refill(p);
            q = p + 1u;
        }
    };
#pragma unroll 1
    for (int i = 0; i < kFreeSteps; i += 2) { step(i, cuda::std::false_type{}); step(i + 1, cuda::std::false_type{}); }
#pragma unroll 1
    for (int i = kFreeSteps; i < 16; i += 2) { step(i, cuda::std::true_type{}); step(i + 1, cuda::std::true_type{}); }
    g.p = q - 1u;
    return complete ? q : 0u;
}

// Decodes the 128 symbols of the lane's group, eight per step (Sec. 4.2, Huffman decode), and hands every step's ranks (nibbles,
// first symbol lowest) to sink(step, ranks, cutting, n_ok).  A codeword that would cross the end bit ends the group: that and
// all later positions are clipped.  cutting (uniform over the warp) says that some lane may have clipped positions in this step, n_ok how
// many of the lane's eight are there (8 if not cutting).  Returns the end bit if all 128 fitted, else 0.  Must be called by all 32 lanes of
// the warp.
// What lies behind the end bit is arbitrary: a codeword that ends by then does not depend on it, and one that does not ends behind it
// whatever it looks like there.
// kEndBit: that bit, counted from the lane's staged stream.  kFreeSteps: that many leading steps carry no end test; the caller
// guarantees that the stream cannot end in them.
// pairs = false (uniform): decode_group_by_one.
// refill(p): called after every step, for a lane that holds a part of its stream only; it may move p, which is LaneGroup::p.
template <uint32_t kEndBit, int kFreeSteps, class Sink, class Refill = NoRefill>
__device__ __forceinline__ uint32_t decode_group(LaneGroup& g, uint32_t bits, bool pairs, Sink&& sink, Refill&& refill = {})
{
    if (!pairs) return decode_group_by_one<kEndBit, kFreeSteps>(g, bits, sink, refill);
    constexpr uint32_t kLastRow = kEndBit / 32;
    bool complete = true;
    // second symbol of an escape entry: its codeword starts 1 + (length of the first) bits into win
    auto resolve = [&](uint32_t e, uint32_t win) {
        const uint32_t b = lds_u8(g.blut ^ ((win >> (1u + (e & 15u))) & 0xffu));
        return (e & 0x078fu) + (b >> 4) + ((b & 15u) << 11);
    };
    auto step = [&](int i, auto tested) {
        constexpr bool kTest = decltype(tested)::value;
        const uint32_t row = bits + (g.p >> 5) * 128;      // past its end a lane reads whatever follows: see kFurthestRow
        const uint32_t w0 = lds_u32(row), w1 = lds_u32(row + 128), w2 = lds_u32(row + 256);
        const uint32_t lo = __funnelshift_r(w0, w1, g.p), hi = __funnelshift_r(w1, w2, g.p);
        // an entry's low bits are the length of its codewords; funnel shifts take their amount modulo 32
        uint32_t e0 = lds_pair(g.plut ^ (lo & g.mask));
        uint32_t x1 = __funnelshift_r(lo, hi, e0);
        uint32_t e1 = lds_pair(g.plut ^ (x1 & g.mask));
        uint32_t n01 = e0 + e1, x2 = __funnelshift_r(lo, hi, n01);
        if ((e0 | e1) & 0x8000u) {
            if (e0 & 0x8000u) {
                e0 = resolve(e0, lo);
                x1 = __funnelshift_r(lo, hi, e0);
                e1 = lds_pair(g.plut ^ (x1 & g.mask));
            }
            if (e1 & 0x8000u) e1 = resolve(e1, x1);
            n01 = e0 + e1;
            x2 = __funnelshift_rc(lo, hi, n01 & 63u);      // up to 32 bits here
        }
        uint32_t e2 = lds_pair(g.plut ^ (x2 & g.mask));
        uint32_t x3 = __funnelshift_r(x2, 0u, e2);
        uint32_t e3 = lds_pair(g.plut ^ (x3 & g.mask));
        if ((e2 | e3) & 0x8000u) {
            // long codewords: the third pair's window is fetched again, the two pairs may need 33 bits of it
            const uint32_t q = g.p + (n01 & 63u);
            const uint32_t r2 = bits + (q >> 5) * 128;
            const uint32_t y0 = lds_u32(r2), y1 = lds_u32(r2 + 128), y2 = lds_u32(r2 + 256);
            const uint32_t l2 = __funnelshift_r(y0, y1, q), h2 = __funnelshift_r(y1, y2, q);
            if (e2 & 0x8000u) {
                e2 = resolve(e2, l2);
                x3 = __funnelshift_r(l2, h2, e2);
                e3 = lds_pair(g.plut ^ (x3 & g.mask));
            }
            if (e3 & 0x8000u) e3 = resolve(e3, __funnelshift_r(l2, h2, e2));
        }
        const uint32_t n = (n01 + e2 + e3) & 0x7fu;
        // two entries side by side and doubled (multiply-adds: the integer pipe is the busier one): ranks in bytes 1 and 3
        const uint32_t e01 = e1 * 0x10000u + e0, e23 = e3 * 0x10000u + e2;
        const uint32_t ranks = prmt(e01 * 2u, e23 * 2u, 0x7531u);
        bool cutting = false;
        int n_ok = 8;
        if (kTest && warp_any(g.p + n >= kEndBit)) {
            // some lane's stream ends in this step: how many of its codewords end by then
            cutting = true;
            const int room = static_cast<int>(kEndBit - 1u) - static_cast<int>(g.p);
            const int c0 = e0 & 31u, c1 = n01 & 63u, c2 = (n01 + e2) & 63u, c3 = n;
            const int start = c0 > room ? 0 : c1 > room ? c0 : c2 > room ? c1 : c2;       // of the first pair that does not fit
            const uint32_t q = g.p + 1u + start, r = bits + min(q >> 5, kLastRow) * 128;
            const int first = lds_u8(g.blut ^ (__funnelshift_r(lds_u32(r), lds_u32(r + 128), q) & 0xffu)) >> 4;
            n_ok = (start + first <= room ? 1 : 0) + (c0 <= room ? 2 : 0) + (c1 <= room ? 2 : 0) + (c2 <= room ? 2 : 0);
            if (c3 <= room) n_ok = 8;
            else complete = false;
        }
        g.p += n;
        sink(i, ranks, cutting, n_ok);
        if constexpr (!cuda::std::is_same_v<cuda::std::remove_reference_t<Refill>, NoRefill>) refill(g.p);
    };
#pragma unroll 1
    for (int i = 0; i < kFreeSteps; i += 2) { step(i, cuda::std::false_type{}); step(i + 1, cuda::std::false_type{}); }
#pragma unroll 1
    for (int i = kFreeSteps; i < 16; i += 2) { step(i, cuda::std::true_type{}); step(i + 1, cuda::std::true_type{}); }
    return complete ? g.p + 1u : 0u;
}
constexpr int kBlockFreeSteps = 6;     // the indices of a block start at bit 22 at the latest: 6 steps end by bit 22 + 6 * 64 = 406

// outlier field j of a block (Sec. 3.2: 7-bit location + FP8 value): bits [512-15(j+1), 512-15j)
__device__ __forceinline__ uint32_t pad_field(uint32_t bits, int j)
{
    const uint32_t pos = kBlockBits - kPadBits * (j + 1), row = bits + (pos >> 5) * 128;
    return __funnelshift_r(lds_u32(row), lds_u32(row + 128), pos) & 0x7fffu;
}
__device__ __forceinline__ int pads_of(uint32_t end) { return end ? min(kMaxPads, static_cast<int>((kBlockBits - end) / kPadBits)) : 0; }

// The outliers of a warp's 32 groups, one per lane.  The groups of a cache have 37 of them together, but one of them usually has
// eight, so lanes that walk their own lists leave most of the warp idle; here the lists are joined and every lane takes one
// outlier, 32 at a time (scores of an [8][32][4096][128] cache with the values' kernel behind them 257.4 -> 250.5 us).  On weights, 16
// together and two or three at most, walking is the cheaper way (batch-1 products of a layer 162.7 against 164.7 us).  A round ends with a whole group,
// so that outliers of one group at the same place (which only a corrupt block has) meet in one round and the last one wins.
//   list     shared address of 64 bytes of scratch
//   take(slot, owner, field, valid)  called by lane `slot` for an outlier of lane owner's group; not valid: overridden by another
//   done(first, count)        called by all lanes after a round: slots first .. first + count - 1 were this lane's (count 0: none)
template <class Take, class Done>
__device__ __forceinline__ void deal_outliers(uint32_t bits, uint32_t list, int n_pad, Take&& take, Done&& done)
{
    constexpr uint32_t kFull = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t upto = n_pad;                                 // outliers of this lane and those before it
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, upto, o);
        if (lane >= static_cast<uint32_t>(o)) upto += v;
    }
    const uint32_t total = __shfl_sync(kFull, upto, 31), from = upto - n_pad;
    for (uint32_t base = 0; base < total;) {               // at least 17 of the rest fit into a round
        const bool mine = from >= base && upto <= base + 32u;
        const uint32_t next = __reduce_max_sync(kFull, mine ? upto : 0u);
        if (mine)
            for (int j = 0; j < n_pad; ++j) sts_u16(list + (from - base + j) * 2, (lane << 4) | j);
        __syncwarp();
        uint32_t owner = 0, field = 0, key = 0x10000u | lane;
        if (lane < next - base) {
            const uint32_t w = lds_u16(list + lane * 2);
            owner = w >> 4;
            field = pad_field(bits + (owner - lane) * 4, w & 15u);
            key = (owner << 7) | (field & 127u);
        }
        const uint32_t same = __match_any_sync(kFull, key);
        if (lane < next - base) take(lane, owner, field, ((same >> lane) >> 1) == 0u);
        __syncwarp();
        done(from - base, mine ? n_pad : 0);
        __syncwarp();
        base = next;
    }
}

}  // namespace
