// bwt_bucket.cu -- the suffix sort of almost every block: the rotations in
// order of their first 44 code bits by one scatter into buckets that fit
// shared memory, then the few ties by further code bits.
//
// Keys. Each block gets order-preserving (alphabetic) prefix codes of the
// byte values, split at the weighted median of a byte sample: one for a
// key's first byte, one for bytes after a zero byte and one for bytes after
// any other (in the (lo, hi) streams that tells the two halves apart). Two
// rotations compare like their concatenated codes, bit by bit, since equal
// bytes so far mean the same code for the next one. 44 code bits reach 9 to
// 16 bytes of the streams this library codes and leave 0.1 to 1 % of their
// rotations tied (8 plain bytes: 48 %). A word holds the 44 key bits above
// the 20-bit rotation start.
//
// Buckets. A sample of the 16-bit key prefixes gives each block at most
// kBuckets splitters with about kBucketTarget rotations between them; a
// prefix with more than that is a bucket of its own. The words are written to
// their buckets (order inside a bucket is free), each bucket is sorted in
// shared memory by 8192 linear sub-bins and a count of the smaller words of
// the sub-bin, and the last column goes out. Groups of equal keys go to a
// list, and one thread per group orders it by the next 44 code bits, and so
// on, read from the block's bytes.
//
// What bounds it: two reads of the bytes, 8 B written and read per rotation
// and one byte gathered per rotation (L2); against the 8 LSD passes over
// 12-byte pairs it replaces (192 B per rotation), a rank scatter and two
// doubling rounds. 12 2040 x 2040 frames (139 blocks, 99 M rotations): plan
// 0.04, counts 0.47, scatter 0.73, buckets 1.45 ms and few ties, where keys,
// passes and rounds took 8.5 ms; one 195 x 195 frame 0.09 ms against 0.26.
//
// Blocks this cannot finish are flagged for bwt.cu: a bucket above the
// largest class's words, in a small pass above the one below (kFlagOver: all
// its words take LSD passes), or groups
// longer than kTieGroup, still tied after kTieRounds more keys, or of a block
// with many that are still tied after a few (kFlagTied: prefix doubling from
// the bytes the groups share).
#include <algorithm>
#include <climits>

#include "lfc_common.cuh"

namespace lfc {

constexpr int kEncThreads = 512;
constexpr int kEncPer = 16;                          // positions of a thread
constexpr int kEncTile = kEncThreads * kEncPer;      // 8192
constexpr int kEncLook = 48;                         // bytes past the tile a key can reach (1 bit each at least)
constexpr int kEncBytes = kEncTile + kEncLook;
constexpr int kEncWords = kEncBytes * kCodeMax / 32 + 8;  // bit stream of a tile, zero padded
constexpr int kPrefixBits = 16;
constexpr int kBucketTarget = 2048;
// size classes of buckets: words, threads, CTAs per SM (shared memory)
constexpr int kBucketClasses = kRsBucketClasses;
__device__ constexpr int kBucketCap[kBucketClasses] = {4096, 8192, 24576};
constexpr int kBucketThreads[kBucketClasses] = {512, 512, 1024};
constexpr int kBucketCtas[kBucketClasses] = {2, 2, 1};
constexpr int kSubBins = 8192;  // 16-bit counters
constexpr int kSubCost = 256;    // words a word is compared with, on average, up to which counting beats the merge network
constexpr int64_t kSmallPass = 4 << 20;  // words of a pass below which 8 LSD passes take less than 0.23 ms
// Frames have few ties and take the same time with any of these. Blocks of
// strings of some hundred bytes several times over decide: groups of up to 8 in
// a thread took up to 40 % longer than of up to 4 (of up to 2 the same); 12 keys
// the same as 24, 48 a tenth less where they resolve the ties (200-byte strings)
// and up to a third longer where they do not (3000-byte strings).
constexpr int kTieGroup = 32;   // longest group ordered by further keys (a warp's lanes)
constexpr int kTieShort = 4;    // longest one that a single thread orders
constexpr int kTieRounds = 24;  // keys a group is compared by
constexpr int kTieFew = 4;      // keys after which the groups still tied are counted, per block
constexpr int kTieMany = 64, kTieShare = 256;  // most of them: kTieMany, or one per kTieShare rotations
constexpr int kTieWaves = 4;    // long groups per warp up to which none is given up
constexpr int kTables = 3;      // codes: after a zero byte, after another byte, first byte of a key
constexpr int kFirst = 512;     // where the last one starts
static_assert(kEncLook >= kKeyBits, "a key reaches at most one byte per bit");
static_assert(kCodeMax <= kPrefixBits, "a bucket of one prefix shares at least one whole byte");

// -------------------------------------------------------------- the code
// One CTA per block: byte sample -> code; prefix sample -> splitters.
constexpr int kPlanThreads = 1024;
constexpr int kPlanHistWords = 32768 + 1024;  // 65536 16-bit counters, one pad word per 32
constexpr size_t kPlanSmem = (size_t)kPlanHistWords * 4;

// Code of byte s: walk down from [0, 256); a node [l, r) splits where the
// weight left of the split is nearest half its weight, moved so that both
// halves still fit the remaining depth.
__device__ __forceinline__ uint32_t alphabetic_code(const uint32_t *cum, int s) {
    int l = 0, r = 256, depth = 0;
    uint32_t code = 0;
    while (r - l > 1) {
        const int cap = 1 << (kCodeMax - depth - 1);
        int a = max(l + 1, r - cap);
        const int lo = a;
        int b = min(r - 1, l + cap);
        const uint32_t t = cum[l] + cum[r];
        while (a < b) {  // first split at or past half the weight
            const int mid = (a + b) >> 1;
            if (2 * cum[mid] >= t) b = mid; else a = mid + 1;
        }
        if (a > lo && 2 * cum[a] >= t && t - 2 * cum[a - 1] <= 2 * cum[a] - t) a--;
        if (s < a) { r = a; code <<= 1; } else { l = a; code = (code << 1) | 1u; }
        depth++;
    }
    return ((uint32_t)depth << 16) | code;
}

__global__ void __launch_bounds__(kPlanThreads) bwt_plan_kernel(const BlockState *__restrict__ st, const uint8_t *__restrict__ rle_all,
                                                                BwtCode *__restrict__ codes, uint32_t *__restrict__ bcount,
                                                                int32_t *__restrict__ bflag, int32_t *__restrict__ bdeep,
                                                                int32_t *__restrict__ rs, int clear_sticky) {
    extern __shared__ __align__(16) uint32_t h16[];
    __shared__ uint32_t hist[512], cum[kTables * 256 + 1], code[kTables * 256];
    __shared__ uint32_t shu[33];
    __shared__ int shi[33];
    const int b = blockIdx.x, t = threadIdx.x;
    const int m = st[b].m;
    const uint8_t *rle = rle_all + (size_t)b * kBlockCap;
    BwtCode &C = codes[b];
    if (b == 0 && t == 0) {  // a new suffix sort: no wait has given up, nothing is flagged or queued
        rs[kRsTied] = rs[kRsTiedMax] = rs[kRsAbort] = 0;
        rs[kRsH] = kBlockCap;  // the least depth of the groups left tied, see leave_tied
        rs[kRsRound] = rs[kRsLongGroup] = 0;
        rs[kRsFlagged] = rs[kRsOver] = rs[kRsTies] = rs[kRsTiesLong] = 0;
        for (int i = 0; i < kBucketClasses; i++) rs[kRsBucketQueue + i] = rs[kRsBucketItems + i] = 0;
        if (clear_sticky) rs[kRsSticky] = 0;
    }
    if (t == 0) bflag[b] = bdeep[b] = 0;
    if (t < 512) hist[t] = 0;
    for (int i = t; i < kPlanHistWords / 4; i += kPlanThreads) reinterpret_cast<uint4 *>(h16)[i] = make_uint4(0, 0, 0, 0);
    for (int i = t; i < kBuckets; i += kPlanThreads) bcount[(size_t)b * kBuckets + i] = 0;
    __syncthreads();
    // byte sample: at most 1024 16-byte pieces spread over the block
    const int nv = m >> 4, vstep = (nv + kPlanThreads - 1) / kPlanThreads;
    for (int q = t; q * vstep < nv; q += kPlanThreads) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(rle) + (size_t)q * vstep);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t prev = w[0] & 255u;
#pragma unroll
        for (int k = 1; k < 16; k++) {
            const uint32_t x = (w[k >> 2] >> (8 * (k & 3))) & 255u;
            atomicAdd(&hist[(prev ? 256u : 0u) + x], 1u);
            prev = x;
        }
    }
    __syncthreads();
    {   // weights 16 x count + 1: a byte the sample missed still has a code
        uint32_t wt = 0;
        if (t < 512) wt = hist[t] * 16u + 1u;
        else if (t < kTables * 256) wt = (hist[t - 512] + hist[t - 256]) * 16u + 1u;
        uint32_t total;
        const uint32_t ex = block_excl_sum<uint32_t>(wt, shu, &total);
        if (t < kTables * 256) cum[t] = ex;  // a table's sums start where the one before ends
        if (t == 0) cum[kTables * 256] = total;
    }
    __syncthreads();
    if (t < kTables * 256) {
        code[t] = alphabetic_code(cum + (t & ~255), t & 255);
        C.code[t] = (uint16_t)((code[t] >> 16 << 12) | (code[t] & 0xFFFu));
    }
    __syncthreads();
    // prefix sample: one rotation of every step, at a scrambled place (a fixed
    // one would follow the (lo, hi) alternation of the stream). The first 12
    // bytes of four rotations are loaded together.
    const int step = max(1, m >> 14), ns = (m + step - 1) / step;
    for (int q0 = t; q0 < ns; q0 += 4 * kPlanThreads) {
        int at[4];
        uint32_t w[4][3];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int q = q0 + i * kPlanThreads;
            at[i] = q < ns ? min(m - 1, q * step + (int)(((uint32_t)q * 2654435761u >> 8) % (uint32_t)step)) : -1;
            const int a4 = at[i] & ~3;
            const bool in = at[i] >= 0 && a4 + 12 <= m;
#pragma unroll
            for (int k = 0; k < 3; k++) w[i][k] = in ? __ldg(reinterpret_cast<const uint32_t *>(rle + a4) + k) : 0u;
            if (at[i] >= 0 && !in)  // the block's end: the bytes one by one, cyclic
                for (int k = 0; k < 12; k++) w[i][k >> 2] |= (uint32_t)rle[(a4 + k) % m] << (8 * (k & 3));
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            if (at[i] < 0) continue;
            int k = at[i] & 3, bits = 0;
            uint32_t acc = 0, tab = kFirst;
            while (bits < kPrefixBits) {
                uint32_t x;
                if (k < 12) x = ((k < 4 ? w[i][0] : k < 8 ? w[i][1] : w[i][2]) >> (8 * (k & 3))) & 255u;
                else x = rle[((at[i] & ~3) + k) % m];
                const uint32_t c = code[tab + x];
                const int l = (int)(c >> 16);
                acc = (acc << l) | (c & 0xFFFFu);
                bits += l;
                tab = x ? 256u : 0u;
                k++;
            }
            const uint32_t p = acc >> (bits - kPrefixBits), h = p >> 1;
            atomicAdd(&h16[h + (h >> 5)], 1u << (16 * (p & 1)));
        }
    }
    __syncthreads();
    // thread t: prefixes 64 t .. 64 t + 63 (words 33 t .. 33 t + 31). A bucket
    // starts at a prefix when the running count crosses a multiple of the
    // target, and around every prefix that exceeds the target by itself.
    const uint32_t *hw = h16 + 33 * t;
    uint32_t sum = 0;
#pragma unroll 8
    for (int i = 0; i < 32; i++) sum += (hw[i] & 0xFFFFu) + (hw[i] >> 16);
    const uint32_t ex = block_excl_sum<uint32_t>(sum, shu, nullptr);
    const uint32_t target = max(1u, (uint32_t)(kBucketTarget / step));
    const uint32_t before = t > 0 ? h16[33 * t - 2] >> 16 : 0u;  // the count of prefix 64 t - 1
    uint64_t flags = t == 0 ? 1u : 0u;
    {
        uint32_t cumc = ex, prev = before;
        uint32_t next = ((ex - before) / target + 1) * target;  // the multiple the running count crosses next
#pragma unroll 4
        for (int i = 0; i < 64; i++) {
            const uint32_t c = (hw[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
            bool flag = max(c, prev) > target;
            if (cumc >= next) {
                flag = true;
                next = (cumc / target + 1) * target;
            }
            flags |= (uint64_t)flag << i;
            prev = c;
            cumc += c;
        }
    }
    int total;
    const int base = block_excl_sum<int>(__popcll(flags), shi, &total);
#pragma unroll
    for (int i = 0; i < 64; i += 16)
        C.base12[4 * t + (i >> 4)] = (uint16_t)min(base + __popcll(flags & ((2ull << i) - 1)) - 1, kBuckets - 1);
    for (int id = base; flags; flags &= flags - 1, id++)
        if (id < kBuckets) C.split[id] = (uint16_t)(64 * t + __ffsll((long long)flags) - 1);
    if (t == 0) {
        const int nb = min(total, kBuckets);
        C.nb = nb;
        C.base12[4096] = (uint16_t)(nb - 1);
    }
}

// ------------------------------------------------------------ tile encoding
struct EncTile {
    __align__(16) uint8_t by[kEncBytes + 16];
    uint32_t bits[kEncWords];
    uint32_t prev;  // the byte before the tile
};

// Splitter tables in shared memory: base[p >> 4] = first bucket of the 12-bit
// prefix | first bucket of the next one << 16.
struct Splitters {
    uint32_t base[4096];
    __align__(16) uint16_t split[kBuckets];
};

__device__ __forceinline__ int bucket_of(uint32_t p16, const Splitters &P) {
    const uint32_t be = P.base[p16 >> 4];
    int k = (int)(be & 0xFFFFu);
    const int e = (int)(be >> 16);
    while (k < e && P.split[k + 1] <= p16) k++;
    return k;
}

__device__ __forceinline__ void load_tables(const BwtCode &C, uint16_t *code, Splitters &P) {
    for (int i = threadIdx.x; i < kTables * 256 / 8; i += blockDim.x)
        reinterpret_cast<uint4 *>(code)[i] = reinterpret_cast<const uint4 *>(C.code)[i];
    for (int i = threadIdx.x; i < 4096; i += blockDim.x) P.base[i] = (uint32_t)C.base12[i] | ((uint32_t)C.base12[i + 1] << 16);
    for (int i = threadIdx.x; i < kBuckets / 8; i += blockDim.x)
        reinterpret_cast<uint4 *>(P.split)[i] = reinterpret_cast<const uint4 *>(C.split)[i];
}

// Appends 16 codes (length << 12 | code, two per word) to the zeroed bit
// stream at bit o (most significant bit first); the first and last word are
// shared with neighbours.
__device__ __forceinline__ void put_codes(const uint32_t (&c2)[kEncPer / 2], uint32_t *bits, uint32_t o) {
    uint32_t w = o >> 5;
    int nb = (int)(o & 31);
    uint64_t acc = 0;
    bool first = true;
#pragma unroll
    for (int q = 0; q < kEncPer; q++) {
        const uint32_t c = (c2[q >> 1] >> (16 * (q & 1))) & 0xFFFFu;
        const int l = (int)(c >> 12);
        acc |= (uint64_t)(c & 0xFFFu) << (64 - nb - l);
        nb += l;
        if (nb >= 32) {
            const uint32_t v = (uint32_t)(acc >> 32);
            if (first) atomicOr(&bits[w], v); else bits[w] = v;
            first = false;
            acc <<= 32;
            nb -= 32;
            w++;
        }
    }
    if (nb > 0) atomicOr(&bits[w], (uint32_t)(acc >> 32));
}

// The codes of 16 bytes after the byte prev; returns their bits.
__device__ __forceinline__ uint32_t get_codes(const uint4 &v4, uint32_t prev, const uint16_t *code, uint32_t (&c2)[kEncPer / 2]) {
    const uint32_t w[4] = {v4.x, v4.y, v4.z, v4.w};
    uint32_t sum = 0;
#pragma unroll
    for (int q = 0; q < kEncPer; q += 2) {
        const uint32_t x = (w[q >> 2] >> (8 * (q & 3))) & 255u, y = (w[q >> 2] >> (8 * (q & 3) + 8)) & 255u;
        const uint32_t a = code[(prev ? 256u : 0u) + x], b = code[(x ? 256u : 0u) + y];
        c2[q >> 1] = a | (b << 16);
        sum += (a >> 12) + (b >> 12);
        prev = y;
    }
    return sum;
}

// Bit stream of positions [t0, t0 + kEncBytes) (cyclic) of a block in E;
// returns the bit offset of this thread's 16 positions, their bytes and their
// codes. The tables must be loaded; syncs.
__device__ __forceinline__ uint32_t encode_tile(const uint8_t *rle, int m, int t0, const uint16_t *code, EncTile &E, uint32_t *sh,
                                                uint4 &v4, uint32_t (&c2)[kEncPer / 2]) {
    const int t = threadIdx.x;
    if (t0 + kEncBytes <= m) {
        const uint4 *src = reinterpret_cast<const uint4 *>(rle + t0);
        for (int i = t; i < kEncBytes / 16; i += kEncThreads) reinterpret_cast<uint4 *>(E.by)[i] = __ldg(src + i);
    } else {
        for (int i = t; i < kEncBytes; i += kEncThreads) E.by[i] = rle[(t0 + i) % m];
    }
    if (t == 0) E.prev = rle[t0 == 0 ? m - 1 : t0 - 1];
    for (int i = t; i < kEncWords; i += kEncThreads) E.bits[i] = 0;
    __syncthreads();
    uint32_t total;
    const uint4 *by4 = reinterpret_cast<const uint4 *>(E.by);
    v4 = by4[t];
    const uint32_t o = block_excl_sum<uint32_t>(get_codes(v4, t ? E.by[kEncPer * t - 1] : E.prev, code, c2), sh, &total);
    put_codes(c2, E.bits, o);
    if (t < kEncLook / kEncPer) {
        uint32_t at = total, x2[kEncPer / 2];
        for (int i = 0; i <= t; i++) {
            const uint32_t l = get_codes(by4[kEncThreads + i], E.by[kEncTile + kEncPer * i - 1], code, x2);
            if (i < t) at += l;
        }
        put_codes(x2, E.bits, at);
    }
    __syncthreads();
    return o;
}

// The bit stream from bit o on as a window of 96 bits (the top 64 valid),
// refilled a word at a time.
struct BitWindow {
    const uint32_t *bits;
    uint32_t a, b, c, next;
    int off;  // bits of a already consumed
    __device__ __forceinline__ BitWindow(const uint32_t *bits_, uint32_t o) : bits(bits_), next((o >> 5) + 3), off((int)(o & 31)) {
        a = bits[o >> 5];
        b = bits[(o >> 5) + 1];
        c = bits[(o >> 5) + 2];
    }
    __device__ __forceinline__ uint32_t hi() const { return __funnelshift_l(b, a, off); }
    __device__ __forceinline__ uint32_t lo() const { return __funnelshift_l(c, b, off); }
    __device__ __forceinline__ void skip(uint32_t l) {
        off += (int)l;
        if (off >= 32) {
            off -= 32;
            a = b;
            b = c;
            c = bits[next++];
        }
    }
};

// Key bits of position q of a thread: the first byte's own code, then the
// stream behind it (W stands on the position's code and moves behind it).
__device__ __forceinline__ uint64_t key_bits(BitWindow &W, const uint4 &v4, const uint32_t (&c2)[kEncPer / 2], int q,
                                             const uint16_t *code) {
    const uint32_t w4[4] = {v4.x, v4.y, v4.z, v4.w};
    const uint32_t f = code[kFirst + ((w4[q >> 2] >> (8 * (q & 3))) & 255u)];
    W.skip((c2[q >> 1] >> (16 * (q & 1) + 12)) & 15u);
    const uint32_t a = W.hi(), b = W.lo(), l = f >> 12;
    return ((uint64_t)__funnelshift_r(a, f & 0xFFFu, l) << 32) | __funnelshift_r(b, a, l);
}

// ------------------------------------------------------- count, offsets
// Words per bucket, a tile per CTA (0.47 ms for 99 M rotations: every
// position's 16 prefix bits are looked up as the scatter does again; keeping
// them would cost 2 B written and read per rotation).
__global__ void __launch_bounds__(kEncThreads) bwt_count_kernel(const BlockState *__restrict__ st, const uint8_t *__restrict__ rle_all,
                                                                const BwtCode *__restrict__ codes, uint32_t *__restrict__ bcount) {
    __shared__ EncTile E;
    __shared__ Splitters P;
    __shared__ uint32_t sh[33], cnt[kBuckets];
    __shared__ __align__(16) uint16_t code[kTables * 256];
    const int b = blockIdx.y, t0 = blockIdx.x * kEncTile;
    const int m = st[b].m;
    if (t0 >= m) return;
    load_tables(codes[b], code, P);
    for (int i = threadIdx.x; i < kBuckets; i += kEncThreads) cnt[i] = 0;
    __syncthreads();
    uint4 v4;
    uint32_t c2[kEncPer / 2];
    BitWindow W(E.bits, encode_tile(rle_all + (size_t)b * kBlockCap, m, t0, code, E, sh, v4, c2));
    const int i0 = t0 + kEncPer * (int)threadIdx.x;
#pragma unroll
    for (int q = 0; q < kEncPer; q++) {
        const uint64_t k = key_bits(W, v4, c2, q, code);
        if (i0 + q < m) atomicAdd(&cnt[bucket_of((uint32_t)(k >> 48), P)], 1u);
    }
    __syncthreads();
    const int nb = codes[b].nb;
    for (int i = threadIdx.x; i < nb; i += kEncThreads)
        if (cnt[i]) atomicAdd(&bcount[(size_t)b * kBuckets + i], cnt[i]);
}

// One CTA per block: bucket starts, scatter cursors, the sort's work lists
// (one per size class); a block with a bucket of more than limit words takes
// the LSD passes. The pending fault of the test hook sends block 0 to
// the LSD passes, whose waits it breaks.
__global__ void __launch_bounds__(256) bwt_offsets_kernel(const BwtCode *__restrict__ codes, const uint32_t *__restrict__ bcount,
                                                          uint32_t *__restrict__ bstart, uint32_t *__restrict__ cursor,
                                                          uint32_t *__restrict__ items_all, size_t items_cap,
                                                          int32_t *__restrict__ bflag, int32_t *__restrict__ rs, uint32_t limit) {
    constexpr int PER = (kBuckets + 255) / 256;
    __shared__ uint32_t shu[33];
    __shared__ int s_base[kBucketClasses];
    const int b = blockIdx.x, t = threadIdx.x;
    const int nb = codes[b].nb;
    uint32_t c[PER], sum = 0;
    bool over = b == 0 && t == 0 && rs[kRsFault] != 0;
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const int k = t * PER + i;
        c[i] = k < nb ? bcount[(size_t)b * kBuckets + k] : 0u;
        sum += c[i];
        over |= c[i] > limit;
    }
    uint32_t total;
    uint32_t ex = block_excl_sum<uint32_t>(sum, shu, &total);
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const int k = t * PER + i;
        if (k < nb) {
            bstart[(size_t)b * kBucketRow + k] = ex;
            cursor[(size_t)b * kBuckets + k] = ex;
        }
        ex += c[i];
    }
    if (t == 0) bstart[(size_t)b * kBucketRow + nb] = total;
    if (__syncthreads_or(over)) {
        if (t == 0) {
            bflag[b] = kFlagOver;
            atomicAdd(&rs[kRsFlagged], 1);
            atomicAdd(&rs[kRsOver], 1);
        }
        return;
    }
#pragma unroll
    for (int cl = 0; cl < kBucketClasses; cl++) {
        const uint32_t lo = cl ? (uint32_t)kBucketCap[cl - 1] : 0u, hi = (uint32_t)kBucketCap[cl];
        uint32_t n = 0, tot;
#pragma unroll
        for (int i = 0; i < PER; i++) n += c[i] > lo && c[i] <= hi;
        uint32_t e = block_excl_sum<uint32_t>(n, shu, &tot);
        if (t == 0) s_base[cl] = tot ? atomicAdd(&rs[kRsBucketItems + cl], (int)tot) : 0;
        __syncthreads();
        uint32_t *items = items_all + cl * items_cap + s_base[cl];
#pragma unroll
        for (int i = 0; i < PER; i++)
            if (c[i] > lo && c[i] <= hi) items[e++] = ((uint32_t)b << 11) | (uint32_t)(t * PER + i);
    }
}

// ------------------------------------------------------------------ scatter
// The tile's words ordered by bucket in shared memory (a counter per bucket),
// each bucket's run reserved with one atomic and written contiguously.
struct ScatterSmem {
    uint64_t w[kEncTile];        // the bit stream lives here until the words are placed
    uint16_t bk[kEncTile];
    uint32_t cnt[kBuckets];
    int32_t adj[kBuckets];       // global minus local index of the tile's run of a bucket
    Splitters P;
    __align__(16) uint16_t code[kTables * 256];
    uint32_t sh[33];
};
static_assert(sizeof(EncTile) <= sizeof(uint64_t) * kEncTile, "the bit stream fits the word array");
static_assert(2 * (sizeof(ScatterSmem) + 1024) <= 228 * 1024, "two CTAs per SM");

__global__ void __launch_bounds__(kEncThreads, 2) bwt_scatter_kernel(const BlockState *__restrict__ st,
                                                                     const uint8_t *__restrict__ rle_all,
                                                                     const BwtCode *__restrict__ codes,
                                                                     uint32_t *__restrict__ cursor, uint64_t *__restrict__ out_all) {
    extern __shared__ __align__(16) uint8_t smraw[];
    ScatterSmem &S = *reinterpret_cast<ScatterSmem *>(smraw);
    EncTile &E = *reinterpret_cast<EncTile *>(smraw);
    const int b = blockIdx.y, t0 = blockIdx.x * kEncTile;
    const int m = st[b].m;
    if (t0 >= m) return;
    load_tables(codes[b], S.code, S.P);
    for (int i = threadIdx.x; i < kBuckets; i += kEncThreads) S.cnt[i] = 0;
    __syncthreads();
    uint4 v4;
    uint32_t c2[kEncPer / 2];
    BitWindow W(E.bits, encode_tile(rle_all + (size_t)b * kBlockCap, m, t0, S.code, E, S.sh, v4, c2));
    const int i0 = t0 + kEncPer * (int)threadIdx.x;
    uint64_t word[kEncPer];
    uint32_t pr[kEncPer];  // bucket << 16 | index among the tile's words of it
#pragma unroll
    for (int q = 0; q < kEncPer; q++) {
        const uint64_t kb = key_bits(W, v4, c2, q, S.code);
        word[q] = (kb & ~(uint64_t)kElemMask) | (uint64_t)(uint32_t)(i0 + q);
        pr[q] = 0xFFFFFFFFu;
        if (i0 + q < m) {
            const int k = bucket_of((uint32_t)(kb >> 48), S.P);
            pr[q] = ((uint32_t)k << 16) | atomicAdd(&S.cnt[k], 1u);
        }
    }
    __syncthreads();  // all keys are in registers: the bit stream may be overwritten
    {
        constexpr int PER = (kBuckets + kEncThreads - 1) / kEncThreads;
        uint32_t c[PER], sum = 0;
#pragma unroll
        for (int i = 0; i < PER; i++) {
            const int k = (int)threadIdx.x * PER + i;
            c[i] = k < kBuckets ? S.cnt[k] : 0u;
            sum += c[i];
        }
        uint32_t ex = block_excl_sum<uint32_t>(sum, S.sh, nullptr);
#pragma unroll
        for (int i = 0; i < PER; i++) {
            const int k = (int)threadIdx.x * PER + i;
            if (k < kBuckets) {
                S.cnt[k] = ex;
                if (c[i]) S.adj[k] = (int32_t)atomicAdd(&cursor[(size_t)b * kBuckets + k], c[i]) - (int32_t)ex;
            }
            ex += c[i];
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kEncPer; q++) {
        if (pr[q] == 0xFFFFFFFFu) continue;
        const uint32_t k = pr[q] >> 16, at = S.cnt[k] + (pr[q] & 0xFFFFu);
        S.w[at] = word[q];
        S.bk[at] = (uint16_t)k;
    }
    __syncthreads();
    const int cnt = min(kEncTile, m - t0);
    uint64_t *out = out_all + (size_t)b * kBlockCap;
    for (int j = threadIdx.x; j < cnt; j += kEncThreads) out[S.adj[S.bk[j]] + j] = S.w[j];
}

// ------------------------------------------------------------- bucket sort
// Code bits of the rotation idx behind its first kKeyBits bits after byte
// depth: skips the whole codes in those (adding them to depth), then returns
// the next kKeyBits. depth 0: the key in the words.
__device__ __forceinline__ uint64_t next_key(const uint8_t *rle, int m, const uint16_t *code, int idx, int &depth) {
    int pos = idx + depth;
    pos -= pos >= m ? m : 0;
    uint32_t tab = depth == 0 ? (uint32_t)kFirst : (rle[pos == 0 ? m - 1 : pos - 1] ? 256u : 0u);
    int used = 0;
    for (;;) {
        const uint32_t x = rle[pos];
        const int l = (int)(code[tab + x] >> 12);
        if (used + l > kKeyBits) break;
        used += l;
        depth++;
        tab = x ? 256u : 0u;
        if (++pos == m) pos = 0;
    }
    uint64_t acc = 0;
    for (used = 0; used < kKeyBits;) {
        const uint32_t x = rle[pos], c = code[tab + x];
        const int l = (int)(c >> 12);
        acc = (acc << l) | (c & 0xFFFu);
        used += l;
        tab = x ? 256u : 0u;
        if (++pos == m) pos = 0;
    }
    return acc >> (used - kKeyBits);
}

// Leaves a group of block b tied after depth equal bytes: prefix doubling
// takes the block, from the least depth of any such group.
__device__ __forceinline__ int ld_flag(const int32_t *p) { return *reinterpret_cast<const volatile int32_t *>(p); }
__device__ __forceinline__ void leave_tied(int32_t *bflag, int32_t *rs, int b, int depth) {
    if (ld_flag(rs + kRsH) > depth) atomicMin(&rs[kRsH], depth);
    if ((ld_flag(bflag + b) & kFlagTied) == 0 && atomicOr(&bflag[b], kFlagTied) == 0) atomicAdd(&rs[kRsFlagged], 1);
}

struct BucketItem {
    int b, start, n, m;
    uint32_t p_lo, p_hi;
};

// A word in shared memory as two 32-bit arrays: with d = key - the bucket's
// first key, hi = (top 12 bits of d) << 20 | start and lo = the other bits of
// d, at most 32 (equal hi >> 20 and equal lo: equal keys).
template <int CAP>
struct BucketSmem {
    uint32_t lo[CAP], hi[CAP];
    __align__(16) uint32_t cnt[2][kSubBins / 2 + 4];  // this bucket's and the next one's
    uint32_t sh[33];
    BucketItem item[3];
    uint32_t cost;  // sum over the sub-bins of their words squared
};

// Persistent CTAs take buckets from the list of their size class. While a
// bucket is ranked and written, the next one's words are loaded (PRE) and the
// one after that is looked up.
template <int CLASS>
__global__ void __launch_bounds__(kBucketThreads[CLASS], kBucketCtas[CLASS])
bwt_bucket_kernel(BlockState *__restrict__ st, const uint8_t *__restrict__ rle_all, const BwtCode *__restrict__ codes,
                  const uint32_t *__restrict__ bstart, const uint32_t *__restrict__ items, const uint64_t *__restrict__ words_all,
                  int32_t *__restrict__ sa_all, uint8_t *__restrict__ L_all, uint64_t *__restrict__ ties, size_t ties_cap,
                  int32_t *__restrict__ bflag, int32_t *__restrict__ rs) {
    constexpr int CAP = kBucketCap[CLASS], TH = kBucketThreads[CLASS], PER = CAP / TH;
    constexpr bool PRE = CLASS == 0;
    extern __shared__ __align__(16) uint8_t smraw[];
    BucketSmem<CAP> &S = *reinterpret_cast<BucketSmem<CAP> *>(smraw);
    const int t = threadIdx.x;
    const int total = rs[kRsBucketItems + CLASS];
    int32_t *queue = rs + kRsBucketQueue + CLASS;
    auto look_up = [&]() {  // one thread
        const int q = atomicAdd(queue, 1);
        BucketItem I{-1, 0, 0, 0, 0, 0};
        if (q < total) {
            const uint32_t item = items[q];
            I.b = (int)(item >> 11);
            const int k = (int)(item & 2047u);
            const uint32_t *row = bstart + (size_t)I.b * kBucketRow + k;
            const BwtCode &C = codes[I.b];
            I.start = (int)row[0];
            I.n = (int)row[1] - I.start;
            I.m = st[I.b].m;
            I.p_lo = C.split[k];
            I.p_hi = k + 1 < C.nb ? (uint32_t)C.split[k + 1] : 65536u;
        }
        return I;
    };
    auto same_key = [&](int i, int j) { return S.lo[i] == S.lo[j] && (S.hi[i] >> 20) == (S.hi[j] >> 20); };
    uint64_t w[PER];
    auto load_words = [&](const BucketItem &I) {
        const uint64_t *in = words_all + (size_t)I.b * kBlockCap + I.start;
#pragma unroll
        for (int r = 0; r < PER; r++) w[r] = r * TH + t < I.n ? in[r * TH + t] : 0ull;
    };
    if (t == 0) {
        S.item[0] = look_up();
        S.item[1] = look_up();
    }
    for (int i = t; i < 2 * (kSubBins / 8 + 1); i += TH) reinterpret_cast<uint4 *>(&S.cnt[0][0])[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    if (PRE && S.item[0].b >= 0) load_words(S.item[0]);
    for (int it = 0;; it++) {
        const BucketItem I = S.item[it % 3];
        if (I.b < 0) return;
        uint32_t *cnt = S.cnt[it & 1];
        const uint16_t *cnt16 = reinterpret_cast<const uint16_t *>(cnt);
        const int n = I.n;
        const uint64_t key_lo = (uint64_t)I.p_lo << (kKeyBits - kPrefixBits);
        const uint64_t range = ((uint64_t)(I.p_hi - I.p_lo) << (kKeyBits - kPrefixBits)) - 1;
        const int low = 64 - __clzll((long long)range) - 12;  // bits of lo: 16 .. 32
        if (!PRE) load_words(I);
        uint32_t lo[PER], hi[PER], pr[PER];
#pragma unroll
        for (int r = 0; r < PER; r++) {
            const uint64_t d = (w[r] >> 20) - key_lo;
            lo[r] = (uint32_t)d & (0xFFFFFFFFu >> (32 - low));
            hi[r] = ((uint32_t)(d >> low) << 20) | ((uint32_t)w[r] & (uint32_t)kElemMask);
            if (r * TH + t >= n) continue;
            const uint32_t sub = (uint32_t)(d >> (low - 1)), sh = 16 * (sub & 1);
            pr[r] = (sub << 16) | ((atomicAdd(&cnt[sub >> 1], 1u << sh) >> sh) & 0xFFFFu);
        }
        if (t == 0) S.cost = 0;
        __syncthreads();  // also: every thread is done with the previous bucket's words
        {
            constexpr int SP = kSubBins / 2 / TH;  // consecutive counter pairs per thread
            uint32_t c[SP], sum = 0, cost = 0;
#pragma unroll
            for (int i = 0; i < SP; i += 4) {
                const uint4 v = reinterpret_cast<const uint4 *>(cnt)[(t * SP + i) / 4];
                c[i] = v.x; c[i + 1] = v.y; c[i + 2] = v.z; c[i + 3] = v.w;
            }
#pragma unroll
            for (int i = 0; i < SP; i++) sum += (c[i] & 0xFFFFu) + (c[i] >> 16);
            uint32_t ex = block_excl_sum<uint32_t>(sum, S.sh, nullptr);
#pragma unroll
            for (int i = 0; i < SP; i++) {
                const uint32_t x = c[i] & 0xFFFFu, y = c[i] >> 16;
                cost += x * x + y * y;
                c[i] = ex | ((ex + x) << 16);
                ex += x + y;
            }
#pragma unroll
            for (int i = 0; i < SP; i += 4)
                reinterpret_cast<uint4 *>(cnt)[(t * SP + i) / 4] = make_uint4(c[i], c[i + 1], c[i + 2], c[i + 3]);
            if (t == 0) cnt[kSubBins / 2] = (uint32_t)n;
            cost = warp_sum(cost);
            if ((t & 31) == 0) atomicAdd(&S.cost, cost);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; r++)
            if (r * TH + t < n) {
                const uint32_t at = cnt16[pr[r] >> 16] + (pr[r] & 0xFFFFu);
                S.lo[at] = lo[r];
                S.hi[at] = hi[r];
            }
        // the next bucket's counters (last read before this bucket's first
        // barrier) are cleared, and S.cost read, before the barrier: behind it
        // threads run ahead into the next bucket
        for (int i = t; i < kSubBins / 8 + 1; i += TH) reinterpret_cast<uint4 *>(S.cnt[(it + 1) & 1])[i] = make_uint4(0, 0, 0, 0);
        const bool big = S.cost > (uint32_t)kSubCost * (uint32_t)n;
        __syncthreads();
        if (PRE && S.item[(it + 1) % 3].b >= 0) load_words(S.item[(it + 1) % 3]);
        if (t == 0) S.item[(it + 2) % 3] = look_up();
        const uint8_t *rle = rle_all + (size_t)I.b * kBlockCap;
        int32_t *sa = sa_all + (size_t)I.b * kBlockCap + I.start;
        uint8_t *L = L_all + (size_t)I.b * kBlockCap + I.start;
        // the word of rank c, the eqb-th of neq equal keys: a group of equal
        // keys is listed by its first word, a long one stays tied (bit 31 of
        // the suffix array on all but its first word)
        auto put = [&](int c, uint32_t h, int eqb, int neq) {
            uint32_t mark = 0;
            if (neq > 1) {
                if (neq > kTieGroup) {
                    if (eqb) {
                        mark = 1u << 31;
                    } else {
                        leave_tied(bflag, rs, I.b, key_depth(rle, I.m, codes[I.b].code, (int)(h & (uint32_t)kElemMask)));
                    }
                } else if (!eqb) {
                    const size_t at = neq <= kTieShort ? (size_t)atomicAdd(&rs[kRsTies], 1)
                                                       : ties_cap - 1 - (size_t)atomicAdd(&rs[kRsTiesLong], 1);
                    ties[at] = ((uint64_t)I.b << 32) | ((uint64_t)neq << 24) | (uint64_t)(I.start + c);
                }
            }
            const int idx = (int)(h & (uint32_t)kElemMask);
            sa[c] = (int32_t)((uint32_t)idx | mark);
            L[c] = rle[idx == 0 ? I.m - 1 : idx - 1];
            if (idx == 0) st[I.b].orig_ptr = I.start + c;
        };
        if (!big) {
            // rank by counting the smaller words of the sub-bin, equal keys by
            // their starts (the later rounds keep that order): neighbouring
            // threads read the same few words and write next to each other
#pragma unroll 2
            for (int i = t; i < n; i += TH) {
                const uint32_t l = S.lo[i], h = S.hi[i];
                const uint32_t sub = ((h >> 20) << 1) | (l >> (low - 1));
                const int b0 = cnt16[sub], b1 = cnt16[sub + 1];
                int lt = 0, le = 0;
#pragma unroll 4
                for (int j = b0; j < b1; j++) {
                    const uint32_t x = S.lo[j];
                    lt += x < l;
                    le += x <= l;
                }
                int eqb = 0;
                if (le - lt > 1)
                    for (int j = b0; j < b1; j++) eqb += S.lo[j] == l && S.hi[j] < h;
                put(b0 + lt + eqb, h, eqb, le - lt);
            }
        } else {
            int np = 1;
            while (np < n) np <<= 1;
            // merge network with all directions ascending (the first step of a
            // merge mirrors the upper half); words past n stand for the largest
            // one and never move
            for (int kk = 2; kk <= np; kk <<= 1)
                for (int j = kk >> 1; j > 0; j >>= 1) {
#pragma unroll 2
                    for (int q = t; q < np / 2; q += TH) {
                        const int o = q & (j - 1), i = 2 * (q - o) + o, l = j == kk >> 1 ? 2 * (q - o) + 2 * j - 1 - o : i + j;
                        if (l < n) {
                            const uint32_t xl = S.lo[i], xh = S.hi[i], yl = S.lo[l], yh = S.hi[l];
                            const bool same = (xh >> 20) == (yh >> 20);
                            if (same ? (xl > yl || (xl == yl && xh > yh)) : xh > yh) {
                                S.lo[i] = yl; S.hi[i] = yh;
                                S.lo[l] = xl; S.hi[l] = xh;
                            }
                        }
                    }
                    __syncthreads();
                }
            for (int i = t; i < n; i += TH) {
                int gs = max(0, i - kTieGroup), ge = min(n, i + kTieGroup + 1);  // the group around i, as far as it counts
                for (int e = i; gs < e;) {
                    const int mid = (gs + e) >> 1;
                    if (same_key(mid, i)) e = mid; else gs = mid + 1;
                }
                for (int f = i + 1; f < ge;) {
                    const int mid = (f + ge) >> 1;
                    if (same_key(mid, i)) f = mid + 1; else ge = mid;
                }
                put(i, S.hi[i], i - gs, ge - gs);
            }
        }
    }
}

// The listed groups: members ordered by further keys, equal ones by start;
// the pieces still tied are taken up to kTieRounds keys deep. Identical
// rotations (the whole block agrees) stay in start order; they are marked as
// tied without a call for prefix doubling, for where a block takes it on
// account of other groups, rotations that differ only by such a piece have to
// find it undivided (ordered by the starts of the piece's members, they could
// come out of start order themselves). One thread orders a group of up to
// kTieShort members (almost all: pairs), one warp a longer one (a lane per
// member: the walks over the bytes are the time it takes). The list holds the
// short groups from its front, the long ones from its end.
// A block with a long repeat takes prefix doubling whatever the number of
// keys, so its groups are not walked far: groups still tied after kTieFew keys
// (streams of frames have next to none) are counted per block, and from the
// count most() on its other groups are left as they are (the long ones by a
// lane each) and those on their way stop at their next key. 24 blocks of
// 100 000 bytes take 2.1 ms a call with 8 copies of a string each and 2.4 with
// 2; with every group walked to kTieRounds it was 7.7 and 4.2. When the whole
// list is few groups a warp, the walks cost less than the doubling rounds they
// may save, and none is given up (300 000 bytes of 200-byte strings twice each
// 0.67 ms, 0.84 without that).
constexpr int kTieThreads = 128;

__global__ void __launch_bounds__(kTieThreads) bwt_tie_kernel(BlockState *__restrict__ st, const uint8_t *__restrict__ rle_all,
                                                              const BwtCode *__restrict__ codes, const uint64_t *__restrict__ ties,
                                                              size_t ties_cap, int32_t *__restrict__ sa_all, uint8_t *__restrict__ L_all,
                                                              int32_t *__restrict__ bflag, int32_t *__restrict__ bdeep,
                                                              int32_t *__restrict__ rs) {
    __shared__ uint64_t sw[kTieThreads / 32][32];
    const int total = rs[kRsTies], total_long = rs[kRsTiesLong];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto out = [&](int b, int m, const uint8_t *rle, int at, uint64_t w, bool tied) {
        const int idx = (int)(w & kElemMask);
        sa_all[(size_t)b * kBlockCap + at] = (int32_t)((uint32_t)idx | (tied ? 1u << 31 : 0u));
        L_all[(size_t)b * kBlockCap + at] = rle[idx == 0 ? m - 1 : idx - 1];
        if (idx == 0) st[b].orig_ptr = at;
    };
    // long groups a warp takes at once: it asks for the block's count once a chunk
    const int warps = gridDim.x * (kTieThreads / 32), chunk = min(8, (total_long + warps - 1) / warps);
    const bool few = total <= warps * 32 && total_long <= kTieWaves * warps;
    auto most = [few](int m) { return few ? INT_MAX : max(kTieMany, m / kTieShare); };
    auto given_up = [&](uint64_t e) { return ld_flag(bdeep + (e >> 32)) >= most(st[e >> 32].m); };
    auto leave = [&](uint64_t e) {  // the group stays as it is, tied (one thread)
        const int b = (int)(e >> 32), len = (int)((e >> 24) & 255u);
        int32_t *sa = sa_all + (size_t)b * kBlockCap + (e & 0xFFFFFFu);
        leave_tied(bflag, rs, b, key_depth(rle_all + (size_t)b * kBlockCap, st[b].m, codes[b].code, sa[0]));
        for (int k = 1; k < len; k++) sa[k] |= (int32_t)(1u << 31);
    };
    auto go_on = [&](int b, int m, int round) {  // whether a group is compared by one more key
        if (!few && round == kTieFew) return ld_flag(bdeep + b) < most(m) && atomicAdd(&bdeep[b], 1) < most(m);
        return round < kTieRounds && (few || round < kTieFew || (ld_flag(bflag + b) & kFlagTied) == 0);
    };
    for (int g = blockIdx.x * kTieThreads + threadIdx.x; g < total; g += gridDim.x * kTieThreads) {
        const uint64_t e = ties[g];
        if (given_up(e)) {
            leave(e);
            continue;
        }
        const int b = (int)(e >> 32), len = (int)((e >> 24) & 255u), at = (int)(e & 0xFFFFFFu);
        const int m = st[b].m;
        const uint8_t *rle = rle_all + (size_t)b * kBlockCap;
        const uint16_t *code = codes[b].code;
        uint64_t w[kTieShort];
        int piece[kTieShort], dep[kTieShort];  // at a piece's first member: its length, the bytes its members share
        for (int k = 0; k < len; k++) w[k] = (uint64_t)(uint32_t)sa_all[(size_t)b * kBlockCap + at + k];
        piece[0] = len;
        dep[0] = 0;
        bool pend = true;
        for (int round = 0; pend && go_on(b, m, round); round++) {
            pend = false;
            for (int p0 = 0; p0 < len;) {
                const int pl = piece[p0];
                if (pl == 1 || dep[p0] >= m) { p0 += pl; continue; }
                int d = 0;
                for (int k = p0; k < p0 + pl; k++) {
                    d = dep[p0];
                    const uint32_t idx = (uint32_t)(w[k] & kElemMask);
                    const uint64_t x = (next_key(rle, m, code, (int)idx, d) << 20) | (uint64_t)idx;
                    int j = k;  // insertion
                    while (j > p0 && w[j - 1] > x) { w[j] = w[j - 1]; j--; }
                    w[j] = x;
                }
                for (int k = p0; k < p0 + pl;) {
                    int q = k + 1;
                    while (q < p0 + pl && (w[q] >> 20) == (w[k] >> 20)) q++;
                    piece[k] = q - k;
                    dep[k] = d;
                    pend |= q - k > 1 && d < m;
                    k = q;
                }
                p0 += pl;
            }
        }
        for (int p0 = 0; p0 < len; p0 += piece[p0]) {
            if (piece[p0] > 1 && dep[p0] < m) leave_tied(bflag, rs, b, dep[p0]);
            for (int k = p0; k < p0 + piece[p0]; k++) out(b, m, rle, at + k, w[k], k > p0);
        }
    }
    for (int g0 = (blockIdx.x * (kTieThreads / 32) + warp) * chunk; g0 < total_long; g0 += warps * chunk) {
        const int gn = min(chunk, total_long - g0);
        const uint64_t mine = lane < gn ? ties[ties_cap - 1 - (size_t)(g0 + lane)] : 0ull;
        bool check = true;  // at first and after a group that went far
        for (uint32_t todo = LFC_FULL >> (32 - gn); todo;) {
            if (check) {
                const bool drop = ((todo >> lane) & 1u) && given_up(mine);  // a lane for each of these
                if (drop) leave(mine);
                todo &= ~__ballot_sync(LFC_FULL, drop);
                if (!todo) break;
            }
            const uint64_t e = __shfl_sync(LFC_FULL, mine, __ffs(todo) - 1);
            todo &= todo - 1;
            const int b = (int)(e >> 32), len = (int)((e >> 24) & 255u), at = (int)(e & 0xFFFFFFu);
            const int m = st[b].m;
            const uint8_t *rle = rle_all + (size_t)b * kBlockCap;
            const uint16_t *code = codes[b].code;
            const bool in = lane < len;
            uint64_t w = in ? (uint64_t)(uint32_t)sa_all[(size_t)b * kBlockCap + at + lane] : ~0ull;
            int p0 = in ? 0 : lane, p1 = in ? len : lane + 1, dep = 0;  // the member's piece, the bytes it shares
            int round = 0;
            for (;; round++) {
                const bool act = p1 - p0 > 1 && dep < m;
                if (!__any_sync(LFC_FULL, act)) break;
                if (!__any_sync(LFC_FULL, lane == 0 && go_on(b, m, round))) break;
                if (act) {
                    const uint32_t idx = (uint32_t)(w & kElemMask);
                    w = (next_key(rle, m, code, (int)idx, dep) << 20) | (uint64_t)idx;
                }
                __syncwarp();
                int to = act ? p0 : lane;
                for (int j = 0; j < len; j++) {
                    const uint64_t x = __shfl_sync(LFC_FULL, w, j);
                    to += act && j >= p0 && j < p1 && x < w;
                }
                sw[warp][to] = w;
                __syncwarp();
                w = sw[warp][lane];  // a piece's members share dep, wherever they stand
                const bool head = lane == p0 || (act && (sw[warp][lane - 1] >> 20) != (w >> 20));
                const uint32_t heads = __ballot_sync(LFC_FULL, head);
                if (act) {
                    const uint32_t above = heads & lanemask_gt();
                    p0 = 31 - __clz(heads & (lanemask_lt() | (1u << lane)));
                    p1 = above ? __ffs(above) - 1 : 32;
                    p1 = min(p1, len);
                }
                __syncwarp();
            }
            if (in) {
                if (p1 - p0 > 1 && lane == p0 && dep < m) leave_tied(bflag, rs, b, dep);
                out(b, m, rle, at + lane, w, lane > p0);
            }
            check = round >= kTieFew;
        }
    }
}

template <int CLASS>
static cudaError_t launch_class(lfc_plan P, int most) {
    Workspace &ws = P->ws;
    const size_t smem = sizeof(BucketSmem<kBucketCap[CLASS]>);
    cudaError_t e = cudaFuncSetAttribute(bwt_bucket_kernel<CLASS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    bwt_bucket_kernel<CLASS><<<std::min(most, kBucketCtas[CLASS] * P->sm_count), kBucketThreads[CLASS], smem, P->stream>>>(
        ws.bstate, ws.rle, ws.bcode, ws.bstart, ws.bitems + CLASS * ws.bitems_cap, ws.keys2, ws.sa, ws.bwt, ws.keys,
        (size_t)P->block_cap * kBlockCap, ws.bflag, ws.act_total);
    return cudaGetLastError();
}

cudaError_t launch_bucket_sort(lfc_plan P, int nblocks, int max_m, bool graph) {
    Workspace &ws = P->ws;
    cudaStream_t s = P->stream;
    cudaError_t e = cudaFuncSetAttribute(bwt_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlanSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(bwt_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterSmem));
    if (e != cudaSuccess) return e;
    const dim3 grid((max_m + kEncTile - 1) / kEncTile, nblocks);
    // A bucket of the largest class is 0.23 ms of one CTA (repetitive text has
    // such buckets); a small pass is sooner done when the blocks with one take
    // the LSD passes (6 blocks of text of up to 400 000 bytes: 1775 us a call
    // against 1590; 30 of up to 700 000: 4.4 ms with the class).
    const int classes = (int64_t)nblocks * max_m < kSmallPass ? 2 : kBucketClasses;
    stage_begin(P, LFC_STAGE_BWT_KEYS);
    // outside graphs the call itself reports a wait that gave up
    bwt_plan_kernel<<<nblocks, kPlanThreads, kPlanSmem, s>>>(ws.bstate, ws.rle, ws.bcode, ws.bcount, ws.bflag, ws.bdeep,
                                                             ws.act_total, graph ? 0 : 1);
    bwt_count_kernel<<<grid, kEncThreads, 0, s>>>(ws.bstate, ws.rle, ws.bcode, ws.bcount);
    bwt_offsets_kernel<<<nblocks, 256, 0, s>>>(ws.bcode, ws.bcount, ws.bstart, ws.bcursor, ws.bitems, ws.bitems_cap, ws.bflag,
                                               ws.act_total, (uint32_t)kBucketCap[classes - 1]);
    stage_end(P, LFC_STAGE_BWT_KEYS);
    stage_begin(P, LFC_STAGE_BWT_SORT8);
    bwt_scatter_kernel<<<grid, kEncThreads, sizeof(ScatterSmem), s>>>(ws.bstate, ws.rle, ws.bcode, ws.bcursor, ws.keys2);
    e = cudaGetLastError();
    const int most = nblocks * std::min(kBuckets, 3 * max_m / kBucketTarget + 4);  // buckets of the pass, at most
    if (e == cudaSuccess) e = launch_class<0>(P, most);
    // a bucket of a larger class needs a block of more words than the class below holds
    if (e == cudaSuccess && max_m > kBucketCap[0]) e = launch_class<1>(P, most);
    if (e == cudaSuccess && max_m > kBucketCap[1] && classes > 2) e = launch_class<2>(P, most);
    if (e != cudaSuccess) return e;
    bwt_tie_kernel<<<8 * P->sm_count, kTieThreads, 0, s>>>(ws.bstate, ws.rle, ws.bcode, ws.keys,
                                                           (size_t)P->block_cap * kBlockCap, ws.sa, ws.bwt, ws.bflag, ws.bdeep,
                                                           ws.act_total);
    e = cudaGetLastError();
    stage_end(P, LFC_STAGE_BWT_SORT8);
    count_launches(P, 5 + 1 + (max_m > kBucketCap[0]) + (max_m > kBucketCap[1] && classes > 2));
    return e;
}

}  // namespace lfc
