// decode.cu -- decompression (Fig. 2b: unpack the header, bzip2-decode every
// block, then the inverse predictor chosen by the header's id).
//
// Every step of a block is spread over many CTAs, so that one frame's few
// blocks fill the GPU as well as a batch does. Every read of the coded stream
// is checked against its length and every write against its buffer, so
// corrupt input ends in an error flag, never an out-of-bounds access.
//  1. Header (a CTA per block): selectors from the positions of the zero bits
//     of their unary codes (a scan), their move-to-front as a scan over
//     permutations of six tables; code lengths and lookup tables.
//  2. Group offsets. A group is 50 codes of one table, so where it ends
//     follows from where it starts. For every bit position and every table
//     the length of 50 codes from there is computed in parallel (lengths of
//     2, 4, 8 and 16 codes by doubling, in shared memory); then one thread
//     per block only adds up a looked-up length per group (EOB lies in the
//     last group, as an encoder writes one selector per group it uses: a
//     stream with more selectors is rejected as corrupt).
//  3. Every group's symbols, a thread per group.
//  4. Inverse RUNA/RUNB and MTF by up to kSegs segments, a thread each with its
//     256-byte list in shared memory: a segment's moves permute list
//     positions whatever the list holds, so the permutations and output
//     lengths come first, the segment-start lists and offsets are chained,
//     and every segment is decoded from its list -> the BWT last column L.
//  5. LF mapping by a stable counting sort over tiles; a word per row holds
//     the next row and the row's byte.
//  6. Inverse BWT: a walker per kWalkStep rows (and one at the origin) follows
//     the rows until it meets another walker's start; the pieces are ranked
//     along their list by pointer doubling; every walker writes its piece. The
//     rows of a block that repeats a shorter string form one cycle per copy:
//     the origin's is the string, and the block is filled with it.
//  7. Inverse RLE1 by tiles from sync points; block CRCs (crc.cu).
// One 1300 x 1300 frame (5 blocks) takes 2.2 ms, 12 frames of 2040 x 2040
// (139 blocks) 10.2 ms; with one CTA per block it was 47 and 58 ms.
#include <algorithm>
#include <climits>

#include "lfc_common.cuh"

namespace lfc {

enum : int32_t {
    DEC_OK = 0, DEC_BAD_MAGIC = 1, DEC_TRUNC = 2, DEC_BAD_TABLE = 3, DEC_BAD_DATA = 4,
    DEC_OVERFLOW = 5, DEC_BAD_ORIG = 6, DEC_BAD_LEN = 7, DEC_BAD_CRC = 8, DEC_BAD_WALK = 9
};

struct DecBlock {
    const uint8_t *src;   // one standalone bzip2 stream
    int64_t src_len;
    uint8_t *dst;         // decoded bytes go here
    int32_t expect;       // decoded length the container promises
    int32_t pad;
};

// What the header says of a block, and how far its decoding has come.
struct DecMeta {
    int32_t status, block_max, orig, n_in_use, alpha, n_groups, n_sel;
    int32_t group, bit;   // next group and its bit offset (group chase)
    int32_t nsym;         // symbols up to and including EOB
    int32_t m;            // bytes of the last column
    int32_t period;       // rows of the origin's cycle: m, or less in a block that repeats a shorter string
    uint32_t stored_crc, crc;
    int32_t pad[6];
};
static_assert(sizeof(DecMeta) == sizeof(BlockState), "the decoder's block records live in the coder's");

// Most bytes of the last column of a block that decodes to `expect` bytes:
// five of them give at least four. A block has at most one symbol per byte and
// EOB. What has more decodes to more than the container promises, and the
// grids of the later steps are sized by it.
__host__ __device__ inline int column_bound(int expect) { return expect + expect / 4; }

constexpr int kJBits = 12;  // prefix bits of the length table
struct DecTab {
    uint2 jlut[1 << kJBits];                 // a byte per table: bits of the code (0: longer)
    uint16_t lut[kMaxGroups][1 << 10];       // symbol << 5 | code length, 0: longer code
    int32_t first[kMaxGroups][22], count[kMaxGroups][22], pidx[kMaxGroups][22];  // laid out as Canon
    uint16_t perm[kMaxGroups][kMaxAlpha];    // symbols by code
    uint8_t seq_to_unseq[256];
};
static_assert(sizeof(DecTab) <= sizeof(int32_t) * kBlockCap, "tables fit a block's slot");

// 32 bits from bit position `bit` on (MSB first), zeros past the end.
__device__ __forceinline__ uint32_t stream_bits32(const uint8_t *p, int64_t nbytes, int64_t bit) {
    const int64_t a = bit >> 3;
    uint64_t w = 0;
    if (a + 5 <= nbytes) {
#pragma unroll
        for (int i = 0; i < 5; i++) w = (w << 8) | __ldg(p + a + i);
    } else {
        for (int i = 0; i < 5; i++) w = (w << 8) | (a + i < nbytes ? __ldg(p + a + i) : 0u);
    }
    return (uint32_t)(w >> (8 - (int)(bit & 7)));
}

// MSB-first bit reader over a bounded byte string: up to 64 bits buffered
// left-aligned, each byte loaded once. get(k) (k <= 32) past the end sets
// err and returns 0; peek(k) pads with zeros past the end.
struct BitReader {
    const uint8_t *p;
    int64_t nbytes, next;  // bytes in the string, next byte to load
    uint64_t buf;          // buffered bits, left-aligned
    int bcnt;              // buffered bit count
    bool err;
    __device__ void init(const uint8_t *src, int64_t n) {
        p = src;
        nbytes = n;
        next = 0;
        buf = 0;
        bcnt = 0;
        err = false;
    }
    __device__ void seek(int64_t bit) {
        next = bit >> 3;
        buf = 0;
        bcnt = 0;
        skip((int)(bit & 7));
    }
    __device__ __forceinline__ int64_t tell() const { return next * 8 - bcnt; }
    // Called with fewer bits buffered than a read needs (at most 32): 32
    // more bits from four independent loads (one memory latency, not four);
    // the last bytes of the string one by one
    __device__ __forceinline__ void refill() {
        if (bcnt <= 32 && next + 4 <= nbytes) {
            const uint32_t w = ((uint32_t)__ldg(p + next) << 24) | ((uint32_t)__ldg(p + next + 1) << 16) |
                               ((uint32_t)__ldg(p + next + 2) << 8) | (uint32_t)__ldg(p + next + 3);
            buf |= (uint64_t)w << (32 - bcnt);
            bcnt += 32;
            next += 4;
            return;
        }
        while (bcnt <= 56 && next < nbytes) {
            buf |= (uint64_t)__ldg(p + next++) << (56 - bcnt);
            bcnt += 8;
        }
    }
    __device__ __forceinline__ uint32_t peek(int k) {
        if (bcnt < k) refill();
        return (uint32_t)(buf >> (64 - k));
    }
    __device__ __forceinline__ bool skip(int k) {
        if (bcnt < k) refill();
        if (bcnt < k) { err = true; bcnt = 0; buf = 0; return false; }
        buf <<= k;
        bcnt -= k;
        return true;
    }
    __device__ __forceinline__ uint32_t get(int k) {
        const uint32_t v = peek(k);
        return skip(k) ? v : 0u;
    }
};

// Canonical tables, per code length.
struct Canon {
    int32_t first[kMaxGroups][22], count[kMaxGroups][22], pidx[kMaxGroups][22];
};

// One Huffman symbol with table t: the 10-bit lookup, else the canonical
// search from 11 bits; -1 for a code that is not in the table or a stream
// that ends first (br.err).
__device__ __forceinline__ int huff_symbol(BitReader &br, const uint16_t *lut, const Canon &C, const DecTab &T, int t) {
    if (br.bcnt < 20) br.refill();
    const uint32_t v = (uint32_t)(br.buf >> 44), e = lut[v >> 10];
    if (e) return br.skip(e & 31) ? (int)(e >> 5) : -1;
    for (int l = 11; l <= 20; l++) {
        const uint32_t d = (uint32_t)((int32_t)(v >> (20 - l)) - C.first[t][l]);
        if (d < (uint32_t)C.count[t][l]) return br.skip(l) ? T.perm[t][C.pidx[t][l] + (int)d] : -1;
    }
    return -1;
}

// ------------------------------------------------------------- 1. header
// A CTA per block, 0.17 ms for one frame and 0.20 ms for 139 blocks: bound by
// the one thread that reads the code lengths, a chain of a few instructions
// per bit.
constexpr int kHdrThreads = 512;

// Lists of six tables as nibbles, entry k in bits 4k .. 4k + 3.
constexpr uint32_t kListId = 0x543210u;
__device__ __forceinline__ uint32_t list_move(uint32_t l, int j) {  // entry j to the front
    const uint32_t v = (l >> (4 * j)) & 15u, keep = ~0u << (4 * j + 4);
    return (l & keep) | ((l << 4) & ~keep & ~15u) | v;
}
__device__ __forceinline__ uint32_t list_after(uint32_t a, uint32_t b) {  // entry k: a[b[k]]
    uint32_t r = 0;
#pragma unroll
    for (int k = 0; k < kMaxGroups; k++) r |= ((a >> (4 * ((b >> (4 * k)) & 15u))) & 15u) << (4 * k);
    return r;
}

__global__ void __launch_bounds__(kHdrThreads) dec_header_kernel(const DecBlock *__restrict__ blocks, DecMeta *__restrict__ meta,
                                                                 DecTab *__restrict__ tabs, size_t tab_stride,
                                                                 uint8_t *__restrict__ sel_all, int32_t *__restrict__ zpos_all) {
    __shared__ uint8_t len[kMaxGroups][kMaxAlpha];
    __shared__ int32_t first[kMaxGroups][22], count[kMaxGroups][22], pidx[kMaxGroups][22];
    __shared__ uint16_t perm[kMaxGroups][kMaxAlpha];
    __shared__ int sh[33];
    __shared__ uint32_t wlist[kHdrThreads / 32];
    __shared__ int s_status, s_alpha, s_ng, s_nsel, s_bit;
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
    const DecBlock D = blocks[b];
    DecMeta &M = meta[b];
    DecTab &T = *reinterpret_cast<DecTab *>(reinterpret_cast<uint8_t *>(tabs) + (size_t)b * tab_stride);
    uint8_t *sel = sel_all + (size_t)b * kMaxSelectors;
    int32_t *zpos = zpos_all + (size_t)b * kBlockCap;
    if (t == 0) {
        BitReader br;
        br.init(D.src, D.src_len);
        int st = DEC_OK;
        do {
            if (br.get(8) != 'B' || br.get(8) != 'Z' || br.get(8) != 'h') { st = DEC_BAD_MAGIC; break; }
            const uint32_t lvl = br.get(8);
            if (lvl < '1' || lvl > '9') { st = DEC_BAD_MAGIC; break; }
            M.block_max = 100000 * (int)(lvl - '0');
            if (br.get(24) != 0x314159u || br.get(24) != 0x265359u) { st = DEC_BAD_MAGIC; break; }
            M.stored_crc = br.get(32);
            if (br.get(1) != 0) { st = DEC_BAD_DATA; break; }
            M.orig = (int)br.get(24);
            const uint32_t used16 = br.get(16);
            int niu = 0;
            for (int i = 0; i < 16; i++) {
                if (!(used16 & (1u << (15 - i)))) continue;
                const uint32_t bits = br.get(16);
                for (int j = 0; j < 16; j++)
                    if (bits & (1u << (15 - j))) T.seq_to_unseq[niu++] = (uint8_t)(i * 16 + j);
            }
            if (br.err) { st = DEC_TRUNC; break; }
            if (niu == 0) { st = DEC_BAD_TABLE; break; }
            const int ng = (int)br.get(3), nsel = (int)br.get(15);
            if (br.err) { st = DEC_TRUNC; break; }
            if (ng < 2 || ng > 6 || nsel < 1 || nsel > kMaxSelectors) { st = DEC_BAD_TABLE; break; }
            M.n_in_use = niu;
            M.alpha = niu + 2;
            M.n_groups = ng;
            M.n_sel = nsel;
            s_alpha = niu + 2;
            s_ng = ng;
            s_nsel = nsel;
            s_bit = (int)br.tell();
        } while (0);
        s_status = st;
    }
    __syncthreads();
    if (s_status != DEC_OK) {
        if (t == 0) M.status = s_status;
        return;
    }
    const int ng = s_ng, nsel = s_nsel, alpha = s_alpha, bit0 = s_bit;
    const int64_t nbits = D.src_len * 8;
    // selector i is a run of ones ended by a zero: zpos[i] = where its zero is
    int found = 0;
    for (int64_t base = bit0; found < nsel && base < nbits; base += 32 * kHdrThreads) {
        const int64_t at = base + 32 * t;
        uint32_t z = at < nbits ? ~stream_bits32(D.src, D.src_len, at) : 0u;
        if (at + 32 > nbits && at < nbits) z &= ~0u << (32 - (int)(nbits - at));
        int total;
        int i = found + block_excl_sum<int>(__popc(z), sh, &total);
        while (z && i < nsel) {
            const int k = __clz(z);
            zpos[i++] = (int32_t)(at + k);
            z &= ~(0x80000000u >> k);
        }
        found += total;
    }
    __syncthreads();
    if (found < nsel) {
        if (t == 0) M.status = DEC_TRUNC;
        return;
    }
    // move-to-front over the tables: a stretch of selectors per thread, its
    // moves as one permutation, a scan over the stretches
    const int per = (nsel + kHdrThreads - 1) / kHdrThreads;
    const int a = min(nsel, t * per), e = min(nsel, a + per);
    uint32_t l = kListId;
    bool bad = false;
    for (int i = a; i < e; i++) {
        const int j = zpos[i] - (i ? zpos[i - 1] : bit0 - 1) - 1;
        bad |= j >= ng;
        l = list_move(l, min(j, 5));
    }
    uint32_t incl = l;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(LFC_FULL, incl, o);
        if (lane >= o) incl = list_after(x, incl);
    }
    if (lane == 31) wlist[w] = incl;
    if (__syncthreads_or(bad)) {
        if (t == 0) M.status = DEC_BAD_TABLE;
        return;
    }
    uint32_t before = __shfl_up_sync(LFC_FULL, incl, 1), cur = kListId;
    for (int i = 0; i < w; i++) cur = list_after(cur, wlist[i]);
    if (lane > 0) cur = list_after(cur, before);
    for (int i = a; i < e; i++) {
        const int j = zpos[i] - (i ? zpos[i - 1] : bit0 - 1) - 1;
        cur = list_move(cur, j);
        sel[i] = (uint8_t)(cur & 15u);
    }
    // code lengths: 5-bit start, then per symbol steps "10" up / "11" down and a "0"
    if (t == 0) {
        BitReader br;
        br.init(D.src, D.src_len);
        br.seek((int64_t)zpos[nsel - 1] + 1);
        int st = DEC_OK;
        for (int g = 0; g < ng && st == DEC_OK; g++) {
            int c = (int)br.get(5);
            for (int v = 0; v < alpha && st == DEC_OK; v++) {
                for (;;) {
                    if (br.bcnt < 2) br.refill();
                    if (c < 1 || c > 20 || br.bcnt < 1) { st = br.bcnt < 1 ? DEC_TRUNC : DEC_BAD_TABLE; break; }
                    if (!(br.buf >> 63)) {
                        br.buf <<= 1;
                        br.bcnt--;
                        break;
                    }
                    if (br.bcnt < 2) { st = DEC_TRUNC; break; }
                    c += (br.buf >> 62) & 1 ? -1 : 1;
                    br.buf <<= 2;
                    br.bcnt -= 2;
                }
                len[g][v] = (uint8_t)c;
            }
        }
        if (br.err) st = DEC_TRUNC;
        s_status = st;
        s_bit = (int)br.tell();
    }
    __syncthreads();
    if (s_status != DEC_OK) {
        if (t == 0) M.status = s_status;
        return;
    }
    // canonical tables: the codes of length l are first[l] .. first[l] +
    // count[l] - 1, in increasing symbol order
    for (int i = t; i < kMaxGroups * 22; i += kHdrThreads) (&count[0][0])[i] = 0;
    __syncthreads();
    for (int i = t; i < ng * alpha; i += kHdrThreads) atomicAdd(&count[i / alpha][len[i / alpha][i % alpha]], 1);
    __syncthreads();
    if (t < ng) {
        int32_t code = 0;
        int np = 0;
        for (int k = 1; k <= 20; k++) {
            first[t][k] = code;
            pidx[t][k] = np;
            np += count[t][k];
            code = (code + count[t][k]) << 1;
        }
    }
    __syncthreads();
    for (int i = t; i < ng * alpha; i += kHdrThreads) {
        const int g = i / alpha, v = i - g * alpha, k = len[g][v];
        int r = 0;
        for (int x = 0; x < v; x++) r += len[g][x] == k;
        perm[g][pidx[g][k] + r] = (uint16_t)v;
    }
    __syncthreads();
    for (int i = t; i < kMaxGroups * kMaxAlpha; i += kHdrThreads) (&T.perm[0][0])[i] = (&perm[0][0])[i];
    for (int i = t; i < kMaxGroups * 22; i += kHdrThreads) {
        (&T.first[0][0])[i] = (&first[0][0])[i];
        (&T.count[0][0])[i] = (&count[0][0])[i];
        (&T.pidx[0][0])[i] = (&pidx[0][0])[i];
    }
    // length of the code that x, n bits, begins with; 0 if it is longer
    auto code_len = [&](int g, uint32_t x, int n) {
        for (int k = 1; k <= n; k++)
            if ((uint32_t)((int32_t)(x >> (n - k)) - first[g][k]) < (uint32_t)count[g][k]) return k;
        return 0;
    };
    for (int x = t; x < 1 << kJBits; x += kHdrThreads) {
        uint32_t k[8] = {};
#pragma unroll
        for (int g = 0; g < kMaxGroups; g++)
            if (g < ng) k[g] = code_len(g, x, kJBits);
        T.jlut[x] = make_uint2(k[0] | (k[1] << 8) | (k[2] << 16) | (k[3] << 24), k[4] | (k[5] << 8));
    }
    for (int i = t; i < ng << 10; i += kHdrThreads) {
        const int g = i >> 10;
        const uint32_t x = i & 1023;
        const int k = code_len(g, x, 10);
        T.lut[g][x] = k ? (uint16_t)((perm[g][pidx[g][k] + ((int32_t)(x >> (10 - k)) - first[g][k])] << 5) | k) : (uint16_t)0;
    }
    if (t == 0) {
        M.group = 0;
        M.bit = s_bit;
        M.nsym = 0;
        M.m = 0;
        M.status = DEC_OK;
    }
}

// ------------------------------------------------------ 2. group offsets
// Lengths of 50 codes from every bit of a stretch of kJRange bits, for every
// table: a tile of kJTile bits per CTA with the bits its groups reach into.
// One 8-byte lookup gives a bit position's code length in all six tables;
// lengths of 2, 4, 8 and 16 codes are bytes (0: there are none, or they are
// too long; such a group is decoded on the chase), four positions a thread:
// one load and one store of a word, four byte gathers and byte-wise sums a
// doubling. Bound by shared memory, about 10 accesses per bit and table: 139
// blocks take 3.06 ms (16-bit lengths, two positions a thread and a lookup per
// table: 6.04), one 1300 x 1300 frame 0.17 ms (0.42).
constexpr int kJTile = 8192;
constexpr int kJHalo = 1024;                  // 2 + 16 + 16 + 16 codes: at most 40 + 3 * 254 bits, and the last code's 20
constexpr int kJSpan = kJTile + kJHalo;
constexpr int kJRange = (kBlockCap * 4 / 3) / kJTile * kJTile;  // bits per round: three tables fill a slot of 8-byte words
constexpr int kJThreads = 768;                // three words each
static_assert((size_t)kJRange * 3 * 2 <= (size_t)kBlockCap * 8, "three tables of one round fit a key slot");
static_assert(kJSpan % (4 * kJThreads) == 0, "whole words per thread");

struct JumpSmem {
    uint2 lut[1 << kJBits];
    __align__(16) uint8_t one[kMaxGroups][kJSpan + 256];             // 256 zeros behind every span
    __align__(16) uint8_t b[kJSpan + 256], c[kJSpan + 256];
    int32_t first[kMaxGroups][20 - kJBits], count[kMaxGroups][20 - kJBits];  // codes longer than the lookup's
    uint32_t bits[kJSpan / 32 + 4];
};

// 0xff for every byte of x whose top bit is set
__device__ __forceinline__ uint32_t top_bytes(uint32_t x) {
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(r) : "r"(x));
    return r;
}
// 0xff for every byte of x, all below 128, that is not 0
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t x) { return top_bytes(x + 0x7f7f7f7fu); }

__global__ void __launch_bounds__(kJThreads, 2) dec_jump_kernel(const DecBlock *__restrict__ blocks, const DecMeta *__restrict__ meta,
                                                                const DecTab *__restrict__ tabs, size_t tab_stride, int64_t range0,
                                                                uint64_t *__restrict__ j0_all, uint64_t *__restrict__ j1_all) {
    extern __shared__ __align__(16) uint8_t smraw[];
    JumpSmem &S = *reinterpret_cast<JumpSmem *>(smraw);
    const int b = blockIdx.y, t = threadIdx.x;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK || M.group >= M.n_sel - 1) return;
    const DecBlock D = blocks[b];
    const int64_t nbits = D.src_len * 8;
    const int64_t w0 = range0 + (int64_t)blockIdx.x * kJTile;
    if (w0 >= nbits || w0 + kJTile <= M.bit) return;
    const DecTab &T = *reinterpret_cast<const DecTab *>(reinterpret_cast<const uint8_t *>(tabs) + (size_t)b * tab_stride);
    const int ng = M.n_groups;
    for (int i = t; i < (1 << kJBits) / 2; i += kJThreads)
        reinterpret_cast<uint4 *>(S.lut)[i] = __ldg(reinterpret_cast<const uint4 *>(T.jlut) + i);
    for (int i = t; i < kJSpan / 32 + 4; i += kJThreads) S.bits[i] = stream_bits32(D.src, D.src_len, w0 + 32 * i);
    for (int i = t; i < kMaxGroups * (20 - kJBits); i += kJThreads) {
        const int g = i / (20 - kJBits), l = kJBits + 1 + i % (20 - kJBits);
        (&S.first[0][0])[i] = T.first[g][l];
        (&S.count[0][0])[i] = g < ng ? T.count[g][l] : 0;
    }
    if (t < 64 * (kMaxGroups + 2)) {
        const int r = t >> 6;
        reinterpret_cast<uint32_t *>((r < kMaxGroups ? S.one[r] : r == kMaxGroups ? S.b : S.c) + kJSpan)[t & 63] = 0;
    }
    __syncthreads();
    for (int i = 4 * t; i < kJSpan; i += 4 * kJThreads) {  // single codes, all tables
        const uint32_t v0 = S.bits[i >> 5], v1 = S.bits[(i >> 5) + 1];
        const uint32_t v = __funnelshift_l(v1, v0, i & 31);  // 20 + 3 bits are looked at
        uint2 e[4];
#pragma unroll
        for (int k = 0; k < 4; k++) e[k] = S.lut[(v << k) >> (32 - kJBits)];
        uint32_t x[kMaxGroups];
        {
            const uint32_t p = __byte_perm(e[0].x, e[1].x, 0x5140), q = __byte_perm(e[2].x, e[3].x, 0x5140);
            const uint32_t r = __byte_perm(e[0].x, e[1].x, 0x7362), u = __byte_perm(e[2].x, e[3].x, 0x7362);
            x[0] = __byte_perm(p, q, 0x5410);
            x[1] = __byte_perm(p, q, 0x7632);
            x[2] = __byte_perm(r, u, 0x5410);
            x[3] = __byte_perm(r, u, 0x7632);
            const uint32_t f = __byte_perm(e[0].y, e[1].y, 0x5140), h = __byte_perm(e[2].y, e[3].y, 0x5140);
            x[4] = __byte_perm(f, h, 0x5410);
            x[5] = __byte_perm(f, h, 0x7632);
        }
#pragma unroll
        for (int g = 0; g < kMaxGroups; g++) {
            if (g >= ng) break;
            uint32_t z = ~nonzero_bytes(x[g]) & 0x01010101u;
            while (z) {  // a longer code, or none
                const int sh = __ffs(z) - 1;
                z &= z - 1;
                const uint32_t y = v << (sh >> 3);
                for (int l = kJBits + 1; l <= 20; l++)
                    if ((uint32_t)((int32_t)(y >> (32 - l)) - S.first[g][l - kJBits - 1]) < (uint32_t)S.count[g][l - kJBits - 1]) {
                        x[g] |= (uint32_t)l << sh;
                        break;
                    }
            }
            *reinterpret_cast<uint32_t *>(S.one[g] + i) = x[g];
        }
    }
    __syncthreads();
    auto twice = [&](const uint8_t *in, uint8_t *out, bool cap) {
#pragma unroll
        for (int r = 0; r < kJSpan / (4 * kJThreads); r++) {
            const int i = 4 * (t + r * kJThreads);
            const uint32_t x = *reinterpret_cast<const uint32_t *>(in + i);
            const uint32_t y0 = in[__dp4a(x, 0x1u, (uint32_t)i)], y1 = in[__dp4a(x, 0x100u, (uint32_t)i) + 1];
            const uint32_t y2 = in[__dp4a(x, 0x10000u, (uint32_t)i) + 2], y3 = in[__dp4a(x, 0x1000000u, (uint32_t)i) + 3];
            const uint32_t y = __byte_perm(__byte_perm(y0, y1, 0x0040), __byte_perm(y2, y3, 0x0040), 0x5410);
            uint32_t v = (x + y) & nonzero_bytes(y);  // x is 0 where y is read at its own place
            if (cap) v &= ~top_bytes(v);  // eight codes of more than 127 bits
            *reinterpret_cast<uint32_t *>(out + i) = v;
        }
        __syncthreads();
    };
    for (int g = 0; g < ng; g++) {
        twice(S.one[g], S.b, false);  // 2: at most 40 bits
        twice(S.b, S.c, false);       // 4: at most 80
        twice(S.c, S.one[g], true);   // 8: at most 127
        twice(S.one[g], S.c, false);  // 16: at most 254
        uint16_t *out = reinterpret_cast<uint16_t *>((g < 3 ? j0_all : j1_all) + (size_t)b * kBlockCap) + (size_t)(g % 3) * kJRange +
                        (size_t)blockIdx.x * kJTile;
#pragma unroll
        for (int r = 0; r < kJSpan / (4 * kJThreads); r++) {  // 2 + 16 + 16 + 16
            const int i = 4 * (t + r * kJThreads);
            if (i >= kJTile) break;
            const uint32_t x = *reinterpret_cast<const uint32_t *>(S.b + i);
            uint32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                uint32_t j = __dp4a(x, 1u << (8 * k), (uint32_t)i) + k;  // a walk that meets a 0 stands still on it
                j += S.c[j];
                j += S.c[j];
                const uint32_t d = S.c[j];
                v[k] = d ? j + d - (i + k) : 0u;
            }
            *reinterpret_cast<uint2 *>(out + i) = make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
        }
        __syncthreads();
    }
}

// One CTA per block: thread 0 adds up the groups' lengths, the other warps
// fetch the next window of them. After the last round also the last group,
// up to EOB. Bound by that chain, about 80 cycles a group: the copying warps
// wait four times as long at the barrier as for their loads (ncu, one frame's
// five blocks). 0.73 ms for one 1300 x 1300 frame and 0.94 ms for 139 blocks
// (with windows of 4096 bits 0.91 and 1.10).
constexpr int kChaseThreads = 256;
constexpr int kChaseWin = 8192;  // bits of a window: long enough that its barriers and copies hide behind 56 groups' adds
constexpr int kChaseBufs = 2;    // one in use, one on its way
struct ChaseSmem {
    __align__(16) uint16_t j[kChaseBufs][kMaxGroups][kChaseWin];
    uint8_t sel[kMaxSelectors + 14];
    int64_t p;
    int g, status;
};
static_assert(kJRange % kChaseWin == 0, "a round holds whole windows");

__device__ __forceinline__ void cp_async16(void *smem, const void *g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(g) : "memory");
}

__global__ void __launch_bounds__(kChaseThreads) dec_chase_kernel(const DecBlock *__restrict__ blocks, DecMeta *__restrict__ meta,
                                                                  const DecTab *__restrict__ tabs, size_t tab_stride, int64_t range0,
                                                                  const uint64_t *__restrict__ j0_all, const uint64_t *__restrict__ j1_all,
                                                                  const uint8_t *__restrict__ sel_all, int32_t *__restrict__ gofs_all) {
    extern __shared__ __align__(16) uint8_t smraw[];
    ChaseSmem &S = *reinterpret_cast<ChaseSmem *>(smraw);
    const int b = blockIdx.x, t = threadIdx.x;
    DecMeta &M = meta[b];
    if (M.status != DEC_OK || M.group >= M.n_sel) return;
    const DecBlock D = blocks[b];
    const int64_t nbits = D.src_len * 8;
    const int last = M.n_sel - 1, ng = M.n_groups;
    const DecTab &T = *reinterpret_cast<const DecTab *>(reinterpret_cast<const uint8_t *>(tabs) + (size_t)b * tab_stride);
    int32_t *gofs = gofs_all + (size_t)b * kBlockCap;
    for (int i = t; i <= last; i += kChaseThreads) S.sel[i] = sel_all[(size_t)b * kMaxSelectors + i];
    if (t == 0) {
        S.p = M.bit;
        S.g = M.group;
        S.status = DEC_OK;
    }
    __syncthreads();
    const int64_t range1 = min(nbits, range0 + kJRange);
    auto fetch = [&](int64_t w, int buf) {  // the window at bit w, by the warps behind the first
        if (t >= 32 && w < range1) {
            const size_t o = (size_t)(w - range0);
            for (int g = 0; g < ng; g++) {
                const uint16_t *in = reinterpret_cast<const uint16_t *>((g < 3 ? j0_all : j1_all) + (size_t)b * kBlockCap) +
                                     (size_t)(g % 3) * kJRange + o;
                for (int q = t - 32; q < kChaseWin / 8; q += kChaseThreads - 32) cp_async16(&S.j[buf][g][8 * q], in + 8 * q);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (S.p < range1 && S.g < last) {
        int64_t w = range0 + (S.p - range0) / kChaseWin * kChaseWin;
        fetch(w, 0);
        for (int buf = 0; w < range1; w += kChaseWin, buf ^= 1) {
            bool stop = false;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();  // the window is there, and the one before is done with
            fetch(w + kChaseWin, buf ^ 1);
            if (t == 0) {
                int g = S.g;
                int q = (int)(S.p - w);
                const int32_t base = (int32_t)w;
                const uint16_t *J = &S.j[buf][0][0];
                int tb = S.sel[g];
                while (g < last && q < kChaseWin) {
                    const int nt = S.sel[g + 1];  // g < last: there is one
                    int d = J[tb * kChaseWin + q];
                    gofs[g] = base + q;
                    if (d == 0) {  // not in the table: decode the group (or find that it cannot be)
                        BitReader br;
                        br.init(D.src, D.src_len);
                        br.seek(w + q);
                        for (int k = 0; k < 50; k++)
                            if (huff_symbol(br, T.lut[tb], *reinterpret_cast<const Canon *>(T.first), T, tb) < 0) { S.status = br.err ? DEC_TRUNC : DEC_BAD_DATA; break; }
                        d = (int)(br.tell() - (w + q));
                        if (S.status != DEC_OK) { g = last; break; }
                    }
                    q += d;
                    tb = nt;
                    g++;
                }
                S.g = g;
                S.p = w + q;
                if (S.p > nbits && S.status == DEC_OK) S.status = DEC_TRUNC;
                stop = g >= last || S.status != DEC_OK;
            }
            if (__syncthreads_or(stop)) break;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    if (t != 0) return;
    M.group = S.g;
    M.bit = (int32_t)S.p;
    if (S.status == DEC_OK && S.g < last && range1 == nbits) S.status = DEC_TRUNC;
    if (S.status != DEC_OK) {
        M.status = S.status;
        return;
    }
    if (S.g != last) return;
    BitReader br;
    br.init(D.src, D.src_len);
    br.seek(S.p);
    const int tb = S.sel[last], alpha = M.alpha;
    gofs[last] = (int32_t)S.p;
    for (int k = 0; k < 50; k++) {
        const int sym = huff_symbol(br, T.lut[tb], *reinterpret_cast<const Canon *>(T.first), T, tb);
        if (sym < 0) { M.status = br.err ? DEC_TRUNC : DEC_BAD_DATA; return; }
        if (sym == alpha - 1) {
            M.nsym = last * 50 + k + 1;
            M.group = last + 1;
            return;
        }
    }
    M.status = DEC_BAD_DATA;  // no EOB
}

// ---------------------------------------------------------- 3. symbols
// 0.03 ms for one frame, 0.22 ms for 139 blocks.
constexpr int kSymGroups = 128;

__global__ void __launch_bounds__(kSymGroups) dec_symbols_kernel(const DecBlock *__restrict__ blocks, DecMeta *__restrict__ meta,
                                                                 const DecTab *__restrict__ tabs, size_t tab_stride,
                                                                 const uint8_t *__restrict__ sel_all, const int32_t *__restrict__ gofs_all,
                                                                 uint16_t *__restrict__ sym_all) {
    __shared__ __align__(16) uint16_t lut[kMaxGroups][1 << 10];
    __shared__ __align__(16) uint16_t out[kSymGroups * 50];
    __shared__ Canon C;
    const int b = blockIdx.y, t = threadIdx.x;
    DecMeta &M = meta[b];
    if (__syncthreads_or(M.status != DEC_OK)) return;  // one answer for the CTA: another one may set it meanwhile
    const int g0 = blockIdx.x * kSymGroups, ns = M.nsym, eob = M.alpha - 1;
    if (g0 * 50 >= ns) return;
    const DecBlock D = blocks[b];
    if (ns - 1 > column_bound(D.expect)) {
        M.status = DEC_BAD_DATA;
        return;
    }
    const DecTab &T = *reinterpret_cast<const DecTab *>(reinterpret_cast<const uint8_t *>(tabs) + (size_t)b * tab_stride);
    for (int i = t; i < M.n_groups * 128; i += kSymGroups)
        reinterpret_cast<uint4 *>(lut)[i] = __ldg(reinterpret_cast<const uint4 *>(T.lut) + i);
    for (int i = t; i < 3 * kMaxGroups * 22; i += kSymGroups) (&C.first[0][0])[i] = (&T.first[0][0])[i];
    __syncthreads();
    const int g = g0 + t;
    if (g * 50 < ns) {
        BitReader br;
        br.init(D.src, D.src_len);
        br.seek(gofs_all[(size_t)b * kBlockCap + g]);
        const int tb = sel_all[(size_t)b * kMaxSelectors + g], cnt = min(50, ns - g * 50);
        bool bad = false;
        for (int k = 0; k < cnt; k++) {
            const int sym = huff_symbol(br, lut[tb], C, T, tb);
            bad |= sym < 0 || (sym == eob) != (g * 50 + k == ns - 1);  // EOB is the last symbol, and only that
            out[t * 50 + k] = (uint16_t)sym;
        }
        if (bad) M.status = DEC_BAD_DATA;
    }
    __syncthreads();
    const int n = min(kSymGroups * 50, ns - g0 * 50);
    uint16_t *sym = sym_all + (size_t)b * (kBlockCap + 64) + g0 * 50;
    for (int i = t; i < n; i += kSymGroups) sym[i] = out[i];
}

// ------------------------------------------- 4. inverse RUNA/RUNB and MTF
// Segments start right after a symbol that is not a run digit, so no run is
// split: segment s begins at the first such place in its share of the symbols
// and ends at the first one past it. A thread's list is 32 words of 8 bytes,
// word i of thread t at [i][t]; moving entry j to the front shifts the words
// below it by a byte.
constexpr int kSegThreadsM = 128;
constexpr int kSegs = 24 * kSegThreadsM;                       // most segments of a block
constexpr int kSegGroup = 48, kSegGroups = kSegs / kSegGroup;  // 64 groups
constexpr int kSegStep = 384;                                  // segment counts are multiples of 3 CTAs and 8 groups
constexpr int kSegSyms = 32;  // symbols of a segment, at least, in the largest block there can be
static_assert(kSegs % kSegStep == 0 && kSegStep % kSegThreadsM == 0 && kSegStep % kSegGroup == 0, "whole CTAs and groups");

struct SegInfo {
    int32_t len, status, off;
};
// a block's slot in the segment buffer: permutations, start lists, records
constexpr size_t kSegPerm = 0, kSegList = (size_t)kSegs * 256, kSegInfo = 2 * (size_t)kSegs * 256,
                 kGroupPerm = kSegInfo + kSegs * sizeof(SegInfo);
static_assert(kGroupPerm + kSegGroups * 256 <= sizeof(int32_t) * (size_t)kBlockCap, "segment records fit a block's slot");

// PASS 0: the permutation of list positions and the output length; PASS 1:
// the output bytes from the segment's starting list. One 1300 x 1300 frame
// takes 0.13 and 0.27 ms, 139 blocks 0.68 and 0.90: a serial chain of shared
// memory accesses per symbol, so the segments are short (768 of them, one
// after the other in the chaining, took 0.49 and 1.02, 0.77 and 1.31).
template <int PASS>
__global__ void __launch_bounds__(kSegThreadsM) dec_mtf_kernel(DecMeta *__restrict__ meta, const uint16_t *__restrict__ sym_all,
                                                               uint8_t *__restrict__ seg_all, uint8_t *__restrict__ L_all, int segs) {
    extern __shared__ __align__(16) uint64_t list_all[];
    const int b = blockIdx.y, t = threadIdx.x, s = blockIdx.x * kSegThreadsM + t;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    uint64_t *list = list_all + t;  // word i at list[i * kSegThreadsM]
    uint8_t *slot = seg_all + (size_t)b * kBlockCap * sizeof(int32_t);
    SegInfo *info = reinterpret_cast<SegInfo *>(slot + kSegInfo) + s;
    const uint16_t *sym = sym_all + (size_t)b * (kBlockCap + 64);
    const int ns = M.nsym, niu = M.n_in_use, alpha = M.alpha, block_max = M.block_max;
    const int per = (ns + segs - 1) / segs, s0 = min(ns, s * per), e0 = min(ns, s0 + per);
    int i = s0;
    if (s > 0)
        while (i < e0 && sym[i - 1] < 2) i++;
    if (i >= e0) {  // empty: its symbols belong to the segment before
        if (PASS == 0) {
            info->len = 0;
            info->status = DEC_OK;
            uint64_t *perm = reinterpret_cast<uint64_t *>(slot + kSegPerm + (size_t)s * 256);
            for (int k = 0; k < 32; k++) perm[k] = 0x0706050403020100ull + 0x0808080808080808ull * (uint64_t)k;
        }
        return;
    }
    const uint64_t *start = reinterpret_cast<const uint64_t *>(slot + kSegList + (size_t)s * 256);
    for (int k = 0; k < 32; k++)
        list[k * kSegThreadsM] = PASS == 0 ? 0x0706050403020100ull + 0x0808080808080808ull * (uint64_t)k : start[k];
    uint8_t *L = L_all + (size_t)b * kBlockCap;
    int out = PASS == 1 ? info->off : 0;
    const int out0 = out, cap = PASS == 1 ? M.m : block_max;
    int st = DEC_OK, run = 0, bit = 0;
    uint64_t acc = 0;  // output bytes of the 8-byte word being filled
    int acc_n = 0;
    auto put = [&](uint32_t v) {  // PASS 1; out < cap
        acc |= (uint64_t)v << (8 * (out & 7));
        acc_n++;
        out++;
        if ((out & 7) == 0) {
            if (acc_n == 8) *reinterpret_cast<uint64_t *>(L + out - 8) = acc;
            else
                for (int k = 8 - acc_n; k < 8; k++) L[out - 8 + k] = (uint8_t)(acc >> (8 * k));
            acc = 0;
            acc_n = 0;
        }
    };
    for (; i < ns; i++) {
        const int x = sym[i];
        if (i >= e0 && sym[i - 1] >= 2) break;  // the next segment starts here
        if (x < 2) {
            if (bit > 20 || (run += (x + 1) << bit) > block_max) { st = DEC_OVERFLOW; break; }
            bit++;
            continue;
        }
        if (run) {
            if (run > cap - out) { st = DEC_OVERFLOW; break; }
            if (PASS == 1) {
                const uint32_t v = (uint32_t)list[0] & 255u;
                while (run && (out & 7)) { put(v); run--; }
                const uint64_t v8 = v * 0x0101010101010101ull;
                for (; run >= 8; run -= 8, out += 8) *reinterpret_cast<uint64_t *>(L + out) = v8;
                while (run) { put(v); run--; }
            } else {
                out += run;
            }
            run = bit = 0;
        }
        if (x == alpha - 1) break;  // EOB
        const int j = x - 1, k = j >> 3, r = j & 7;
        if (j >= niu) { st = DEC_BAD_DATA; break; }
        if (out >= cap) { st = DEC_OVERFLOW; break; }
        const uint64_t wk = list[k * kSegThreadsM], v = (wk >> (8 * r)) & 255u;
        uint64_t carry = v;
        for (int q = 0; q < k; q++) {
            const uint64_t w = list[q * kSegThreadsM];
            list[q * kSegThreadsM] = (w << 8) | carry;
            carry = w >> 56;
        }
        const uint64_t keep = r == 7 ? 0ull : ~0ull << (8 * (r + 1));
        list[k * kSegThreadsM] = (wk & keep) | (((wk << 8) | carry) & ~keep);
        if (PASS == 1) put((uint32_t)v); else out++;
    }
    if (PASS == 0) {
        info->len = out;
        info->status = st;
        uint64_t *perm = reinterpret_cast<uint64_t *>(slot + kSegPerm + (size_t)s * 256);
        for (int k = 0; k < 32; k++) perm[k] = list[k * kSegThreadsM];
    } else {
        if (acc_n) {
            const int o = out & 7;
            for (int k = o - acc_n; k < o; k++) L[out - o + k] = (uint8_t)(acc >> (8 * k));
        }
        if (st != DEC_OK || out - out0 != info->len) meta[b].status = st != DEC_OK ? st : DEC_BAD_DATA;
    }
}

// The lists at the segments' starts. A segment takes the list entry at
// position perm[q] to position q, so the segments compose as gathers: per
// group of 48 the whole group's permutation, per block the list at every
// group's start (and the segments' output offsets), per group the list at
// every segment's start. One after the other over 3072 segments it would be
// 0.2 ms.
__global__ void __launch_bounds__(256) dec_seg_group_kernel(const DecMeta *__restrict__ meta, uint8_t *__restrict__ seg_all) {
    __shared__ __align__(16) uint8_t perm[kSegGroup * 256];
    __shared__ uint8_t cur[2][256];
    const int b = blockIdx.y, g = blockIdx.x, t = threadIdx.x;
    if (meta[b].status != DEC_OK) return;
    uint8_t *slot = seg_all + (size_t)b * kBlockCap * sizeof(int32_t);
    const uint4 *in = reinterpret_cast<const uint4 *>(slot + kSegPerm + (size_t)g * kSegGroup * 256);
    for (int i = t; i < kSegGroup * 16; i += 256) reinterpret_cast<uint4 *>(perm)[i] = in[i];
    cur[0][t] = (uint8_t)t;
    __syncthreads();
    for (int k = 0; k < kSegGroup; k++) {
        cur[(k & 1) ^ 1][t] = cur[k & 1][perm[k * 256 + t]];
        __syncthreads();
    }
    slot[kGroupPerm + g * 256 + t] = cur[kSegGroup & 1][t];
}

__global__ void __launch_bounds__(256) dec_seg_chain_kernel(const DecBlock *__restrict__ blocks, DecMeta *__restrict__ meta,
                                                            const DecTab *__restrict__ tabs, size_t tab_stride,
                                                            uint8_t *__restrict__ seg_all, int segs) {
    constexpr int PER = kSegs / 256;
    const int groups_n = segs / kSegGroup;
    __shared__ __align__(16) uint8_t perm[kSegGroups * 256];
    __shared__ uint8_t cur[2][256];
    __shared__ int sh[33];
    const int b = blockIdx.x, t = threadIdx.x;
    DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    const DecTab &T = *reinterpret_cast<const DecTab *>(reinterpret_cast<const uint8_t *>(tabs) + (size_t)b * tab_stride);
    uint8_t *slot = seg_all + (size_t)b * kBlockCap * sizeof(int32_t);
    SegInfo *info = reinterpret_cast<SegInfo *>(slot + kSegInfo);
    uint4 *groups = reinterpret_cast<uint4 *>(slot + kGroupPerm);
    for (int i = t; i < groups_n * 16; i += 256) reinterpret_cast<uint4 *>(perm)[i] = groups[i];
    // output offsets; a segment has at most block_max bytes, so the sum of
    // 3072 lengths fits 32 bits unsigned
    uint32_t c[PER], sum = 0;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < PER; i++) {
        c[i] = 0;
        if (t * PER + i >= segs) continue;
        const SegInfo I = info[t * PER + i];
        c[i] = (uint32_t)I.len;
        sum += c[i];
        bad |= I.status != DEC_OK;
    }
    uint32_t total;
    uint32_t off = block_excl_sum<uint32_t>(sum, reinterpret_cast<uint32_t *>(sh), &total);
    if (__syncthreads_or(bad) || total > (uint32_t)M.block_max || total > (uint32_t)column_bound(blocks[b].expect) ||
        (uint32_t)M.orig >= total) {
        if (t == 0) M.status = total <= (uint32_t)M.block_max && (uint32_t)M.orig >= total ? DEC_BAD_ORIG : DEC_BAD_DATA;
        return;
    }
#pragma unroll
    for (int i = 0; i < PER; i++) {
        if (t * PER + i < segs) info[t * PER + i].off = (int32_t)off;
        off += c[i];
    }
    if (t == 0) M.m = (int32_t)total;
    cur[0][t] = t < M.n_in_use ? T.seq_to_unseq[t] : (uint8_t)0;
    __syncthreads();
    for (int k = 0; k < groups_n; k++) {
        slot[kGroupPerm + k * 256 + t] = cur[k & 1][t];  // the group's permutation is in shared memory
        cur[(k & 1) ^ 1][t] = cur[k & 1][perm[k * 256 + t]];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) dec_seg_lists_kernel(const DecMeta *__restrict__ meta, uint8_t *__restrict__ seg_all) {
    __shared__ __align__(16) uint8_t perm[kSegGroup * 256];
    __shared__ uint8_t cur[2][256];
    const int b = blockIdx.y, g = blockIdx.x, t = threadIdx.x;
    if (meta[b].status != DEC_OK) return;
    uint8_t *slot = seg_all + (size_t)b * kBlockCap * sizeof(int32_t);
    const uint4 *in = reinterpret_cast<const uint4 *>(slot + kSegPerm + (size_t)g * kSegGroup * 256);
    for (int i = t; i < kSegGroup * 16; i += 256) reinterpret_cast<uint4 *>(perm)[i] = in[i];
    cur[0][t] = slot[kGroupPerm + g * 256 + t];
    __syncthreads();
    uint8_t *lists = slot + kSegList + (size_t)g * kSegGroup * 256;
    for (int k = 0; k < kSegGroup; k++) {
        lists[k * 256 + t] = cur[k & 1][t];
        cur[(k & 1) ^ 1][t] = cur[k & 1][perm[k * 256 + t]];
        __syncthreads();
    }
}

// -------------------------------------------------------- 5. LF mapping
// next[j] = C[L[j]] + rank of j among equal bytes; a row's word holds it with
// the row's byte above (bits 20 .. 27) and whether a walker of the inverse BWT
// starts at the next row (bit 28).
constexpr int kLfThreads = 256;
constexpr int kRowStart = 28;
constexpr int kWalkStep = 48;  // rows between walkers: as few as the ranking's shared memory allows

// Walker 0 starts at the origin row, walker k > 0 in stretch k - 1 of kWalkStep
// rows, at a scrambled place: in a block that nearly repeats a string n times
// a row's next one has the same place among n rows throughout a copy, so with
// a fixed place and n a multiple of kWalkStep a walk met no start for many
// copies (64 copies of 2812 bytes, starts at every 64th row: one piece of 174 587
// of 179 968 rows, 44 ms). A piece is as long as its walker's luck, and a call of
// few blocks takes as long as its longest one: 550 to 750 rows of a 1300 x 1300
// frame with 64 rows between walkers, whatever the multiplier; with 48 such a
// frame takes 2.19 to 2.25 ms (2.22 to 2.27 with 64).
__device__ __forceinline__ int walk_place(uint32_t stretch) { return (int)__umulhi(stretch * 0x85EBCA6Bu, kWalkStep); }
__device__ __forceinline__ int walk_start(int k, int orig) { return k == 0 ? orig : (k - 1) * kWalkStep + walk_place(k - 1); }
__device__ __forceinline__ bool is_walk_start(uint32_t r) { return r % kWalkStep == (uint32_t)walk_place(r / kWalkStep); }

__global__ void __launch_bounds__(kLfThreads) dec_lf_count_kernel(const DecMeta *__restrict__ meta, const uint8_t *__restrict__ L_all,
                                                                  uint32_t *__restrict__ hist_all) {
    __shared__ uint32_t h[256];
    const int b = blockIdx.y, tile = blockIdx.x, t = threadIdx.x;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK || tile * kTile >= M.m) return;
    h[t] = 0;
    __syncthreads();
    const int a = tile * kTile + 16 * t, m = M.m;
    const uint8_t *L = L_all + (size_t)b * kBlockCap;
    if (a + 16 <= m) {
        const uint4 v = *reinterpret_cast<const uint4 *>(L + a);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 16; k++) atomicAdd(&h[(w[k >> 2] >> (8 * (k & 3))) & 255u], 1u);
    } else {
        for (int k = a; k < m; k++) atomicAdd(&h[L[k]], 1u);
    }
    __syncthreads();
    hist_all[(size_t)b * kBlockCap + (size_t)tile * 256 + t] = h[t];
}

// One CTA per block: per tile and byte, the row of the tile's first such byte.
__global__ void __launch_bounds__(256) dec_lf_scan_kernel(const DecMeta *__restrict__ meta, uint32_t *__restrict__ hist_all) {
    __shared__ uint32_t sh[33];
    const int b = blockIdx.x, t = threadIdx.x;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    uint32_t *h = hist_all + (size_t)b * kBlockCap;
    const int nt = (M.m + kTile - 1) / kTile;
    uint32_t sum = 0;
#pragma unroll 8
    for (int i = 0; i < nt; i++) sum += h[i * 256 + t];
    uint32_t at = block_excl_sum<uint32_t>(sum, sh, nullptr);
#pragma unroll 8
    for (int i = 0; i < nt; i++) {
        const uint32_t c = h[i * 256 + t];
        h[i * 256 + t] = at;
        at += c;
    }
}

__global__ void __launch_bounds__(kLfThreads) dec_lf_map_kernel(const DecMeta *__restrict__ meta, const uint8_t *__restrict__ L_all,
                                                                const uint32_t *__restrict__ hist_all, uint32_t *__restrict__ P_all) {
    constexpr int NW = kLfThreads / 32;
    __shared__ uint32_t wc[NW][256];
    __shared__ __align__(16) uint8_t by[kTile];
    const int b = blockIdx.y, tile = blockIdx.x, t = threadIdx.x, w = t >> 5, lane = t & 31;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK || tile * kTile >= M.m) return;
    const int cnt = min(kTile, M.m - tile * kTile), orig = M.orig;
    const uint8_t *L = L_all + (size_t)b * kBlockCap + (size_t)tile * kTile;
    reinterpret_cast<uint4 *>(by)[t] = *reinterpret_cast<const uint4 *>(L + 16 * t);  // the slot holds whole tiles
    for (int i = t; i < NW * 256; i += kLfThreads) (&wc[0][0])[i] = 0;
    __syncthreads();
    // warp w: bytes [512 w, 512 w + 512) of the tile, 32 at a time in order
    uint32_t rk[kTile / kLfThreads];
#pragma unroll
    for (int r = 0; r < kTile / kLfThreads; r++) {
        const int k = w * 512 + r * 32 + lane;
        const bool ok = k < cnt;
        const uint32_t c = by[k];
        const uint32_t mm = __match_any_sync(LFC_FULL, ok ? c : 256u + lane);
        uint32_t before = 0;
        if (ok) before = wc[w][c];
        __syncwarp();
        if (ok && (mm & lanemask_gt()) == 0) wc[w][c] = before + __popc(mm);
        __syncwarp();
        rk[r] = before + __popc(mm & lanemask_lt());
    }
    __syncthreads();
    uint32_t at = hist_all[(size_t)b * kBlockCap + (size_t)tile * 256 + t];
#pragma unroll
    for (int i = 0; i < NW; i++) {
        const uint32_t c = wc[i][t];
        wc[i][t] = at;
        at += c;
    }
    __syncthreads();
    uint32_t *P = P_all + (size_t)b * kBlockCap + (size_t)tile * kTile;
#pragma unroll
    for (int r = 0; r < kTile / kLfThreads; r++) {
        const int k = w * 512 + r * 32 + lane;
        if (k >= cnt) continue;
        const uint32_t next = wc[w][by[k]] + rk[r];
        const bool start = is_walk_start(next) || (int)next == orig;
        P[k] = next | ((uint32_t)by[k] << 20) | ((uint32_t)start << kRowStart);
    }
}

// ------------------------------------------------------- 6. inverse BWT
// Bound by the latency of dependent 4-byte gathers from L2, about 48 a walker
// and two walks (the bytes can only be placed once the pieces are ranked): 0.10 +
// 0.12 ms for one 1300 x 1300 frame, 0.50 + 0.67 ms for 139 blocks.
constexpr int kWalkMax = kBlockCap / kWalkStep + 2;       // walkers of a block
constexpr uint32_t kRowMask = (1u << 20) - 1u;
// walker records in a block's slot: length, next walker, output position
constexpr size_t kWalkLen = 0, kWalkNext = kWalkMax, kWalkPos = 2 * (size_t)kWalkMax;

__global__ void __launch_bounds__(256) dec_walk_kernel(const DecMeta *__restrict__ meta, const uint32_t *__restrict__ P_all,
                                                       int32_t *__restrict__ rec_all) {
    const int b = blockIdx.y, k = blockIdx.x * 256 + (int)threadIdx.x;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    const int m = M.m, orig = M.orig, K = (m + kWalkStep - 1) / kWalkStep + 1;
    if (k >= K) return;
    const uint32_t *P = P_all + (size_t)b * kBlockCap;
    int32_t *rec = rec_all + (size_t)b * kBlockCap;
    int r = walk_start(k, orig), steps = 0;
    if (k > 0 && (r == orig || r >= m)) {  // walker 0's row, or none in the last stretch
        rec[kWalkLen + k] = 0;
        rec[kWalkNext + k] = 0;
        return;
    }
    uint32_t p;
    do {  // the rows form cycles, so a walk ends at its own row at the latest
        p = P[r];
        r = (int)(p & kRowMask);
        steps++;
    } while ((p >> kRowStart) == 0);
    rec[kWalkLen + k] = steps;
    rec[kWalkNext + k] = r == orig ? 0 : r / kWalkStep + 1;
}

// One CTA per block: where each walker's piece goes, from its distance to
// the end of the list (walker 0 first, ended by the return to it). The list
// holds the rows of the origin's cycle. Identical rotations are neighbouring
// rows in the same order everywhere, so in a block of r copies of a string
// every copy has a cycle of its own, of m / r rows; a cycle whose length does
// not divide m is no encoder's. Walkers off the list write nothing.
struct RankSmem {
    uint32_t d[2][kWalkMax + 1];
    uint16_t nx[2][kWalkMax + 1];
};
__global__ void __launch_bounds__(1024) dec_rank_kernel(DecMeta *__restrict__ meta, int32_t *__restrict__ rec_all) {
    extern __shared__ __align__(16) uint8_t smraw[];
    RankSmem &S = *reinterpret_cast<RankSmem *>(smraw);
    const int b = blockIdx.x, t = threadIdx.x;
    DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    const int m = M.m, K = (m + kWalkStep - 1) / kWalkStep + 1;
    int32_t *rec = rec_all + (size_t)b * kBlockCap;
    for (int k = t; k <= K; k += 1024) {
        const int nx = k < K ? rec[kWalkNext + k] : 0;
        S.d[0][k] = k < K ? (uint32_t)rec[kWalkLen + k] : 0u;
        S.nx[0][k] = (uint16_t)(k == K || nx == 0 ? K : nx);
    }
    __syncthreads();
    int cur = 0;
    for (int span = 1; span < K; span <<= 1, cur ^= 1) {
        for (int k = t; k <= K; k += 1024) {
            const int nx = S.nx[cur][k];
            S.d[cur ^ 1][k] = min(S.d[cur][k] + S.d[cur][nx], 1u << 30);  // off the list the sums only have to stay finite
            S.nx[cur ^ 1][k] = S.nx[cur][nx];
        }
        __syncthreads();
    }
    const int period = (int)S.d[cur][0];
    if (S.nx[cur][0] != K || m % period != 0) {
        if (t == 0) M.status = DEC_BAD_WALK;
        return;
    }
    if (t == 0) M.period = period;
    for (int k = t; k < K; k += 1024) {
        if (S.nx[cur][k] == K) rec[kWalkPos + k] = period - (int)S.d[cur][k];
        else rec[kWalkLen + k] = 0;
    }
}

__global__ void __launch_bounds__(256) dec_emit_kernel(const DecMeta *__restrict__ meta, const uint32_t *__restrict__ P_all,
                                                       const int32_t *__restrict__ rec_all, uint8_t *__restrict__ blk_all) {
    const int b = blockIdx.y, k = blockIdx.x * 256 + (int)threadIdx.x;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    const int m = M.m, K = (m + kWalkStep - 1) / kWalkStep + 1;
    if (k >= K) return;
    const uint32_t *P = P_all + (size_t)b * kBlockCap;
    const int32_t *rec = rec_all + (size_t)b * kBlockCap;
    uint8_t *blk = blk_all + (size_t)b * kBlockCap;
    const int len = rec[kWalkLen + k];
    int r = walk_start(k, M.orig);
    int at = m - rec[kWalkPos + k];  // bytes go to at - 1, at - 2, ...
    uint64_t acc = 0;
    int n = 0;  // bytes of the 8-byte word being filled, from its end
    for (int s = 0; s < len; s++) {
        const uint32_t p = P[r];
        r = (int)(p & kRowMask);
        at--;
        acc |= (uint64_t)((p >> 20) & 255u) << (8 * (at & 7));
        n++;
        if ((at & 7) == 0) {
            if (n == 8) *reinterpret_cast<uint64_t *>(blk + at) = acc;
            else
                for (int q = 0; q < n; q++) blk[at + q] = (uint8_t)(acc >> (8 * q));
            acc = 0;
            n = 0;
        }
    }
    for (int q = 0; q < n; q++) blk[at + q] = (uint8_t)(acc >> (8 * ((at & 7) + q)));
}

// The bytes before the last period of a block that repeats it (any other
// block is left at once, so the grid is small).
constexpr int kRepeatCtas = 8;
__global__ void __launch_bounds__(256) dec_repeat_kernel(const DecMeta *__restrict__ meta, uint8_t *__restrict__ blk_all) {
    const int b = blockIdx.y;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK || M.period == M.m) return;
    const int period = M.period, start = M.m - period;
    uint8_t *blk = blk_all + (size_t)b * kBlockCap;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < start; i += kRepeatCtas * 256) blk[i] = blk[start + i % period];
}

// ----------------------------------------------------- 7. inverse RLE1
// A position q is a sync point when bytes q-2 and q-1 differ and bytes q-5 ..
// q-2 are not all equal: byte q-1 is then a literal (a count byte follows
// four equal literals) that starts a run, so decoding can start at q from
// (run 1, last = byte q-1). A thread starts at the first sync point of its 16
// bytes (the block's first thread at 0, fresh) and stops at the first one
// past them.
constexpr int kUnThreads = 256;
constexpr int kUnStage = 3 * kTile;  // output bytes of a tile staged in shared memory

__device__ __forceinline__ bool rle_sync(const uint8_t *blk, int q) {
    const uint8_t b1 = blk[q - 1], b2 = blk[q - 2];
    return b1 != b2 && !(blk[q - 5] == b2 && blk[q - 4] == b2 && blk[q - 3] == b2);
}

// Walks the thread's bytes; put(byte, count) takes each literal (count 1) and
// repeat. Returns the output bytes, or -1 for a missing count byte.
template <typename Put>
__device__ __forceinline__ int rle_walk(const uint8_t *blk, int m, int a, Put put) {
    const int e = min(m, a + 16);
    int p = a;
    if (a > 0) {
        for (p = max(a, 5); p < e && !rle_sync(blk, p); p++) {}
        if (p >= e) return 0;
    }
    int o = 0, same = p == 0 ? 0 : 1, last = p == 0 ? -1 : (int)blk[p - 1];
    for (int i = p; i < m; i++) {
        if (i >= max(a + 16, 5) && rle_sync(blk, i)) break;
        const uint8_t v = blk[i];
        put(v, 1, o);
        o++;
        same = (int)v == last ? same + 1 : 1;
        last = v;
        if (same == 4) {
            if (i + 1 >= m) return -1;
            const int extra = blk[++i];
            put(v, extra, o);
            o += extra;
            same = 0;
            last = -1;
        }
    }
    return o;
}

__global__ void __launch_bounds__(kUnThreads) dec_unrle_count_kernel(DecMeta *__restrict__ meta, const uint8_t *__restrict__ blk_all,
                                                                     int32_t *__restrict__ aux_all) {
    __shared__ int sh[33];
    const int b = blockIdx.y, tile = blockIdx.x;
    DecMeta &M = meta[b];
    if (__syncthreads_or(M.status != DEC_OK) || tile * kTile >= M.m) return;  // one answer for the CTA, as above
    const int a = tile * kTile + 16 * (int)threadIdx.x;
    int n = a < M.m ? rle_walk(blk_all + (size_t)b * kBlockCap, M.m, a, [](uint8_t, int, int) {}) : 0;
    if (__syncthreads_or(n < 0)) {
        if (threadIdx.x == 0) M.status = DEC_BAD_DATA;
        n = 0;
    }
    int total;
    block_excl_sum<int>(n, sh, &total);
    if (threadIdx.x == 0) aux_all[((size_t)b * kTilesPerBlock + tile) * 4] = total;
}

__global__ void __launch_bounds__(256) dec_unrle_scan_kernel(const DecBlock *__restrict__ blocks, DecMeta *__restrict__ meta,
                                                             int32_t *__restrict__ aux_all) {
    __shared__ int sh[33];
    const int b = blockIdx.x, t = threadIdx.x;
    DecMeta &M = meta[b];
    if (M.status != DEC_OK) return;
    const int nt = (M.m + kTile - 1) / kTile;  // <= 220
    int32_t *aux = aux_all + (size_t)b * kTilesPerBlock * 4;
    int total;
    const int off = block_excl_sum<int>(t < nt ? aux[t * 4] : 0, sh, &total);
    if (t < nt) aux[t * 4 + 1] = off;
    if (t == 0 && total != blocks[b].expect) M.status = DEC_BAD_LEN;
}

__global__ void __launch_bounds__(kUnThreads) dec_unrle_write_kernel(const DecBlock *__restrict__ blocks, const DecMeta *__restrict__ meta,
                                                                     const uint8_t *__restrict__ blk_all,
                                                                     const int32_t *__restrict__ aux_all) {
    __shared__ int sh[33];
    __shared__ uint8_t ob[kUnStage];
    const int b = blockIdx.y, tile = blockIdx.x;
    const DecMeta &M = meta[b];
    if (M.status != DEC_OK || tile * kTile >= M.m) return;
    const uint8_t *blk = blk_all + (size_t)b * kBlockCap;
    const int a = tile * kTile + 16 * (int)threadIdx.x;
    const int n = a < M.m ? rle_walk(blk, M.m, a, [](uint8_t, int, int) {}) : 0;
    int total;
    const int o = block_excl_sum<int>(n, sh, &total);
    uint8_t *dst = blocks[b].dst + aux_all[((size_t)b * kTilesPerBlock + tile) * 4 + 1];
    const bool staged = total <= kUnStage;
    uint8_t *to = (staged ? ob : dst) + o;  // the scan checked the block's total against the promised length
    if (n)
        rle_walk(blk, M.m, a, [&](uint8_t v, int cnt, int at) {
            for (int k = 0; k < cnt; k++) to[at + k] = v;
        });
    if (!staged) return;
    __syncthreads();
    for (int k = threadIdx.x; k < total; k += kUnThreads) dst[k] = ob[k];
}

// Final status per block: what failed, or the CRC check.
__global__ void dec_status_kernel(const DecMeta *__restrict__ meta, int nblocks, int32_t *__restrict__ status) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nblocks) return;
    const DecMeta &M = meta[b];
    status[b] = M.status != DEC_OK ? M.status : (M.crc == M.stored_crc ? DEC_OK : DEC_BAD_CRC);
}

cudaError_t launch_bzip2_decode(lfc_plan P, const DecBlockHost *h_blocks, const void *d_blocks, int nblocks, const uint8_t *d_crc,
                                const CrcRun &crc, int32_t *d_status) {
    Workspace &ws = P->ws;
    cudaStream_t s = P->stream;
    const DecBlock *blocks = reinterpret_cast<const DecBlock *>(d_blocks);
    DecMeta *meta = reinterpret_cast<DecMeta *>(ws.bstate);
    DecTab *tabs = reinterpret_cast<DecTab *>(ws.act2);
    const size_t ts = sizeof(int32_t) * (size_t)kBlockCap;
    uint8_t *seg_buf = reinterpret_cast<uint8_t *>(ws.act);
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws.val);  // the group offsets' slot, free once the symbols are out
    uint32_t *rows = reinterpret_cast<uint32_t *>(ws.sa);
    const size_t list_smem = (size_t)256 * kSegThreadsM;
    cudaError_t e = cudaFuncSetAttribute(dec_chase_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ChaseSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(dec_jump_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(JumpSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(dec_rank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RankSmem));
    if (e != cudaSuccess) return e;
    int64_t max_bits = 0;
    int max_m = 0;  // of the last columns
    for (int b = 0; b < nblocks; b++) {
        if (h_blocks[b].src_len * 8 > max_bits) max_bits = h_blocks[b].src_len * 8;
        if (column_bound(h_blocks[b].expect) > max_m) max_m = column_bound(h_blocks[b].expect);
    }
    // Grids for the largest block there can be, not for the largest of the
    // format: 338 blocks of 900 bytes took 1.3 ms with 3072 segments, 220
    // tiles and 141 CTAs of groups each.
    const int max_groups = (max_m + 1 + 49) / 50, max_tiles = (max_m + kTile - 1) / kTile;
    const int segs = kSegStep * std::min(kSegs / kSegStep, (max_m + kSegStep * kSegSyms) / (kSegStep * kSegSyms));
    dec_header_kernel<<<nblocks, kHdrThreads, 0, s>>>(blocks, meta, tabs, ts, ws.sel, ws.val);
    int launches = 17;
    for (int64_t r0 = 0; r0 < max_bits; r0 += kJRange, launches += 2) {
        const int64_t n = max_bits - r0 < kJRange ? max_bits - r0 : kJRange;
        dec_jump_kernel<<<dim3((unsigned)((n + kJTile - 1) / kJTile), nblocks), kJThreads, sizeof(JumpSmem), s>>>(
            blocks, meta, tabs, ts, r0, ws.keys, ws.keys2);
        dec_chase_kernel<<<nblocks, kChaseThreads, sizeof(ChaseSmem), s>>>(blocks, meta, tabs, ts, r0, ws.keys, ws.keys2, ws.sel, ws.val);
    }
    dec_symbols_kernel<<<dim3((max_groups + kSymGroups - 1) / kSymGroups, nblocks), kSymGroups, 0, s>>>(blocks, meta, tabs, ts, ws.sel,
                                                                                                          ws.val, ws.sym);
    const dim3 seg_grid(segs / kSegThreadsM, nblocks), groups(segs / kSegGroup, nblocks), tiles(max_tiles, nblocks);
    const dim3 walkers((max_m / kWalkStep + 2 + 255) / 256, nblocks);
    dec_mtf_kernel<0><<<seg_grid, kSegThreadsM, list_smem, s>>>(meta, ws.sym, seg_buf, ws.bwt, segs);
    dec_seg_group_kernel<<<groups, 256, 0, s>>>(meta, seg_buf);
    dec_seg_chain_kernel<<<nblocks, 256, 0, s>>>(blocks, meta, tabs, ts, seg_buf, segs);
    dec_seg_lists_kernel<<<groups, 256, 0, s>>>(meta, seg_buf);
    dec_mtf_kernel<1><<<seg_grid, kSegThreadsM, list_smem, s>>>(meta, ws.sym, seg_buf, ws.bwt, segs);
    dec_lf_count_kernel<<<tiles, kLfThreads, 0, s>>>(meta, ws.bwt, hist);
    dec_lf_scan_kernel<<<nblocks, 256, 0, s>>>(meta, hist);
    dec_lf_map_kernel<<<tiles, kLfThreads, 0, s>>>(meta, ws.bwt, hist, rows);
    dec_walk_kernel<<<walkers, 256, 0, s>>>(meta, rows, ws.sa2);
    dec_rank_kernel<<<nblocks, 1024, sizeof(RankSmem), s>>>(meta, ws.sa2);
    dec_emit_kernel<<<walkers, 256, 0, s>>>(meta, rows, ws.sa2, ws.rle);
    dec_repeat_kernel<<<dim3(kRepeatCtas, nblocks), 256, 0, s>>>(meta, ws.rle);
    dec_unrle_count_kernel<<<tiles, kUnThreads, 0, s>>>(meta, ws.rle, ws.tileaux);
    dec_unrle_scan_kernel<<<nblocks, 256, 0, s>>>(blocks, meta, ws.tileaux);
    dec_unrle_write_kernel<<<tiles, kUnThreads, 0, s>>>(blocks, meta, ws.rle, ws.tileaux);
    e = launch_crc(P, d_crc, crc, &meta[0].crc, (int)(sizeof(DecMeta) / 4));
    if (e != cudaSuccess) return e;
    dec_status_kernel<<<(nblocks + 127) / 128, 128, 0, s>>>(meta, nblocks, d_status);
    count_launches(P, launches);
    return cudaGetLastError();
}

// ------------------------------------------------------ inverse predictor
__device__ __forceinline__ int32_t as_s16(uint32_t v) { return (int32_t)(int16_t)(uint16_t)v; }
__device__ __forceinline__ uint32_t unzig(uint32_t z) { return (uint32_t)(((z >> 1) ^ (0u - (z & 1u))) & 0xFFFFu); }

__device__ __forceinline__ int32_t jp(int f, int32_t A, int32_t B, int32_t C) {
    switch (f) {
    case 1: return A;
    case 2: return B;
    case 3: return C;
    case 4: return A + B - C;
    case 5: return A + ((B - C) >> 1);
    case 6: return B + ((A - C) >> 1);
    case 7: return (A + B) >> 1;
    default: return 0;
    }
}
__device__ __forceinline__ int32_t gp(int f, int row, int col, int32_t A, int32_t B, int32_t C) {
    if (row == 0) return col == 0 ? 0 : A;
    if (col == 0) return B;
    return jp(f, A, B, C);
}


__device__ __forceinline__ size_t stream_index(const InvFrame &F, int y, int x) {
    if (!((F.id >> 6) & 1)) return (size_t)y * F.W + x;
    const int Nx = F.W / F.p, Ny = F.H / F.p;
    const int t = y / F.p, v = y % F.p, s = x / F.p, u = x % F.p;
    return (size_t)(v * Ny + t) * F.W + (size_t)u * Nx + s;
}

// Residual field e at every pixel (raw for f == 0 without temporal).
__global__ void inv_residual_kernel(const InvFrame *__restrict__ frames) {
    const InvFrame F = frames[blockIdx.y];
    const int64_t n = (int64_t)F.W * F.H;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int y = (int)(k / F.W), x = (int)(k % F.W);
        const size_t si = stream_index(F, y, x);
        // planar layout: high bytes of all symbols, then their low bytes
        const uint8_t *Z8 = reinterpret_cast<const uint8_t *>(F.Z);
        const uint32_t z = id_planar(F.id) ? ((uint32_t)Z8[si] << 8) | Z8[(size_t)n + si] : F.Z[si];
        const int f = id_f(F.id);
        const bool tmp = id_tmp(F.id);
        F.E[k] = (f == 0 && !tmp) ? (int32_t)z : as_s16(unzig(z));
    }
}

// Inter-lenslet inverse over the view grid of every (u, v): one CTA per
// view restores its Ny x Nx grid by anti-diagonals (cell (t, s) needs the
// cells left, above and above-left, all on the two previous diagonals), one
// thread per cell of a diagonal. The result stays a signed 16-bit field for
// the phase stage and temporal frames. The grid is staged in shared memory
// (its cells are p pixels apart in memory, and a diagonal is one dependent
// step: 60 against 600 cycles); one that does not fit is restored in place.
constexpr int kInterThreads = 256;

__global__ void __launch_bounds__(kInterThreads) inv_inter_kernel(const InvFrame *__restrict__ frames, int smem_cells) {
    extern __shared__ __align__(16) uint16_t cells[];
    const InvFrame F = frames[blockIdx.y];
    const int p = F.p, Nx = F.W / p, Ny = F.H / p;
    const int view = blockIdx.x;
    const int f = id_f(F.id), dom = id_dom(F.id);
    if (f == 0 || dom == 0 || view >= p * p) return;
    const bool signed_field = dom == 2 || id_tmp(F.id);
    const int v = view / p, u = view % p;
    int32_t *E = F.E + (size_t)v * F.W + u;
    const size_t row = (size_t)p * F.W;
    const bool staged = Nx * Ny <= smem_cells;
    if (staged) {
        for (int q = threadIdx.x; q < Nx * Ny; q += kInterThreads) {
            const int t = q / Nx, s = q - t * Nx;
            cells[q] = (uint16_t)E[t * row + (size_t)s * p];
        }
        __syncthreads();
    }
    auto get = [&](int t, int s) -> int32_t {
        if (!staged) return E[t * row + (size_t)s * p];
        const uint32_t x = cells[t * Nx + s];
        return signed_field ? as_s16(x) : (int32_t)x;
    };
    for (int d = 0; d < Nx + Ny - 1; d++) {
        const int t_lo = max(0, d - (Nx - 1)), t_hi = min(Ny - 1, d);
        for (int t = t_lo + (int)threadIdx.x; t <= t_hi; t += kInterThreads) {
            const int s = d - t;
            const int32_t A = s > 0 ? get(t, s - 1) : 0;
            const int32_t B = t > 0 ? get(t - 1, s) : 0;
            const int32_t C = (s > 0 && t > 0) ? get(t - 1, s - 1) : 0;
            const uint32_t val = ((uint32_t)get(t, s) + (uint32_t)gp(f, t, s, A, B, C)) & 0xFFFFu;
            if (staged) cells[t * Nx + s] = (uint16_t)val;
            else E[t * row + (size_t)s * p] = signed_field ? as_s16(val) : (int32_t)val;
        }
        __syncthreads();
    }
    if (staged)
        for (int q = threadIdx.x; q < Nx * Ny; q += kInterThreads) {
            const int t = q / Nx, s = q - t * Nx;
            E[t * row + (size_t)s * p] = get(t, s);
        }
}

// Intra-lenslet inverse: one thread per lenslet, raster order inside it.
__global__ void inv_intra_kernel(const InvFrame *__restrict__ frames) {
    const InvFrame F = frames[blockIdx.y];
    const int p = F.p, Nx = F.W / p, Ny = F.H / p;
    const int lens = blockIdx.x * blockDim.x + threadIdx.x;
    const int f = id_f(F.id);
    if (f == 0 || id_dom(F.id) == 1 || lens >= Nx * Ny) return;
    const bool signed_field = id_tmp(F.id);
    const int t = lens / Nx, s = lens % Nx;
    for (int v = 0; v < p; v++) {
        for (int u = 0; u < p; u++) {
            const size_t k = (size_t)(t * p + v) * F.W + s * p + u;
            const int32_t A = u > 0 ? F.E[k - 1] : 0;
            const int32_t B = v > 0 ? F.E[k - F.W] : 0;
            const int32_t C = (u > 0 && v > 0) ? F.E[k - F.W - 1] : 0;
            const uint32_t val = ((uint32_t)F.E[k] + (uint32_t)gp(f, v, u, A, B, C)) & 0xFFFFu;
            F.E[k] = signed_field ? as_s16(val) : (int32_t)val;
        }
    }
}

// Base field -> raw counts (adds the previous frame for temporal ids).
__global__ void inv_finish_kernel(const InvFrame *__restrict__ frame) {
    const InvFrame F = *frame;
    const int64_t n = (int64_t)F.W * F.H;
    const bool tmp = (F.id >> 7) & 1;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        uint32_t v = (uint32_t)F.E[k];
        if (tmp) v += F.prev[k];
        F.X[k] = (uint16_t)(v & 0xFFFFu);
    }
}

// The frames of a call at once: residual fields, then the inverse
// predictors of the frames that have each stage. The last step runs frame by
// frame, as a temporal frame may need the one before.
cudaError_t launch_inverse_predict(lfc_plan P, const InvFrame *h_frames, const InvFrame *d_frames, int n) {
    cudaStream_t s = P->stream;
    int lenslets = 0, views = 0, cells = 0;
    constexpr int kCellsMax = 100 * 1024;  // 16-bit cells of a view's grid in shared memory
    bool inter = false, intra = false;
    for (int i = 0; i < n; i++) {
        const InvFrame &F = h_frames[i];
        const int f = id_f(F.id), dom = id_dom(F.id);
        inter |= f != 0 && dom != 0;
        intra |= f != 0 && dom != 1;
        const int nl = (F.W / F.p) * (F.H / F.p), nv = F.p * F.p;
        lenslets = nl > lenslets ? nl : lenslets;
        views = nv > views ? nv : views;
        if (nl <= kCellsMax && nl > cells) cells = nl;
    }
    const cudaError_t e = cudaFuncSetAttribute(inv_inter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCellsMax * 2);
    if (e != cudaSuccess) return e;
    inv_residual_kernel<<<dim3(1216, n), 256, 0, s>>>(d_frames);
    if (inter) inv_inter_kernel<<<dim3(views, n), kInterThreads, 2 * (size_t)cells, s>>>(d_frames, cells);
    if (intra) inv_intra_kernel<<<dim3((lenslets + 127) / 128, n), 128, 0, s>>>(d_frames);
    for (int i = 0; i < n; i++) inv_finish_kernel<<<1216, 256, 0, s>>>(d_frames + i);
    count_launches(P, 1 + inter + intra + n);
    return cudaGetLastError();
}

}  // namespace lfc
