// mtf_huff.cu -- move-to-front, zero-run coding, Huffman table choice and bit
// packing of every bzip2 block (Sec. 2.1.3; public bzip2 block format).
//
// MTF is sequential per block, so each block's BWT output is cut into
// segments handled by one warp each. A segment's effect on the MTF list is
// "its distinct bytes by most recent use, then the old list without them".
// These records compose, and composing is associative: the records of groups
// of segments are composed in parallel, one CTA per block chains the groups'
// starting lists, and every group's CTA steps through its segments for
// theirs. Lists hold byte values; only the bytes in use stand in them.
#include <climits>

#include "lfc_common.cuh"

namespace lfc {

constexpr int kSymStride = kBlockCap + 64;  // uint16 symbols per block slot

// ---------------------------------------------------- MTF: segment lists
// The records (distinct bytes of a segment of L by last use, latest first,
// and the bitmap of these bytes) come from the BWT output kernel.
constexpr int kMtfGroup = 32;  // most segments of a group
constexpr int kMtfGroupsMax = (kMtfSegs + 15) / 16;

// Applies a record (length rl, this thread's byte r, bitmap pres) to the list
// cur of n bytes, a byte per thread (256 threads); returns the new length.
// wc: 8 words. Two barriers.
__device__ __forceinline__ int list_apply(uint8_t (*lst)[256], int cur, int n, int rl, uint8_t r, const uint32_t *pres, int *wc) {
    const int t = threadIdx.x, w = t >> 5;
    const uint8_t x = lst[cur][t];
    const bool keep = t < n && !((pres[x >> 5] >> (x & 31)) & 1u);
    const uint32_t kept = __ballot_sync(LFC_FULL, keep);
    if ((t & 31) == 0) wc[w] = __popc(kept);
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        before += i < w ? wc[i] : 0;
        total += wc[i];
    }
    if (keep) lst[cur ^ 1][rl + before + __popc(kept & lanemask_lt())] = x;
    if (t < rl) lst[cur ^ 1][t] = r;
    __syncthreads();
    return rl + total;
}

struct MtfGroupSmem {
    __align__(16) uint8_t rec[kMtfGroup][256];
    uint32_t pres[kMtfGroup][8];
    int32_t len[kMtfGroup];
    uint8_t lst[2][256];
    int wc[8];
};

// The records of segments [s0, s0 + n) of block b into shared memory.
__device__ __forceinline__ void load_records(MtfGroupSmem &S, int b, int s0, int n, const uint8_t *rec_all, const uint32_t *pres_all,
                                             const int32_t *len_all) {
    const size_t seg0 = (size_t)b * kMtfSegs + s0;
    for (int i = threadIdx.x; i < n * 16; i += 256)
        reinterpret_cast<uint4 *>(&S.rec[0][0])[i] = __ldg(reinterpret_cast<const uint4 *>(rec_all + seg0 * 256) + i);
    for (int i = threadIdx.x; i < n * 8; i += 256) (&S.pres[0][0])[i] = pres_all[seg0 * 8 + i];
    for (int i = threadIdx.x; i < n; i += 256) S.len[i] = len_all[seg0 + i];
    __syncthreads();
}

// (1) one CTA per group: its segments' records composed.
__global__ void __launch_bounds__(256) mtf_group_kernel(const BlockState *__restrict__ st, int seg_log2, int group,
                                                        const uint8_t *__restrict__ rec_all, const uint32_t *__restrict__ pres_all,
                                                        const int32_t *__restrict__ len_all, uint8_t *__restrict__ grec_all,
                                                        uint32_t *__restrict__ gpres_all, int32_t *__restrict__ glen_all) {
    __shared__ MtfGroupSmem S;
    const int b = blockIdx.y, g = blockIdx.x, t = threadIdx.x;
    const int nseg = (st[b].m + (1 << seg_log2) - 1) >> seg_log2, s0 = g * group, n = min(group, nseg - s0);
    if (n <= 0) return;
    load_records(S, b, s0, n, rec_all, pres_all, len_all);
    int cur = 0, len = 0;
    for (int i = 0; i < n; i++, cur ^= 1) len = list_apply(S.lst, cur, len, S.len[i], S.rec[i][t], S.pres[i], S.wc);
    const size_t go = (size_t)b * kMtfGroupsMax + g;
    grec_all[go * 256 + t] = S.lst[cur][t];
    if (t < 8) {
        uint32_t p = 0;
        for (int i = 0; i < n; i++) p |= S.pres[i][t];
        gpres_all[go * 8 + t] = p;
    }
    if (t == 0) glen_all[go] = len;
}

// (2) one CTA per block: the list at every group's start (in place of the
// group's record), from the bytes in use in ascending order.
__global__ void __launch_bounds__(256) mtf_chain_kernel(const BlockState *__restrict__ st, int seg_log2, int group,
                                                        uint8_t *__restrict__ grec_all, const uint32_t *__restrict__ gpres_all,
                                                        const int32_t *__restrict__ glen_all) {
    __shared__ uint8_t lst[2][256];
    __shared__ uint32_t pres[kMtfGroupsMax][8];
    __shared__ int32_t lens[kMtfGroupsMax];
    __shared__ int wc[8];
    const int b = blockIdx.x, t = threadIdx.x;
    const int nseg = (st[b].m + (1 << seg_log2) - 1) >> seg_log2, ng = (nseg + group - 1) / group;
    uint8_t *grec = grec_all + (size_t)b * kMtfGroupsMax * 256;
    for (int i = t; i < ng * 8; i += 256) (&pres[0][0])[i] = gpres_all[(size_t)b * kMtfGroupsMax * 8 + i];
    for (int i = t; i < ng; i += 256) lens[i] = glen_all[(size_t)b * kMtfGroupsMax + i];
    int n = 0, at = 0;  // bytes in use, those below t
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const uint32_t w = st[b].in_use[i];
        at += i < (t >> 5) ? __popc(w) : (i == (t >> 5) ? __popc(w & lanemask_lt()) : 0);
        n += __popc(w);
    }
    if ((st[b].in_use[t >> 5] >> (t & 31)) & 1u) lst[0][at] = (uint8_t)t;
    uint8_t r = ng > 0 ? grec[t] : (uint8_t)0;
    __syncthreads();
    int cur = 0;
    for (int g = 0; g < ng; g++, cur ^= 1) {
        const uint8_t next = g + 1 < ng ? grec[(g + 1) * 256 + t] : (uint8_t)0;
        grec[g * 256 + t] = lst[cur][t];
        list_apply(lst, cur, n, lens[g], r, pres[g], wc);
        r = next;
    }
}

// (3) one CTA per group: the list at every segment's start.
__global__ void __launch_bounds__(256) mtf_lists_kernel(const BlockState *__restrict__ st, int seg_log2, int group,
                                                        const uint8_t *__restrict__ rec_all, const uint32_t *__restrict__ pres_all,
                                                        const int32_t *__restrict__ len_all, const uint8_t *__restrict__ grec_all,
                                                        uint8_t *__restrict__ lists_all) {
    __shared__ MtfGroupSmem S;
    const int b = blockIdx.y, g = blockIdx.x, t = threadIdx.x;
    const int nseg = (st[b].m + (1 << seg_log2) - 1) >> seg_log2, s0 = g * group, n = min(group, nseg - s0);
    if (n <= 0) return;
    int in_use = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) in_use += __popc(st[b].in_use[i]);
    S.lst[0][t] = grec_all[((size_t)b * kMtfGroupsMax + g) * 256 + t];
    load_records(S, b, s0, n, rec_all, pres_all, len_all);
    uint8_t *lists = lists_all + ((size_t)b * kMtfSegs + s0) * 256;
    int cur = 0;
    for (int i = 0; i < n; i++, cur ^= 1) {
        lists[i * 256 + t] = S.lst[cur][t];
        if (i + 1 < n) list_apply(S.lst, cur, in_use, S.len[i], S.rec[i][t], S.pres[i], S.wc);
    }
}

// One warp per segment: MTF indices from the segment's starting list, 32
// positions per step. With the list (lst) and its inverse (posof) in shared
// memory at the window start, lane k with symbol s:
//  - s also at an earlier lane j of the window (the latest such j): s was at
//    the front after j and each lane i in (j, k) pushed it back one place iff
//    i's symbol was not moved to the front after j, i.e. prev(i) <= j, where
//    prev(i) is the latest earlier lane with i's symbol (-1 if none);
//  - otherwise: s is still in the old part of the list, behind the distinct
//    symbols of lanes < k, so its index is P + #{first-occurrence lanes
//    i < k with P_i > P}, P = posof[s].
// Both counts compare one value per lane with every other lane's: done
// bit-sliced over ballots of the values' bits. The list then becomes the
// window's symbols by last use, then the old list without them; entries
// behind the deepest window symbol keep their places.
__global__ void __launch_bounds__(32) mtf_encode_kernel(const BlockState *__restrict__ st, int seg_log2,
                                                        const uint8_t *__restrict__ L_all, const uint8_t *__restrict__ lists_all,
                                                        uint8_t *__restrict__ idx_all) {
    __shared__ __align__(8) uint8_t lst[256];
    __shared__ uint8_t posof[256];
    __shared__ uint32_t WP[8];
    __shared__ __align__(16) uint8_t seg[kTile];  // the segment's bytes, loaded at once
    const int b = blockIdx.y, g = blockIdx.x;
    const int m = st[b].m;
    const int s0 = g << seg_log2;
    if (s0 >= m) return;
    const int s1 = min(m, s0 + (1 << seg_log2));
    const int lane = threadIdx.x;
    {
        const uint8_t *Lb = L_all + (size_t)b * kBlockCap + s0;  // 16-byte aligned (block slots and tiles are)
        const int nb = s1 - s0;
        for (int q = lane; q < (nb >> 4); q += 32)
            reinterpret_cast<uint4 *>(seg)[q] = __ldg(reinterpret_cast<const uint4 *>(Lb) + q);
        for (int q = (nb & ~15) + lane; q < nb; q += 32) seg[q] = Lb[q];
    }
    int n_in_use = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) n_in_use += __popc(st[b].in_use[i]);
    const uint64_t *start = reinterpret_cast<const uint64_t *>(lists_all + ((size_t)b * kMtfSegs + g) * 256);
    reinterpret_cast<uint64_t *>(lst)[lane] = start[lane];
    __syncwarp();
    for (int q = lane; q < n_in_use; q += 32) posof[lst[q]] = (uint8_t)q;
    __syncwarp();
    uint8_t *out = idx_all + (size_t)b * kBlockCap;
    const uint32_t lt = lanemask_lt(), gt = lanemask_gt();
    for (int w0 = s0; w0 < s1; w0 += 32) {
        const int i = w0 + lane;
        const bool valid = i < s1;
        const uint32_t s = valid ? (uint32_t)seg[i - s0] : 256u + lane;
        const uint32_t grp = __match_any_sync(LFC_FULL, s);
        const uint32_t lower = grp & lt;
        const bool fo = valid && lower == 0;
        const uint32_t FO = __ballot_sync(LFC_FULL, fo);
        const uint32_t LAST = __ballot_sync(LFC_FULL, valid && (grp & gt) == 0);
        const uint32_t P = fo ? (uint32_t)posof[s] : 0u;
        const uint32_t maxP = __reduce_max_sync(LFC_FULL, P);
        const int pbits = 32 - __clz(maxP | 1u);  // bits of the deepest list position
        uint32_t gtm = 0, eqm = LFC_FULL;  // lanes with P_i > P
        for (int bb = pbits - 1; bb >= 0; bb--) {
            const uint32_t Bb = __ballot_sync(LFC_FULL, (P >> bb) & 1u);
            if ((P >> bb) & 1u) {
                eqm &= Bb;
            } else {
                gtm |= eqm & Bb;
                eqm &= ~Bb;
            }
        }
        const int j = lower ? 31 - __clz(lower) : -1;
        const uint32_t pp = lower ? (uint32_t)(j + 1) : 0u;  // prev + 1, in 0..31 (j <= 30)
        const uint32_t T = (uint32_t)(j + 1);
        uint32_t gt2 = 0, eq2 = LFC_FULL;  // lanes with prev_i + 1 > j + 1
#pragma unroll
        for (int bb = 4; bb >= 0; bb--) {
            const uint32_t Bb = __ballot_sync(LFC_FULL, (pp >> bb) & 1u);
            if ((T >> bb) & 1u) {
                eq2 &= Bb;
            } else {
                gt2 |= eq2 & Bb;
                eq2 &= ~Bb;
            }
        }
        uint32_t idx;
        if (lower == 0) idx = P + __popc(gtm & FO & lt);
        else idx = __popc(lt & ~((2u << j) - 1u) & ~gt2);
        if (valid) out[i] = (uint8_t)idx;
        // list update
        const uint32_t D = __popc(FO);
        if (lane < 8) WP[lane] = 0;
        __syncwarp();
        if (fo) atomicOr(&WP[P >> 5], 1u << (P & 31));
        __syncwarp();
        uint32_t mv[8];  // (new position << 8 | symbol) of the moved old entries, 0xFFFFFFFF if none
        uint32_t before = 0;  // window positions in earlier words
#pragma unroll
        for (int r = 0; r < 8; r++) {
            mv[r] = 0xFFFFFFFFu;
            const uint32_t q = (uint32_t)lane + 32u * r;
            if (32u * r > maxP) continue;
            const uint32_t wd = WP[r];
            if (q <= maxP && ((wd >> lane) & 1u) == 0) {
                const uint32_t rank = before + __popc(wd & lt);
                mv[r] = ((D + q - rank) << 8) | lst[q];
            }
            before += __popc(wd);
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 8; r++) {
            if (mv[r] == 0xFFFFFFFFu) continue;
            const uint32_t np = mv[r] >> 8, x = mv[r] & 0xFFu;
            lst[np] = (uint8_t)x;
            posof[x] = (uint8_t)np;
        }
        if ((LAST >> lane) & 1u) {
            const uint32_t np = __popc(LAST & gt);
            lst[np] = (uint8_t)s;
            posof[s] = (uint8_t)np;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ RLE2
// Zero runs of length r -> bijective base-2 digits RUNA(0)/RUNB(1): digit k
// is bit k of r + 1, floor(log2(r + 1)) digits, emitted at the run's last
// position. Index j > 0 -> j + 1. As for RLE1, a scan over 4096-position
// tiles in three kernels: per tile the first / last nonzero index and the
// symbols of the positions after the first nonzero (1); per block the last
// nonzero before each tile, the symbols of each tile's leading zero run and
// the tiles' symbol offsets (2); per tile the symbols and their frequencies (3).
constexpr int kRle2Tile = 4096;
constexpr int kRle2Threads = 256;

__device__ __forceinline__ int run_digits(int r) { return 31 - __clz(r + 1); }

// Nonzero mask of a thread's 16 positions [a, a + 16) of the tile, a run-end
// mask (zero followed by a nonzero or by the end of the block) and the
// thread's first / last nonzero position (absolute; INT_MAX / -1 if none).
__device__ __forceinline__ void rle2_masks(const uint8_t *idx, int a, int te, int m, uint32_t &nz, uint32_t &end,
                                           int &first, int &last, uint8_t (&v)[16]) {
    *reinterpret_cast<uint4 *>(v) = *reinterpret_cast<const uint4 *>(idx + a);
    const uint32_t nxt = a + 16 < m ? idx[a + 16] : 0u;
    nz = 0; end = 0; first = INT_MAX; last = -1;
#pragma unroll
    for (int q = 0; q < 16; q++) {
        if (a + q >= te) break;
        if (v[q]) {
            nz |= 1u << q;
            first = min(first, a + q);
            last = a + q;
        } else {
            const bool next_nz = q < 15 ? (a + q + 1 < m && v[q + 1] != 0) : (a + 16 < m && nxt != 0);
            if (a + q == m - 1 || next_nz) end |= 1u << q;
        }
    }
}

__global__ void __launch_bounds__(kRle2Threads) rle2_tile_kernel(const BlockState *__restrict__ st,
                                                                 const uint8_t *__restrict__ idx_all,
                                                                 int32_t *__restrict__ aux_all) {
    __shared__ int sh[33];
    __shared__ int sfirst, slast;
    const int b = blockIdx.y, tile = blockIdx.x;
    const int m = st[b].m;
    const int ts = tile * kRle2Tile;
    if (ts >= m) return;
    const int te = min(m, ts + kRle2Tile);
    if (threadIdx.x == 0) { sfirst = INT_MAX; slast = -1; }
    const uint8_t *idx = idx_all + (size_t)b * kBlockCap;
    const int a = ts + 16 * (int)threadIdx.x;
    uint32_t nz = 0, end = 0;
    int first = INT_MAX, last = -1;
    uint8_t v[16];
    if (a < te) rle2_masks(idx, a, te, m, nz, end, first, last, v);
    int lz = block_excl_max(last, sh);   // last nonzero of the tile before this thread, or -1
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 16; q++) {
        if ((nz >> q) & 1u) { cnt++; lz = a + q; }
        else if (((end >> q) & 1u) && lz >= ts) cnt += run_digits(a + q - lz);
    }
    int total;
    block_excl_sum<int>(cnt, sh, &total);
    if (first != INT_MAX) atomicMin(&sfirst, first);
    if (last >= 0) atomicMax(&slast, last);
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t *aux = aux_all + ((size_t)b * kTilesPerBlock + tile) * 4;
        aux[0] = sfirst != INT_MAX ? sfirst : te;
        aux[1] = slast;
        aux[2] = total;
    }
}

// One warp per block: aux[tile][1] = last nonzero before the tile (-1 if
// none), aux[tile][2] = the tile's symbol offset; symbol count, EOB and the
// frequency table's start.
__global__ void __launch_bounds__(32) rle2_scan_kernel(BlockState *__restrict__ st, int32_t *__restrict__ aux_all,
                                                       uint16_t *__restrict__ sym_all, uint32_t *__restrict__ freq_all) {
    const int b = blockIdx.x;
    const int m = st[b].m;
    const int ntile = (m + kRle2Tile - 1) / kRle2Tile;
    int32_t *aux = aux_all + (size_t)b * kTilesPerBlock * 4;
    const int lane = (int)lane_id();
    int carryR = -1, carryO = 0;
    for (int base = 0; base < ntile; base += 32) {
        const int t = base + lane;
        const bool valid = t < ntile;
        const int ts = t * kRle2Tile, te = min(m, ts + kRle2Tile);
        const int fs = valid ? aux[t * 4 + 0] : 0;
        const int ls = valid ? aux[t * 4 + 1] : -1;
        const int lo = valid ? aux[t * 4 + 2] : 0;
        const int imax = warp_incl_max(ls);
        int ex = __shfl_up_sync(LFC_FULL, imax, 1);
        if (lane == 0) ex = -1;
        const int R = max(carryR, ex);
        int pre = 0;  // the zero run the tile starts with, if it ends in the tile
        if (valid && fs > ts) {
            if (fs < te) {
                pre = run_digits(fs - 1 - R);
            } else if (te == m || (t + 1 < ntile && aux[(t + 1) * 4 + 0] == te)) {
                // no nonzero in the tile: the run ends at its last position when the
                // block ends there or the next tile starts with a nonzero
                pre = run_digits(te - 1 - R);
            }
        }
        const int out = valid ? pre + lo : 0;
        const int incl = warp_incl_sum(out);
        if (valid) {
            aux[t * 4 + 1] = R;
            aux[t * 4 + 2] = carryO + incl - out;
        }
        carryR = max(carryR, __shfl_sync(LFC_FULL, imax, 31));
        carryO += __shfl_sync(LFC_FULL, incl, 31);
    }
    int n_in_use = 0;
    for (int i = 0; i < 8; i++) n_in_use += __popc(st[b].in_use[i]);
    uint32_t *freq = freq_all + (size_t)b * kMaxAlpha;
    for (int i = lane; i < kMaxAlpha; i += 32) freq[i] = i == n_in_use + 1 ? 1u : 0u;
    if (lane == 0) {
        sym_all[(size_t)b * kSymStride + carryO] = (uint16_t)(n_in_use + 1);
        st[b].n_mtf = carryO + 1;
        st[b].n_in_use = n_in_use;
    }
}

__global__ void __launch_bounds__(kRle2Threads) rle2_write_kernel(const BlockState *__restrict__ st,
                                                                  const uint8_t *__restrict__ idx_all,
                                                                  const int32_t *__restrict__ aux_all,
                                                                  uint16_t *__restrict__ sym_all, uint32_t *__restrict__ freq_all) {
    __shared__ int sh[33];
    __shared__ uint32_t fq[kMaxAlpha];
    // the tile's symbols: a zero run of r codes to at most r digits, and only
    // the first run ending in the tile can hold zeros of earlier tiles (at
    // most 20 digits: a block is below 2^20 positions)
    __shared__ uint16_t ssym[kRle2Tile + 32];
    const int b = blockIdx.y, tile = blockIdx.x;
    const int m = st[b].m;
    const int ts = tile * kRle2Tile;
    if (ts >= m) return;
    const int te = min(m, ts + kRle2Tile);
    for (int i = threadIdx.x; i < kMaxAlpha; i += kRle2Threads) fq[i] = 0;
    const uint8_t *idx = idx_all + (size_t)b * kBlockCap;
    const int32_t *aux = aux_all + ((size_t)b * kTilesPerBlock + tile) * 4;
    const int R = aux[1], off = aux[2];
    const int a = ts + 16 * (int)threadIdx.x;
    uint32_t nz = 0, end = 0;
    int first = INT_MAX, last = -1;
    uint8_t v[16];
    if (a < te) rle2_masks(idx, a, te, m, nz, end, first, last, v);
    const int lz0 = max(block_excl_max(last, sh), R);
    int lz = lz0, cnt = 0;
#pragma unroll
    for (int q = 0; q < 16; q++) {
        if ((nz >> q) & 1u) { cnt++; lz = a + q; }
        else if ((end >> q) & 1u) cnt += run_digits(a + q - lz);
    }
    // symbols staged in shared memory at their tile-local offsets, then
    // written by consecutive threads on consecutive positions
    int total = 0;
    int o = block_excl_sum<int>(cnt, sh, &total);
    uint16_t *sym = sym_all + (size_t)b * kSymStride;
    lz = lz0;
#pragma unroll
    for (int q = 0; q < 16; q++) {
        if ((nz >> q) & 1u) {
            const uint32_t s = (uint32_t)v[q] + 1u;
            ssym[o++] = (uint16_t)s;
            atomicAdd(&fq[s], 1u);
            lz = a + q;
        } else if ((end >> q) & 1u) {
            const uint32_t r1 = (uint32_t)(a + q - lz);  // run length r, digits of r + 1
            const int nd = run_digits((int)r1);
            for (int k = 0; k < nd; k++) {
                const uint32_t d = ((r1 + 1u) >> k) & 1u;
                ssym[o++] = (uint16_t)d;
                atomicAdd(&fq[d], 1u);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < total; i += kRle2Threads) sym[off + i] = ssym[i];
    uint32_t *freq = freq_all + (size_t)b * kMaxAlpha;
    for (int i = threadIdx.x; i < kMaxAlpha; i += kRle2Threads)
        if (fq[i]) atomicAdd(&freq[i], fq[i]);
}

// --------------------------------------------------------------- Huffman
// Code lengths of one table by one CTA (a thread per symbol): weights
// max(freq, 1); the two nodes with the smallest (weight, key) are joined (leaf
// key = symbol, k-th joined node key = alpha + k; the two-queue method
// reproduces that order because leaves are pre-sorted by (weight, symbol) and
// joined nodes appear in non-decreasing weight); over-long codes halve the
// weights (1 + w/2).
constexpr int kHuffThreads = 288;
static_assert(kHuffThreads >= kMaxAlpha, "a thread per symbol");

struct HuffScratch {
    uint32_t w[kHuffThreads];
    uint32_t lw[kMaxAlpha];          // leaf weights in (weight, symbol) order
    uint32_t nw[kMaxAlpha];          // joined-node weights
    uint32_t pair[kMaxAlpha];        // weights of a round's items in order
    uint16_t order[kMaxAlpha];       // leaves sorted by (w, symbol)
    uint16_t par[2 * kMaxAlpha];     // parent of a node (leaves, then joined nodes)
    uint16_t dist[2 * kMaxAlpha];    // pointer-jumping distance to par
    int longest;
};

// Two-queue merge by one warp, in rounds: the pair of the two smallest
// (weight, key) items makes a node of weight n0, and every item at hand of
// weight <= n0 comes before it (a leaf before a joined node of equal weight, a
// joined node before a later one: the keys), so all of them pair up in order
// at once. An item's place among them is its index plus the count of the
// other queue's items before it. About 20 rounds for the counts of one table
// instead of 257 dependent steps.
__device__ void huff_merge(int alpha, HuffScratch &S) {
    constexpr uint32_t kEmpty = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    int la = 0, lb = 0, k = 0;  // queue heads, joined nodes made
    while (k < alpha - 1) {
        const uint32_t a0 = la < alpha ? S.lw[la] : kEmpty, a1 = la + 1 < alpha ? S.lw[la + 1] : kEmpty;
        const uint32_t b0 = lb < k ? S.nw[lb] : kEmpty, b1 = lb + 1 < k ? S.nw[lb + 1] : kEmpty;
        const uint32_t n0 = a0 <= b0 ? a0 + min(a1, b0) : b0 + min(a0, b1);
        int ca = 0, cb = 0;  // items of weight <= n0 (the queues ascend)
        for (uint32_t more = LFC_FULL; more == LFC_FULL;) {
            const int i = la + ca + lane;
            more = __ballot_sync(LFC_FULL, i < alpha && S.lw[i] <= n0);
            ca += __popc(more);
        }
        for (uint32_t more = LFC_FULL; more == LFC_FULL;) {
            const int i = lb + cb + lane;
            more = __ballot_sync(LFC_FULL, i < k && S.nw[i] <= n0);
            cb += __popc(more);
        }
        const int n = (ca + cb) & ~1;  // items that pair up; an odd last one waits
        int used = 0;                  // leaves among them
        for (int i0 = 0; i0 < ca; i0 += 32) {
            const int i = i0 + lane;
            bool mine = false;
            if (i < ca) {
                const uint32_t x = S.lw[la + i];
                int lo = 0, hi = cb;  // joined nodes below x
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (S.nw[lb + mid] < x) lo = mid + 1; else hi = mid;
                }
                mine = i + lo < n;
                if (mine) {
                    S.pair[i + lo] = x;
                    S.par[S.order[la + i]] = (uint16_t)(alpha + k + ((i + lo) >> 1));
                }
            }
            used += __popc(__ballot_sync(LFC_FULL, mine));
        }
        for (int i = lane; i < cb; i += 32) {
            const uint32_t x = S.nw[lb + i];
            int lo = 0, hi = ca;  // leaves up to x
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (S.lw[la + mid] <= x) lo = mid + 1; else hi = mid;
            }
            if (i + lo < n) {
                S.pair[i + lo] = x;
                S.par[alpha + lb + i] = (uint16_t)(alpha + k + ((i + lo) >> 1));
            }
        }
        __syncwarp();
        for (int i = lane; i < n / 2; i += 32) S.nw[k + i] = S.pair[2 * i] + S.pair[2 * i + 1];
        __syncwarp();
        la += used;
        lb += n - used;
        k += n / 2;
    }
}

// The length of symbol threadIdx.x (w: its weight). Keys (w << 9 | symbol)
// are distinct, so a key's rank is the count of smaller keys; w < 2^21
// (counts of one block), so the key fits 30 bits. Node depths by pointer
// jumping: after r rounds par[n] is n's 2^r-th ancestor (capped at the root)
// and dist[n] the distance to it.
__device__ int huff_length(uint32_t w, int alpha, int max_len, HuffScratch &S) {
    const int v = threadIdx.x;
    const int nodes = 2 * alpha - 1, root = 2 * alpha - 2;
    for (;;) {
        S.w[v] = w;
        if (v == 0) S.longest = 0;
        __syncthreads();
        if (v < alpha) {
            const uint32_t key = (w << 9) | (uint32_t)v;
            int r = 0;
#pragma unroll 8
            for (int j = 0; j < alpha; j++) r += ((S.w[j] << 9) | (uint32_t)j) < key;
            S.order[r] = (uint16_t)v;
            S.lw[r] = w;
        }
        __syncthreads();
        if (v < 32) huff_merge(alpha, S);
        if (v == 0) S.par[root] = (uint16_t)root;
        const int n0 = v, n1 = v + kHuffThreads;
        if (n0 < nodes) S.dist[n0] = n0 == root ? 0 : 1;
        if (n1 < nodes) S.dist[n1] = n1 == root ? 0 : 1;
        __syncthreads();
        for (int span = 1; span < alpha; span <<= 1) {
            int p0 = 0, d0 = 0, p1 = 0, d1 = 0;
            if (n0 < nodes) {
                const int p = S.par[n0];
                d0 = S.dist[n0] + S.dist[p];
                p0 = S.par[p];
            }
            if (n1 < nodes) {
                const int p = S.par[n1];
                d1 = S.dist[n1] + S.dist[p];
                p1 = S.par[p];
            }
            __syncthreads();
            if (n0 < nodes) { S.dist[n0] = (uint16_t)d0; S.par[n0] = (uint16_t)p0; }
            if (n1 < nodes) { S.dist[n1] = (uint16_t)d1; S.par[n1] = (uint16_t)p1; }
            __syncthreads();
        }
        const int len = v < alpha ? S.dist[v] : 0;
        const int longest = __reduce_max_sync(LFC_FULL, (unsigned)len);
        if ((v & 31) == 0) atomicMax(&S.longest, longest);
        __syncthreads();
        if (S.longest <= max_len) return len;
        w = 1u + w / 2u;
        __syncthreads();
    }
}

constexpr int kPackGroups = 128;                                           // selector groups per tile = threads
constexpr int kPackTiles = (kMaxSelectors + kPackGroups - 1) / kPackGroups;  // 141
constexpr int kTileSyms = kPackGroups * 50;                                   // symbols of a tile

// Stage the symbols of a tile of selector groups in shared memory with
// coalesced 16-byte loads (tile starts are 16-byte aligned); returns their count.
__device__ __forceinline__ int stage_tile_syms(const uint16_t *sym, int tile, int n_mtf, uint16_t *ssym) {
    const int a = tile * kTileSyms;
    const int cnt = min(kTileSyms, n_mtf - a);
    const int n8 = cnt >> 3;
    const uint4 *src = reinterpret_cast<const uint4 *>(sym + a);
    uint4 *dst = reinterpret_cast<uint4 *>(ssym);
    for (int i = threadIdx.x; i < n8; i += blockDim.x) dst[i] = src[i];
    for (int i = (n8 << 3) + threadIdx.x; i < cnt; i += blockDim.x) ssym[i] = sym[a + i];
    return cnt;
}

// Table choice per block, in launches: the table count and the initial
// partition by cumulative frequency (init); four refinement passes, each
// "every 50-symbol group picks the cheapest table, ties to the lower" over
// many CTAs (select) followed by "every table is rebuilt from its groups'
// counts with a 17-bit limit" (build), the last of them with the canonical
// codes.
__global__ void __launch_bounds__(kHuffThreads) huff_init_kernel(BlockState *__restrict__ st, const uint32_t *__restrict__ freq_all,
                                                                     uint8_t *__restrict__ lens_all, uint32_t *__restrict__ rfreq_all) {
    __shared__ uint32_t sh[33];
    const int b = blockIdx.x, v = threadIdx.x;
    const int n_mtf = st[b].n_mtf;
    const int alpha = st[b].n_in_use + 2;
    const int ng = n_mtf < 200 ? 2 : n_mtf < 600 ? 3 : n_mtf < 1200 ? 4 : n_mtf < 2400 ? 5 : 6;
    for (int i = v; i < kMaxGroups * kMaxAlpha; i += blockDim.x) rfreq_all[(size_t)b * kMaxGroups * kMaxAlpha + i] = 0;
    const uint32_t f = v < alpha ? freq_all[(size_t)b * kMaxAlpha + v] : 0u;
    const uint32_t cum = block_excl_sum<uint32_t>(f, sh, nullptr);  // cum * ng < 2^23
    if (v < alpha) {
        const int gsel = min((int)(cum * (uint32_t)ng / (uint32_t)n_mtf), ng - 1);
        uint8_t *len = lens_all + (size_t)b * kMaxGroups * kMaxAlpha;
        for (int t = 0; t < ng; t++) len[t * kMaxAlpha + v] = (uint8_t)(t == gsel ? 0 : 15);
    }
    if (v == 0) {
        st[b].n_groups = ng;
        st[b].n_sel = (n_mtf + 49) / 50;
    }
}

// Thread per 50-symbol group: cost under every table (10-bit fields of one
// 64-bit word per symbol; <= 50 x 17 bits), the cheapest table, and the
// group's symbols added to that table's counts (RUNA / RUNB, the most common
// symbols, in registers; the rest through shared memory, flushed per CTA).
__global__ void __launch_bounds__(kPackGroups) huff_select_kernel(const BlockState *__restrict__ st,
                                                                  const uint16_t *__restrict__ sym_all,
                                                                  const uint8_t *__restrict__ lens_all,
                                                                  uint8_t *__restrict__ sel_all, uint32_t *__restrict__ rfreq_all) {
    __shared__ uint64_t packed[kMaxAlpha];
    __shared__ uint32_t rf[kMaxGroups][kMaxAlpha];
    __shared__ __align__(16) uint16_t ssym[kTileSyms];
    const int b = blockIdx.y, tile = blockIdx.x;
    const BlockState S = st[b];
    const int ng = S.n_groups, nsel = S.n_sel, n_mtf = S.n_mtf, alpha = S.n_in_use + 2;
    if (tile * kPackGroups >= nsel) return;
    stage_tile_syms(sym_all + (size_t)b * kSymStride, tile, n_mtf, ssym);
    const uint8_t *len = lens_all + (size_t)b * kMaxGroups * kMaxAlpha;
    for (int v = threadIdx.x; v < alpha; v += blockDim.x) {
        uint64_t pk = 0;
        for (int t = 0; t < ng; t++) pk |= (uint64_t)len[t * kMaxAlpha + v] << (10 * t);
        packed[v] = pk;
    }
    for (int i = threadIdx.x; i < kMaxGroups * kMaxAlpha; i += blockDim.x) (&rf[0][0])[i] = 0;
    __syncthreads();
    const int gi = tile * kPackGroups + (int)threadIdx.x;
    int bt = -1;
    uint32_t c0 = 0, c1 = 0;
    if (gi < nsel) {
        const uint16_t *sym = ssym - tile * kTileSyms;  // indexed by block position
        const int a = gi * 50, e = min(n_mtf, a + 50);
        uint64_t acc = 0;
        for (int i = a; i < e; i++) acc += packed[sym[i]];
        bt = 0;
        uint32_t bc = (uint32_t)(acc & 1023u);
        for (int t = 1; t < ng; t++) {
            const uint32_t c = (uint32_t)((acc >> (10 * t)) & 1023u);
            if (c < bc) { bc = c; bt = t; }
        }
        sel_all[(size_t)b * kMaxSelectors + gi] = (uint8_t)bt;
        for (int i = a; i < e; i++) {
            const uint32_t v = sym[i];
            if (v == 0) c0++;
            else if (v == 1) c1++;
            else atomicAdd(&rf[bt][v], 1u);
        }
        if (c0) atomicAdd(&rf[bt][0], c0);
        if (c1) atomicAdd(&rf[bt][1], c1);
    }
    __syncthreads();
    uint32_t *rfreq = rfreq_all + (size_t)b * kMaxGroups * kMaxAlpha;
    for (int i = threadIdx.x; i < ng * kMaxAlpha; i += blockDim.x) {
        const uint32_t c = (&rf[0][0])[i];
        if (c) atomicAdd(&rfreq[i], c);
    }
}

// CTA per table: code lengths from the pass's counts, which are then cleared
// for the next pass. The last pass also writes the canonical codes (by
// length, then symbol): a symbol's code is its length's first one plus the
// symbols before it of the same length.
__global__ void __launch_bounds__(kHuffThreads) huff_build_kernel(const BlockState *__restrict__ st, uint32_t *__restrict__ rfreq_all,
                                                                  uint8_t *__restrict__ lens_all, uint32_t *__restrict__ codes_all,
                                                                  int last) {
    __shared__ HuffScratch S;
    __shared__ uint8_t ls[kHuffThreads];
    __shared__ uint32_t first[32];
    const int b = blockIdx.y, g = blockIdx.x, v = threadIdx.x;
    if (g >= st[b].n_groups) return;
    const int alpha = st[b].n_in_use + 2;
    const size_t at = ((size_t)b * kMaxGroups + g) * kMaxAlpha + v;
    uint32_t w = 0xFFFFFFFFu >> 9;
    if (v < alpha) {
        w = max(rfreq_all[at], 1u);
        rfreq_all[at] = 0;
    }
    const int len = huff_length(w, alpha, 17, S);
    if (v < alpha) lens_all[at] = (uint8_t)len;
    if (!last) return;
    ls[v] = (uint8_t)len;
    if (v < 32) first[v] = 0;
    __syncthreads();
    if (v < alpha) atomicAdd(&first[len], 1u);
    __syncthreads();
    if (v == 0) {
        uint32_t c = 0;
        for (int l = 1; l <= 20; l++) {
            const uint32_t n = first[l];
            first[l] = c;
            c = (c + n) << 1;
        }
    }
    __syncthreads();
    if (v < alpha) {
        uint32_t r = first[len];
#pragma unroll 8
        for (int j = 0; j < v; j++) r += ls[j] == len;
        codes_all[at] = r;
    }
}

// ------------------------------------------------------------ bit packing
// Bits are numbered from the start of the stream; bit P lands in word P/32 at
// bit 31 - P%32 (MSB first). Words are stored byte-swapped (so the bytes
// come out in stream order); swapping commutes with OR, so partial words
// from different writers are swapped first and OR-ed into zeroed memory.
__device__ __forceinline__ uint32_t bswap32(uint32_t w) { return __byte_perm(w, 0u, 0x0123); }

__device__ __forceinline__ void put_bits(uint32_t *words, uint64_t pos, uint32_t value, int nbits) {
    if (nbits == 0) return;
    const int sh = (int)(pos & 31);
    const uint64_t v = (uint64_t)value << (64 - nbits - sh);
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    if (hi) atomicOr(&words[pos >> 5], bswap32(hi));
    if (lo) atomicOr(&words[(pos >> 5) + 1], bswap32(lo));
}

// MTF index of a selector of table s (tables listed 0..ng-1 initially),
// given last[t] = position of the latest earlier selector of table t (-1 if
// none): the number of tables used since s was last used, or, before its
// first use, the tables used so far plus the unused tables below s.
__device__ __forceinline__ int selector_mtf(int s, const int (&last)[kMaxGroups], int ng) {
    int ls = -1;
#pragma unroll
    for (int t = 0; t < kMaxGroups; t++)
        if (t == s) ls = last[t];
    int j = 0;
#pragma unroll
    for (int t = 0; t < kMaxGroups; t++) {
        if (t >= ng || t == s) continue;
        j += ls >= 0 ? (last[t] > ls) : (last[t] >= 0 || t < s);
    }
    return j;
}

__device__ __forceinline__ void set_last(int (&last)[kMaxGroups], int s, int i) {
#pragma unroll
    for (int t = 0; t < kMaxGroups; t++)
        if (t == s) last[t] = i;
}

// Data packing is a scan over tiles of 128 selector groups (50 symbols each):
// group bit lengths and tile sums (1); per block the stream layout, the tile
// offsets, the header, selector, code-length and trailer sections (2); each
// group's codes from its bit offset, whole words stored, the two boundary
// words OR-ed (3).
static_assert(kPackTiles <= kTilesPerBlock, "pack tile records live in the per-block tile scratch");
constexpr int kLayoutThreads = 1024;

__device__ __forceinline__ void load_tables(const uint8_t *lens_all, const uint32_t *codes_all, int b, int ng,
                                            uint8_t (*len)[kMaxAlpha], uint32_t (*code)[kMaxAlpha]) {
    for (int i = threadIdx.x; i < ng * kMaxAlpha; i += blockDim.x) {
        const int t = i / kMaxAlpha, v = i - t * kMaxAlpha;
        len[t][v] = lens_all[((size_t)b * kMaxGroups + t) * kMaxAlpha + v];
        if (code) code[t][v] = codes_all[((size_t)b * kMaxGroups + t) * kMaxAlpha + v];
    }
}

__global__ void __launch_bounds__(kPackGroups) pack_bits_kernel(const BlockState *__restrict__ st,
                                                                const uint16_t *__restrict__ sym_all,
                                                                const uint8_t *__restrict__ sel_all,
                                                                const uint8_t *__restrict__ lens_all,
                                                                uint16_t *__restrict__ gbits_all,
                                                                int32_t *__restrict__ aux_all) {
    __shared__ uint8_t len[kMaxGroups][kMaxAlpha];
    __shared__ int sh[33];
    __shared__ __align__(16) uint16_t ssym[kTileSyms];
    const int b = blockIdx.y, tile = blockIdx.x;
    const BlockState S = st[b];
    if (tile * kPackGroups >= S.n_sel) return;
    load_tables(lens_all, nullptr, b, S.n_groups, len, nullptr);
    stage_tile_syms(sym_all + (size_t)b * kSymStride, tile, S.n_mtf, ssym);
    __syncthreads();
    const int gi = tile * kPackGroups + (int)threadIdx.x;
    int bits = 0;
    if (gi < S.n_sel) {
        const uint16_t *sym = ssym - tile * kTileSyms;
        const uint8_t *lt = len[sel_all[(size_t)b * kMaxSelectors + gi]];
        const int a = gi * 50, e = min(S.n_mtf, a + 50);
        for (int i = a; i < e; i++) bits += lt[sym[i]];
        gbits_all[(size_t)b * (kBlockCap / 2) + gi] = (uint16_t)bits;
    }
    int total;
    block_excl_sum<int>(bits, sh, &total);
    if (threadIdx.x == 0) aux_all[((size_t)b * kTilesPerBlock + tile) * 4] = total;
}

__global__ void __launch_bounds__(kLayoutThreads) pack_layout_kernel(BlockState *__restrict__ st,
                                                                     const uint8_t *__restrict__ sel_all,
                                                                     const uint8_t *__restrict__ lens_all,
                                                                     int32_t *__restrict__ aux_all,
                                                                     uint32_t *__restrict__ packed_all, int64_t stream_words) {
    __shared__ uint8_t len[kMaxGroups][kMaxAlpha];
    __shared__ uint64_t sh64[33];
    __shared__ int shi[33];
    __shared__ uint32_t tbl_bits[kMaxGroups];
    __shared__ uint64_t base_bits[4];
    const int b = blockIdx.x;
    const BlockState S = st[b];
    const int ng = S.n_groups, nsel = S.n_sel, alpha = S.n_in_use + 2;
    const uint8_t *sel = sel_all + (size_t)b * kMaxSelectors;
    uint32_t *words = packed_all + (size_t)b * stream_words;
    int32_t *aux = aux_all + (size_t)b * kTilesPerBlock * 4;
    load_tables(lens_all, nullptr, b, ng, len, nullptr);
    uint32_t used16 = 0;
    for (int i = 0; i < 16; i++) {
        const uint32_t half = (S.in_use[i >> 1] >> ((i & 1) * 16)) & 0xFFFFu;
        if (half) used16 |= 1u << (15 - i);
    }
    __syncthreads();
    // data tiles: exclusive offsets (one tile per thread, <= 141 tiles)
    const int ntiles = (nsel + kPackGroups - 1) / kPackGroups;
    const uint64_t tb = (int)threadIdx.x < ntiles ? (uint64_t)(uint32_t)aux[threadIdx.x * 4] : 0ull;
    uint64_t data_total;
    const uint64_t toff = block_excl_sum<uint64_t>(tb, sh64, &data_total);
    if ((int)threadIdx.x < ntiles) aux[threadIdx.x * 4 + 1] = (int32_t)toff;
    // selector MTF: each thread's span starts from the last use of every table
    // before it (exclusive max-scans), then replays its span
    const int T = blockDim.x;
    const int sper = (nsel + T - 1) / T;
    const int sa = min(nsel, (int)threadIdx.x * sper), se = min(nsel, sa + sper);
    int last0[kMaxGroups];
#pragma unroll
    for (int t = 0; t < kMaxGroups; t++) last0[t] = -1;
    for (int i = sa; i < se; i++) set_last(last0, sel[i], i);
#pragma unroll
    for (int t = 0; t < kMaxGroups; t++) last0[t] = block_excl_max(last0[t], shi);
    int last[kMaxGroups];
#pragma unroll
    for (int t = 0; t < kMaxGroups; t++) last[t] = last0[t];
    uint64_t sbits = 0;
    for (int i = sa; i < se; i++) {
        const int sv = sel[i];
        sbits += (uint64_t)selector_mtf(sv, last, ng) + 1;
        set_last(last, sv, i);
    }
    uint64_t sel_total;
    const uint64_t sel_off = block_excl_sum<uint64_t>(sbits, sh64, &sel_total);
    // code-length section bits per table (warp t)
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < ng) {
        uint32_t bits = 0;
        for (int v = lane; v < alpha; v += 32) {
            const int d = v == 0 ? 0 : (int)len[w][v] - (int)len[w][v - 1];
            bits += 2u * (uint32_t)abs(d) + 1u;
        }
        bits = warp_sum(bits);
        if (lane == 0) tbl_bits[w] = bits + 5u;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t p = 32 + 48 + 32 + 1 + 24 + 16 + 16ull * __popc(used16) + 3 + 15;
        base_bits[0] = p;                       // selectors start
        p += sel_total;
        for (int t = 0; t < ng; t++) p += tbl_bits[t];
        base_bits[1] = p;                       // data start
        p += data_total;
        base_bits[2] = p;                       // trailer start
        p += 48 + 32;
        p = (p + 7) & ~7ull;
        base_bits[3] = p;                       // total bits
    }
    __syncthreads();
    const uint64_t total_bits = base_bits[3];
    const int64_t nwords = (int64_t)((total_bits + 31) >> 5);
    for (int64_t i = threadIdx.x; i < nwords + 1 && i < stream_words; i += blockDim.x) words[i] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t p = 0;
        put_bits(words, p, 0x425A6839u, 32); p += 32;  // "BZh9"
        put_bits(words, p, 0x314159u, 24); p += 24;
        put_bits(words, p, 0x265359u, 24); p += 24;
        put_bits(words, p, S.crc, 32); p += 32;
        put_bits(words, p, 0, 1); p += 1;
        put_bits(words, p, (uint32_t)S.orig_ptr, 24); p += 24;
        put_bits(words, p, used16, 16); p += 16;
        for (int i = 0; i < 16; i++) {
            if (!(used16 & (1u << (15 - i)))) continue;
            const uint32_t half = (S.in_use[i >> 1] >> ((i & 1) * 16)) & 0xFFFFu;
            put_bits(words, p, __brev(half) >> 16, 16);  // byte 16i+j -> bit 15-j
            p += 16;
        }
        put_bits(words, p, (uint32_t)ng, 3); p += 3;
        put_bits(words, p, (uint32_t)nsel, 15); p += 15;
        uint64_t q = base_bits[2];
        put_bits(words, q, 0x177245u, 24); q += 24;
        put_bits(words, q, 0x385090u, 24); q += 24;
        put_bits(words, q, S.crc, 32);
        st[b].stream_bits = (uint32_t)total_bits;
        st[b].stream_bytes = (uint32_t)(total_bits >> 3);
        st[b].data_bit0 = (uint32_t)base_bits[1];
    }
    {   // selectors: j ones then a zero
        uint64_t p = base_bits[0] + sel_off;
        for (int t = 0; t < kMaxGroups; t++) last[t] = last0[t];
        for (int i = sa; i < se; i++) {
            const int sv = sel[i];
            const int j = selector_mtf(sv, last, ng);
            set_last(last, sv, i);
            put_bits(words, p, ((1u << j) - 1u) << 1, j + 1);
            p += (uint64_t)j + 1;
        }
    }
    if (w < ng) {  // code lengths: 5-bit start, then per symbol |d| x ("10" up or "11" down) and a '0'
        uint64_t p = base_bits[0] + sel_total;
        for (int t = 0; t < w; t++) p += tbl_bits[t];
        if (lane == 0) put_bits(words, p, (uint32_t)len[w][0], 5);
        p += 5;
        for (int v0 = 0; v0 < alpha; v0 += 32) {
            const int v = v0 + lane;
            const int d = v < alpha ? (v == 0 ? 0 : (int)len[w][v] - (int)len[w][v - 1]) : 0;
            const uint32_t nb = v < alpha ? 2u * (uint32_t)abs(d) + 1u : 0u;
            const uint32_t incl = warp_incl_sum(nb);
            uint64_t q = p + incl - nb;
            for (int k = 0; k < abs(d); k++, q += 2) put_bits(words, q, d > 0 ? 2u : 3u, 2);
            p += __shfl_sync(LFC_FULL, incl, 31);
        }
    }
}

__global__ void __launch_bounds__(kPackGroups) pack_data_kernel(const BlockState *__restrict__ st,
                                                                const uint16_t *__restrict__ sym_all,
                                                                const uint8_t *__restrict__ sel_all,
                                                                const uint8_t *__restrict__ lens_all,
                                                                const uint32_t *__restrict__ codes_all,
                                                                const uint16_t *__restrict__ gbits_all,
                                                                const int32_t *__restrict__ aux_all,
                                                                uint32_t *__restrict__ packed_all, int64_t stream_words) {
    __shared__ uint8_t len[kMaxGroups][kMaxAlpha];
    __shared__ uint32_t code[kMaxGroups][kMaxAlpha];
    __shared__ int sh[33];
    __shared__ __align__(16) uint16_t ssym[kTileSyms];
    const int b = blockIdx.y, tile = blockIdx.x;
    const BlockState S = st[b];
    if (tile * kPackGroups >= S.n_sel) return;
    load_tables(lens_all, codes_all, b, S.n_groups, len, code);
    stage_tile_syms(sym_all + (size_t)b * kSymStride, tile, S.n_mtf, ssym);
    const int gi = tile * kPackGroups + (int)threadIdx.x;
    const int bits = gi < S.n_sel ? (int)gbits_all[(size_t)b * (kBlockCap / 2) + gi] : 0;
    const int off = block_excl_sum<int>(bits, sh, nullptr);  // also orders the table loads
    if (gi >= S.n_sel || bits == 0) return;
    uint32_t *words = packed_all + (size_t)b * stream_words;
    const uint64_t p0 = (uint64_t)S.data_bit0 + (uint32_t)aux_all[((size_t)b * kTilesPerBlock + tile) * 4 + 1] + off;
    const int t = sel_all[(size_t)b * kMaxSelectors + gi];
    const uint16_t *sym = ssym - tile * kTileSyms;
    const int a = gi * 50, e = min(S.n_mtf, a + 50);
    uint64_t acc = 0;                 // pending bits, left-aligned
    uint64_t wpos = p0 & ~31ull;      // bit position of the word being built
    int nacc = (int)(p0 - wpos);      // leading bits owned by the previous group (zeros)
    for (int i = a; i < e; i++) {
        const uint32_t sv = sym[i];
        const int l = len[t][sv];
        acc |= (uint64_t)code[t][sv] << (64 - nacc - l);
        nacc += l;
        if (nacc >= 32) {
            const uint32_t word = bswap32((uint32_t)(acc >> 32));
            if (wpos < p0) atomicOr(&words[wpos >> 5], word);  // shared with the previous group
            else words[wpos >> 5] = word;
            acc <<= 32;
            nacc -= 32;
            wpos += 32;
        }
    }
    if (nacc > 0) atomicOr(&words[wpos >> 5], bswap32((uint32_t)(acc >> 32)));  // shared with the next
}

cudaError_t launch_mtf_rle2(lfc_plan P, int nblocks, int max_m) {
    Workspace &ws = P->ws;
    cudaStream_t s = P->stream;
    const int seg_log2 = mtf_seg_log2(P, nblocks, max_m);
    const int segs = (max_m + (1 << seg_log2) - 1) >> seg_log2;
    const int group = seg_log2 == 12 ? 16 : kMtfGroup, groups = (segs + group - 1) / group;
    const dim3 ggrid(groups, nblocks);
    mtf_group_kernel<<<ggrid, 256, 0, s>>>(ws.bstate, seg_log2, group, ws.mtfrec, ws.mtfpres, ws.mtfreclen, ws.mtfgrec, ws.mtfgpres,
                                           ws.mtfglen);
    mtf_chain_kernel<<<nblocks, 256, 0, s>>>(ws.bstate, seg_log2, group, ws.mtfgrec, ws.mtfgpres, ws.mtfglen);
    mtf_lists_kernel<<<ggrid, 256, 0, s>>>(ws.bstate, seg_log2, group, ws.mtfrec, ws.mtfpres, ws.mtfreclen, ws.mtfgrec, ws.mtflists);
    mtf_encode_kernel<<<dim3(segs, nblocks), 32, 0, s>>>(ws.bstate, seg_log2, ws.bwt, ws.mtflists, ws.mtfidx);
    const dim3 g2((max_m + kRle2Tile - 1) / kRle2Tile, nblocks);
    rle2_tile_kernel<<<g2, kRle2Threads, 0, s>>>(ws.bstate, ws.mtfidx, ws.tileaux);
    rle2_scan_kernel<<<nblocks, 32, 0, s>>>(ws.bstate, ws.tileaux, ws.sym, ws.freq);
    rle2_write_kernel<<<g2, kRle2Threads, 0, s>>>(ws.bstate, ws.mtfidx, ws.tileaux, ws.sym, ws.freq);
    count_launches(P, 7);
    return cudaGetLastError();
}

// Tiles of selector groups of a block with max_m positions: at most a symbol
// per position and EOB.
static int pack_tiles(int max_m) { return (max_m + 1 + kTileSyms - 1) / kTileSyms; }

cudaError_t launch_huffman(lfc_plan P, int nblocks, int max_m) {
    Workspace &ws = P->ws;
    cudaStream_t s = P->stream;
    huff_init_kernel<<<nblocks, kHuffThreads, 0, s>>>(ws.bstate, ws.freq, ws.lens, ws.rfreq);
    const dim3 grid(pack_tiles(max_m), nblocks);
    for (int iter = 0; iter < 4; iter++) {
        huff_select_kernel<<<grid, kPackGroups, 0, s>>>(ws.bstate, ws.sym, ws.lens, ws.sel, ws.rfreq);
        huff_build_kernel<<<dim3(kMaxGroups, nblocks), kHuffThreads, 0, s>>>(ws.bstate, ws.rfreq, ws.lens, ws.codes, iter == 3);
    }
    count_launches(P, 9);
    return cudaGetLastError();
}

cudaError_t launch_pack(lfc_plan P, int nblocks, int max_m) {
    Workspace &ws = P->ws;
    // group bit lengths live in the MTF index slots, free once RLE2 has run
    uint16_t *gbits = reinterpret_cast<uint16_t *>(ws.mtfidx);
    const dim3 grid(pack_tiles(max_m), nblocks);
    pack_bits_kernel<<<grid, kPackGroups, 0, P->stream>>>(ws.bstate, ws.sym, ws.sel, ws.lens, gbits, ws.tileaux);
    pack_layout_kernel<<<nblocks, kLayoutThreads, 0, P->stream>>>(ws.bstate, ws.sel, ws.lens, ws.tileaux, ws.packed,
                                                                  ws.stream_words);
    pack_data_kernel<<<grid, kPackGroups, 0, P->stream>>>(ws.bstate, ws.sym, ws.sel, ws.lens, ws.codes, gbits,
                                                          ws.tileaux, ws.packed, ws.stream_words);
    count_launches(P, 3);
    return cudaGetLastError();
}

}  // namespace lfc
