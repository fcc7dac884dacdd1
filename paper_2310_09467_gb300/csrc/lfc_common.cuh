// lfc_common.cuh -- internal declarations shared by the liblfc CUDA sources.
// Nothing here is part of the public ABI (include/lfc.h is).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include <cstring>
#include <string>
#include <vector>

#include "lfc.h"

namespace lfc {

// ---------------------------------------------------------------- constants
constexpr int kMaxBlockBytes = LFC_MAX_BLOCK_BYTES;  // input bytes per bzip2 block
constexpr int kTile = 4096;                          // elements per sort tile
constexpr int kRleCap = 900000;                      // RLE1 output bound (5/4 of 720000)
constexpr int kBlockCap = 901120;                    // 220 tiles of 4096, >= kRleCap
constexpr int kTilesPerBlock = kBlockCap / kTile;    // 220
constexpr int kMaxAlpha = 258;                       // bzip2 symbols: 256 MTF + RUNA/RUNB... + EOB
constexpr int kMaxGroups = 6;
constexpr int kMaxSelectors = 18002;
constexpr int kHistBins = 65536;
constexpr int kMtfSegs = kBlockCap / 1024;           // most MTF segments of a block
constexpr int kMaxCand = 104;                        // candidates per frame: 26 default ids x 2 byte layouts x 2 (temporal)

// Sort state in device memory (rs): tied elements after a round, their
// per-block maximum, the shift h, the round number; the abort word (nonzero
// once a bounded wait has given up in this suffix sort: every later sort
// kernel returns at once), the fault-injection word (test hook), the two work
// queues of the radix passes (by pass parity), the work items of the current
// pass, the sticky status (kept until the host reads it), the blocks the
// bucket sort flagged and those with kFlagOver, the queues and item counts of
// the bucket classes, the tied groups (short, long), and from kRsTileOff on the per-block tile counts.
enum : int {
    kRsTied = 0, kRsTiedMax = 1, kRsH = 2, kRsRound = 3, kRsAbort = 4, kRsFault = 5, kRsQueue = 6, kRsItems = 8,
    kRsSticky = 9, kRsFlagged = 10, kRsOver = 11, kRsBucketQueue = 12, kRsBucketClasses = 3,
    kRsBucketItems = kRsBucketQueue + kRsBucketClasses, kRsTies = kRsBucketItems + kRsBucketClasses,
    kRsTiesLong = kRsTies + 1, kRsEnter = kRsTiesLong + 1,
    kRsLongGroup = kRsEnter + 1, kRsTileOff = kRsLongGroup + 1
};
constexpr int kSortCtlHead = kRsTileOff;             // sort state words before the per-block tile counts
constexpr int kFlagTied = 1, kFlagOver = 2;  // block flags of the bucket sort (bwt_bucket.cu)
constexpr uint64_t kElemMask = (1u << 20) - 1u;      // rotation start in a sort word, below its key
constexpr int kCodeMax = 12;                         // longest code of the order-preserving byte code
constexpr int kKeyBits = 44;                         // code bits in a sort word
constexpr int kBuckets = 1408;                       // most buckets of a block
constexpr int kBucketRow = kBuckets + 8;             // bucket starts of a block (one more than buckets)

#define LFC_FULL 0xffffffffu

// One block's byte codes (length << 12 | code; after a zero byte, after
// another byte, first byte of a key), the first bucket of every 12-bit key
// prefix, and the 16-bit key prefix where each bucket starts.
struct BwtCode {
    uint16_t code[3 * 256];
    uint16_t base12[4104];  // 4097 used
    uint16_t split[kBuckets];
    int32_t nb, pad[3];
};
static_assert(sizeof(BwtCode) % 16 == 0, "BwtCode rows stay 16-byte aligned");

// Whole codes (bytes) in the key of a rotation.
static __device__ __noinline__ int key_depth(const uint8_t *rle, int m, const uint16_t *code, int idx) {
    int pos = idx, used = 0, depth = 0;
    uint32_t tab = 512;  // the first byte's table
    for (;;) {
        const uint32_t x = rle[pos];
        used += (int)(code[tab + x] >> 12);
        if (used > kKeyBits) return depth;
        depth++;
        tab = x ? 256u : 0u;
        if (++pos == m) pos = 0;
    }
}

// ------------------------------------------------------------ warp helpers
__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ uint32_t lanemask_lt() { return (1u << lane_id()) - 1u; }
__device__ __forceinline__ uint32_t lanemask_gt() { return lane_id() == 31 ? 0u : (~0u << (lane_id() + 1)); }

template <typename T>
__device__ __forceinline__ T warp_incl_sum(T v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(LFC_FULL, v, o);
        if ((int)lane_id() >= o) v += t;
    }
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(LFC_FULL, v, o);
    return v;
}

__device__ __forceinline__ int warp_incl_max(int v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(LFC_FULL, v, o);
        if ((int)lane_id() >= o) v = max(v, t);
    }
    return v;
}

// Block-wide exclusive sum over blockDim.x threads (<= 1024). `sh` needs 33
// entries. Returns the exclusive prefix; *total gets the block sum.
template <typename T>
__device__ __forceinline__ T block_excl_sum(T v, T *sh, T *total) {
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    T incl = warp_incl_sum(v);
    if (lane_id() == 31) sh[w] = incl;
    __syncthreads();
    if (w == 0) {
        T s = lane_id() < (uint32_t)nw ? sh[lane_id()] : T(0);
        T si = warp_incl_sum(s);
        if (lane_id() < (uint32_t)nw) sh[lane_id()] = si - s;
        if (lane_id() == 31) sh[32] = si;
    }
    __syncthreads();
    T r = sh[w] + incl - v;
    if (total) *total = sh[32];
    __syncthreads();
    return r;
}

// Block-wide exclusive max over blockDim.x threads (identity -1).
__device__ __forceinline__ int block_excl_max(int v, int *sh) {
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    int incl = warp_incl_max(v);
    if (lane_id() == 31) sh[w] = incl;
    __syncthreads();
    if (w == 0) {
        int s = lane_id() < (uint32_t)nw ? sh[lane_id()] : -1;
        int si = warp_incl_max(s);
        int ex = __shfl_up_sync(LFC_FULL, si, 1);
        if (lane_id() == 0) ex = -1;
        if (lane_id() < (uint32_t)nw) sh[lane_id()] = ex;
    }
    __syncthreads();
    int ex_in_warp = __shfl_up_sync(LFC_FULL, incl, 1);
    if (lane_id() == 0) ex_in_warp = -1;
    int r = max(sh[w], ex_in_warp);
    __syncthreads();
    return r;
}

// ------------------------------------------------------------ candidate ids
// Fields of a candidate id (include/lfc.h): f bits 0-2, byte layout bit 3
// (1: planar, high bytes then low bytes), domain bits 4-5, ordering bit 6,
// temporal bit 7.
__host__ __device__ __forceinline__ int id_f(int id) { return id & 7; }
__host__ __device__ __forceinline__ int id_planar(int id) { return (id >> 3) & 1; }
__host__ __device__ __forceinline__ int id_dom(int id) { return (id >> 4) & 3; }
__host__ __device__ __forceinline__ int id_ord(int id) { return (id >> 6) & 1; }
__host__ __device__ __forceinline__ int id_tmp(int id) { return (id >> 7) & 1; }

// ------------------------------------------------------------- descriptors
// One frame as the kernels see it.
struct FrameDev {
    const uint16_t *X;     // raw counts, row-major H x W
    const uint16_t *prev;  // previous raw frame or nullptr
    int32_t W, H, p, Nx, Ny;
};

// Judge work description of one frame.
struct JudgeFrame {
    FrameDev F;
    int32_t K;             // candidates judged
    int32_t cand_off;      // first entry in the candidate id table
    int32_t segs;          // segments (CTAs) per candidate
    int32_t rows_per_seg;  // stream rows per segment
    int64_t cta_base;      // first CTA index of this frame
    int64_t hist_off;      // first histogram (in units of 65536 bins)
    int64_t summ_off;      // first segment summary
    const uint64_t *mask;  // candidate mask (4 words) from the proposal, or nullptr = all
};

__device__ __forceinline__ bool cand_on(const JudgeFrame &J, int id) {
    return J.mask == nullptr || ((J.mask[id >> 6] >> (id & 63)) & 1ull);
}

// One bzip2 block: input bytes at src[0 .. len).
struct BlockDesc {
    const uint8_t *src;
    int32_t len;
    int32_t frame;         // owning frame (-1 for raw block encodes)
};

// Per-block coder state on the device (sizes the host never reads).
struct BlockState {
    int32_t m;             // RLE1 output length
    int32_t orig_ptr;      // BWT origin row
    int32_t n_act;         // active elements in the current doubling round
    int32_t n_act_next;    // active elements after the round
    int32_t n_mtf;         // bzip2 symbols including EOB
    int32_t n_in_use;      // distinct bytes in the block
    int32_t n_groups;
    int32_t n_sel;
    uint32_t crc;          // CRC-32/BZIP2 of the block input (word 8)
    uint32_t stream_bytes; // packed stream length
    uint32_t stream_bits;
    uint32_t data_bit0;    // first bit of the Huffman-coded data in the stream
    uint32_t in_use[8];    // bytes present in the block
};
static_assert(sizeof(BlockState) == 80, "BlockState layout");

// ------------------------------------------------------------------ plan
struct Workspace {
    // judge
    uint32_t *hist = nullptr;      // judge_frames_cap * K * 65536
    uint16_t *summ = nullptr;      // per judge CTA: first[256], last[256]
    uint8_t *chain_first = nullptr;  // per SM: the chain kernel's first-predecessor bytes
    int chain_nsm = 0;               // SM slots of chain_first (%nsmid)
    uint64_t *scores = nullptr;    // max_frames * 256
    uint8_t *choice = nullptr;     // max_frames
    JudgeFrame *jframes = nullptr; // judge_frames_cap
    uint8_t *cand = nullptr;       // judge_frames_cap * kMaxCand
    uint64_t *l2tab = nullptr;     // 65536
    int64_t summ_cap = 0;
    uint8_t *cstream = nullptr;    // candidate streams: judge_frames_cap * cstream_kmax slots
    // lfc_compress_host staging, allocated on its first call: frames, previous
    // frames, containers, sizes, given ids
    uint8_t *hx_frames = nullptr, *hx_prev = nullptr, *hx_out = nullptr, *hx_choice = nullptr;
    uint64_t *hx_sizes = nullptr;
    size_t hx_out_cap = 0;
    uint64_t *masks = nullptr;     // proposal candidate masks, max_frames x 4
    uint8_t *class_ids = nullptr;  // proposal class -> candidate id (64)
    int64_t cstream_slot = 0;
    int cstream_kmax = 0;
    // symbol streams of the frames being compressed
    uint8_t *stream = nullptr;     // max_frames * stream_slot
    int64_t stream_slot = 0;
    // coder, per block slot
    BlockDesc *blocks = nullptr;
    BlockState *bstate = nullptr;
    uint8_t *rle = nullptr;        // block_cap * kBlockCap
    int32_t *sa = nullptr;         // block_cap * kBlockCap
    int32_t *sa2 = nullptr;
    int32_t *rank = nullptr;
    int32_t *act = nullptr;        // active SA positions
    int32_t *act2 = nullptr;
    int32_t *val = nullptr;        // SA values of the active elements
    uint64_t *keys = nullptr;      // sort words, block_cap * kBlockCap
    uint64_t *keys2 = nullptr;
    uint32_t *lbstat = nullptr;    // radix look-back status, 2 arrays of block_cap * kTilesPerBlock * 256
    size_t lbstat_words = 0;       // words of one of those arrays
    uint32_t *dhist = nullptr;     // per block and radix pass: digit totals, block_cap * 8 * 256
    int32_t *segbig = nullptr;     // per block: a doubling round has a group longer than the segmented sort's window
    BwtCode *bcode = nullptr;      // bucket sort: byte code and splitters per block
    uint32_t *bcount = nullptr;    // rotations per bucket, block_cap * kBuckets
    uint32_t *bcursor = nullptr;   // scatter cursors, same shape
    uint32_t *bstart = nullptr;    // bucket starts, block_cap * kBucketRow
    uint32_t *bitems = nullptr;    // bucket work lists, one of bitems_cap entries per size class
    size_t bitems_cap = 0;
    int32_t *bflag = nullptr;      // kFlag* per block
    int32_t *bdeep = nullptr;      // per block: groups still tied after some further keys (bwt_bucket.cu)
    int32_t *tileaux = nullptr;    // block_cap * kTilesPerBlock * 4
    uint8_t *bwt = nullptr;        // L column
    uint8_t *mtfidx = nullptr;
    uint8_t *mtflists = nullptr;   // starting list per MTF segment, block_cap * kMtfSegs * 256
    uint8_t *mtfrec = nullptr;     // recency records, same shape
    int32_t *mtfreclen = nullptr;  // block_cap * kMtfSegs
    uint32_t *mtfpres = nullptr;   // bytes of a record as a bitmap, block_cap * kMtfSegs * 8
    uint8_t *mtfgrec = nullptr;    // records, then starting lists, of groups of segments (a sixteenth of the segments)
    uint32_t *mtfgpres = nullptr;
    int32_t *mtfglen = nullptr;
    uint16_t *sym = nullptr;       // block_cap * (kBlockCap + 1)
    uint32_t *freq = nullptr;      // block_cap * kMaxAlpha
    uint32_t *rfreq = nullptr;     // block_cap * kMaxGroups * kMaxAlpha, counts of a refinement pass
    uint8_t *sel = nullptr;        // block_cap * kMaxSelectors
    uint8_t *lens = nullptr;       // block_cap * 6 * 258
    uint32_t *codes = nullptr;     // block_cap * 6 * 258
    uint32_t *packed = nullptr;    // block_cap * stream_words
    int64_t stream_words = 0;
    int32_t *act_total = nullptr;  // sort state: kSortCtlHead words + block_cap + 1 tile offsets
    int32_t *h_act_total = nullptr;// pinned host mirror of the first kSortCtlHead words
    // container assembly
    uint64_t *block_dst = nullptr;     // block_cap: stream destination offsets
    uint32_t *frame_crc = nullptr;     // max_frames
    uint32_t *crc_part = nullptr;      // CRC partial remainders
    uint32_t *crc_part2 = nullptr;   // partial remainders of the frame CRCs (side stream)
    int64_t crc_part_cap = 0;
    void *chunk_desc = nullptr;        // descriptor staging (CRC chunks, frame tables)
    size_t chunk_desc_bytes = 0;
};

}  // namespace lfc

struct lfc_plan_s {
    lfc_config cfg;
    cudaStream_t stream = nullptr;
    cudaStream_t aux_stream = nullptr;  // capture of conditional-node bodies
    cudaStream_t side_stream = nullptr; // CRCs, overlapped with the judge and the BWT
    cudaEvent_t side_fork = nullptr, side_join = nullptr;
    cudaStream_t cap_stream = nullptr;  // capture of batches
    int device = 0;
    int sm_count = 0;  // streaming multiprocessors of the device
    std::string err;
    std::vector<uint8_t> ids_spatial;   // judged for every frame
    std::vector<uint8_t> ids_temporal;  // judged for frames with prev
    int judge_frames_cap = 0;           // frames per judge launch (allocated)
    lfc_tuning tune{16, 262144, 0, 0};    // autotuned judge knobs
    lfc_cnn cnn = nullptr;              // learned proposal (optional)
    int topk = 0;
    float tau = 0.f;
    int block_cap = 0;                  // blocks per coder pass
    lfc::Workspace ws;
    // tracing: CUDA events around stages, harvested by lfc_plan_timing
    bool timing = false;
    int64_t launches = 0;
    struct Span { int stage; cudaEvent_t a, b; };
    std::vector<Span> spans;
    std::vector<cudaEvent_t> event_pool;
    cudaEvent_t open_ev[LFC_NUM_STAGES] = {};
    double stage_ms[LFC_NUM_STAGES] = {};
    int64_t bwt_calls = 0, bwt_rounds = 0, bwt_tied_total = 0, bwt_elements = 0, bwt_elements_in = 0;
    int64_t bwt_round_tied[32] = {};
    long long wait_cycles = 0;          // bounded device waits: budget in SM clock cycles
    int sm_clock_khz = 0;
    bool bwt_timed_out = false;         // a wait of the last suffix sort gave up
    int64_t stage_spans[LFC_NUM_STAGES] = {};
};

namespace lfc {

// cnn.cu
int cnn_propose(lfc_cnn C, const lfc_frame *frames, int n, const uint8_t *d_class_ids, int topk, float tau,
                uint64_t *d_masks, cudaStream_t s);
int cnn_classes(lfc_cnn C);
int cnn_max_batch(lfc_cnn C);

// ---------------------------------------------------------------- tracing
void stage_begin(lfc_plan P, int stage);
void stage_end(lfc_plan P, int stage);
inline void count_launches(lfc_plan P, int n) { P->launches += n; }

// ------------------------------------------------------- internal launchers
// judge.cu
cudaError_t init_l2_table(uint64_t *tab, cudaStream_t s);
size_t judge_smem_bytes(int maxW);
// judge_stream.cu
size_t emit_all_smem_bytes(int p, int ts, int nslots);
size_t chain_smem_bytes();
int64_t chain_seg_bytes(int range_bytes);  // stream bytes one chain CTA covers
size_t chain_first_bytes(int nsm);          // chain_first bytes for nsm SM slots
cudaError_t query_nsmid(cudaStream_t s, int *nsm);
cudaError_t launch_emit_all(lfc_plan P, const JudgeFrame *d_frames, int nframes, const uint8_t *d_cand, int max_tiles,
                            int TS, int nslots_max, int any_temporal, int max_p);
cudaError_t launch_chain_hist(lfc_plan P, const JudgeFrame *d_frames, int nframes, const uint8_t *d_cand, int64_t total_ctas,
                              int range_bytes);
struct JudgeLaunch {
    int max_tiles, TS, nslots_max, any_temporal, max_p, range_bytes;
};
cudaError_t launch_judge(lfc_plan P, const JudgeFrame *d_frames, int nframes, int64_t total_ctas,
                         const JudgeLaunch &L, const uint8_t *d_cand, int64_t nhist,
                         uint64_t *d_scores, uint8_t *d_choice);
cudaError_t launch_copy_chosen(lfc_plan P, const JudgeFrame *d_frames, int nframes, const uint8_t *d_cand,
                               const uint8_t *d_choice, uint8_t *const *d_dst);
cudaError_t launch_emit(const FrameDev *h_frames, const uint8_t *d_choice, int nframes,
                        uint8_t *const *h_dst, cudaStream_t s);
cudaError_t launch_symbols_one(const FrameDev &F, int id, uint16_t *dst, cudaStream_t s);

// crc.cu
struct CrcRun {
    int nchunks = 0, nranges = 0;
    size_t off_first = 0, off_len = 0;
};
int crc_count_chunks(const int64_t *len, int n);
size_t crc_table_bytes(int nchunks, int n);
void crc_build_tables(const uint8_t *const *ptr, const int64_t *len, int n, uint8_t *out, CrcRun *run);
cudaError_t launch_crc(lfc_plan P, const uint8_t *d_tables, const CrcRun &run, uint32_t *out, int out_stride_words,
                       cudaStream_t stream = nullptr, uint32_t *part = nullptr);

// bwt.cu
cudaError_t launch_rle1(lfc_plan P, int nblocks, const BlockDesc *d_blocks);
cudaError_t launch_bwt(lfc_plan P, int nblocks, int max_m);
// bwt_bucket.cu: sorts every block's rotations, writes last columns; flags the blocks it could not finish
cudaError_t launch_bucket_sort(lfc_plan P, int nblocks, int max_m, bool graph);
cudaError_t launch_copy_bwt(lfc_plan P, int nblocks, uint8_t *d_L, size_t stride, uint32_t *d_len, uint32_t *d_orig);

// mtf_huff.cu
// max_m: the largest RLE1 length a block of the pass can have
cudaError_t launch_mtf_rle2(lfc_plan P, int nblocks, int max_m);
cudaError_t launch_huffman(lfc_plan P, int nblocks, int max_m);
cudaError_t launch_pack(lfc_plan P, int nblocks, int max_m);

// MTF segment length (log2) of a pass. A segment is one warp's serial work
// (112 us for 4096 bytes), so a pass that cannot fill the SMs with 32 warps
// twice over takes segments of 1024 bytes (30 us); a larger one is bound by
// issue and keeps 4096 (fewer starting lists).
inline int mtf_seg_log2(lfc_plan P, int nblocks, int max_m) {
    return (int64_t)nblocks * ((max_m + 4095) / 4096) < (int64_t)64 * P->sm_count ? 10 : 12;
}

// container.cu
struct FrameOut {
    uint64_t out_off;    // container offset in d_out
    int32_t block0, nblocks;
    int32_t W, H, p, pad;
};
cudaError_t launch_container(lfc_plan P, int nframes, int nblocks, const FrameOut *d_fo, const uint8_t *d_choice,
                             const uint32_t *d_frame_crc, uint8_t *d_out, uint64_t *d_out_sizes, int block_bytes);
cudaError_t launch_copy_streams(lfc_plan P, int nblocks, uint8_t *d_out, size_t stride, uint32_t *d_sizes);

// decode.cu
struct DecBlockHost {
    const uint8_t *src;
    int64_t src_len;
    uint8_t *dst;
    int32_t expect;
    int32_t pad;
};
// d_crc / crc: a CRC run over the blocks' output ranges, laid out by the caller
cudaError_t launch_bzip2_decode(lfc_plan P, const DecBlockHost *h_blocks, const void *d_blocks, int nblocks, const uint8_t *d_crc,
                                const CrcRun &crc, int32_t *d_status);
struct InvFrame {
    const uint16_t *Z;      // symbol stream (stream order)
    const uint16_t *prev;   // previous raw frame or nullptr
    uint16_t *X;            // output frame
    int32_t *E;             // int32 scratch field (W*H)
    int32_t W, H, p, id;
};
cudaError_t launch_inverse_predict(lfc_plan P, const InvFrame *h_frames, const InvFrame *d_frames, int n);

}  // namespace lfc
