// Dequant-GEMM on the Blackwell tensor cores: y = x W^T with W^ = code * scale.
//
// The tensor cores never see a scale: the B operand holds the integer codes as fp16 (exact; int8 in the integer-activation
// variant), every scale group (128 fan-in elements for W4, the whole row for W8) is accumulated on its own in TMEM, and
// each finished group is folded into fp32 registers, y += scale[n][g] * acc_g, while the tensor core is already on the
// next groups.
//
// A CTA computes tiles of 128 rows x BN columns.  K is walked in pairs of blocks of 64 elements (128 for int8) through two
// rings of shared-memory stages: activation tiles (128 rows x 128 bytes per block, by TMA) and expanded weight tiles (BN rows
// x 128 bytes per block), both in the 128-byte swizzle.  Every step has warps of its own, so that none of them is behind
// another one in program order:
//   producer  one thread issues the TMA loads of the activation tiles;
//   MMA       owns the TMEM allocation; one thread issues tcgen05.mma (M=128, N=BN, K=32 bytes) and commits;
//   scales    (2 warps) bring the scales and biases of a tile;
//   builders  (8 or 16 warps) fetch the packed codes straight from global memory into registers, one pair of blocks ahead,
//             and expand them into the weight tiles;
//   folders   (16 or 8 warps) one thread per row (TMEM lane) and HC = 40 or 32 columns: fold finished groups into registers
//             and run the epilogue: bias / fp16 conversion, or the per-(row, head) int8 quantization Q_a of Eq. 2, or the
//             mixed int8 / fp16 K~, V~ of Eq. 2 together with the attention kernel's operand images.
// Launches of more tiles than SMs are persistent: a CTA walks several tiles, and the epilogue of one runs under the K loop of
// the next (most of those with fp16 rows in and no fp32 rows out run on pairs of CTAs instead: taq_linear_pair_sm100.cuh).  The packed weights
// stay packed in HBM.
//
// What bounds it.  A 64-wide K block of a 160-column tile is 320 cycles of tensor time; the MMA thread needs 60 cycles per wait
// on a complete barrier, 60 per commit and 45 per MMA (measured), hence barriers per pair of blocks, looked at one pair ahead.
// A register spilled in a loop is a round trip to L2, since beside 200 KB of shared memory there is next to no L1 (a first version
// with 120 bytes of spills ran at half the speed), hence the register split.  What `-Xptxas -v` still reports at 72
// registers: 4 to 64 bytes stored and up to 108 loaded in most 160-wide kernels and some of the others, none in the rest.  Whether such a
// kernel pays for them is told by its time only: the unsplit 160-wide K/V kernels went from 8 / 8 bytes to 44 / 100 when their epilogue was
// shortened, and two prompts at 1280 channels from 15.3 to 14.0 us.
#pragma once
#include "taq_ptx.cuh"
#include "taq_sm100.cuh"
#include "taq_sm100_parts.cuh"
#include "taq_prof.cuh"
#include <atomic>
#include <cstddef>
#include <cstring>
#include <type_traits>

namespace taq {
namespace linear {

using namespace parts;

constexpr int BM = 128;
constexpr int BK = 64;                     // fp16 elements per 128-byte operand row; the int8 variant has 2 BK
constexpr int A_TILE_BYTES = BM * 128;     // 16 KB
constexpr int MAX_STAGE = 6;               // ring depths, in pairs of k-blocks
constexpr int MAX_SLOT = 8;                // accumulators in TMEM
constexpr int SMEM_LIMIT = 227 * 1024;

// Tile shapes: 160 columns (a multiple of every SD head width), 80 for launches with few rows, 128 and 64 for heads of 64 channels
// and matrices that are no multiple of 80.  One CTA per SM: what a launch costs beyond its K loop is the latency of a few
// hand-overs between warps, and more warps per role shorten it more than a second CTA hides it.
template <int BN_>
struct Tile {
    static constexpr int BN = BN_;
    // Folder warps and builder warps: the wide tiles have sixteen and eight (a thread of eight folder warps would hold 80 sums, which
    // spills, and two warps per scheduler hide neither TMEM nor shared-memory latency: a group took them 950 cycles), the
    // narrow ones, which live for one tile, eight and sixteen (their weight tiles are all built before the activations arrive).
    static constexpr bool BIG = BN >= 128;
    static constexpr int NCG = BIG ? 4 : 2;                                   // column groups: folder threads per row
    static constexpr int HC = BN / NCG;                                       // columns per folder thread: 40 or 32
    static constexpr int NF = 4 * NCG, NFOLD = 32 * NF;                       // folder warps, threads
    static constexpr int NB = 24 - NF, NBUILD = 32 * NB;                      // builder warps, threads
    // Warpgroups keep one role each, and registers go where they are needed.  What the block is launched with covers it:
    //   896 threads x 72 = 128 x (56 + 4 x 88 + 2 x 48) = 128 x (56 + 2 x 128 + 4 x 48)
    static constexpr int NTHREADS = 128 + NFOLD + NBUILD;
    static constexpr int W_PROD = 0, W_MMA = 1, W_AUX = 2, W_FOLD = 4, W_BUILD = W_FOLD + NF;
    static constexpr int R_FOLD = BIG ? 88 : 128, R_BUILD = 48, R_REST = 56;
    static_assert(128 * (R_REST + NF / 4 * R_FOLD + NB / 4 * R_BUILD) == NTHREADS * 72, "register split");
    // ... and of the K~/V~ epilogue's second half, one for both roles (they run the same code): the 72 of the launch.
    static constexpr int R_KV = 72;
    static_assert((NF + NB) * R_KV <= NF * R_FOLD + NB * R_BUILD, "register split");
    static constexpr uint32_t TMEM_COLS = 512;
    static constexpr int NSLOT = TMEM_COLS / BN;                              // accumulators in TMEM: 3 to 8
    static constexpr int B_TILE = BN * 128;                                   // one k-block
    static constexpr int NCH = BN * 16 / (NBUILD / 2);                        // 16-byte tile chunks per builder thread and pair of k-blocks
    static constexpr int PIECE = 32 * HC * 4;                                 // a warp's partial sums in transit
    static_assert(BN * 16 % (NBUILD / 2) == 0 && HC % 8 == 0 && NSLOT <= MAX_SLOT && NSLOT >= 3, "tile shape");
};

// The K~/V~ epilogue's fp32 tile in shared memory.
__host__ __device__ constexpr int kv_tile_bytes(int bn) { return (128 * (bn + 4) + 16 * 8) * 4; }

struct Bars {
    uint64_t full_a[MAX_STAGE], empty_a[MAX_STAGE], full_b[MAX_STAGE], empty_b[MAX_STAGE];
    uint64_t acc_full[MAX_SLOT], acc_free[MAX_SLOT];
    uint64_t scale_full[2], scale_free[2];
    uint64_t tmem_ready, peer_ready, part_full[16], pair_full[4];
    uint32_t tmem_base;
    volatile int abort_flag;
};
constexpr int N_BARS = 4 * MAX_STAGE + 2 * MAX_SLOT + 4 + 2 + 16 + 4;       // the barriers above, one after the other
static_assert(offsetof(Bars, tmem_base) == N_BARS * 8, "barriers are contiguous");

// Shared-memory plan of one launch (host and device agree through these numbers).
struct Plan { int ring_bytes, off_scales, scale_bytes, off_bias, off_xchg, off_bars, total; };

// nsa, nsb: pairs of k-blocks in the rings; persistent: a CTA walks several tiles.
template <int BN>
inline Plan make_plan(int n_groups, int nsa, int nsb, bool persistent, int x_bytes) {
    Plan p;
    p.ring_bytes = 2 * (nsa * x_bytes + nsb * Tile<BN>::B_TILE);
    p.off_scales = p.ring_bytes;                                              // (two buffers of) float [n_groups][BN], then bias [BN]
    p.scale_bytes = (n_groups + 1) * BN * 4;
    p.off_bias = p.off_scales + n_groups * BN * 4;
    p.off_xchg = p.off_scales + (persistent ? 2 : 1) * p.scale_bytes;         // float [4][128], then (K~/V~) the slots [128] and the bitmap [4]
    p.off_bars = p.off_xchg + 5 * 128 * 4 + 128;
    p.total = p.off_bars + 1024 + 1024;                                       // barriers + slack to align the base to 1024
    return p;
}

// How a launch is laid out: CTAs that share the K loop of a tile, ring depths in pairs of k-blocks, heads of 160 channels on two
// tiles, tiles; and what every thread would otherwise work out for itself at the start (a third of a small launch's prologue):
// the blob's layout, the shared-memory plan, multipliers for the divisions by n_cols and n_rows.
struct LinearLayout {
    int nsplit, nsa, nsb, head_pair, persistent;
    int d, per_head;                        // per-head outputs: head width, folder threads per (row, head) (four divisions less per thread:
    uint32_t mul_d;                         // 2048 x 1280 x 1280 14.7 -> 13.8 us, 8192 x 320 x 320 8.1 -> 7.3)
    int n_tiles, n_cols, n_rows;            // tiles of the launch: n_cols column tiles (K's and V's) per row tile, n_rows row tiles per z
    uint32_t mul_cols, mul_rows, mul_groups;            // see quotient()
    int n_groups, kb_per_group, n_kb;
    uint32_t row_bytes;
    unsigned long long off_scales, off_bias;
    Plan plan;
    // K~/V~: the block of a sequence (kv_layout) and its images (operand_geom), offsets below 2^31.  (At the end: in the middle of what
    // every launch reads it cost a small launch 0.3 us.)
    struct {
        uint32_t off_v_codes, off_k_scales, off_v_scales, off_k_trigger, off_v_trigger, off_trig_slot, off_operands, head_bytes, k_bytes, vt_bytes;
        unsigned long long block_bytes;
        int images, dp, kbq, n_heads;       // n_heads: of a tile
        uint32_t mul_dp;
        float logit_unit;                   // log2(e) / sqrt(d)
        uint32_t x_bytes;                   // of an activation tile: 128 rows, or the 80 that images have (the MMA's other rows are whatever lies behind them, and used by nobody)
    } kv;
    uint32_t prefetch_ctas, prefetch_bytes, blob_bytes;      // CTAs that ask for a share of the packed weights each (0: none)
};

// t / d by a multiplication (mul = 2^32 / d + 1, exact for t and d below 2^16; 0: divide).
__device__ __forceinline__ int quotient(int t, int d, uint32_t mul) { return mul ? (int)__umulhi((uint32_t)t, mul) : d == 1 ? t : t / d; }
inline uint32_t multiplier(int d, long long n) { return d > 1 && d < 65536 && n < 65536 ? (uint32_t)((1ull << 32) / (unsigned)d + 1) : 0u; }

__device__ __forceinline__ void ffma2(unsigned long long& acc, uint32_t lo, uint32_t hi, unsigned long long s) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(v), "l"(s));
}

// Packed codes of one 16-byte chunk of a weight tile, as they lie in the blob.
template <bool I8, bool W8> struct Code { using T = typename std::conditional<I8 && W8, uint4, typename std::conditional<I8 || W8, uint2, uint32_t>::type>::type; };
template <bool I8, bool W8>
__device__ __forceinline__ uint4 expand_chunk(const typename Code<I8, W8>::T& p) {
    if constexpr (I8 && W8) return p;
    else if constexpr (I8) { const uint2 lo = codes_w4_to_i8(p.x), hi = codes_w4_to_i8(p.y); return make_uint4(lo.x, lo.y, hi.x, hi.y); }
    else if constexpr (W8) return codes_w8_to_half(p);
    else return codes_w4_to_half(p);
}
template <bool I8, bool W8>
__device__ __forceinline__ typename Code<I8, W8>::T zero_codes() {
    if constexpr (I8 && W8) return make_uint4(0, 0, 0, 0);
    else if constexpr (I8) return make_uint2(0x88888888u, 0x88888888u);      // nibble 8 = code 0
    else if constexpr (W8) return make_uint2(0, 0);
    else return 0x88888888u;
}

// The output and the CTAs' share of the work are compiled in, not looked up: most launches last 6 to 9 us, and a kernel without
// the other outputs' code took 0.3 to 0.6 us less of them than one kernel for all (2048 x 640 x 640: Q~ 6.8 -> 6.1 us, fp16
// 6.25 -> 5.8 us; 8192 rows, Q~: 16.2 -> 15.6 us.  Since a launch that does not know its predecessor waits for its weights, and over
// buffers larger than L2, the three take 6.7, 6.2 and 17.4 us.)
enum class Out { F16, F32, Q8, KV };     // fp16 or fp32 rows; int8 rows with a scale per head; K~/V~
enum class Ctas { ONE, MANY, SPLIT };    // a tile per CTA; several tiles per CTA; a cluster of two or four CTAs per tile

// I8: the integer-activation variant (the literal W/A reading of Table 1).  The A operand is the int8 codes of the
// per-token-quantized activations, the B operand the int8 weight codes, the accumulators are exact int32; a K block is
// 128 elements (one W4 scale group), and the row's activation scale multiplies the folded sum at the end.
// Out::KV: the K and the V projection are one launch: the first half of the column tiles is K's.
// Ctas::SPLIT: for launches with few tiles and a long K loop, two or four CTAs (a cluster) share one output tile: each
// takes a share of the scale groups (of the k-blocks, when there is one group); then they exchange folded fp32 partial sums
// through stores into each other's shared memory, every CTA adding and storing its share of the tile's rows.
template <int BN, bool I8, bool W8, Out OUT, Ctas CTAS>
__global__ void __launch_bounds__(Tile<BN>::NTHREADS, 1)
linear_sm100_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ LinearArgs a, const __grid_constant__ LinearLayout lay) {
    using TL = Tile<BN>;
    constexpr bool KV = OUT == Out::KV;
    constexpr bool clustered = CTAS == Ctas::SPLIT;
    constexpr bool persistent = CTAS == Ctas::MANY;
    const bool head_pair = clustered && (!KV || BN == 80) && lay.head_pair;      // heads of 160 channels on the 80-wide tiles of two CTAs
    using CodeT = typename Code<I8, W8>::T;
    constexpr int HC = TL::HC, NCG = TL::NCG, NSLOT = TL::NSLOT, NCH = TL::NCH;
    constexpr int BKE = I8 ? 2 * BK : BK;             // elements per K block
    constexpr int FC = TL::BIG ? 8 : HC;            // columns of a group that are loaded at a time while it is folded
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* smem = smem_dyn + ((1024u - (ptx::smem_u32(smem_dyn) & 1023u)) & 1023u);   // 1024-byte aligned, still provably shared

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nsplit = clustered ? lay.nsplit : 1, nsa = lay.nsa, nsb = lay.nsb;
    const int rank = clustered ? (int)(blockIdx.x % (unsigned)nsplit) : 0;
    const int n_groups = lay.n_groups;
    const Plan& P = lay.plan;
    static_assert(sizeof(Bars) <= 1024, "barrier block");
    Bars* bars = reinterpret_cast<Bars*>(smem + P.off_bars);
    const uint32_t XT = KV ? lay.kv.x_bytes : (uint32_t)A_TILE_BYTES;      // an activation tile
    const int n_kb_all = lay.n_kb;                      // (int8: the last block may be ragged; TMA and the expansion zero-fill)
    const int kb_per_group = lay.kb_per_group;          // k-blocks in a full group (the last group may be shorter)
    // this CTA's share of the K loop: a run of whole scale groups, or (one scale per output channel) of k-blocks
    int g_begin = 0, g_end = n_groups, kb_begin = 0, kb_stop = n_kb_all;
    if (clustered) {
        if (n_groups == 1) {
            kb_begin = n_kb_all * rank / nsplit; kb_stop = n_kb_all * (rank + 1) / nsplit;
        } else {
            g_begin = n_groups * rank / nsplit; g_end = n_groups * (rank + 1) / nsplit;
            kb_begin = g_begin * kb_per_group; kb_stop = min(n_kb_all, g_end * kb_per_group);
        }
    }
    const int n_kb = kb_stop - kb_begin;
    const bool with_bias = (OUT == Out::F16 || OUT == Out::F32) && (I8 || rank == 0);   // (of CTAs that share a tile one starts from the bias)
    // Tiles: column tile fastest, so that the CTAs running at one time share rows of x; then row tile, then z.
    const int tile0 = (int)blockIdx.x / nsplit, tile_step = persistent ? (int)gridDim.x : lay.n_tiles;      // (several tiles: never split)
    auto tile_of = [&](int t, int& z, int& row0, int& col0, int& kv_which) {
        const int cz = quotient(t, lay.n_cols, lay.mul_cols);
        int c = t - cz * lay.n_cols;
        z = quotient(cz, lay.n_rows, lay.mul_rows);
        row0 = (cz - z * lay.n_rows) * BM;
        kv_which = KV && 2 * c >= lay.n_cols ? 1 : 0;
        if (kv_which) c -= lay.n_cols >> 1;
        col0 = c * BN;
    };

    TAQ_PROF_INIT
    if (tid == 0) { TAQ_PROF(0); TAQ_GPROF(30); }
    if (warp == TL::W_PROD) {
        // (one lane per barrier: sixty in a row by one thread took a fifth of a small launch's start)
        uint64_t* all = bars->full_a;
        constexpr int FULL_B = 2 * MAX_STAGE, EMPTY_B = 3 * MAX_STAGE, ACC_FREE = 4 * MAX_STAGE + MAX_SLOT, SCALE_FULL = ACC_FREE + MAX_SLOT, SCALE_FREE = SCALE_FULL + 2;
#pragma unroll
        for (int i = lane; i < N_BARS; i += 32) {
            const int count = i >= FULL_B && i < EMPTY_B ? TL::NB / 2 : i < ACC_FREE ? 1 : i < SCALE_FULL ? TL::NF : i < SCALE_FREE ? 2 : i < SCALE_FREE + 2 ? TL::NF :
                              i == SCALE_FREE + 3 && clustered ? max(nsplit - 1, 1) : 1;       // (the last: peer_ready)
            ptx::mbar_init(all + i, (uint32_t)count);
        }
        ptx::mbar_fence_init();
        __syncwarp();
        if (lane == 0) {
            bars->abort_flag = 0;
            if (clustered) {
                const int per_cta = 4 / nsplit;              // lane quarters whose rows a CTA finishes
                for (int cg = 0; cg < NCG; ++cg)             // the warps of those quarters receive a piece from every other CTA
                    for (int i = 0; i < per_cta; ++i) ptx::mbar_arrive_expect_tx(&bars->part_full[cg * 4 + rank * per_cta + i], (uint32_t)((nsplit - 1) * TL::PIECE));
                if (head_pair)
                    for (int i = 0; i < per_cta; ++i) ptx::mbar_arrive_expect_tx(&bars->pair_full[rank * per_cta + i], 128u);
            }
        }
    } else if (warp == TL::W_AUX && lane == 0) {
        ptx::tma_prefetch_desc(&tmap_x);
    }
    // Every role passes this barrier before it touches another role's state; the builders do so with their first codes under way,
    // and the producer, whose own barriers are all it needs, only announces itself and starts to load.
    auto start = [&](bool wait) {
        if (wait) asm volatile("bar.sync 14, %0;" ::"n"(TL::NTHREADS) : "memory");
        else asm volatile("bar.arrive 14, %0;" ::"n"(TL::NTHREADS) : "memory");
        if (clustered) ptx::cluster_arrive_relaxed();        // waited for right before the first operation on another CTA
    };
    auto blob_of = [&](int z, int kv_which) { return (const uint8_t*)(a.reqs ? ((KV ? kv_which : a.which) == 0 ? a.reqs[z].Wq : a.reqs[z].Wout) : kv_which ? a.w2 : a.w); };
    auto give_up = [&]() { raise_status(a.status, TAQ_ERR_TIMEOUT); bars->abort_flag = 1; };

    // K~/V~, second half: all folders and builders, once the fp32 tile and the scales of its rows are in shared memory.  Short loops
    // over 8-element chunks, neighbouring lanes on neighbouring chunks, write everything in runs.  (With a row per lane straight
    // from the registers this epilogue took 15 000 - 24 000 cycles: 32 sectors per store, 20 KB of unrolled code that runs
    // once.  With the eight folder warps alone these loops took 9 000: two warps on a scheduler hide no latency.
    // With the block's layout worked out here, 2 300 cycles went by before the first load; it comes from the host now: two
    // prompts of 77 x 768, W4, 320 channels 10.0 -> 8.6 us, 1280 channels 15.3 -> 14.0.)
    // Row t of the fp32 tile: 16-byte accesses by a row per lane, and reads of eight columns by four groups of eight rows, hit all banks
    // (with 4-byte accesses and an odd row length 2 prompts, W4, 320 channels took 8.70 us, 8.55 so; 32 prompts, 1280 channels, 52.0 and 50.1).
    auto kv_row = [](int t) { return t * (BN + 4) + (t >> 3) * 8; };
    auto kv_store = [&](int w) {
        constexpr int NT = TL::NFOLD + TL::NBUILD, NC8 = BN / 8;
        int z, row0, col0, kv_which;
        tile_of(tile0, z, row0, col0, kv_which);
        const auto& G = lay.kv;
        const int T = a.n_ctx, d = lay.d, head0 = quotient(col0, d, lay.mul_d), ch0 = head_pair ? col0 - head0 * d : 0;      // (ch0: the second half of a head on two tiles)
        uint8_t* blk = a.reqs ? (uint8_t*)a.reqs[z].kv : (uint8_t*)a.y + (size_t)z * G.block_bytes;
        uint8_t* img0 = blk + G.off_operands + (uint32_t)head0 * G.head_bytes;
        const int* slots = reinterpret_cast<const int*>(smem + P.off_xchg) + 512;
        const float* ys = reinterpret_cast<const float*>(smem);
        const float2* hs = reinterpret_cast<const float2*>(smem + kv_tile_bytes(BN));
        const int own_shift = nsplit == 1 ? 7 : nsplit == 2 ? 6 : 5;         // (CTAs that share the tile finish the rows of some lane quarters each)
        auto own = [&](int key) { return key >> own_shift == rank; };
        {                                                    // codes, trigger rows and K~'s image: 8 channels of a token
            const int c = (w % NC8) * 8, hl = quotient(ch0 + c, d, lay.mul_d), ch = ch0 + c - hl * d, h = head0 + hl;
            uint8_t* codes = blk + (kv_which ? G.off_v_codes : 0u) + (uint32_t)(h * T * d + ch);
            uint8_t* trigs = blk + (kv_which ? G.off_v_trigger : G.off_k_trigger) + (uint32_t)(h * d + ch) * 2;
            uint8_t* k_img = img0 + (uint32_t)hl * G.head_bytes + (ch >> 6) * (kOperandKeys * 128);
            for (int t = w / NC8; t < T && w < NT / NC8 * NC8; t += NT / NC8) {
                if (!own(t)) continue;
                const int slot = slots[t];
                const float rs = hs[hl * 128 + t].y;
                const float4* row = reinterpret_cast<const float4*>(ys + kv_row(t) + c);
                const float4 lo = row[0], hi = row[1];
                const float f[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                const uint2 code = slot == -1 ? quant8(f, rs) : make_uint2(0, 0);
                *reinterpret_cast<uint2*>(codes + t * d) = code;
                uint4 k8 = codes_w8_to_half(code);
                if (slot >= 0) {
                    k8 = pack8(f);
                    *reinterpret_cast<uint4*>(trigs + (size_t)slot * a.n_out * 2) = k8;
                }
                if (G.images && !kv_which) *reinterpret_cast<uint4*>(k_img + ptx::sw128_offset(t, (ch >> 3) & 7)) = k8;
            }
        }
        if (!G.images) return;
        if (!kv_which) {                                     // K~'s padding: keys T..79, and the channels behind the head's last
            const int cc0 = ch0 >> 3, ncc = head_pair && ch0 == 0 ? NC8 : G.kbq * 8;       // (of a head on two tiles this CTA's)
            for (int line = w >> 3; line < G.n_heads * kOperandKeys; line += NT / 8) {
                const int hl = line / kOperandKeys, t = line - hl * kOperandKeys;
                if (!own(t)) continue;
                for (int cc = (w & 7) + (t >= T || d >= 64 ? 0 : d / 8 & ~7); cc < ncc; cc += 8)
                    if ((t >= T && cc >= cc0) || cc * 8 >= d) *reinterpret_cast<uint4*>(img0 + (uint32_t)hl * G.head_bytes + (cc >> 3) * (kOperandKeys * 128) + ptx::sw128_offset(t, cc & 7)) = make_uint4(0, 0, 0, 0);
            }
        } else {
            // V~^T: 8 keys of a channel per lane; a warp takes 8 channels x 4 chunks of keys (reads of the fp32 tile without bank
            // conflicts, stores of 64 contiguous bytes).  Everything is read first (rows and columns beyond the last token and
            // channel, too: something of the tile, not used), so that a chunk costs one round trip to shared memory.
            const int wl = w & 31;
            for (int u = w >> 5; u < (head_pair ? BN : G.n_heads * G.dp) / 2; u += NT / 32) {
                const int jc = (u & 3) * 4 + (wl >> 3), line = ch0 + (u >> 2) * 8 + (wl & 7), hl = quotient(line, G.dp, G.mul_dp), ch = line - hl * G.dp;
                if (!own(jc * 8)) continue;
                const float* col = ys + kv_row(jc * 8) + hl * d + min(ch, d - 1) - ch0;
                const float4* sc4 = reinterpret_cast<const float4*>(hs + hl * 128 + jc * 8);
                const int n_real = ch < d ? T - jc * 8 : 0;
                float x[8];
                float4 sc[4];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = col[e * (BN + 4)];
#pragma unroll
                for (int e = 0; e < 4; ++e) sc[e] = sc4[e];
                __half v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float s1 = e & 1 ? sc[e / 2].z : sc[e / 2].x, rs = e & 1 ? sc[e / 2].w : sc[e / 2].y;
                    const float quantized = __fmul_rn(fmaf(x[e], rs, 12582912.0f) - 12582912.0f, s1);
                    v[e] = __float2half_rn(e >= n_real ? 0.f : rs < 0.f ? x[e] : quantized);      // (rs < 0: a trigger row)
                }
                *reinterpret_cast<uint4*>(img0 + (uint32_t)hl * G.head_bytes + G.k_bytes + (jc >> 3) * (G.dp * 128) + ptx::sw128_offset(ch, jc & 7)) = *reinterpret_cast<const uint4*>(v);
            }
        }
    };
    if (warp >= TL::W_FOLD && warp < TL::W_BUILD) {
        // ---------------- folders ----------------
        start(true);
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(TL::R_FOLD));
        const int ft = tid - 32 * TL::W_FOLD;
        const int q = warp & 3;                              // TMEM lane quarter this warp may read
        const int cg = (warp - TL::W_FOLD) >> 2;             // column group
        const int fw = cg * 4 + q;
        const int r = q * 32 + lane;
        const int cb = cg * HC;                              // first owned column inside the tile
        int slot = 0, sbuf = 0;
        uint32_t ph_acc = 0, ph_scale = 0;
        bool alive = true;                                   // no wait has run out (a warp skips work then, never a barrier)
        uint32_t tmem_base = 0;
        if (ptx::mbar_wait(&bars->tmem_ready, 0)) tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base); else give_up();
        ptx::pdl_wait();                                     // (nothing to fold before the activations have come anyway) orders the stores below
        __syncwarp();
        if (clustered) ptx::cluster_wait();                  // the other CTAs' barriers exist
        for (int tile = tile0; tile < lay.n_tiles; tile += tile_step) {
            int z, row0, col0, kv_which;
            tile_of(tile, z, row0, col0, kv_which);
            const float* scales = reinterpret_cast<const float*>(smem + P.off_scales + sbuf * P.scale_bytes) + cb;
            const float* bias = scales + n_groups * BN;
            unsigned long long y2[HC / 2];
            bool ok = alive && ptx::mbar_wait(&bars->scale_full[sbuf], ph_scale);
#pragma unroll
            for (int c = 0; c < HC; c += 4) {                // the sums start from the bias (zero where there is none; int8: added last)
                const ulonglong2 b4 = *reinterpret_cast<const ulonglong2*>(bias + c);
                y2[c / 2] = I8 ? 0ull : b4.x; y2[c / 2 + 1] = I8 ? 0ull : b4.y;
            }
            // y += scale[g] * accumulator of group g (this thread's HC columns of its row)
            for (int g = g_begin; g < g_end && ok; ++g) {
                ok = ptx::mbar_wait(&bars->acc_full[slot], ph_acc);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + slot * BN + cb;
                const float* sg = scales + g * BN;
                // (the next columns are on their way from TMEM while these are multiplied and added: a group of 80 columns took
                // 850 cycles one load after the other, and the folders, not the tensor core, set the pace of a large launch)
                uint32_t v[2][FC / 8][8];
#pragma unroll
                for (int i = 0; i < FC / 8; ++i) ptx::tmem_ld8(taddr + i * 8, v[0][i]);
#pragma unroll
                for (int c0 = 0; c0 < HC; c0 += FC) {
                    const int k = (c0 / FC) & 1;
                    ptx::tmem_ld_wait(v[k][0]);
#pragma unroll
                    for (int i = 1; i < FC / 8; ++i) ptx::reg_fence8(v[k][i]);
                    if (c0 + FC < HC) {
#pragma unroll
                        for (int i = 0; i < FC / 8; ++i) ptx::tmem_ld8(taddr + c0 + FC + i * 8, v[k ^ 1][i]);
                    } else {                                 // the accumulator is in registers: the tensor core may have it back
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(&bars->acc_free[slot]);
                    }
#pragma unroll
                    for (int i = 0; i < FC / 8; ++i) {
                        const ulonglong2 s0 = *reinterpret_cast<const ulonglong2*>(sg + c0 + i * 8), s1 = *reinterpret_cast<const ulonglong2*>(sg + c0 + i * 8 + 4);
                        uint32_t (&w)[8] = v[k][i];
                        if (I8) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(__int2float_rn((int)w[e]));
                        }
                        unsigned long long* yy = y2 + (c0 + i * 8) / 2;
                        ffma2(yy[0], w[0], w[1], s0.x); ffma2(yy[1], w[2], w[3], s0.y);
                        ffma2(yy[2], w[4], w[5], s1.x); ffma2(yy[3], w[6], w[7], s1.y);
                    }
                }
                if (++slot == NSLOT) { slot = 0; ph_acc ^= 1; }
            }
            if (!ok && alive) { give_up(); alive = false; }
            if (ft == 0) TAQ_PROF(7);
            if (!I8 && lane == 0) ptx::mbar_arrive(&bars->scale_free[sbuf]);     // scales and biases of this tile have been read

            float y[HC];
#pragma unroll
            for (int c = 0; c < HC / 2; ++c) asm("mov.b64 {%0, %1}, %2;" : "=f"(y[2 * c]), "=f"(y[2 * c + 1]) : "l"(y2[c]));

            bool mine = alive;                               // this CTA finishes the warp's rows
            if (clustered) {
                // All of this CTA's MMAs are complete (every group was folded), so its rings are free: they take the partial sums that
                // come in.  CTA `owner` of the cluster finishes the rows of 4 / nsplit lane quarters: a folder warp either
                // stores its 32 rows into that CTA's shared memory, straight from the registers (16 bytes a lane, the lanes
                // of a store next to each other, no staging, no bank conflicts), or receives a piece from every other CTA and
                // adds them in rank order, so that every output is the same sum whoever computes it.  Rows beyond the last one
                // stay where they are (the exchange goes at about 25 bytes a cycle, and a launch of 64 rows is half padding).
                const bool padding = !KV && (long long)row0 + q * 32 >= a.rows;          // (K~/V~: rows beyond the last are keys of the images)
                const int per_cta = 4 / nsplit, owner = q / per_cta;
                const uint32_t base = ptx::cluster_ctarank() - (uint32_t)rank;        // ranks along x are consecutive
                mine = alive && owner == rank && !padding;
                if (ft < nsplit && ft != rank) ptx::mbar_arrive_cluster_relaxed(ptx::map_to_cta(ptx::smem_u32(&bars->peer_ready), base + (uint32_t)ft));
                auto piece = [&](int cta, int from) { return smem + ((cg * per_cta + q - cta * per_cta) * (nsplit - 1) + (from < cta ? from : from - 1)) * TL::PIECE + lane * 16; };
                if (padding || nsplit == 1) {
                    // nothing to send, nothing comes
                } else if (owner != rank) {
                    if (alive && ptx::mbar_wait(&bars->peer_ready, 0)) {                 // the other CTAs' rings are free, too
                        const uint32_t dst = ptx::map_to_cta(ptx::smem_u32(piece(owner, rank)), base + (uint32_t)owner);
                        const uint32_t bar = ptx::map_to_cta(ptx::smem_u32(&bars->part_full[fw]), base + (uint32_t)owner);
#pragma unroll
                        for (int c = 0; c < HC; c += 4)
                            ptx::store_to_cta(dst + c * 128, __float_as_uint(y[c]), __float_as_uint(y[c + 1]), __float_as_uint(y[c + 2]), __float_as_uint(y[c + 3]), bar);
                    } else give_up();
                } else if (!ptx::mbar_wait(&bars->part_full[fw], 0) || !ptx::mbar_wait(&bars->peer_ready, 0)) {      // (peer_ready: no arrival may come in after the CTA has left)
                    give_up();
                } else {
                    const unsigned char* in = smem + (cg * per_cta + q - rank * per_cta) * (nsplit - 1) * TL::PIECE + lane * 16;
                    if (nsplit == 2) {
#pragma unroll
                        for (int c = 0; c < HC; c += 4) {
                            const float4 p4 = *reinterpret_cast<const float4*>(in + c * 128);
                            y[c] += p4.x; y[c + 1] += p4.y; y[c + 2] += p4.z; y[c + 3] += p4.w;
                        }
                    } else {
                        // rank order, ((p0 + p1) + p2) + p3, with this CTA's own sum in its place (o: the others')
                        auto sum4 = [&](float own, float o0, float o1, float o2) {
                            const float s01 = o0 + (rank <= 1 ? own : o1);
                            return (s01 + (rank <= 1 ? o1 : rank == 2 ? own : o2)) + (rank == 3 ? own : o2);
                        };
#pragma unroll
                        for (int c = 0; c < HC; c += 4) {
                            const float4 o0 = *reinterpret_cast<const float4*>(in + c * 128), o1 = *reinterpret_cast<const float4*>(in + TL::PIECE + c * 128),
                                         o2 = *reinterpret_cast<const float4*>(in + 2 * TL::PIECE + c * 128);
                            y[c] = sum4(y[c], o0.x, o1.x, o2.x); y[c + 1] = sum4(y[c + 1], o0.y, o1.y, o2.y);
                            y[c + 2] = sum4(y[c + 2], o0.z, o1.z, o2.z); y[c + 3] = sum4(y[c + 3], o0.w, o1.w, o2.w);
                        }
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"n"(TL::NFOLD) : "memory");     // pieces read: the epilogue stages output where they were
                if (ft == 0) TAQ_PROF(10);
                mine = mine && !bars->abort_flag;
            }
            unsigned char* staging = smem;

            const long long row = (long long)row0 + r;
            const bool live = mine && row < a.rows;
            if (I8) {                                        // x~ = code * s_x: the row's activation scale
                const float sx = live ? a.x_scales[(size_t)z * a.rows + row] : 0.f;
#pragma unroll
                for (int c = 0; c < HC; c += 4) {
                    const float4 b4 = *reinterpret_cast<const float4*>(bias + c);
                    y[c] = fmaf(y[c], sx, b4.x); y[c + 1] = fmaf(y[c + 1], sx, b4.y); y[c + 2] = fmaf(y[c + 2], sx, b4.z); y[c + 3] = fmaf(y[c + 3], sx, b4.w);
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&bars->scale_free[sbuf]);
            }

            // ---------------- epilogue on this thread's HC columns ----------------
            // Dense outputs.  A CTA with one tile stages each warp's rows in shared memory (its rings are free) and stores them with
            // neighbouring lanes on neighbouring chunks of a row; a CTA that walks several tiles stores a row per lane straight from
            // the registers, in pieces of 32 bytes.  (TMA stores cost a one-tile CTA 1 000 cycles of waiting until the box was
            // read, and the folders of the others 2 600 per tile of fences and waits for the box before.)
            auto put = [&](const uint32_t* w, auto bytes_c) {                        // the thread's columns, `bytes` in w
                constexpr int ROW = decltype(bytes_c)::value, ESZ = ROW / HC, CHUNK = ROW % 16 == 0 ? 16 : 8, N = ROW / CHUNK;
                using V = typename std::conditional<CHUNK == 16, uint4, uint2>::type;
                uint8_t* dst = (uint8_t*)a.y + (((size_t)z * a.rows + row0 + q * 32) * a.n_out + col0 + cb) * ESZ;
                const uint32_t pitch = (uint32_t)a.n_out * ESZ;
                const long long left = mine ? a.rows - ((long long)row0 + q * 32) : 0;
                if (persistent) {
                    if (lane >= left) return;
                    dst += (size_t)lane * pitch;
                    const uint32_t odd = (uint32_t)reinterpret_cast<uintptr_t>(dst) & 31u;
                    if constexpr (ROW == 40) {               // 8 + 16 + 16 or 16 + 16 + 8 bytes
                        const uint2 *w2 = reinterpret_cast<const uint2*>(w);
                        if (odd & 8u) {
                            *reinterpret_cast<uint2*>(dst) = w2[0];
#pragma unroll
                            for (int i = 0; i < 2; ++i) reinterpret_cast<uint4*>(dst + 8)[i] = make_uint4(w[2 + 4 * i], w[3 + 4 * i], w[4 + 4 * i], w[5 + 4 * i]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 2; ++i) reinterpret_cast<uint4*>(dst)[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
                            *reinterpret_cast<uint2*>(dst + 32) = w2[4];
                        }
                    } else if (odd == 0) {
#pragma unroll
                        for (int i = 0; i < ROW / 32; ++i) ptx::store_32b(dst + i * 32, w + i * 8);
                        if constexpr (ROW % 32 == 16) *reinterpret_cast<uint4*>(dst + ROW - 16) = *reinterpret_cast<const uint4*>(w + ROW / 4 - 4);
                    } else if (odd == 16 && ROW % 32 == 16) {
                        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(w);
#pragma unroll
                        for (int i = 0; i < ROW / 32; ++i) ptx::store_32b(dst + 16 + i * 32, w + 4 + i * 8);
                    } else {
#pragma unroll
                        for (int i = 0; i < N; ++i) reinterpret_cast<V*>(dst)[i] = reinterpret_cast<const V*>(w)[i];
                    }
                } else {
                    unsigned char* st = staging + (size_t)fw * 32 * ROW;
#pragma unroll
                    for (int i = 0; i < N; ++i) reinterpret_cast<V*>(st + lane * ROW)[i] = reinterpret_cast<const V*>(w)[i];
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < N; ++i) {
                        const int j = lane + 32 * i, rr = j / N, part = j - rr * N;
                        if (rr < left) *reinterpret_cast<V*>(dst + (size_t)rr * pitch + part * CHUNK) = *reinterpret_cast<const V*>(st + j * CHUNK);
                    }
                }
            };
            if constexpr (OUT == Out::F16) {
                alignas(16) uint32_t w[HC / 2];
#pragma unroll
                for (int c = 0; c < HC; c += 2) {
                    const __half2 h = __floats2half2_rn(y[c], y[c + 1]);
                    w[c / 2] = *reinterpret_cast<const uint32_t*>(&h);
                }
                put(w, std::integral_constant<int, HC * 2>{});
            } else if constexpr (OUT == Out::F32) {
                alignas(16) uint32_t w[HC];
#pragma unroll
                for (int c = 0; c < HC; ++c) w[c] = __float_as_uint(y[c]);
                put(w, std::integral_constant<int, HC * 4>{});
            } else {
                // Per-(row, head) symmetric int8.  A thread's columns are one head or a half or a quarter of one.  On 32-column threads
                // heads are 64 wide, which is compiled in where it shortens the code (8192 x 1280 x 1280 of int8 rows and W8, heads of
                // 64: 25.1 -> 23.2 us; with fp16 rows and W4 the persistent kernel would spill: 8192 x 640 x 640 15.8 -> 16.6; int8
                // rows and W8, a tile per CTA: 1294 x 1280 x 1280 7.67 -> 7.77).
                constexpr bool D64 = !KV && HC == 32 && (I8 != W8 || (I8 && persistent));
                const int d = D64 ? 64 : lay.d;
                const int colg = col0 + cb;
                const int h0 = D64 ? colg / 64 : quotient(colg, d, lay.mul_d);
                float am = 0.f;
#pragma unroll
                for (int c = 0; c < HC; ++c) am = fmaxf(am, fabsf(y[c]));
                if (d > HC) {                                // the row's threads with columns of the same head combine their absmax
                    float* xc = reinterpret_cast<float*>(smem + P.off_xchg);     // [NCG][128], and at 384 the absmax of a head pair's other half
                    // (the partners by exclusive or in the persistent kernels of int8 rows, which spill less: 8192 x 1280 x 1280, W8,
                    // heads of 160, 27.0 -> 26.3 us; the others spill more that way)
                    constexpr bool PARTNERS = I8 && persistent;
                    const int per_head = D64 ? 2 : lay.per_head, first = cg & ~(per_head - 1);
                    xc[cg * 128 + r] = am;
                    asm volatile("bar.sync %0, %1;" ::"r"(2 + q), "n"(NCG * 32) : "memory");
#pragma unroll
                    for (int k = PARTNERS ? 1 : 0; k < NCG; ++k) if (k < per_head) am = fmaxf(am, xc[(PARTNERS ? cg ^ k : first + k) * 128 + r]);
                    if (persistent) asm volatile("bar.sync %0, %1;" ::"r"(6 + q), "n"(NCG * 32) : "memory");      // (read before the next tile's are written)
                    if (head_pair && mine) {
                        // The head's other columns belong to a CTA of the same cluster (same rows, same share of the K loop):
                        // each sends its rows' absmax over.
                        const uint32_t me = ptx::cluster_ctarank();
                        const uint32_t other = me < (uint32_t)nsplit ? me + nsplit : me - nsplit;
                        if (cg == 0) ptx::store_to_cta(ptx::map_to_cta(ptx::smem_u32(xc + 384 + r), other), __float_as_uint(am), ptx::map_to_cta(ptx::smem_u32(&bars->pair_full[q]), other));
                        if (ptx::mbar_wait(&bars->pair_full[q], 0)) am = fmaxf(am, xc[384 + r]);
                        else give_up();
                        __syncwarp();
                    }
                }
                const float qmax = KV && a.kv_qmax ? (float)a.kv_qmax : 127.f;
                const float s = quant_scale(am, qmax), rs = s > 0.f ? __frcp_rn(s) : 0.f;
                const bool owner = colg == h0 * d;           // holds the head's first column: writes its scale
                if constexpr (!KV) {
                    // Q~ = Q_a(Q), Eq. 2 third line
                    alignas(16) uint32_t w[HC / 4];
#pragma unroll
                    for (int c = 0; c < HC; c += 8) {
                        const uint2 code = quant8(y + c, rs);
                        w[c / 4] = code.x; w[c / 4 + 1] = code.y;
                    }
                    put(w, std::integral_constant<int, HC>{});
                    if (live && owner) a.scales[((size_t)z * a.rows + row) * a.heads + h0] = s;
                } else {
                    // Eq. 2 for K or V of one sequence (a row tile is one sequence; rows beyond its T tokens are the padding keys of
                    // the images): rows of ordinary tokens -> int8 codes + scale, rows of trigger tokens -> fp16; and the same
                    // rows once more as the attention kernel's operand images (taq_kv_operands.cu rebuilds them for blocks
                    // that were not written here): K~ as a row of fp16 integers, V~ as a column of fp16(code * scale).  The
                    // fp32 tile goes through shared memory to kv_store below.
                    const int T = a.n_ctx;
                    const int* slots = reinterpret_cast<const int*>(smem + P.off_xchg) + 512;      // [128] and the bitmap [4], by the scales' warps
                    const auto& G = lay.kv;
                    uint8_t* blk = a.reqs ? (uint8_t*)a.reqs[z].kv : (uint8_t*)a.y + (size_t)z * G.block_bytes;
                    const int head0 = quotient(col0, d, lay.mul_d);
                    float* ys = reinterpret_cast<float*>(staging);                   // see kv_row
                    float2* hs = reinterpret_cast<float2*>(staging + kv_tile_bytes(BN));   // [heads][128] scale and its reciprocal (trigger rows: 0 and -1)
                    if (mine) {
                        const int slot = slots[r];           // >= 0: trigger row, -1: ordinary (or padding), -2: a trigger row beyond the capacity
                        const bool plain = r < T && slot == -1;
#pragma unroll
                        for (int c = 0; c < HC; c += 4) *reinterpret_cast<float4*>(ys + kv_row(r) + cb + c) = make_float4(y[c], y[c + 1], y[c + 2], y[c + 3]);
                        const float sk = plain ? s : 0.f;
                        if (owner || (head_pair && cg == 0)) hs[(h0 - head0) * 128 + r] = make_float2(sk, plain ? rs : slot >= 0 ? -1.f : 0.f);
                        if (owner) {
                            if (r < T) reinterpret_cast<float*>(blk + (kv_which ? G.off_v_scales : G.off_k_scales))[(uint32_t)(h0 * T + r)] = sk;
                            if (!kv_which && h0 == 0) reinterpret_cast<int32_t*>(blk + G.off_trig_slot)[r] = slot >= 0 ? slot : -1;
                            if (!kv_which && G.images && r < kOperandKeys) {
                                OperandConsts* cst = reinterpret_cast<OperandConsts*>(blk + G.off_operands + (uint32_t)h0 * G.head_bytes + G.k_bytes + G.vt_bytes);
                                cst->logit_factor[r] = (slot >= 0 ? 1.0f : sk) * G.logit_unit;
                                if (r < 4) cst->trig_bits[r] = (uint32_t)slots[128 + r];
                            }
                        }
                    }
                }
            }
            sbuf ^= 1;
            if (sbuf == 0) ph_scale ^= 1;
        }
        __syncwarp();
    } else if (warp >= TL::W_BUILD && warp < TL::W_BUILD + TL::NB) {
        // ---------------- builders ----------------
        const int bt = (tid - 32 * TL::W_BUILD) & (TL::NBUILD / 2 - 1), group = (warp - TL::W_BUILD) / (TL::NB / 2);
        unsigned char* b_ring = smem + 2 * nsa * XT;
        // The two halves of the builders take the pairs of k-blocks in turn: a pair costs its warps about 900 cycles of latency
        // (barrier, expansion, proxy fence), half of which is somebody else's turn.  16 chunks per weight row; sixteen
        // consecutive lanes take one row, so that a warp's loads are two runs of 64 (128) consecutive bytes and its stores
        // of a tile row hit all banks.
        constexpr int CB = (int)sizeof(CodeT);
        const int c16 = bt & 15, n0 = bt >> 4;
        const uint32_t row_step = (uint32_t)(TL::NBUILD / 32) * lay.row_bytes;
        const int n_pair = (n_kb + 1) / 2;
        // Codes are fetched one turn ahead, across tile boundaries: as many of a pair's chunks as twenty registers hold (more would
        // spill), the rest when they are needed.
        constexpr int NPRE = NCH * (CB / 4) <= 20 ? NCH : NCH * (CB / 4) <= 40 ? NCH / 2 : NCH / 4;
        static_assert(NCH % NPRE == 0, "rounds");
        CodeT pw[NPRE];
        const uint8_t* src = nullptr;                        // codes of the fetched pair
        int tile = tile0, pair = group;                      // the fetched pair
        // (Weights that the previous kernel in the stream is known not to write are fetched and expanded under its tail.)
        auto load = [&](int j) {
            const int i = 2 * pair + (c16 >> 3);
            const bool have = i < n_kb && (!I8 || (kb_begin + 2 * pair) * BKE + c16 * 16 < a.k_in);
            return have ? ptx::load_global(reinterpret_cast<const CodeT*>(src + (uint32_t)j * row_step)) : zero_codes<I8, W8>();
        };
        auto fetch = [&](bool new_tile) {
            while (pair >= n_pair) { pair -= n_pair; tile += tile_step; new_tile = true; }
            if (tile >= lay.n_tiles) return;
            if (new_tile) {
                int z, row0, col0, kv_which;
                tile_of(tile, z, row0, col0, kv_which);
                src = blob_of(z, kv_which) + 128 + (size_t)(col0 + n0) * lay.row_bytes + (size_t)(kb_begin + 2 * pair) * (8 * CB) + c16 * CB;
            }
#pragma unroll
            for (int j = 0; j < NPRE; ++j) pw[j] = load(j);
        };
        if (a.early_weights) fetch(true);
        start(true);
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TL::R_BUILD));
        if (!a.early_weights) { ptx::pdl_wait(); fetch(true); }
        int s = group;
        uint32_t ph = 1;
        bool passed = false, ok = true;                      // passed: the ring has been passed once
        while (tile < lay.n_tiles) {
            while (s >= nsb) { s -= nsb; ph ^= 1; passed = true; }
            if (passed && !ptx::mbar_wait(&bars->empty_b[s], ph)) { ok = false; break; }
            unsigned char* tile_b = b_ring + (2 * s + (c16 >> 3)) * TL::B_TILE;
            if (c16 < 8 || 2 * pair + 1 < n_kb) {
#pragma unroll
                for (int j = 0; j < NPRE; ++j) *reinterpret_cast<uint4*>(tile_b + ptx::sw128_offset(n0 + j * (TL::NBUILD / 32), c16 & 7)) = expand_chunk<I8, W8>(pw[j]);
#pragma unroll
                for (int j0 = NPRE; j0 < NCH; j0 += NPRE) {
#pragma unroll
                    for (int j = 0; j < NPRE; ++j) pw[j] = load(j0 + j);
#pragma unroll
                    for (int j = 0; j < NPRE; ++j) *reinterpret_cast<uint4*>(tile_b + ptx::sw128_offset(n0 + (j0 + j) * (TL::NBUILD / 32), c16 & 7)) = expand_chunk<I8, W8>(pw[j]);
                }
            }
            if (bt == 0 && pair < 10) TAQ_PROF(60 + 2 * pair);
            pair += 2; src += 32 * CB;
            fetch(false);
            ptx::fence_proxy_async_smem();                   // make the generic-proxy writes visible to the tensor core
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars->full_b[s]);
            s += 2;
        }
        if (!ok) give_up();
        __syncwarp();
        if (!KV && clustered) ptx::cluster_wait();
    } else {
        start(warp != TL::W_PROD);
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TL::R_REST));
        if (warp == TL::W_PROD) {
            // ---------------- producer: activation tiles ----------------
            if (lane == 0) {
                ptx::pdl_wait();                             // the activations may come from the previous kernel
                // (Not before the wait: the successor's early reads, K~/V~ images and weights, may be of data that whatever ran before
                // this kernel wrote.)
                ptx::pdl_trigger();
                TAQ_PROF(1); TAQ_GPROF(28);
                int s = 0, issued = 0;
                uint32_t ph = 1;
                bool passed = false, ok = true;
                for (int tile = tile0; tile < lay.n_tiles && ok; tile += tile_step) {
                    int z, row0, col0, kv_which;
                    tile_of(tile, z, row0, col0, kv_which);
                    for (int i = 0; i < n_kb; i += 2) {
                        if (passed && !ptx::mbar_wait(&bars->empty_a[s], ph)) { give_up(); ok = false; break; }
                        unsigned char* dst = smem + 2 * s * XT;
                        const bool two = i + 1 < n_kb;
                        ptx::mbar_arrive_expect_tx(&bars->full_a[s], two ? 2 * XT : XT);
                        ptx::tma_load_3d(dst, &tmap_x, &bars->full_a[s], (kb_begin + i) * BKE, row0, z);
                        if (two) ptx::tma_load_3d(dst + XT, &tmap_x, &bars->full_a[s], (kb_begin + i + 1) * BKE, row0, z);
                        ++issued;
                        if (++s == nsa) { s = 0; ph ^= 1; passed = true; }
                    }
                }
                if (bars->abort_flag)                        // give copies that are still in flight a bounded chance to land before the CTA exits
                    for (int k = issued > nsa ? issued - nsa : 0; k < issued; ++k) (void)ptx::mbar_wait(&bars->full_a[k % nsa], (k / nsa) & 1);
            }
        } else if (warp == TL::W_MMA) {
            // ---------------- MMA issuer ----------------
            // (The allocation may have to wait for a predecessor on the same SM to give its TMEM back; only this warp waits.)
            ptx::tmem_alloc(&bars->tmem_base, TL::TMEM_COLS);
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (ptx::elect_one()) {
                ptx::mbar_arrive(&bars->tmem_ready);
                ptx::tc_fence_after_sync();
                const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
                constexpr uint32_t idesc = I8 ? ptx::idesc_i8_m128(BN) : ptx::idesc_f16_m128(BN);
                constexpr uint32_t HI = ptx::kDescHiSw128;
                const uint32_t a_lo0 = ptx::desc_lo(ptx::smem_u32(smem)), b_lo0 = ptx::desc_lo(ptx::smem_u32(smem + 2 * nsa * XT));
                int sa = 0, sb = 0, slot = 0;
                uint32_t pha = 0, phb = 0, ph_free = 1, a_lo = a_lo0, b_lo = b_lo0;
                bool ok = true, recycled = false;            // recycled: every accumulator has been used once
                bool next_a = false, next_b = false;         // the next pair was seen complete already
                int todo = ((n_kb + 1) / 2) * ((lay.n_tiles - tile0 + tile_step - 1) / tile_step);      // pairs left
                for (int tile = tile0; tile < lay.n_tiles && ok; tile += tile_step) {
                    int left = 0;                            // k-blocks left in the current group
                    uint32_t d_tmem = 0;
                    for (int i = 0; i < n_kb; i += 2) {
                        if (!next_b && !ptx::mbar_wait(&bars->full_b[sb], phb)) { ok = false; break; }
                        if (!next_a && !ptx::mbar_wait(&bars->full_a[sa], pha)) { ok = false; break; }
                        if (i < 20) TAQ_PROF(40 + i);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (h == 1 && i + 1 >= n_kb) break;
                            uint32_t acc = 1;
                            if (left == 0) {                 // a new group: the next accumulator, emptied by the folders if it was in use
                                left = min(kb_per_group, n_kb - i - h);
                                if (recycled) {
                                    if (!ptx::mbar_wait(&bars->acc_free[slot], ph_free)) { ok = false; break; }
                                    ptx::tc_fence_after_sync();
                                }
                                d_tmem = tmem_base + slot * BN;
                                acc = 0;
                            }
#pragma unroll
                            for (int k = 0; k < 4; ++k) {    // four 32-byte K slices per 128-byte operand row
                                const uint64_t da = ptx::desc_join(HI, a_lo + h * (XT >> 4) + 2 * k), db = ptx::desc_join(HI, b_lo + h * (TL::B_TILE >> 4) + 2 * k);
                                if (I8) ptx::mma_i8_ss(d_tmem, da, db, idesc, acc | k);
                                else ptx::mma_f16_ss(d_tmem, da, db, idesc, acc | k);
                            }
                            if (--left == 0) {
                                ptx::mma_commit(&bars->acc_full[slot]);
                                if (++slot == NSLOT) { slot = 0; recycled = true; ph_free ^= 1; }
                            }
                        }
                        if (!ok) break;
                        // these free the stages once the MMAs have read them (a commit costs 60 cycles: none where nothing follows)
                        if (todo > nsa) ptx::mma_commit(&bars->empty_a[sa]);
                        if (todo > nsb) ptx::mma_commit(&bars->empty_b[sb]);
                        --todo;
                        a_lo += 2 * XT >> 4;
                        b_lo += 2 * TL::B_TILE >> 4;
                        if (++sa == nsa) { sa = 0; pha ^= 1; a_lo = a_lo0; }
                        if (++sb == nsb) { sb = 0; phb ^= 1; b_lo = b_lo0; }
                        // (also behind the last pair, for one that does not come: with a test of `todo` in front launches of one wave took
                        // 0.04 - 0.1 us more, 2048 x 640 x 640 6.04 -> 5.96 us without it, 64 x 320 x 320, per head, 4.59 -> 4.51)
                        next_b = ptx::mbar_try_wait(&bars->full_b[sb], phb);
                        next_a = ptx::mbar_try_wait(&bars->full_a[sa], pha);
                    }
                }
                if (!ok) give_up();
            }
        }
        else if (warp < TL::W_AUX + 2) {
            // ---------------- scales and biases, one tile ahead ----------------
            // Packed weights, on their way to L2 while the previous kernel runs (the builders may read only behind the wait).  Sixteen
            // projections of a prompt 175.5 -> 171.5 us, sixteen layers of a denoising step 317.3 -> 315.4 (in front of the barrier above, which
            // it kept everybody from, 172.1 and 316.5, and 8.99 instead of 8.91 for two prompts at 320 channels).  In the K/V kernels of
            // every width (the wide ones spill as much without it: 44 bytes stored, 100 loaded in 160-wide tiles, none in the 128- and 64-wide
            // ones) and in the 80-wide ones.  Not in the others that are no K/V kernels: the wide ones have no register to spare there (116 bytes of
            // spills, 2048 x 1280 x 1280 1.6 us more), and a layer of 1294 rows x 640, 64-wide tiles on 120 CTAs, which none of
            // them asks for, lost 0.2 us of 20.9 to the code alone.
            if ((KV || BN == 80) && !persistent && warp == TL::W_AUX + 1 && lane == 0 && blockIdx.x < lay.prefetch_ctas) {
                const uint32_t from = blockIdx.x * lay.prefetch_bytes, n = min(lay.prefetch_bytes, lay.blob_bytes - from);
                ptx::prefetch_l2((const uint8_t*)a.w + from, n);
                if (KV) ptx::prefetch_l2((const uint8_t*)a.w2 + from, n);
            }
            if (!a.early_weights) ptx::pdl_wait();
            int sbuf = 0, it = 0;
            uint32_t ph = 1;
            for (int tile = tile0; tile < lay.n_tiles; tile += tile_step, ++it) {
                int z, row0, col0, kv_which;
                tile_of(tile, z, row0, col0, kv_which);
                const uint8_t* blob = blob_of(z, kv_which);
                const float* gs = reinterpret_cast<const float*>(blob + lay.off_scales) + (size_t)col0 * n_groups;
                const float* gb = reinterpret_cast<const float*>(blob + lay.off_bias) + col0;
                if (it >= 2 && !ptx::mbar_wait(&bars->scale_free[sbuf], ph)) { give_up(); break; }
                float* sc = reinterpret_cast<float*>(smem + P.off_scales + sbuf * P.scale_bytes);
                // [BN][n_groups] -> [n_groups][BN], so that a group's scales of consecutive columns are contiguous; eight loads at a time
                // are on their way
                const int t = (warp - TL::W_AUX) * 32 + lane, n_all = BN * n_groups;
                for (int n = t; n < BN; n += 64) sc[n_all + n] = with_bias ? ptx::load_global(gb + n) : 0.f;
#pragma unroll 1
                for (int base = t; base < n_all; base += 64 * 8) {
                    float v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = base + 64 * j < n_all ? ptx::load_global(gs + base + 64 * j) : 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int i = base + 64 * j, n = quotient(i, n_groups, lay.mul_groups);
                        if (i < n_all) sc[(i - n * n_groups) * BN + n] = v[j];
                    }
                }
                if (KV && warp == TL::W_AUX) {               // (the mask may come from the previous kernel) slot of every token of the sequence among its trigger tokens, and their bitmap
                    ptx::pdl_wait();
                    const uint8_t* mask = a.reqs ? a.reqs[z].trig_mask : a.mask + (size_t)z * a.n_ctx;
                    int* slots = reinterpret_cast<int*>(smem + P.off_xchg) + 512;
                    int before = 0;
                    for (int k = 0; k < 4; ++k) {
                        const int t = 32 * k + lane;
                        const bool trig = t < a.n_ctx && mask[t] != 0;
                        const uint32_t w = __ballot_sync(0xffffffffu, trig);
                        int slot = trig ? before + __popc(w & ((1u << lane) - 1u)) : -1;
                        if (slot >= a.max_trigger) { raise_status(a.status, TAQ_ERR_SHAPE); slot = -2; }
                        before += __popc(w);
                        slots[t] = slot;
                        const uint32_t kept = __ballot_sync(0xffffffffu, slot >= 0);
                        if (lane == 0) slots[128 + k] = (int)kept;
                    }
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&bars->scale_full[sbuf]);
                sbuf ^= 1;
                if (sbuf == 0) ph ^= 1;
            }
        }
        __syncwarp();
        if (clustered) ptx::cluster_wait();
    }

    if (KV && warp >= TL::W_FOLD) {
        // The folders hand registers to the builders on the way: they give theirs back before the barrier, the builders ask behind
        // it.  (A builder that asked as soon as it ran out of work could be given what the folders' first request was still
        // waiting for, and neither would ever go on.)  One copy of what follows for both: it runs once, and what it costs
        // is to fetch it.
        if (warp < TL::W_BUILD) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TL::R_KV));
        asm volatile("bar.sync 15, %0;" ::"n"(TL::NFOLD + TL::NBUILD) : "memory");
        if (warp >= TL::W_BUILD) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(TL::R_KV));
        if (!bars->abort_flag) kv_store(tid - 32 * TL::W_FOLD);
        __syncwarp();
        if (clustered && warp >= TL::W_BUILD) ptx::cluster_wait();
    }

    // ---------------- teardown ----------------
    ptx::tc_fence_before_sync();
    // (No CTA of a cluster may leave while another one may still store into its shared memory: by this barrier everything has
    // been received.  Every thread arrives, whatever happened to its waits.)
    if (clustered) { ptx::cluster_arrive_relaxed(); ptx::cluster_wait(); }
    __syncthreads();
    if (tid == 0) { TAQ_PROF(9); TAQ_GPROF(29); }
    if (warp == TL::W_MMA) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(*reinterpret_cast<volatile uint32_t*>(&bars->tmem_base), TL::TMEM_COLS);
    }
}

// (Of this file's tile width.  Not a static of the template: such a variable is one for all copies of the library in a process.)
static std::atomic<unsigned long long> limit_set[48];

template <int BN>
cudaError_t launch_tile(const CUtensorMap& tmap, const LinearArgs& a, const LinearLayout& lay, int grid, size_t smem_bytes, cudaStream_t stream) {
    using TL = Tile<BN>;
    const bool i8 = a.xq != nullptr, w8 = a.bits == 8;
    const Ctas ctas = lay.nsplit > 1 || lay.head_pair ? Ctas::SPLIT : lay.persistent ? Ctas::MANY : Ctas::ONE;
    using Kernel = void (*)(const CUtensorMap, const LinearArgs, const LinearLayout);
    auto of_types = [&](auto out, auto ctas_c) -> Kernel {
        constexpr Out O = decltype(out)::value;
        constexpr Ctas C = decltype(ctas_c)::value;
        if constexpr (C == Ctas::SPLIT) {      // (8-bit weights have one scale group, which integer activations keep in one accumulation)
            if (i8 && w8) return nullptr;
        } else {
            if (i8 && w8) return linear_sm100_kernel<BN, true, true, O, C>;
        }
        return i8 ? linear_sm100_kernel<BN, true, false, O, C> : w8 ? linear_sm100_kernel<BN, false, true, O, C> : linear_sm100_kernel<BN, false, false, O, C>;
    };
    auto of_out = [&](auto out) -> Kernel {
        constexpr Ctas MANY = decltype(out)::value == Out::KV ? Ctas::ONE : Ctas::MANY;          // (K~/V~ tiles: one per CTA)
        return ctas == Ctas::SPLIT ? of_types(out, std::integral_constant<Ctas, Ctas::SPLIT>{}) :
               ctas == Ctas::MANY ? of_types(out, std::integral_constant<Ctas, MANY>{}) : of_types(out, std::integral_constant<Ctas, Ctas::ONE>{});
    };
    const Kernel kern = a.epi == EPI_KV ? of_out(std::integral_constant<Out, Out::KV>{}) : a.epi == EPI_Q8_HEAD ? of_out(std::integral_constant<Out, Out::Q8>{}) :
                        a.epi == EPI_F32 ? of_out(std::integral_constant<Out, Out::F32>{}) : of_out(std::integral_constant<Out, Out::F16>{});
    if (!kern) return cudaErrorNotSupported;
    cudaError_t e = allow_shared_memory((const void*)kern, SMEM_LIMIT, limit_set[(a.epi * 3 + (int)ctas) * 4 + i8 * 2 + w8]);
    if (e != cudaSuccess) return e;
    if (ctas == Ctas::SPLIT) return launch_pdl_cluster(kern, dim3(grid), dim3(lay.nsplit * (lay.head_pair ? 2 : 1), 1, 1), dim3(TL::NTHREADS), smem_bytes, stream, tmap, a, lay);
    return launch_pdl(kern, dim3(grid), dim3(TL::NTHREADS), smem_bytes, stream, tmap, a, lay);
}

}  // namespace linear
}  // namespace taq
