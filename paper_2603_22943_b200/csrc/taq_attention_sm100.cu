// Fused TAQ attention on the Blackwell tensor cores (tcgen05 + TMEM): Q~ in, O out, nothing else touches HBM.
//   S = Q~ K~^T             tcgen05.mma; the fp16 operands hold the int8 codes exactly (trigger rows: fp16 values)
//   A = softmax(S * scale)  one thread per query row; the row's 80 scores live in its registers (TMEM lane)
//   A^ (Eq. 3)              ordinary columns -> uint8 code, trigger columns -> fp16, both in units of 1/255
//   O = A^ V~               tcgen05.mma with the probabilities as the A operand and V~^T (fp16) as B; O = acc/255
// A CTA owns 128 query rows of one sequence and walks over a group of heads, software-pipelined:
//   warps 0-7  two threads per query row (TMEM lane), one per half of the keys: stage the row's Q~ codes of the next
//              head as an fp16 operand tile, softmax + Eq. 3 of the current head (the two threads of a row exchange
//              their partial maximum and sum once per head), epilogue of the previous head;
//   warp 8     one thread issues the MMAs: S of head h+1 is in flight while the rows are in the softmax of head h;
//   warp 9     one thread fetches each head's K~/V~ operand image (written once per prompt by the K/V projection)
//              by bulk copies, one head ahead: the whole image into the second buffer (head widths up to 64), or,
//              with a single buffer, K~ as soon as this head's S is complete and V~^T as soon as its PV is (heads of 80 with
//              int8 Q~: K~ into a second buffer, V~^T by a thread of warp 10).
// Head widths up to 64: two CTAs share an SM, and the row threads read Q~ and write O themselves.  Head widths 80 and
// 160: one CTA per SM; Q~ tiles arrive and O tiles leave by TMA, and from the second head on warps of their own do that work:
//   warps 12-15  expand the next head's codes (fp16 Q~: load it straight into the operand tile);
//   warps 16-19  bring the previous head's O from TMEM to global memory.
// (With the row warps doing everything in turn a head of 160 channels took 5 700 cycles: softmax 1 650, codes 1 100, O 2 250,
// probabilities 600.)
#include "taq_prof.cuh"
#include "taq_ptx.cuh"
#include "taq_sm100.cuh"
#include "taq_sm100_parts.cuh"
#include <algorithm>
#include <cstddef>
#include <cstring>

namespace taq {

TAQ_PROF_DEFINE(attention)

namespace {

using namespace parts;

constexpr int ROWS = 128;
constexpr int MISC_BYTES = 4608;     // barriers and small tables
constexpr int ROW_WARPS = 8;         // two threads per query row
constexpr int MMA_WARP = 8, COPY_WARP = 9, V_WARP = 10;
// Three warpgroups: two of row warps, and one of the MMA and copy warps with two idle ones, which gives registers to the rows where
// two CTAs share an SM (384 threads launched with 80 each = 128 x (2 x 104 + 32); with 96 for everybody the softmax spilled).
constexpr int R_ROWS = 104, R_REST = 32;
// Wide heads: five warpgroups, 640 threads launched with 96 registers each >= 128 x (2 x 128 + 40 + 72 + 104).
constexpr int Q_WARP = 12, O_WARP = 16;
constexpr int R_WIDE_ROWS = 128, R_WIDE_REST = 40, R_WIDE_Q = 72, R_WIDE_O = 104;
static_assert(2 * R_WIDE_ROWS + R_WIDE_REST + R_WIDE_Q + R_WIDE_O <= 5 * 96, "register split");

// Heads of 80 channels with int8 Q~ (K2) have two K~ buffers, so that a head's K~ is there long before its S may start: with one it
// was asked for when the S before it was complete, and S came 400 - 800 cycles after the rows were ready for it (16 x 1024 rows, 8 heads of
// 80, inputs in L2: 17.4 -> 16.1 us, 3 x 1872 8.65 -> 8.22).  The last 16 channels of their Q~ and the last 16 keys of everybody's P are tiles
// of 32-byte rows of their own instead of half-empty 128-byte ones.
// At 160 channels a K~ asked for that early is in the way of the V~^T that is needed first (30 and 40 KB at some 20 bytes a cycle): one
// buffer, and K~ behind V~^T in the order of one thread, takes 21.6 us for 16 x 1024 rows, 8 heads of 160, 12.5 for 2 x 4096 and 10.6 for 3 x
// 1872, two buffers 22.9, 13.3 and 10.95.  (64 x 256 rows, where two row tiles and no more share an image, 24.4 and 24.2.)
template <int D, bool Q8>
struct Cfg {
    static constexpr int DP = (D + 15) / 16 * 16;            // head width padded to the MMA K / N granule
    static constexpr int KBQ = (DP + 63) / 64;               // 64-wide k-blocks of the Q~ and K~ tiles
    static constexpr int A_BLOCK = ROWS * 128;
    static constexpr int K_BLOCK = TP * 128;
    static constexpr int VT_BLOCK = DP * 128;
    static constexpr int K_BYTES = KBQ * K_BLOCK;
    static constexpr int VT_BYTES = 2 * VT_BLOCK;
    static constexpr int HEAD_BYTES = K_BYTES + VT_BYTES + kOperandConstBytes;
    static constexpr int KVBUF = D <= 64 ? 2 : 1;            // K~/V~ images in flight
    static constexpr int OBUF = D == 64 ? 1 : 2;             // O accumulators in TMEM
    static constexpr bool K2 = D == 80 && Q8;
    static constexpr int QFULL = K2 ? DP / 64 : KBQ, QTAIL = K2 ? DP % 64 : 0;     // 64-wide blocks of the Q~ tile, channels of its narrow one (16)
    static constexpr int OFF_KV = 0;                         // images; wide heads: K~ (twice if K2), V~^T
    static constexpr int OFF_V = OFF_KV + (K2 ? 2 : 1) * K_BYTES;
    static constexpr int OFF_Q = D <= 64 ? OFF_KV + KVBUF * HEAD_BYTES : OFF_V + VT_BYTES;
    static constexpr int OFF_P = OFF_Q + QFULL * A_BLOCK + ROWS * QTAIL * 2;
    static constexpr int P_BYTES = D >= 80 ? A_BLOCK + ROWS * 32 : 2 * A_BLOCK;
    // One image buffer (wide heads): the next head's K~ loads as soon as this head's S is complete and its V~^T as soon
    // as this head's PV is, each with a barrier of its own; the constants of a head then live in a rotating slot of their
    // own (three slots: the softmax of head h - 1 may still read its slot when the constants of head h + 1 arrive; with two K~
    // buffers they arrive a head earlier, hence four).
    static constexpr bool SPLIT_KV = KVBUF == 1;
    static constexpr int CST_SLOT = 384, CST_SLOTS = K2 ? 4 : 3;
    static constexpr int OFF_CST = OFF_P + P_BYTES;
    // Wide heads move Q~ and O by TMA (a row's codes or outputs of one head are 80 to 320
    // bytes at a stride of the whole channel width: per-thread global accesses of that shape keep the load/store
    // unit busy for longer than the arithmetic takes): O through one staging buffer, int8 codes through a second one, fp16 Q~
    // straight into the operand tile.
    static constexpr bool TMA_IO = D >= 80;
    static constexpr int THREADS = TMA_IO ? 640 : 384;
    static constexpr int OFF_U = OFF_CST + (SPLIT_KV ? CST_SLOTS * CST_SLOT : 0);
    static constexpr int UO_BYTES = ROWS * D * 2;                  // an O tile
    static constexpr int U_BYTES = TMA_IO ? UO_BYTES + ROWS * D : 0; // + a raw int8 Q~ tile
    static constexpr int OFF_MISC = OFF_U + U_BYTES;
    static constexpr int TOTAL = OFF_MISC + MISC_BYTES + 1024;   // misc block + slack for 1024-byte alignment
    static constexpr uint32_t TMEM_S = 0, TMEM_O = 2 * TP;
    static constexpr uint32_t TMEM_COLS = (2 * TP + OBUF * DP) <= 256 ? 256 : 512;
    static constexpr int CTAS_PER_SM = (2 * (TOTAL + 1024) <= 232448 && TMEM_COLS == 256) ? 2 : 1;
    static_assert(HEAD_BYTES % 1024 == 0 && K_BYTES % 1024 == 0 && VT_BLOCK % 1024 == 0, "operand tiles must keep 1024-byte alignment");
    static_assert(TOTAL <= 232448 && OFF_MISC % 16 == 0, "shared memory budget");
    static_assert(QTAIL == 0 || QTAIL == 16, "narrow tile of Q~: 32-byte rows");
    static_assert(OFF_Q % 1024 == 0 && OFF_P % 1024 == 0 && OFF_U % 128 == 0, "tile alignment");
    // 16-byte chunk cc ^ flip (8 channels; flip 0 or 2) of a row of the Q~ tile; chunk of a row of P (8 keys)
    static __device__ __forceinline__ uint32_t q_offset(int row, int cc, int flip = 0) {
        if (QTAIL == 0 || cc < 8 * QFULL) return (cc >> 3) * A_BLOCK + (ptx::sw128_offset(row, cc & 7) ^ (flip << 4));
        return QFULL * A_BLOCK + ptx::sw32_offset(row, cc - 8 * QFULL);
    }
    static __device__ __forceinline__ uint32_t p_offset(int row, int chunk) {
        if (D < 80) return (chunk >> 3) * A_BLOCK + ptx::sw128_offset(row, chunk & 7);
        return chunk < 8 ? ptx::sw128_offset(row, chunk) : A_BLOCK + ptx::sw32_offset(row, chunk - 8);
    }
};

struct Misc {
    uint64_t kv_full[2], kv_free[2], q_full, s_full[2], p_full, o_full[2], drain, qraw_full, o_free[2], u_free, k_odd;
    uint32_t tmem_base;
    volatile int abort_flag;
    float2 xchg[2][2][ROWS];     // [head parity][half][row]: (max, sum) of a thread's half of the softmax
    alignas(16) float pad[TP];   // 0, or -inf for the keys at and beyond T
};
constexpr int N_BARS = (int)(offsetof(Misc, tmem_base) / 8);
static_assert(sizeof(Misc) <= MISC_BYTES && N_BARS <= 32 && offsetof(Misc, pad) % 16 == 0 && offsetof(Misc, xchg) % 8 == 0, "misc block");
static_assert(sizeof(OperandConsts) % 16 == 0 && sizeof(OperandConsts) <= 384, "constants slot");

// What the softmax takes for a row's scale: its sign is with the codes (SignOf), and beside the smallest number above 0 any logit is 0.
__device__ __forceinline__ float size_of(float scale) { return scale == 0.f ? __int_as_float(1) : fabsf(scale); }

// Half of the query codes (or fp16 values) of one row and head, held in registers between the global load and
// the store into the operand tile: the row's two threads take the lower and the upper half of the 16-byte chunks.
template <int D, bool Q8>
struct QRegs {
    static constexpr int CH2 = (Cfg<D, Q8>::DP / 8 + 1) / 2;      // chunks (8 channels) per thread
    uint4 v[Q8 ? (CH2 + 1) / 2 : CH2];
    // (Heads of 64: 32 bytes at a time where the address allows.  A load or store of a row per lane keeps the load/store unit for 64 cycles whatever
    // its width, and 8 bytes of codes in and 16 bytes of O out at a time paced these launches: 8192 rows x 10 heads 15.7 -> 13.3 us.  Heads of 40: 24 and 16 codes
    // in as few pieces as the address allows.)
    __device__ __forceinline__ void load(const void* q, size_t elem_off, bool valid, int half) {
        const int c0 = half * CH2;
        if constexpr (D == 64) {
            constexpr int N = Q8 ? 1 : 2;                    // pieces of 32 bytes
            const uint8_t* src = (const uint8_t*)q + (elem_off + c0 * 8) * (Q8 ? 1 : 2);
            const bool wide = (reinterpret_cast<uintptr_t>(q) & 31u) == 0;       // (rows and heads are multiples of 32 bytes)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                v[2 * i] = v[2 * i + 1] = make_uint4(0, 0, 0, 0);
                if (valid && wide) ptx::load_32b(src + 32 * i, v[2 * i], v[2 * i + 1]);
                else if (valid) { v[2 * i] = *reinterpret_cast<const uint4*>(src + 32 * i); v[2 * i + 1] = *reinterpret_cast<const uint4*>(src + 32 * i + 16); }
            }
        } else if constexpr (D == 40 && Q8) {
            const uint8_t* src = (const uint8_t*)q + elem_off + c0 * 8;
            v[0] = v[1] = make_uint4(0, 0, 0, 0);
            if (valid) {
                const bool wide = (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
                if (wide) v[0] = *reinterpret_cast<const uint4*>(src);
                else { const uint2 w = *reinterpret_cast<const uint2*>(src); v[0].x = w.x; v[0].y = w.y; }
                if (half == 0) {
                    if (wide) { const uint2 w = *reinterpret_cast<const uint2*>(src + 16); v[1].x = w.x; v[1].y = w.y; }
                    else { const uint4 w = *reinterpret_cast<const uint4*>(src + 8); v[0].z = w.x; v[0].w = w.y; v[1].x = w.z; v[1].y = w.w; }
                } else if (!wide) { const uint2 w = *reinterpret_cast<const uint2*>(src + 8); v[0].z = w.x; v[0].w = w.y; }
            }
        } else if (Q8) {
#pragma unroll
            for (int i = 0; i < (CH2 + 1) / 2; ++i) {
                uint2 lo = make_uint2(0, 0), hi = make_uint2(0, 0);
                if (valid && (c0 + 2 * i) * 8 < D) lo = *reinterpret_cast<const uint2*>((const int8_t*)q + elem_off + (c0 + 2 * i) * 8);
                if (valid && 2 * i + 1 < CH2 && (c0 + 2 * i + 1) * 8 < D) hi = *reinterpret_cast<const uint2*>((const int8_t*)q + elem_off + (c0 + 2 * i + 1) * 8);
                v[i] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
        } else {
#pragma unroll
            for (int i = 0; i < CH2; ++i) {
                v[i] = make_uint4(0, 0, 0, 0);
                if (valid && (c0 + i) * 8 < D) v[i] = *reinterpret_cast<const uint4*>((const __half*)q + elem_off + (c0 + i) * 8);
            }
        }
    }
    // local chunk i (8 channels) as fp16 operands; channels beyond D are zero (a zero int8 code maps to fp16 zero)
    __device__ __forceinline__ uint4 chunk(int i, const SignOf& sign) const {
        if (Q8) {
            const uint4 w = v[i / 2];
            return codes_w8_to_half((i & 1) ? make_uint2(w.z, w.w) : make_uint2(w.x, w.y), sign);
        }
        return v[i];
    }
};

template <int D, bool Q8, bool TAIL_ONLY>
__global__ void __launch_bounds__(Cfg<D, Q8>::THREADS, Cfg<D, Q8>::CTAS_PER_SM) attention_sm100_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_o, const AttnArgs a) {
    using C = Cfg<D, Q8>;
    constexpr int DP = C::DP;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* smem = smem_dyn + ((1024u - (ptx::smem_u32(smem_dyn) & 1023u)) & 1023u);   // 1024-byte aligned, still provably shared
    Misc* misc = reinterpret_cast<Misc*>(smem + C::OFF_MISC);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = a.n_ctx, H = a.heads, Cch = a.channels;
    const int zb = blockIdx.z;
    const int b = a.reqs ? 0 : zb;
    const int row0 = blockIdx.x * ROWS;
    const int h_begin = H * (int)blockIdx.y / (int)gridDim.y;         // the heads dealt out as evenly as they go
    const int HG = H * ((int)blockIdx.y + 1) / (int)gridDim.y - h_begin;

    TAQ_PROF_INIT
    if (tid == 0) { TAQ_PROF(0); TAQ_GPROF(126); }
    if (tid < TP) misc->pad[tid] = tid < T ? 0.f : -INFINITY;
    if (warp == COPY_WARP) {                          // one lane per barrier
        uint64_t* all = misc->kv_full;
        // one arrival per row warp; q_full of an fp16 tile that TMA loads: one; o_free: one per warp of the O warps
        const uint64_t* bar = all + lane;
        const int count = bar == &misc->p_full ? ROW_WARPS : bar == &misc->q_full ? (C::TMA_IO && !Q8 ? 1 : ROW_WARPS) : bar == &misc->o_free[0] || bar == &misc->o_free[1] ? 4 : 1;
        if (lane < N_BARS) ptx::mbar_init(all + lane, (uint32_t)count);
        if (lane == 0) misc->abort_flag = 0;
        ptx::mbar_fence_init();
        if (C::TMA_IO && lane == 0) { ptx::tma_prefetch_desc(&tmap_q); ptx::tma_prefetch_desc(&tmap_o); }
    }
    if (warp == MMA_WARP) ptx::tmem_alloc(&misc->tmem_base, C::TMEM_COLS);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = misc->tmem_base;
    ptx::pdl_trigger();

    const taq_kv_layout KL = kv_layout(H, T, D, a.max_trigger);

    // Raw tiles of even and odd heads complete barriers of their own: who waits for the second head only must not take the phase
    // before the first one for it.  (Wide heads have one image buffer, the second kv_free is theirs to use.)
    auto qraw_full = [&](int hi) { return hi & 1 ? &misc->kv_free[1] : &misc->qraw_full; };
    auto k_full = [&](int hi) { return C::K2 && (hi & 1) ? &misc->k_odd : &misc->kv_full[0]; };      // (K~ of wide heads)
    auto k_parity = [&](int hi) { return (uint32_t)(C::K2 ? hi >> 1 : hi) & 1u; };

    constexpr bool REG_SPLIT = C::CTAS_PER_SM == 2;
    if (C::TMA_IO && warp >= Q_WARP) {
        if constexpr (C::TMA_IO) {
        if (warp < O_WARP) {
            // ---------------- Q~ of the second head and on ----------------
            asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_WIDE_Q));
            bool alive = true;
            if constexpr (Q8) {
                // A thread is a row: sixteen codes per load, and every place in the operand tile is a constant beside the row's.  Rows of 80
                // bytes are free of bank conflicts; of rows of 160 bytes four start 32 bytes apart and the next four at the same
                // banks, so these take their chunks in pairs the other way round (`swap`: 16 x 1024 rows, 8 heads of 160, 21.5 -> 21.3 us, 64
                // x 256 24.4 -> 24.1).  They are read before S of the head before is complete (its operand
                // tile is free then), and the raw tile of the head after next lands under all that.  (With the chunks dealt out in
                // linear order, row and place worked out for each, S of a head of 160 channels was 2 500 cycles later.)
                constexpr int N = D / 16;
                const unsigned char* UQ = smem + C::OFF_U + C::UO_BYTES;
                const int t = tid - 32 * Q_WARP, swap = D == 160 ? (t >> 2) & 1 : 0;
                static_assert(D != 160 || (N % 2 == 0 && C::QTAIL == 0), "pairs of chunks");
                ptx::pdl_wait();                                         // (scales; one thread loads Q~ of the third head and on, too)
                const float* scales = a.q_scales + ((size_t)zb * a.n_query + min(row0 + t, a.n_query - 1)) * H + h_begin;
                float scale = HG > 1 ? scales[1] : 0.f;
                for (int hi = 1; hi < HG; ++hi) {
                    alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(qraw_full(hi), (hi >> 1) & 1));
                    uint4 raw[N];
#pragma unroll
                    for (int i = 0; i < N; ++i) raw[i] = *reinterpret_cast<const uint4*>(UQ + t * D + (i ^ swap) * 16);
                    ptx::fence_proxy_async_smem();                           // (generic reads before the TMA load that overwrites them)
                    asm volatile("bar.sync 6, 128;" ::: "memory");           // the raw tile has been read
                    if (t == 0 && alive && hi + 1 < HG) {
                        ptx::mbar_arrive_expect_tx(qraw_full(hi + 1), (uint32_t)(ROWS * D));
                        ptx::tma_load_3d(smem + C::OFF_U + C::UO_BYTES, &tmap_q, qraw_full(hi + 1), (h_begin + hi + 1) * D, row0, zb);
                    }
                    __syncwarp();
                    SignOf sign(scale);
                    alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(&misc->s_full[(hi - 1) & 1], ((hi - 1) >> 1) & 1));
                    if (alive) {
#pragma unroll
                        for (int i = 0; i < N; ++i) {
                            *reinterpret_cast<uint4*>(smem + C::OFF_Q + C::q_offset(t, 2 * i, 2 * swap)) = codes_w8_to_half(make_uint2(raw[i].x, raw[i].y), sign);
                            *reinterpret_cast<uint4*>(smem + C::OFF_Q + C::q_offset(t, 2 * i + 1, 2 * swap)) = codes_w8_to_half(make_uint2(raw[i].z, raw[i].w), sign);
                        }
                        ptx::fence_proxy_async_smem();
                    }
                    __syncwarp();
                    if (alive && lane < ROW_WARPS / 4) ptx::mbar_arrive(&misc->q_full);      // (two lanes of each of four warps: as many as row warps)
                    if (hi + 1 < HG) scale = scales[hi + 1];
                }
            } else if (warp == Q_WARP && lane == 0) {
                // (channels behind the head's last in its last 64-wide block are never multiplied)
                ptx::pdl_wait();
                for (int hi = 0; hi < HG && alive; ++hi) {
                    if (hi > 0) alive = ptx::mbar_wait(&misc->s_full[(hi - 1) & 1], ((hi - 1) >> 1) & 1);
                    if (!alive) break;
                    ptx::mbar_arrive_expect_tx(&misc->q_full, (uint32_t)(C::KBQ * C::A_BLOCK));
                    for (int kb = 0; kb < C::KBQ; ++kb) ptx::tma_load_3d(smem + C::OFF_Q + kb * C::A_BLOCK, &tmap_q, &misc->q_full, (h_begin + hi) * D + kb * 64, row0, zb);
                }
            }
            if (!alive) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
        } else {
            // ---------------- O of all heads but the last ----------------
            asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R_WIDE_O));
            unsigned char* U = smem + C::OFF_U;
            const int q4 = warp & 3, r = q4 * 32 + lane, t = tid - 32 * O_WARP;
            const float inv255 = 1.0f / (a.p_log ? 256.0f : a.p_bits == 4 ? 15.0f : 255.0f);
            bool alive = true;
            ptx::pdl_wait();
            for (int hi = 0; hi + 1 < HG; ++hi) {
                alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(&misc->o_full[hi & 1], (hi >> 1) & 1));
                if (t == 0) ptx::bulk_store_wait_read();     // (the tile of the head before)
                __syncwarp();
                asm volatile("bar.sync 7, 128;" ::: "memory");
                if (alive) {
                    ptx::tc_fence_after_sync();
                    const uint32_t t_o = tmem_base + C::TMEM_O + (hi & 1) * DP + ((uint32_t)(q4 * 32) << 16);
                    // (a loop of 40 instructions: beside the softmax the instructions of all roles do not fit the cache near the schedulers,
                    // and unrolled, 400 of them a head, this took 100 - 200 cycles from every softmax)
#pragma unroll 1
                    for (int c0 = 0; c0 < D; c0 += 16) {
                        uint32_t v[2][8];
                        ptx::tmem_ld8(t_o + c0, v[0]);
                        ptx::tmem_ld8(t_o + c0 + 8, v[1]);
                        ptx::tmem_ld_wait(v[0]);
                        ptx::reg_fence8(v[1]);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            uint32_t pk[4];
#pragma unroll
                            for (int e2 = 0; e2 < 4; ++e2) {
                                __half2 hv = __floats2half2_rn(__uint_as_float(v[i][2 * e2]) * inv255, __uint_as_float(v[i][2 * e2 + 1]) * inv255);
                                pk[e2] = *reinterpret_cast<uint32_t*>(&hv);
                            }
                            *reinterpret_cast<uint4*>(U + ((size_t)r * D + c0 + i * 8) * 2) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                    }
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&misc->o_free[hi & 1]);
                    ptx::fence_proxy_async_smem();
                }
                asm volatile("bar.sync 7, 128;" ::: "memory");
                if (t == 0 && alive) {
                    ptx::tma_store_3d(&tmap_o, U, (h_begin + hi) * D, row0, zb);
                    ptx::bulk_store_commit();
                }
            }
            if (t == 0) {
                ptx::bulk_store_wait_read();
                ptx::mbar_arrive(&misc->u_free);
                ptx::bulk_store_wait();                      // (a successor that waits for this kernel reads O as soon as it may)
            }
            if (!alive) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
        }
        }
    } else if (warp >= MMA_WARP) {
    if constexpr (C::TMA_IO) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_WIDE_REST));
    if constexpr (REG_SPLIT) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_REST));
    if (warp == COPY_WARP) {
        // ---------------- K~/V~ operand images, one head ahead ----------------
        if (lane == 0) {
            if (!a.early_kv) ptx::pdl_wait();             // in general the images may come from the previous kernel
            const uint8_t* blk = a.reqs ? (const uint8_t*)a.reqs[zb].kv : (const uint8_t*)a.kv + (size_t)b * KL.block_bytes;
            const uint8_t* img = blk + KL.off_operands + (size_t)h_begin * KL.operand_head_bytes;
            int issued = 0;
            if (C::K2) {
                for (int hi = 0; hi < HG; ++hi) {            // a buffer is free when the S before last is complete
                    if (hi >= 2 && !ptx::mbar_wait(&misc->s_full[hi & 1], ((hi - 2) >> 1) & 1)) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
                    if (misc->abort_flag) break;
                    const uint8_t* src = img + (size_t)hi * KL.operand_head_bytes;
                    ptx::mbar_arrive_expect_tx(k_full(hi), C::K_BYTES + (uint32_t)sizeof(OperandConsts));
                    ptx::bulk_load(smem + C::OFF_KV + (hi & 1) * C::K_BYTES, src, C::K_BYTES, k_full(hi));
                    ptx::bulk_load(smem + C::OFF_CST + (hi % C::CST_SLOTS) * C::CST_SLOT, src + C::K_BYTES + C::VT_BYTES, (uint32_t)sizeof(OperandConsts), k_full(hi));
                    issued = hi + 1;
                }
                if (misc->abort_flag)     // let copies that were issued land before the CTA goes away
                    for (int hi = issued > 2 ? issued - 2 : 0; hi < issued; ++hi) (void)ptx::mbar_wait(k_full(hi), k_parity(hi));
            } else
            if (C::SPLIT_KV) {
                // kv_full[0]: K~ and the constants of a head; kv_full[1]: its V~^T
                int issued_v = 0;
                for (int hi = 0; hi < HG; ++hi) {
                    if (hi >= 1 && !ptx::mbar_wait(&misc->s_full[(hi - 1) & 1], ((hi - 1) >> 1) & 1)) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
                    if (misc->abort_flag) break;
                    const uint8_t* src = img + (size_t)hi * KL.operand_head_bytes;
                    ptx::mbar_arrive_expect_tx(&misc->kv_full[0], C::K_BYTES + (uint32_t)sizeof(OperandConsts));
                    ptx::bulk_load(smem + C::OFF_KV, src, C::K_BYTES, &misc->kv_full[0]);
                    ptx::bulk_load(smem + C::OFF_CST + (hi % C::CST_SLOTS) * C::CST_SLOT, src + C::K_BYTES + C::VT_BYTES, (uint32_t)sizeof(OperandConsts), &misc->kv_full[0]);
                    issued = hi + 1;
                    if (hi >= 1 && !ptx::mbar_wait(&misc->kv_free[0], (hi - 1) & 1)) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
                    if (misc->abort_flag) break;
                    ptx::mbar_arrive_expect_tx(&misc->kv_full[1], C::VT_BYTES);
                    ptx::bulk_load(smem + C::OFF_V, src + C::K_BYTES, C::VT_BYTES, &misc->kv_full[1]);
                    issued_v = hi + 1;
                }
                if (misc->abort_flag) {   // let copies that were issued land before the CTA goes away
                    if (issued) (void)ptx::mbar_wait(&misc->kv_full[0], (issued - 1) & 1);
                    if (issued_v) (void)ptx::mbar_wait(&misc->kv_full[1], (issued_v - 1) & 1);
                }
            } else {
            for (int hi = 0; hi < HG; ++hi) {
                const int buf = hi % C::KVBUF;
                if (hi >= C::KVBUF && !ptx::mbar_wait(&misc->kv_free[buf], ((hi / C::KVBUF) - 1) & 1)) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
                if (misc->abort_flag) break;
                ptx::mbar_arrive_expect_tx(&misc->kv_full[buf], C::HEAD_BYTES);
                ptx::bulk_load(smem + C::OFF_KV + buf * C::HEAD_BYTES, img + (size_t)hi * KL.operand_head_bytes, C::HEAD_BYTES, &misc->kv_full[buf]);
                issued = hi + 1;
            }
            if (misc->abort_flag) {   // let copies that were issued land before the CTA goes away
                for (int hi = issued > C::KVBUF ? issued - C::KVBUF : 0; hi < issued; ++hi) (void)ptx::mbar_wait(&misc->kv_full[hi % C::KVBUF], (hi / C::KVBUF) & 1);
            }
            }
        }
    } else if (C::K2 && warp == V_WARP) {
        // ---------------- V~^T of heads with two K~ buffers: as soon as the PV before it is complete ----------------
        if (lane == 0) {
            if (!a.early_kv) ptx::pdl_wait();
            const uint8_t* blk = a.reqs ? (const uint8_t*)a.reqs[zb].kv : (const uint8_t*)a.kv + (size_t)b * KL.block_bytes;
            const uint8_t* img = blk + KL.off_operands + (size_t)h_begin * KL.operand_head_bytes + C::K_BYTES;
            int issued = 0;
            for (int hi = 0; hi < HG; ++hi) {
                if (hi >= 1 && !ptx::mbar_wait(&misc->kv_free[0], (hi - 1) & 1)) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
                if (misc->abort_flag) break;
                ptx::mbar_arrive_expect_tx(&misc->kv_full[1], C::VT_BYTES);
                ptx::bulk_load(smem + C::OFF_V, img + (size_t)hi * KL.operand_head_bytes, C::VT_BYTES, &misc->kv_full[1]);
                issued = hi + 1;
            }
            if (misc->abort_flag && issued) (void)ptx::mbar_wait(&misc->kv_full[1], (issued - 1) & 1);
        }
    } else if (warp == MMA_WARP) {
        // ---------------- MMA issuer ----------------
        // One elected thread walks it alone (a wait on a complete barrier costs it 60 cycles; a vote of the whole warp and a poll
        // of the abort flag made it 190).
        if (ptx::elect_one()) {
        auto wait = [&](uint64_t* bar, uint32_t parity) -> bool { return ptx::mbar_wait(bar, parity); };
        constexpr uint32_t HI = ptx::kDescHiSw128;
        const uint32_t q_lo0 = ptx::desc_lo(ptx::smem_u32(smem + C::OFF_Q)), p_lo0 = ptx::desc_lo(ptx::smem_u32(smem + C::OFF_P));
        const uint32_t kv_lo0 = ptx::desc_lo(ptx::smem_u32(smem + C::OFF_KV));
        auto issue_s = [&](int hi) -> bool {
            const int buf = hi % C::KVBUF;
            if (C::SPLIT_KV ? !wait(k_full(hi), k_parity(hi)) : !wait(&misc->kv_full[buf], (hi / C::KVBUF) & 1)) return false;
            if (!wait(&misc->q_full, hi & 1)) return false;
            ptx::tc_fence_after_sync();
            {
                if (hi < 8) TAQ_PROF(80 + hi);
                const uint32_t k_lo = kv_lo0 + (C::SPLIT_KV ? (C::K2 ? (hi & 1) * (C::K_BYTES >> 4) : 0) : buf * (C::HEAD_BYTES >> 4));
#pragma unroll
                for (int ks = 0; ks < DP / 16; ++ks) {
                    const uint64_t qd = ks < 4 * C::QFULL ? ptx::desc_join(HI, q_lo0 + (ks / 4) * (C::A_BLOCK >> 4) + (ks % 4) * 2)
                                                          : ptx::desc_join(ptx::kDescHiSw32, q_lo0 + C::QFULL * (C::A_BLOCK >> 4) + (ks - 4 * C::QFULL) * 2);
                    ptx::mma_f16_ss(tmem_base + C::TMEM_S + (hi & 1) * TP, qd, ptx::desc_join(HI, k_lo + (ks / 4) * (C::K_BLOCK >> 4) + (ks % 4) * 2), ptx::idesc_f16_m128(TP), ks != 0);
                }
                ptx::mma_commit(&misc->s_full[hi & 1]);
            }
            return true;
        };
        auto issue_pv = [&](int hi) -> bool {
            const int buf = hi % C::KVBUF;
            if (C::SPLIT_KV && !wait(&misc->kv_full[1], hi & 1)) return false;
            if (!wait(&misc->p_full, hi & 1)) return false;
            if (C::TMA_IO && hi >= 2 && !wait(&misc->o_free[hi & 1], ((hi >> 1) - 1) & 1)) return false;     // (the O warps have read the head before last)
            ptx::tc_fence_after_sync();
            {
                if (hi < 8) TAQ_PROF(96 + hi);
                const uint32_t vt_lo = C::SPLIT_KV ? kv_lo0 + ((C::OFF_V - C::OFF_KV) >> 4) : kv_lo0 + ((buf * C::HEAD_BYTES + C::K_BYTES) >> 4);
#pragma unroll
                for (int ks = 0; ks < TP / 16; ++ks) {
                    const uint64_t pd = C::TMA_IO && ks >= 4 ? ptx::desc_join(ptx::kDescHiSw32, p_lo0 + (C::A_BLOCK >> 4)) : ptx::desc_join(HI, p_lo0 + (ks / 4) * (C::A_BLOCK >> 4) + (ks % 4) * 2);
                    ptx::mma_f16_ss(tmem_base + C::TMEM_O + (hi % C::OBUF) * DP, pd, ptx::desc_join(HI, vt_lo + (ks / 4) * (C::VT_BLOCK >> 4) + (ks % 4) * 2), ptx::idesc_f16_m128(DP), ks != 0);
                }
                ptx::mma_commit(&misc->o_full[hi % C::OBUF]);
                ptx::mma_commit(&misc->kv_free[buf]);
            }
            return true;
        };
        bool ok = issue_s(0);
        for (int hi = 0; hi < HG && ok; ++hi) {
            if (C::KVBUF == 2 || C::K2) { // S of the next head first: it runs under this head's softmax
                if (hi + 1 < HG) ok = issue_s(hi + 1);
                if (ok) ok = issue_pv(hi);
            } else {
                // one image buffer: the next head's K~ arrives some time after this head's S; its S goes as soon as K~ and Q~
                // are there (it then runs under this head's softmax), at the latest after this head's PV.  Nothing to look out for once it
                // is under way, nor behind the last head (while this loop waited for the probabilities there, too, a CTA of one
                // head took 0.1 us longer).
                bool s_next = hi + 1 >= HG;
                for (const long long t0 = clock64(); ok && !s_next;) {
                    if (ptx::mbar_try_wait(&misc->kv_full[0], (hi + 1) & 1) && ptx::mbar_try_wait(&misc->q_full, (hi + 1) & 1)) ok = s_next = issue_s(hi + 1);
                    if (ptx::mbar_try_wait(&misc->p_full, hi & 1)) break;
                    if (clock64() - t0 > ptx::kWaitCycles) ok = false;
                }
                if (ok) ok = issue_pv(hi);
                if (ok && !s_next) ok = issue_s(hi + 1);
            }
        }
        if (!ok) {                        // wait (bounded) for whatever was issued before TMEM is given back
            raise_status(a.status, TAQ_ERR_TIMEOUT);
            misc->abort_flag = 1;
            ptx::mma_commit(&misc->drain);
            (void)ptx::mbar_wait(&misc->drain, 0);
        }
        }
        __syncwarp();
    }
    } else {
        if constexpr (C::TMA_IO) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R_WIDE_ROWS));
        if constexpr (REG_SPLIT) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R_ROWS));
        // ---------------- row threads: two per query row (TMEM lane), each with half of the keys ----------------
        const int q4 = warp & 3, half = warp >> 2;
        const int r = q4 * 32 + lane;
        const int n = row0 + r;
        const bool valid = n < a.n_query;
        const size_t grow = (size_t)zb * a.n_query + (valid ? n : 0);
        const uint32_t lane_addr = (uint32_t)(q4 * 32) << 16;
        const int key0 = half * HK;
        const float cmax = a.p_bits == 4 ? 15.0f : 255.0f;     // last code
        const float pmax = a.p_log ? 256.0f : cmax;            // probabilities are held in units of 1 / pmax (linear codes: 1 / last code)
        const float inv255 = 1.0f / pmax;
        auto p_place = [&](int chunk) { return smem + C::OFF_P + C::p_offset(r, chunk); };
        constexpr int CH2 = QRegs<D, Q8>::CH2;
        constexpr int OC = DP / 2;                       // O columns per thread
        bool alive = true;
        ptx::pdl_wait();                                 // Q~ comes from the previous kernel in the stream
        if (tid == 0) TAQ_PROF(1);

        if constexpr (C::TMA_IO) {
            // ---- the first head's Q~ in and the last head's O out; the heads between are others' work ----
            // Every warp walks every barrier of the loop, whatever happened to its waits: a warp whose wait ran out
            // skips the work, never a barrier.
            unsigned char* U = smem + C::OFF_U;
            auto all256 = [&]() { asm volatile("bar.sync 5, 256;" ::: "memory"); };
            // raw tile of the first head -> fp16 operand tile: half a row per thread
            auto stage_q_u = [&](float scale) {
                constexpr int N = D / 16, N2 = (N + 1) / 2;  // sixteen codes at a time
                unsigned char* UQ = U + C::UO_BYTES;
                auto load_q = [&](int hi) {                  // one thread: raw Q~ tile of head hi (rows beyond n_query read as zero)
                    ptx::mbar_arrive_expect_tx(qraw_full(hi), (uint32_t)(ROWS * D));
                    ptx::tma_load_3d(UQ, &tmap_q, qraw_full(hi), (h_begin + hi) * D, row0, zb);
                };
                if (tid == 0) load_q(0);
                alive = __all_sync(0xffffffffu, ptx::mbar_wait(qraw_full(0), 0));
                if (alive) {
                    const SignOf sign(scale);
#pragma unroll
                    for (int i = 0; i < N2; ++i) {
                        if (half * N2 + i < N) {
                            const uint4 raw = *reinterpret_cast<const uint4*>(UQ + r * D + (half * N2 + i) * 16);
                            *reinterpret_cast<uint4*>(smem + C::OFF_Q + C::q_offset(r, 2 * (half * N2 + i))) = codes_w8_to_half(make_uint2(raw.x, raw.y), sign);
                            *reinterpret_cast<uint4*>(smem + C::OFF_Q + C::q_offset(r, 2 * (half * N2 + i) + 1)) = codes_w8_to_half(make_uint2(raw.z, raw.w), sign);
                        }
                    }
                    ptx::fence_proxy_async_smem();
                }
                __syncwarp();
                if (alive && lane == 0) ptx::mbar_arrive(&misc->q_full);
                all256();                                    // the raw tile has been read by everybody
                if (tid == 0 && HG > 1 && alive) load_q(1);
            };
            // this thread's half of O of head hi: acc / 255 -> fp16 into U (the dense [128][D] tile)
            auto stage_o_u = [&](int hi) {
                const uint32_t t_o = tmem_base + C::TMEM_O + (hi % C::OBUF) * DP + half * OC + lane_addr;
                uint32_t v[OC / 8][8];
#pragma unroll
                for (int i = 0; i < OC / 8; ++i) ptx::tmem_ld8(t_o + i * 8, v[i]);
                ptx::tmem_ld_wait(v[0]);
#pragma unroll
                for (int i = 1; i < OC / 8; ++i) ptx::reg_fence8(v[i]);
#pragma unroll
                for (int i = 0; i < OC / 8; ++i) {
                    if (half * OC + i * 8 < D) {
                        uint32_t pk[4];
#pragma unroll
                        for (int e2 = 0; e2 < 4; ++e2) {
                            __half2 hv = __floats2half2_rn(__uint_as_float(v[i][2 * e2]) * inv255, __uint_as_float(v[i][2 * e2 + 1]) * inv255);
                            pk[e2] = *reinterpret_cast<uint32_t*>(&hv);
                        }
                        *reinterpret_cast<uint4*>(U + ((size_t)r * D + half * OC + i * 8) * 2) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                }
                ptx::tc_fence_before_sync();
                ptx::fence_proxy_async_smem();
            };
            auto send_o = [&](int hi) {          // one thread, after the barrier that follows stage_o_u
                ptx::tma_store_3d(&tmap_o, U, (h_begin + hi) * D, row0, zb);
                ptx::bulk_store_commit();
            };

            float sq = 1.0f, sq_next = 1.0f;
            if (Q8) {
                sq = valid ? a.q_scales[grow * H + h_begin] : 0.f;
                stage_q_u(sq);
            }

            for (int hi = 0; hi < HG; ++hi) {
                const uint32_t ph = hi & 1;
                const bool more = hi + 1 < HG;
                if (Q8 && more) sq_next = valid ? a.q_scales[grow * H + h_begin + hi + 1] : 0.f;
                alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(&misc->s_full[ph], (hi >> 1) & 1));
                if (tid == 0 && hi < 8) TAQ_PROF(16 + hi);
                float e[HK];
                float k255 = 0.f;
                unsigned long long trig = 0;
                if (alive) {
                    ptx::tc_fence_after_sync();
                    uint32_t u[HK];
                    {
                        const uint32_t t_s = tmem_base + C::TMEM_S + ph * TP + key0 + lane_addr;
                        uint32_t (&u8)[HK / 8][8] = *reinterpret_cast<uint32_t (*)[HK / 8][8]>(&u);
#pragma unroll
                        for (int i = 0; i < HK / 8; ++i) ptx::tmem_ld8(t_s + i * 8, u8[i]);
                        ptx::tmem_ld_wait(u8[0]);
#pragma unroll
                        for (int i = 1; i < HK / 8; ++i) ptx::reg_fence8(u8[i]);
                    }
                    ptx::tc_fence_before_sync();
                    const OperandConsts* cst = reinterpret_cast<const OperandConsts*>(smem + C::OFF_CST + (hi % C::CST_SLOTS) * C::CST_SLOT);
                    float m_loc, l_loc;
                    softmax_half<TAIL_ONLY>(u, cst->logit_factor + key0, misc->pad + key0, size_of(sq), e, m_loc, l_loc);
                    trig = half == 0 ? ((unsigned long long)cst->trig_bits[0] | ((unsigned long long)(cst->trig_bits[1] & 0xFFu) << 32))
                                     : ((unsigned long long)(cst->trig_bits[1] >> 8) | ((unsigned long long)cst->trig_bits[2] << 24));
                    misc->xchg[ph][half][r] = make_float2(m_loc, l_loc);
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + q4) : "memory");
                    const float2 other = misc->xchg[ph][half ^ 1][r];
                    const float m_all = fmaxf(m_loc, other.x);
                    const float c_self = ex2_approx(m_loc - m_all), c_other = ex2_approx(other.x - m_all);
                    k255 = __fdividef(pmax * c_self, fmaf(l_loc, c_self, other.y * c_other));
                } else {
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + q4) : "memory");
                }
                if (tid == 0 && hi < 8) TAQ_PROF(32 + hi);
                // the P tile is free once the previous head's PV has completed
                if (hi > 0) {
                    alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(&misc->o_full[(hi - 1) & 1], ((hi - 1) >> 1) & 1));
                    ptx::tc_fence_after_sync();
                }
                if (tid == 0 && hi < 8) TAQ_PROF(48 + hi);
                if (alive) {
                    if (a.p_log) write_p_half_log(e, k255, cmax, trig, half * (HK / 8), p_place);
                    else write_p_half(e, k255, trig, half * (HK / 8), p_place);
                    ptx::fence_proxy_async_smem();
                    ptx::tc_fence_before_sync();
                }
                __syncwarp();
                if (alive && lane == 0) ptx::mbar_arrive(&misc->p_full);
                if (tid == 0 && hi < 8) TAQ_PROF(64 + hi);
                sq = sq_next;
            }
            alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(&misc->o_full[(HG - 1) % C::OBUF], ((HG - 1) / C::OBUF) & 1));
            alive = alive && __all_sync(0xffffffffu, ptx::mbar_wait(&misc->u_free, 0));      // the store of the head before has read U
            if (alive) {
                ptx::tc_fence_after_sync();
                stage_o_u(HG - 1);
            }
            all256();
            if (tid == 0) {
                if (alive) send_o(HG - 1);
                ptx::bulk_store_wait();
            }
            if (!alive) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
        } else {
        static_assert(D == 64 || (D == 40 && OC == 24), "pieces of Q~ and O");
        auto store_o = [&](int hi) {        // this thread's half of O of head hi: acc / 255 -> fp16
            __half* orow = a.o + grow * Cch + (h_begin + hi) * D + half * OC;
            const uint32_t t_o = tmem_base + C::TMEM_O + (hi % C::OBUF) * DP + half * OC + lane_addr;
            uint32_t v[OC / 8][8];
#pragma unroll
            for (int i = 0; i < OC / 8; ++i) ptx::tmem_ld8(t_o + i * 8, v[i]);
            ptx::tmem_ld_wait(v[0]);
#pragma unroll
            for (int i = 1; i < OC / 8; ++i) ptx::reg_fence8(v[i]);
            if constexpr (D == 64) {
                const bool wide = (reinterpret_cast<uintptr_t>(a.o) & 31u) == 0;
#pragma unroll
                for (int i = 0; i < OC / 16; ++i) {
                    uint32_t pk[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        __half2 hv = __floats2half2_rn(__uint_as_float(v[2 * i + e / 4][2 * (e & 3)]) * inv255, __uint_as_float(v[2 * i + e / 4][2 * (e & 3) + 1]) * inv255);
                        pk[e] = *reinterpret_cast<uint32_t*>(&hv);
                    }
                    if (valid && wide) ptx::store_32b(orow + i * 16, pk);
                    else if (valid) {
                        *reinterpret_cast<uint4*>(orow + i * 16) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        *reinterpret_cast<uint4*>(orow + i * 16 + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                    }
                }
            } else {                                         // heads of 40: 24 or 16 channels
                uint32_t pk[12];
#pragma unroll
                for (int e = 0; e < 12; ++e) {
                    __half2 hv = __floats2half2_rn(__uint_as_float(v[e / 4][2 * (e & 3)]) * inv255, __uint_as_float(v[e / 4][2 * (e & 3) + 1]) * inv255);
                    pk[e] = *reinterpret_cast<uint32_t*>(&hv);
                }
                if (valid) {
                    const bool wide = (reinterpret_cast<uintptr_t>(orow) & 31u) == 0;
                    if (wide) ptx::store_32b(orow, pk);
                    else *reinterpret_cast<uint4*>(orow) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    if (half == 0) {
                        if (wide) *reinterpret_cast<uint4*>(orow + 16) = make_uint4(pk[8], pk[9], pk[10], pk[11]);
                        else ptx::store_32b(orow + 8, pk + 4);
                    } else if (!wide) *reinterpret_cast<uint4*>(orow + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                }
            }
            ptx::tc_fence_before_sync();
        };
        auto stage_q = [&](const QRegs<D, Q8>& qr, float scale) {
            const SignOf sign(scale);
#pragma unroll
            for (int i = 0; i < CH2; ++i) {
                const int cc = half * CH2 + i;
                if (cc < DP / 8) *reinterpret_cast<uint4*>(smem + C::OFF_Q + (cc >> 3) * C::A_BLOCK + ptx::sw128_offset(r, cc & 7)) = qr.chunk(i, sign);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&misc->q_full);
        };

        QRegs<D, Q8> qr;
        qr.load(a.q, grow * Cch + (size_t)h_begin * D, valid, half);
        float sq = 1.0f, sq_next = 1.0f;
        if (Q8) sq = valid ? a.q_scales[grow * H + h_begin] : 0.f;
        stage_q(qr, sq);

        for (int hi = 0; hi < HG; ++hi) {
            const uint32_t ph = hi & 1;
            const bool more = hi + 1 < HG;
            if (more) {                         // next head's query codes: in flight while this head's S is awaited
                qr.load(a.q, grow * Cch + (size_t)(h_begin + hi + 1) * D, valid, half);
                if (Q8) sq_next = valid ? a.q_scales[grow * H + h_begin + hi + 1] : 0.f;
            }
            alive = __all_sync(0xffffffffu, ptx::mbar_wait(&misc->s_full[ph], (hi >> 1) & 1));
            if (!alive) break;
            if (tid == 0 && hi < 8) TAQ_PROF(16 + hi);
            ptx::tc_fence_after_sync();
            uint32_t u[HK];
            {
                const uint32_t t_s = tmem_base + C::TMEM_S + ph * TP + key0 + lane_addr;
                uint32_t (&u8)[HK / 8][8] = *reinterpret_cast<uint32_t (*)[HK / 8][8]>(&u);
#pragma unroll
                for (int i = 0; i < HK / 8; ++i) ptx::tmem_ld8(t_s + i * 8, u8[i]);
                ptx::tmem_ld_wait(u8[0]);
#pragma unroll
                for (int i = 1; i < HK / 8; ++i) ptx::reg_fence8(u8[i]);
            }
            ptx::tc_fence_before_sync();

            // ---- this thread's half of the softmax; the row's two threads then exchange (max, sum) ----
            const OperandConsts* cst = reinterpret_cast<const OperandConsts*>(smem + C::OFF_KV + (hi % C::KVBUF) * C::HEAD_BYTES + C::K_BYTES + C::VT_BYTES);
            float e[HK];
            float m_loc, l_loc;
            softmax_half<TAIL_ONLY>(u, cst->logit_factor + key0, misc->pad + key0, size_of(sq), e, m_loc, l_loc);
            const unsigned long long trig = half == 0 ? ((unsigned long long)cst->trig_bits[0] | ((unsigned long long)(cst->trig_bits[1] & 0xFFu) << 32))
                                                      : ((unsigned long long)(cst->trig_bits[1] >> 8) | ((unsigned long long)cst->trig_bits[2] << 24));
            misc->xchg[ph][half][r] = make_float2(m_loc, l_loc);
            asm volatile("bar.sync %0, 64;" ::"r"(1 + q4) : "memory");
            const float2 other = misc->xchg[ph][half ^ 1][r];
            const float m_all = fmaxf(m_loc, other.x);
            const float c_self = ex2_approx(m_loc - m_all), c_other = ex2_approx(other.x - m_all);
            const float k255 = __fdividef(pmax * c_self, fmaf(l_loc, c_self, other.y * c_other));

            // S of this head is complete, so the Q~ tile is free again; the next head's codes, asked for at the top of this
            // iteration, have had the softmax to arrive
            if (more) stage_q(qr, sq_next);
            if (tid == 0 && hi < 8) TAQ_PROF(32 + hi);
            // the P tile is free once the previous head's PV has completed
            if (hi > 0) {
                alive = __all_sync(0xffffffffu, ptx::mbar_wait(&misc->o_full[(hi - 1) % C::OBUF], ((hi - 1) / C::OBUF) & 1));
                if (!alive) break;
                ptx::tc_fence_after_sync();
                if (C::OBUF == 1) store_o(hi - 1);   // one O accumulator: empty it before the next PV may start
            }
            if (tid == 0 && hi < 8) TAQ_PROF(48 + hi);
            if (a.p_log) write_p_half_log(e, k255, cmax, trig, half * (HK / 8), p_place);
            else write_p_half(e, k255, trig, half * (HK / 8), p_place);
            ptx::fence_proxy_async_smem();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&misc->p_full);
            if (tid == 0 && hi < 8) TAQ_PROF(64 + hi);

            if (hi > 0 && C::OBUF == 2) store_o(hi - 1);    // under this head's PV
            sq = sq_next;
        }
        if (alive) {
            alive = __all_sync(0xffffffffu, ptx::mbar_wait(&misc->o_full[(HG - 1) % C::OBUF], ((HG - 1) / C::OBUF) & 1));
            if (alive) {
                ptx::tc_fence_after_sync();
                store_o(HG - 1);
            }
        }
        if (!alive) { raise_status(a.status, TAQ_ERR_TIMEOUT); misc->abort_flag = 1; }
        }
    }

    if (tid == 0) TAQ_PROF(9);
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (tid == 0) TAQ_GPROF(127);
    if (warp == MMA_WARP) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, C::TMEM_COLS);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn3() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess && qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// CTAs per row tile, among which the heads are dealt out: the number with the shortest estimated time, in units of a head: a CTA's
// heads and its start and end (two heads' time; where two CTAs share an SM the second one hides most of it), times the waves.
// A partial last wave of two CTAs per SM costs less than a full one.  (Measured, 64 row tiles x 10 heads of 64: five CTAs of
// two heads each, 320 in two waves, 17.4 us; four of two or three heads, one wave, 14.9.  45 tiles x 8 heads of 80: two CTAs
// of four heads 11.5 us, three of two or three 9.4.)
template <typename C>
int pick_head_groups(const AttnArgs& a, int n_z) {
    const long long tiles = (long long)((a.n_query + ROWS - 1) / ROWS) * n_z;
    int best = 1;
    double best_cost = 1e30;
    for (int groups = 1; groups <= a.heads; ++groups) {
        const long long ctas = tiles * groups, places = 148 * C::CTAS_PER_SM, waves = (ctas + places - 1) / places;
        const int most = (a.heads + groups - 1) / groups;
        const double cost = C::CTAS_PER_SM == 2 ? (0.75 * (double)waves + 0.25 * std::max(1.0, (double)ctas / (double)places)) * (0.4 + most) : (double)waves * (2.0 + most);
        if (cost <= best_cost) { best_cost = cost; best = groups; }
    }
    return best;
}

template <int D, bool Q8, bool TAIL_ONLY>
cudaError_t launch_k(const AttnArgs& a, int n_z, cudaStream_t stream) {
    using C = Cfg<D, Q8>;
    static std::atomic<unsigned long long> limit_set;
    cudaError_t e = allow_shared_memory((const void*)attention_sm100_kernel<D, Q8, TAIL_ONLY>, C::TOTAL, limit_set);
    if (e != cudaSuccess) return e;
    dim3 grid((a.n_query + ROWS - 1) / ROWS, pick_head_groups<C>(a, n_z), n_z);
    CUtensorMap tmap_q, tmap_o;
    memset(&tmap_q, 0, sizeof(tmap_q));
    memset(&tmap_o, 0, sizeof(tmap_o));
    if (C::TMA_IO) {      // Q~ and O as [n_z][n_query][channels] in boxes of 128 rows x one head (fp16 Q~: x 64 channels, as the operand tile has them)
        EncodeTiledFn enc = encode_tiled_fn3();
        if (!enc) return cudaErrorNotSupported;
        const cuuint64_t qesz = Q8 ? 1 : 2;
        const cuuint64_t dims[3] = {(cuuint64_t)a.channels, (cuuint64_t)a.n_query, (cuuint64_t)n_z};
        const cuuint64_t qstr[2] = {(cuuint64_t)a.channels * qesz, (cuuint64_t)a.channels * qesz * (cuuint64_t)a.n_query};
        const cuuint64_t ostr[2] = {(cuuint64_t)a.channels * 2, (cuuint64_t)a.channels * 2 * (cuuint64_t)a.n_query};
        const cuuint32_t box[3] = {(cuuint32_t)D, ROWS, 1}, qbox[3] = {(cuuint32_t)(Q8 ? D : 64), ROWS, 1}, estr[3] = {1, 1, 1};
        if (enc(&tmap_q, Q8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(a.q), dims, qstr, qbox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                Q8 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return cudaErrorInvalidValue;
        if (enc(&tmap_o, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, (void*)a.o, dims, ostr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    return launch_pdl(attention_sm100_kernel<D, Q8, TAIL_ONLY>, grid, dim3(C::THREADS), (size_t)C::TOTAL, stream, tmap_q, tmap_o, a);
}

template <int D>
cudaError_t launch_d(const AttnArgs& a, int n_z, cudaStream_t stream) {
    const bool q8 = a.q_bits == 8, tail = a.n_ctx > 64;
    if (q8) return tail ? launch_k<D, true, true>(a, n_z, stream) : launch_k<D, true, false>(a, n_z, stream);
    return tail ? launch_k<D, false, true>(a, n_z, stream) : launch_k<D, false, false>(a, n_z, stream);
}

}  // namespace

bool sm100_attention_supported(const AttnArgs& a) {
    OperandGeom g;
    if (!operand_geom(a.channels / a.heads, a.n_ctx, &g)) return false;
    if (a.p_bits != 8 && a.p_bits != 4) return false;
    if (a.heads > 65535) return false;
    return true;
}

cudaError_t launch_attention_sm100(const AttnArgs& a, int n_z, cudaStream_t stream) {
    if (a.n_query == 0 || n_z == 0) return cudaSuccess;
    switch (a.channels / a.heads) {
        case 40: return launch_d<40>(a, n_z, stream);
        case 64: return launch_d<64>(a, n_z, stream);
        case 80: return launch_d<80>(a, n_z, stream);
        case 160: return launch_d<160>(a, n_z, stream);
    }
    return cudaErrorNotSupported;
}

}  // namespace taq
