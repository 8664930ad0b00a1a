// Dequant-GEMM on pairs of CTAs, for launches of many rows: y = x W^T with W^ = code * scale, as in taq_linear_sm100.cuh.
//
// Two CTAs (a cluster) compute tiles of 256 rows x BN columns with `cta_group::2` MMAs: each CTA loads 128 rows of x and expands half
// of the tile's weight rows, and one thread of the CTA of rank 0 issues for both.  The same thread of the other CTA tells it which
// stages are complete there.  CTAs walk several tiles; roles are those of taq_linear_sm100.cuh.
//
// Why pairs.  With a CTA per tile nothing single bounded a large launch (8192 x 1280 x 1280, W4: 43.3 us; without the expansion 40.5, without
// the folds 40.8, without MMAs 38.0, without loads of x 40.7), but the two weight and activation rings left room for two pairs of k-blocks of
// activations.  Half of the weight rows per CTA halve the expansion and its shared memory: three stages of both, and room for an output tile.
//
// What bounds it.  Shared-memory bandwidth while a tile lasts: a 128-wide group costs the 160-wide tile 256 cycles of incoming activations, 416
// of the MMAs' operands, 160 of expanded weights and 160 of scales at 128 bytes a cycle, 992 for 640 cycles of tensor time; 1 150 to 1 220
// are measured.  At a tile's end the folders are away for 3 200 cycles, of which the accumulators in TMEM cover three groups.
// Measured, a CTA per tile -> pairs (buffers larger than L2): W4, fp16 rows: 8192 x 640 x 640 16.7 -> 12.1 us, 2048 x 1280 x 1280 13.6 -> 12.0,
// 8192 x 1280 x 1280 44.6 -> 32.7, 32768 x 640 x 640 45.0 -> 32.8; per-head rows of 80: 8192 x 640 x 640 17.4 -> 11.9, 32768 50.6 -> 33.4, of 64: 16.9 ->
// 13.5 and 44.5 -> 35.8; W8, fp16 rows: 8192 x 640 x 640 15.3 -> 12.1.
// Taken back: weights in TMEM as the A operand, channels on its lanes (two accumulators beside them are too few: 33.9 us at 8192 x 1280 x
// 1280, 18.0 at 640 channels); a warp of its own that sends the output off (one tile per pair 0.3 us more, seven 4 % less).
#pragma once
#include "taq_linear_sm100.cuh"

namespace taq {
namespace linear {

constexpr int PAIR_STAGES = 3;             // ring depth in pairs of k-blocks, activations and weights together
// Long sums in the tensor core's accumulator lose bits.  Root mean square error of the scales of per-head rows, W8: 8192 x 640 x 640 7.0e-7 from
// sums of 640 elements, 3.7e-7 from three pairs, 2.4e-7 from two; 64 x 1280 x 1280 2.8e-7 from a K loop in quarters, 3.3e-7 and 2.2e-7.  (8.47 us
// with three pairs, 8.67 with two; 8192 x 640 x 640 11.44 and 11.53.)
constexpr int ONE_GROUP_PAIRS = 2;
constexpr int PAIR_DONE = 4;               // barriers of finished pairs of k-blocks, taken in turn: at least the accumulators in TMEM
// The stages (a CTA has half of the weight rows) and, behind them, the output tile on its way out.
template <int BN> constexpr int pair_ring_bytes() { return PAIR_STAGES * (2 * A_TILE_BYTES + Tile<BN>::B_TILE); }
template <int BN> constexpr int pair_staged_bytes() { return pair_ring_bytes<BN>() + BM * BN * 2; }

struct PairBars {
    uint64_t full[PAIR_STAGES], done[PAIR_DONE], acc_full[MAX_SLOT], acc_free[MAX_SLOT], scale_full[2], scale_free[2], tmem_ready;
    uint32_t tmem_base;
    volatile int abort_flag;
};
constexpr int N_PAIR_BARS = PAIR_STAGES + PAIR_DONE + 2 * MAX_SLOT + 5;
static_assert(offsetof(PairBars, tmem_base) == N_PAIR_BARS * 8 && sizeof(PairBars) <= 1024, "barriers are contiguous");

template <int BN, bool W8, Out OUT>
__global__ void __launch_bounds__(Tile<BN>::NTHREADS, 1)
linear_pair_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_y, const __grid_constant__ LinearArgs a, const __grid_constant__ LinearLayout lay) {
    using TL = Tile<BN>;
    using CodeT = typename Code<false, W8>::T;
    constexpr int HC = TL::HC, NCG = TL::NCG, NSLOT = TL::NSLOT, NS = PAIR_STAGES, ND = PAIR_DONE;
    constexpr int B_TILE = TL::B_TILE / 2;                   // a CTA's half of a weight tile, one k-block
    constexpr int NCH = TL::NCH / 2;                         // 16-byte chunks per builder thread and pair of k-blocks
    static_assert(TL::BIG && TL::NB == 8 && ND >= NSLOT && ND >= NS, "wide tiles");
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* smem = smem_dyn + ((1024u - (ptx::smem_u32(smem_dyn) & 1023u)) & 1023u);   // 1024-byte aligned, still provably shared

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)(blockIdx.x & 1u);
    const int n_groups = lay.n_groups, n_kb = lay.n_kb, n_pair = (n_kb + 1) / 2;
    const Plan& P = lay.plan;
    PairBars* bars = reinterpret_cast<PairBars*>(smem + P.off_bars);
    // Pairs of k-blocks per accumulator: a scale group; of one group for the whole row ONE_GROUP_PAIRS, each folded with the same scale.
    const int group_pairs = n_groups == 1 ? min(n_pair, ONE_GROUP_PAIRS) : lay.kb_per_group / 2;
    const int n_folds = (n_pair + group_pairs - 1) / group_pairs;
    // A pair's MMAs complete one barrier for everybody: the stage's next writers and, where an accumulator is one pair, the folders.
    // (Longer ones have a barrier of their own: folders may be more than ND pairs behind.)
    const bool long_groups = group_pairs != 1;
    const int tile0 = (int)(blockIdx.x >> 1), tile_step = (int)(gridDim.x >> 1);
    const int n_all = n_pair * ((lay.n_tiles - tile0 + tile_step - 1) / tile_step);      // pairs of all tiles
    auto tile_of = [&](int t, int& z, int& row0, int& col0) {
        const int cz = quotient(t, lay.n_cols, lay.mul_cols);
        z = quotient(cz, lay.n_rows, lay.mul_rows);
        row0 = (cz - z * lay.n_rows) * (2 * BM) + rank * BM;
        col0 = (t - cz * lay.n_cols) * BN;
    };

    TAQ_PROF_INIT
    if (tid == 0) { TAQ_PROF(0); TAQ_GPROF(30); }
    if (warp == TL::W_PROD) {
        uint64_t* all = bars->full;
        constexpr int DONE = NS, ACC_FREE = NS + ND + MAX_SLOT, SCALE_FULL = ACC_FREE + MAX_SLOT, SCALE_FREE = SCALE_FULL + 2;
        for (int i = lane; i < N_PAIR_BARS; i += 32) {
            // (a full stage: the builders' warps that have the pair, the producer, and at rank 0 the other CTA's stage)
            const int count = i < DONE ? TL::NB / 2 + 1 + (rank == 0) : i < ACC_FREE ? 1 : i < SCALE_FULL ? 2 * TL::NF : i < SCALE_FREE ? 2 : i < SCALE_FREE + 2 ? TL::NF : 1;
            ptx::mbar_init(all + i, (uint32_t)count);
        }
        ptx::mbar_fence_init();
        __syncwarp();
        if (lane == 0) bars->abort_flag = 0;
    } else if (warp == TL::W_AUX && lane == 0) {
        ptx::tma_prefetch_desc(&tmap_x);
        ptx::tma_prefetch_desc(&tmap_y);
    }
    auto start = [&](bool wait) {
        if (wait) asm volatile("bar.sync 14, %0;" ::"n"(TL::NTHREADS) : "memory");
        else asm volatile("bar.arrive 14, %0;" ::"n"(TL::NTHREADS) : "memory");
        ptx::cluster_arrive_relaxed();                       // waited for right before the first operation on the other CTA
    };
    auto blob_of = [&](int z) { return (const uint8_t*)(a.reqs ? (a.which == 0 ? a.reqs[z].Wq : a.reqs[z].Wout) : a.w); };
    auto give_up = [&]() { raise_status(a.status, TAQ_ERR_TIMEOUT); bars->abort_flag = 1; };

    if (warp >= TL::W_FOLD && warp < TL::W_BUILD) {
        // ---------------- folders ----------------
        start(true);
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(TL::R_FOLD));
        const int ft = tid - 32 * TL::W_FOLD;
        const int q = warp & 3;                              // TMEM lane quarter this warp may read
        const int cg = (warp - TL::W_FOLD) >> 2;             // column group
        const int r = q * 32 + lane;
        const int cb = cg * HC;                              // first owned column inside the tile
        int slot = 0, done = 0, sbuf = 0;
        uint32_t ph_acc = 0, ph_done = 0, ph_scale = 0;
        bool alive = true;                                   // no wait has run out (a warp skips work then, never a barrier)
        uint32_t tmem_base = 0;
        if (ptx::mbar_wait(&bars->tmem_ready, 0)) tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base); else give_up();
        ptx::pdl_wait();                                     // orders the stores below
        __syncwarp();
        ptx::cluster_wait();
        const uint32_t acc_free = ptx::map_to_cta(ptx::smem_u32(bars->acc_free), 0);     // (the folders of both CTAs tell the thread that issues)
        unsigned char* staging = smem + pair_ring_bytes<BN>() + q * (32 * BN * 2);       // the quarter's rows
        const bool storer = cg == 0 && lane == 0;            // sends the quarter's rows off
        for (int tile = tile0; tile < lay.n_tiles; tile += tile_step) {
            int z, row0, col0;
            tile_of(tile, z, row0, col0);
            const float* scales = reinterpret_cast<const float*>(smem + P.off_scales + sbuf * P.scale_bytes) + cb;
            const float* bias = scales + n_groups * BN;
            unsigned long long y2[HC / 2];
            bool ok = alive && ptx::mbar_wait(&bars->scale_full[sbuf], ph_scale);
#pragma unroll
            for (int c = 0; c < HC; c += 4) {                // the sums start from the bias (zero where there is none)
                const ulonglong2 b4 = OUT == Out::F16 ? *reinterpret_cast<const ulonglong2*>(bias + c) : make_ulonglong2(0, 0);
                y2[c / 2] = b4.x; y2[c / 2 + 1] = b4.y;
            }
            // y += scale[g] * accumulator g (this thread's HC columns of its row)
            for (int g = 0; g < n_folds && ok; ++g) {
                ok = long_groups ? ptx::mbar_wait(&bars->acc_full[slot], ph_acc) : ptx::mbar_wait(&bars->done[done], ph_done);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + slot * BN + cb;
                const float* sg = scales + (n_groups == 1 ? 0 : g * BN);
                // (sixteen columns at a time, the next on their way while these are multiplied and added)
                uint32_t v[2][2][8];
                ptx::tmem_ld8(taddr, v[0][0]); ptx::tmem_ld8(taddr + 8, v[0][1]);
#pragma unroll
                for (int c0 = 0; c0 < HC; c0 += 16) {
                    const int k = (c0 / 16) & 1;
                    ptx::tmem_ld_wait(v[k][0]);
                    ptx::reg_fence8(v[k][1]);
                    if (c0 + 16 < HC) {
                        ptx::tmem_ld8(taddr + c0 + 16, v[k ^ 1][0]);
                        if (c0 + 24 < HC) ptx::tmem_ld8(taddr + c0 + 24, v[k ^ 1][1]);
                    } else {                                 // the accumulator is in registers: the tensor core may have it back
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive_cluster(acc_free + 8 * slot);
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (c0 + 8 * i >= HC) break;
                        const ulonglong2 s0 = *reinterpret_cast<const ulonglong2*>(sg + c0 + 8 * i), s1 = *reinterpret_cast<const ulonglong2*>(sg + c0 + 8 * i + 4);
                        uint32_t (&w)[8] = v[k][i];
                        unsigned long long* yy = y2 + (c0 + 8 * i) / 2;
                        ffma2(yy[0], w[0], w[1], s0.x); ffma2(yy[1], w[2], w[3], s0.y);
                        ffma2(yy[2], w[4], w[5], s1.x); ffma2(yy[3], w[6], w[7], s1.y);
                    }
                }
                if (++slot == NSLOT) { slot = 0; ph_acc ^= 1; }
                if (++done == ND) { done = 0; ph_done ^= 1; }
            }
            if (!ok && alive) { give_up(); alive = false; }
            if (ft == 0) TAQ_PROF(7);
            if (lane == 0) ptx::mbar_arrive(&bars->scale_free[sbuf]);            // scales and biases of this tile have been read

            float y[HC];
#pragma unroll
            for (int c = 0; c < HC / 2; ++c) asm("mov.b64 {%0, %1}, %2;" : "=f"(y[2 * c]), "=f"(y[2 * c + 1]) : "l"(y2[c]));

            // The quarter's 32 rows leave by TMA through shared memory: nobody waits until memory has taken them (stored by the threads themselves
            // they kept the folders 3 800 cycles per tile).  The storing thread makes sure that the tile before has been read.
            if (storer) ptx::bulk_store_wait_read();
            if constexpr (OUT == Out::F16) {
                asm volatile("bar.sync %0, %1;" ::"r"(2 + q), "n"(NCG * 32) : "memory");
#pragma unroll
                for (int c = 0; c < HC; c += 8) {            // boxes of 32 columns, rows of 64 bytes
                    const int cc = (cb + c) >> 3;
                    *reinterpret_cast<uint4*>(staging + (cc >> 2) * 2048 + ptx::sw64_offset(lane, cc & 3)) = pack8(*reinterpret_cast<const float (*)[8]>(y + c));
                }
            } else {
                // Q~ = Q_a(Q), Eq. 2 third line: per-(row, head) symmetric int8.  A thread's columns are one head or a half or a quarter of one.
                constexpr bool D64 = HC == 32;
                const int d = D64 ? 64 : lay.d;
                const int colg = col0 + cb;
                const int h0 = D64 ? colg / 64 : quotient(colg, d, lay.mul_d);
                float am = 0.f;
#pragma unroll
                for (int c = 0; c < HC; ++c) am = fmaxf(am, fabsf(y[c]));
                float* xc = reinterpret_cast<float*>(smem + P.off_xchg);                 // [NCG][128]
                xc[cg * 128 + r] = am;
                asm volatile("bar.sync %0, %1;" ::"r"(2 + q), "n"(NCG * 32) : "memory");
                if (d > HC) {                                // the row's threads with columns of the same head combine their absmax
                    const int per_head = D64 ? 2 : lay.per_head, first = cg & ~(per_head - 1);
#pragma unroll
                    for (int k = 0; k < NCG; ++k) if (k < per_head) am = fmaxf(am, xc[(first + k) * 128 + r]);
                }
                const float s = quant_scale(am, 127.f), rs = s > 0.f ? __frcp_rn(s) : 0.f;
#pragma unroll
                for (int c = 0; c < HC; c += 8) {
                    const int b = cb + c;                    // 160 columns: rows of 160 bytes; 128: swizzled
                    *reinterpret_cast<uint2*>(staging + (BN == 128 ? ptx::sw128_offset(lane, b >> 4) + (b & 8) : lane * BN + b)) = quant8(y + c, rs);
                }
                const long long row = (long long)row0 + r;
                if (alive && row < a.rows && colg == h0 * d) a.scales[((size_t)z * a.rows + row) * a.heads + h0] = s;      // (holds the head's first column)
            }
            ptx::fence_proxy_async_smem();
            asm volatile("bar.sync %0, %1;" ::"r"(6 + q), "n"(NCG * 32) : "memory");
            if (storer && alive && (long long)row0 + q * 32 < a.rows) {
                if constexpr (OUT == Out::F16) {
#pragma unroll
                    for (int i = 0; i < BN / 32; ++i) ptx::tma_store_3d(&tmap_y, staging + i * 2048, col0 + 32 * i, row0 + q * 32, z);
                } else {
                    ptx::tma_store_3d(&tmap_y, staging, col0, row0 + q * 32, z);
                }
                ptx::bulk_store_commit();
            }
            sbuf ^= 1;
            if (sbuf == 0) ph_scale ^= 1;
        }
        if (storer) ptx::bulk_store_wait();
        __syncwarp();
    } else if (warp >= TL::W_BUILD) {
        // ---------------- builders ----------------
        // The two halves of the builders take the pairs of k-blocks in turn.  16 chunks per weight row; sixteen consecutive lanes take one row,
        // so that a warp's loads are two runs of 64 (128) consecutive bytes and its stores of a tile row hit all banks.
        const int bt = (tid - 32 * TL::W_BUILD) & (TL::NBUILD / 2 - 1), group = (warp - TL::W_BUILD) / (TL::NB / 2);
        unsigned char* b_ring = smem + 2 * NS * A_TILE_BYTES;
        constexpr int CB = (int)sizeof(CodeT);
        const int c16 = bt & 15, n0 = bt >> 4;
        const uint32_t row_step = (uint32_t)(TL::NBUILD / 32) * lay.row_bytes;
        CodeT pw[NCH];
        const uint8_t* src = nullptr;                        // codes of the fetched pair
        int tile = tile0, pair = group;                      // the fetched pair
        auto fetch = [&](bool new_tile) {
            while (pair >= n_pair) { pair -= n_pair; tile += tile_step; new_tile = true; }
            if (tile >= lay.n_tiles) return;
            if (new_tile) {
                int z, row0, col0;
                tile_of(tile, z, row0, col0);
                src = blob_of(z) + 128 + (size_t)(col0 + rank * (BN / 2) + n0) * lay.row_bytes + (size_t)(2 * pair) * (8 * CB) + c16 * CB;
            }
            const bool have = 2 * pair + (c16 >> 3) < n_kb;
#pragma unroll
            for (int j = 0; j < NCH; ++j) pw[j] = have ? ptx::load_global(reinterpret_cast<const CodeT*>(src + (uint32_t)j * row_step)) : zero_codes<false, W8>();
        };
        if (a.early_weights) fetch(true);
        start(true);
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TL::R_BUILD));
        if (!a.early_weights) { ptx::pdl_wait(); fetch(true); }
        int sb = group;
        bool ok = true;
        for (int n = group; tile < lay.n_tiles; n += 2, sb += 2) {                       // n: the pair's number in the CTA's walk
            if (sb >= NS) sb -= NS;
            if (n >= NS && !ptx::mbar_wait(&bars->done[(n - NS) % ND], ((n - NS) / ND) & 1)) { ok = false; break; }
            unsigned char* tile_b = b_ring + (2 * sb + (c16 >> 3)) * B_TILE;
#pragma unroll
            for (int j = 0; j < NCH; ++j) *reinterpret_cast<uint4*>(tile_b + ptx::sw128_offset(n0 + j * (TL::NBUILD / 32), c16 & 7)) = expand_chunk<false, W8>(pw[j]);
            if (bt == 0 && pair < 10) TAQ_PROF(60 + 2 * pair);
            ptx::fence_proxy_async_smem();                   // make the generic-proxy writes visible to the tensor core
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars->full[sb]);
            pair += 2; src += 32 * CB;
            fetch(false);
        }
        if (!ok) give_up();
        __syncwarp();
        ptx::cluster_wait();
    } else {
        start(warp != TL::W_PROD);
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TL::R_REST));
        if (warp == TL::W_PROD) {
            // ---------------- producer: activation tiles ----------------
            if (lane == 0) {
                ptx::pdl_wait();                             // the activations may come from the previous kernel
                ptx::pdl_trigger();
                TAQ_PROF(1); TAQ_GPROF(28);
                int s = 0, issued = 0;
                bool ok = true;
                for (int tile = tile0; tile < lay.n_tiles && ok; tile += tile_step) {
                    int z, row0, col0;
                    tile_of(tile, z, row0, col0);
                    for (int i = 0; i < n_kb; i += 2) {
                        const int before = issued - NS;      // the stage's previous pair
                        if (before >= 0 && !ptx::mbar_wait(&bars->done[before % ND], (before / ND) & 1)) { give_up(); ok = false; break; }
                        unsigned char* dst = smem + 2 * s * A_TILE_BYTES;
                        const bool two = i + 1 < n_kb;
                        ptx::mbar_arrive_expect_tx(&bars->full[s], two ? 2 * A_TILE_BYTES : A_TILE_BYTES);
                        ptx::tma_load_3d(dst, &tmap_x, &bars->full[s], i * BK, row0, z);
                        if (two) ptx::tma_load_3d(dst + A_TILE_BYTES, &tmap_x, &bars->full[s], (i + 1) * BK, row0, z);
                        ++issued;
                        if (++s == NS) s = 0;
                    }
                }
                if (bars->abort_flag)                        // give copies that are still in flight a bounded chance to land before the CTA exits
                    for (int k = issued > NS ? issued - NS : 0; k < issued; ++k) (void)ptx::mbar_wait(&bars->full[k % NS], (k / NS) & 1);
            }
            __syncwarp();
            ptx::cluster_wait();
        } else if (warp == TL::W_MMA) {
            // ---------------- MMA issuer (rank 0); rank 1: tells rank 0 which stages are complete here ----------------
            ptx::tmem_alloc_pair(&bars->tmem_base, TL::TMEM_COLS);
            ptx::tc_fence_before_sync();
            __syncwarp();
            ptx::cluster_wait();                             // the other CTA's barriers exist
            if (ptx::elect_one()) {
                ptx::mbar_arrive(&bars->tmem_ready);
                ptx::tc_fence_after_sync();
                const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
                constexpr uint32_t idesc = ptx::idesc_f16_m256(BN);
                constexpr uint32_t HI = ptx::kDescHiSw128;
                const uint32_t a_lo = ptx::desc_lo(ptx::smem_u32(smem)), b_lo = ptx::desc_lo(ptx::smem_u32(smem + 2 * NS * A_TILE_BYTES));
                const uint32_t peer_full = ptx::map_to_cta(ptx::smem_u32(bars->full), 0);
                const int odd_pair = n_kb & 1 ? n_pair - 1 : n_pair;                     // the tile's pair that is one k-block
                int slot = 0, left = 0, j = 0;               // left: pairs left in the current group; j: pair of the tile
                uint32_t ph = 0, ph_free = 1, d_tmem = 0;
                bool ok = true, recycled = false;            // recycled: every accumulator has been used once
                for (int pair = 0; pair < n_all && ok; pair += NS, ph ^= 1) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) {           // (one copy per stage: addresses are constants)
                        if (pair + s >= n_all) break;
                        uint32_t acc = 1;
                        if (left == 0) {                     // a new group: the next accumulator, emptied by the folders if it was in use
                            left = min(group_pairs, n_pair - j);
                            if (rank == 0 && recycled && !ptx::mbar_wait(&bars->acc_free[slot], ph_free)) { ok = false; break; }
                            d_tmem = tmem_base + slot * BN;
                            acc = 0;
                        }
                        if (!ptx::mbar_wait(&bars->full[s], ph)) { ok = false; break; }
                        if (s == 0 && j < 20) TAQ_PROF(40 + j);
                        const bool last = --left == 0;
                        if (rank == 0) {
                            ptx::tc_fence_after_sync();
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if (h == 1 && j == odd_pair) break;
#pragma unroll
                                for (int k = 0; k < 4; ++k)  // four 32-byte K slices per 128-byte operand row
                                    ptx::mma_f16_ss_pair(d_tmem, ptx::desc_join(HI, a_lo + ((2 * s + h) * A_TILE_BYTES >> 4) + 2 * k),
                                                         ptx::desc_join(HI, b_lo + ((2 * s + h) * B_TILE >> 4) + 2 * k), idesc, acc | h | k);
                            }
                            // (what nobody waits for any more must not arrive: the other CTA may have left)
                            if (!long_groups || pair + s + NS < n_all) ptx::mma_commit_pair(&bars->done[(pair + s) % ND]);
                            if (long_groups && last) ptx::mma_commit_pair(&bars->acc_full[slot]);
                        } else {
                            ptx::mbar_arrive_cluster(peer_full + 8 * s);
                        }
                        if (last && ++slot == NSLOT) { slot = 0; recycled = true; ph_free ^= 1; }
                        if (++j == n_pair) j = 0;
                    }
                }
                // The last arrivals on acc_free, half of them the other CTA's, are seen here, too: nothing may arrive in a CTA that has left.  (Release
                // instead of relaxed in the barrier below would do, and wait for the stores of every thread: 0.2 to 0.6 us a launch.)
                if (rank == 0)
                    for (int s = 0; s < NSLOT && ok; ++s)
                        if (s < slot || recycled) ok = ptx::mbar_wait(&bars->acc_free[s], s < slot ? ph_free ^ 1 : ph_free);
                if (!ok) give_up();
            }
            __syncwarp();
        } else {
            // ---------------- scales and biases, one tile ahead ----------------
            if (!a.early_weights) ptx::pdl_wait();
            int sbuf = 0, it = 0;
            uint32_t ph = 1;
            for (int tile = tile0; tile < lay.n_tiles; tile += tile_step, ++it) {
                int z, row0, col0;
                tile_of(tile, z, row0, col0);
                const uint8_t* blob = blob_of(z);
                const float* gs = reinterpret_cast<const float*>(blob + lay.off_scales) + (size_t)col0 * n_groups;
                const float* gb = reinterpret_cast<const float*>(blob + lay.off_bias) + col0;
                if (it >= 2 && !ptx::mbar_wait(&bars->scale_free[sbuf], ph)) { give_up(); break; }
                float* sc = reinterpret_cast<float*>(smem + P.off_scales + sbuf * P.scale_bytes);
                // [BN][n_groups] -> [n_groups][BN], so that a group's scales of consecutive columns are contiguous
                const int t = (warp - TL::W_AUX) * 32 + lane, n_all_scales = BN * n_groups;
                if (OUT == Out::F16)
                    for (int n = t; n < BN; n += 64) sc[n_all_scales + n] = ptx::load_global(gb + n);
#pragma unroll 1
                for (int base = t; base < n_all_scales; base += 64 * 8) {
                    float v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = base + 64 * j < n_all_scales ? ptx::load_global(gs + base + 64 * j) : 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int i = base + 64 * j, n = quotient(i, n_groups, lay.mul_groups);
                        if (i < n_all_scales) sc[(i - n * n_groups) * BN + n] = v[j];
                    }
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&bars->scale_full[sbuf]);
                sbuf ^= 1;
                if (sbuf == 0) ph ^= 1;
            }
            __syncwarp();
            ptx::cluster_wait();
        }
    }

    // ---------------- teardown ----------------
    ptx::tc_fence_before_sync();
    // (Neither CTA may leave, or free its TMEM, while the other may still read or write its shared memory.  Every thread arrives, whatever
    // happened to its waits.)
    ptx::cluster_arrive_relaxed();
    ptx::cluster_wait();
    if (tid == 0) { TAQ_PROF(9); TAQ_GPROF(29); }
    if (warp == TL::W_MMA) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(*reinterpret_cast<volatile uint32_t*>(&bars->tmem_base), TL::TMEM_COLS);
    }
}

static std::atomic<unsigned long long> pair_limit_set[4];

template <int BN>
cudaError_t launch_pair(const CUtensorMap& tmap, const LinearArgs& a, const LinearLayout& lay, const CUtensorMap& tmap_y, int grid, size_t smem_bytes, cudaStream_t stream) {
    const bool w8 = a.bits == 8, q8 = a.epi == EPI_Q8_HEAD;
    const auto kern = q8 ? (w8 ? linear_pair_kernel<BN, true, Out::Q8> : linear_pair_kernel<BN, false, Out::Q8>)
                         : (w8 ? linear_pair_kernel<BN, true, Out::F16> : linear_pair_kernel<BN, false, Out::F16>);
    cudaError_t e = allow_shared_memory((const void*)kern, SMEM_LIMIT, pair_limit_set[q8 * 2 + w8]);
    if (e != cudaSuccess) return e;
    return launch_pdl_cluster(kern, dim3(grid), dim3(2, 1, 1), dim3(Tile<BN>::NTHREADS), smem_bytes, stream, tmap, tmap_y, a, lay);
}

}  // namespace linear
}  // namespace taq
