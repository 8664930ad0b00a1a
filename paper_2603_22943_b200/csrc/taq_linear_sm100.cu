// Dequant-GEMM on the Blackwell tensor cores, host side: which tile, how many CTAs per tile, how shared memory is laid out.  The
// kernel is in taq_linear_sm100.cuh; every tile width is compiled in a file of its own (taq_linear_sm100_n*.cu).
#include "taq_prof.cuh"
TAQ_PROF_DEFINE(linear)
#include "taq_linear_pair_sm100.cuh"
#include <algorithm>
#include <cmath>

namespace taq {

namespace linear {
extern template cudaError_t launch_tile<64>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, int, size_t, cudaStream_t);
extern template cudaError_t launch_tile<80>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, int, size_t, cudaStream_t);
extern template cudaError_t launch_tile<128>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, int, size_t, cudaStream_t);
extern template cudaError_t launch_tile<160>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, int, size_t, cudaStream_t);
extern template cudaError_t launch_pair<128>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, const CUtensorMap&, int, size_t, cudaStream_t);
extern template cudaError_t launch_pair<160>(const CUtensorMap&, const LinearArgs&, const LinearLayout&, const CUtensorMap&, int, size_t, cudaStream_t);
}  // namespace linear

namespace {

using namespace linear;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess && qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// How a launch is laid out.
struct Choice { int bn, grid; LinearLayout lay; int total, ring, staged; bool pair; };      // grid in CTAs; staged: bytes the epilogue stages in the rings; pair: linear_pair_kernel

struct Problem {                       // what the choice depends on
    int n_groups, group_len, bke, n_kb, d, ncols_factor;
    bool i8;
    long long row_tiles;
    WeightLayout L;
};
Problem problem_of(const LinearArgs& a) {
    const WeightLayout L = weight_layout(a.n_out, a.k_in, a.bits, a.group);
    Problem p;
    p.i8 = a.xq != nullptr;
    p.bke = p.i8 ? 2 * BK : BK;
    p.n_groups = L.n_groups; p.group_len = L.group_len;
    p.n_kb = (a.k_in + p.bke - 1) / p.bke;
    p.d = a.epi == EPI_Q8_HEAD || a.epi == EPI_KV ? a.n_out / a.heads : 0;
    p.ncols_factor = a.epi == EPI_KV ? 2 : 1;
    p.row_tiles = (a.rows + BM - 1) / BM;
    p.L = L;
    return p;
}
// k-blocks of the longest share when the K loop is split
int share_of(const Problem& p, int nsplit) {
    if (nsplit == 1) return p.n_kb;
    if (p.n_groups == 1) return (p.n_kb + nsplit - 1) / nsplit;
    const int kbs = ((p.n_groups + nsplit - 1) / nsplit) * (p.group_len / p.bke);
    return kbs < p.n_kb ? kbs : p.n_kb;
}

// Ring depths of a tile width, or false when it does not fit: as many of a tile's weight blocks as shared memory holds (they are
// expanded before the activations arrive), activations two pairs of blocks deep, or three.
template <int BN>
bool rings(const LinearArgs& a, const Problem& p, int nsplit, int head_pair, bool persistent, Choice& c) {
    using TL = Tile<BN>;
    const int n_pair = (share_of(p, nsplit) + 1) / 2;
    int staged = 0;
    const int tile_bytes = a.epi == EPI_F16 ? BM * BN * 2 : a.epi == EPI_F32 ? BM * BN * 4 : a.epi == EPI_Q8_HEAD ? BM * BN : kv_tile_bytes(BN) + std::max(1, BN / p.d) * 1024;      // (K~/V~: the fp32 tile and the rows' scales)
    if (persistent) {
        // (stored from the registers)
    } else if (nsplit == 1) {
        staged = tile_bytes;
    } else {
        staged = std::max(TL::NCG * (4 - 4 / nsplit) * TL::PIECE, tile_bytes);                  // (the pieces of the other CTAs, then the output)
    }
    // (K~/V~ of fp16 contexts: the images' 80 rows and not 128: 0.1 - 0.2 us of every such launch; with int8 contexts W4 lost as much)
    const int xb = a.epi == EPI_KV && !p.i8 && a.n_ctx <= kOperandKeys ? kOperandKeys * 128 : A_TILE_BYTES;
    int nsa = n_pair < 2 ? 1 : 2, nsb = n_pair < 2 ? 1 : 2;
    while (make_plan<BN>(p.n_groups, nsa, nsb, persistent, xb).ring_bytes < staged) { if (nsa < nsb) ++nsa; else ++nsb; if (nsb > MAX_STAGE) return false; }
    auto fits = [&](int na, int nb) { return make_plan<BN>(p.n_groups, na, nb, persistent, xb).total <= SMEM_LIMIT; };
    while (nsb < (persistent ? MAX_STAGE : n_pair) && nsb < MAX_STAGE && fits(nsa, nsb + 1)) ++nsb;
    while (nsa < 3 && nsa < n_pair && fits(nsa + 1, nsb)) ++nsa;
    const Plan P = make_plan<BN>(p.n_groups, nsa, nsb, persistent, xb);
    if (P.total > SMEM_LIMIT || P.ring_bytes < staged) return false;
    c.bn = BN;
    c.lay.kv.x_bytes = (uint32_t)xb;
    c.lay.nsplit = nsplit; c.lay.nsa = nsa; c.lay.nsb = nsb; c.lay.head_pair = head_pair; c.lay.persistent = persistent;
    c.lay.plan = P;
    c.lay.n_groups = p.n_groups; c.lay.n_kb = p.n_kb; c.lay.mul_groups = multiplier(p.n_groups, (long long)BN * p.n_groups);
    c.lay.kb_per_group = p.n_groups == 1 ? p.n_kb : p.group_len / p.bke;
    c.lay.row_bytes = (uint32_t)p.L.row_bytes; c.lay.off_scales = p.L.off_scales; c.lay.off_bias = p.L.off_bias;
    if (p.d) {
        c.lay.d = p.d; c.lay.mul_d = multiplier(p.d, a.n_out);
        c.lay.per_head = std::max(1, std::min(TL::NCG, p.d / TL::HC));
    }
    if (a.epi == EPI_KV) {
        const taq_kv_layout KL = kv_layout(a.heads, a.n_ctx, p.d, a.max_trigger);
        if (KL.block_bytes >= (1ull << 31)) return false;
        auto& G = c.lay.kv;
        G.off_v_codes = (uint32_t)KL.off_v_codes; G.off_k_scales = (uint32_t)KL.off_k_scales; G.off_v_scales = (uint32_t)KL.off_v_scales;
        G.off_k_trigger = (uint32_t)KL.off_k_trigger; G.off_v_trigger = (uint32_t)KL.off_v_trigger; G.off_trig_slot = (uint32_t)KL.off_trig_slot;
        G.off_operands = (uint32_t)KL.off_operands; G.block_bytes = KL.block_bytes;
        OperandGeom g{};
        G.images = operand_geom(p.d, a.n_ctx, &g);
        G.head_bytes = (uint32_t)g.head_bytes; G.k_bytes = (uint32_t)g.k_bytes; G.vt_bytes = (uint32_t)g.vt_bytes;
        G.dp = g.dp; G.kbq = g.kbq; G.n_heads = std::max(1, BN / p.d);
        G.mul_dp = g.dp ? multiplier(g.dp, G.n_heads * g.dp) : 0;
        G.logit_unit = 1.4426950408889634f / sqrtf((float)p.d);
    }
    c.total = P.total; c.ring = P.ring_bytes; c.staged = staged;
    return true;
}
bool rings_of(const LinearArgs& a, const Problem& p, int bn, int nsplit, int head_pair, bool persistent, Choice& c) {
    switch (bn) {
        case 64: return rings<64>(a, p, nsplit, head_pair, persistent, c);
        case 80: return rings<80>(a, p, nsplit, head_pair, persistent, c);
        case 128: return rings<128>(a, p, nsplit, head_pair, persistent, c);
        case 160: return rings<160>(a, p, nsplit, head_pair, persistent, c);
    }
    return false;
}

// Pairs of CTAs (taq_linear_pair_sm100.cuh): fp16 rows in, fp16 or per-head int8 rows out, scale groups that end with a pair of k-blocks.
template <int BN>
bool pair_rings(const LinearArgs& a, const Problem& p, Choice& c) {
    if (p.i8 || (a.epi != EPI_F16 && a.epi != EPI_Q8_HEAD) || (p.n_groups > 1 && p.group_len / p.bke % 2 != 0)) return false;
    if (!rings<BN>(a, p, 1, 0, true, c)) return false;                        // (the layout's other fields)
    Plan& P = c.lay.plan;
    const int ring = pair_staged_bytes<BN>(), shift = ring - P.ring_bytes;
    P.ring_bytes = ring; P.off_scales += shift; P.off_bias += shift; P.off_xchg += shift; P.off_bars += shift; P.total += shift;
    c.lay.nsa = c.lay.nsb = PAIR_STAGES;
    c.total = P.total; c.ring = ring; c.staged = BM * BN * 2; c.pair = true;          // (behind the stages)
    return P.total <= SMEM_LIMIT;
}

constexpr int SMS = 148;                                 // of a B200

// Whether a tile of bn columns can carry the epilogue: per-head outputs want a thread's 80 or 64 columns to be whole heads, or a
// head of 160 channels on the two threads of a row.
bool tile_carries(const LinearArgs& a, const Problem& p, int bn) {
    if (a.n_out % bn) return false;
    switch (p.d) {
        case 0: return true;
        case 40: return bn == 160 || bn == 80;
        case 80: return bn == 160 || bn == 80;
        case 160: return bn == 160;                      // (80: head pairs, below)
        case 64: return bn == 128 || bn == 64;
    }
    return false;
}

// The cheapest layout by a small model, in microseconds: a fixed part (launch, barriers, first loads, epilogue), the K loop per k-block
// and scale group, what a tile costs a CTA that walks several, and the exchange of partial sums when the K loop is split (a
// part that grows with the CTAs that exchange at one time).  The numbers are a least-squares fit to 351 measured launches of
// 64 to 8192 rows, 640 and 1280 channels, W4 and W8, every width and split that can carry them (5 % rms); the layouts it picks
// are on average 0.5 % slower than the best one measured.  It decides beyond that, too.  320 channels, 32 to 8192 rows, W4 and W8,
// fp16 and per-head int8 rows: of 20 launches 17 are within 2 % of the best layout, two within 4 %, and 8192 W8 rows per head
// take 7.6 us where 80-wide tiles take 6.9.  Two terms are set by hand: 0.2 us more for four CTAs than for two, and for K~/V~ an
// epilogue that grows with the tile's width (0.008 us a column).  Of 30 projections of 1, 2 and 8 prompts, 320 to 1280 channels,
// contexts of 768 and 2048, W4 and W8, 28 are within 2 % of the best layout; the other two (1280 channels, W4, 1 and 2
// prompts) the rule on narrow contexts below keeps from it.
struct Pace { int bn; double fixed, kb, group, tile, q8, split, exchange; };
constexpr Pace PACES[4] = {
    {160, 3.08, 0.320, 0.248, 1.54, 0.72, 0.95, 1.72},
    {128, 3.17, 0.274, 0.150, 0.49, 0.05, 1.30, 1.66},
    {80, 2.49, 0.200, 0.131, 0.52, 0.35, 1.05, 1.04},
    {64, 2.56, 0.192, 0.106, 0.24, 0.18, 1.00, 0.87},
};
Choice& finish(Choice& c, const LinearArgs& a, const Problem& p, long long tiles, long long ctas) {
    c.lay.n_tiles = (int)tiles;
    c.lay.n_cols = a.n_out / c.bn * p.ncols_factor; c.lay.n_rows = (int)p.row_tiles;
    c.lay.mul_cols = multiplier(c.lay.n_cols, tiles); c.lay.mul_rows = multiplier(c.lay.n_rows, tiles);
    c.grid = (int)ctas;
    // Packed weights asked for ahead of time, a share by each of up to 16 CTAs: where all CTAs of the launch find room beside its
    // predecessor's, at most half the SMs.  Weights of requests are known behind the wait only.
    if (!a.reqs && ctas <= SMS / 2 && p.L.total < (1u << 31)) {
        const uint32_t n = (uint32_t)std::min(ctas, 16LL), bytes = (uint32_t)align_up((p.L.total + n - 1) / n, 128);
        c.lay.blob_bytes = (uint32_t)p.L.total; c.lay.prefetch_bytes = bytes;
        c.lay.prefetch_ctas = (uint32_t)((p.L.total + bytes - 1) / bytes);
    }
    return c;
}

Choice choose_single(const LinearArgs& a, int n_z, double& best_cost) {
    const Problem p = problem_of(a);
    Choice best{};
    best_cost = 1e30;
    // Heads of 160 channels in a launch of few rows: two 80-wide tiles per head whose CTAs exchange the rows' absmax, the K loop in
    // halves (with integer activations: halves of the scale groups).
    if (a.epi == EPI_Q8_HEAD && p.d == 160 && a.bits == 4 && (p.n_groups >= 2 || (!p.i8 && p.n_kb >= 2))) {
        const long long tiles = p.row_tiles * (a.n_out / 80) * (long long)n_z;
        Choice c{};
        if (tiles * 2 <= SMS && rings_of(a, p, 80, 2, 1, false, c)) { best_cost = 0; return finish(c, a, p, tiles, tiles * 2); }      // (faster than pairs, too)
    }
    // K~/V~ with heads of 160 channels: the same, the K loop whole, where the CTAs are one wave (two prompts of 77 x 768, 1280 channels: W4 13.4 ->
    // 9.5 us, W8 12.8 -> 9.1, against one 160-wide tile per head on half as many).  Wider contexts are split below, and their sums stay as short as
    // that makes them: whole, the scales' root mean square error of W8 rises from 3.4e-7 to 8.1e-7 at 1024 (12.9 -> 10.2 us) and from 3.1e-7 to
    // 1.8e-6 at 2048 (13.8 -> 13.3), and 4096 takes 21.1 us instead of 19.1.
    if (a.epi == EPI_KV && p.d == 160 && a.k_in < 1024 && !(p.i8 && a.bits == 8)) {
        const long long tiles = p.row_tiles * (a.n_out / 80) * 2 * (long long)n_z;
        Choice c{};
        if (tiles <= SMS && rings_of(a, p, 80, 1, 1, false, c)) { best_cost = 0; return finish(c, a, p, tiles, tiles); }
    }
    for (const Pace& m : PACES) {
        const int bn = m.bn;
        if (!tile_carries(a, p, bn)) continue;
        const long long tiles = p.row_tiles * (a.n_out / bn) * p.ncols_factor * (long long)n_z;
        if (tiles > (1 << 30)) continue;
        for (int ns : {1, 2, 4}) {
            // (K~/V~: the line lies between the two widths of text contexts in use.  From a 768-wide context a split gains 0 to 2 % at
            // 320 and 640 channels (one prompt, W4: 9.8 us, in halves 9.7) and at 1280 10 % with W4, nothing with W8 (14.7
            // and 13.3 us, 13.2 and 13.1); unsplit, a prompt's bits are the same in every batch.  Of a 2048-wide one four CTAs take
            // 14.6 us to 11.2 at 640 channels.)
            if (ns > 1 && a.epi == EPI_KV && a.k_in < 1024) continue;
            if (ns > 1 && ((p.i8 && p.n_groups == 1) || (p.n_groups == 1 ? p.n_kb : p.n_groups) < ns || tiles * ns > SMS)) continue;    // (integer activations: a group's sum stays one exact int32 accumulation)
            const bool persistent = a.epi != EPI_KV && tiles * ns > SMS;           // (K~/V~ tiles are assembled in the rings: one per CTA)
            Choice c{};
            if (!rings_of(a, p, bn, ns, 0, persistent, c)) continue;
            const long long per = (tiles * ns + SMS - 1) / SMS;                                            // tiles per CTA
            const long long ctas = persistent ? (tiles + per - 1) / per : tiles * ns;
            const int share = share_of(p, ns);
            const double fixed = m.fixed + (a.epi == EPI_KV ? 0.008 * bn : 0), tile = persistent ? m.tile : 0;
            const double groups = p.n_groups == 1 ? 1 : (double)share * p.n_groups / p.n_kb;
            const double cost = (persistent ? 1 : per) * fixed + (double)per * (share * m.kb + groups * m.group + tile + (a.epi == EPI_Q8_HEAD ? m.q8 : 0)) +
                                (ns > 1 ? m.split + 0.1 * (ns - 2) + m.exchange * (ns - 1) * (double)(tiles * ns) / SMS : 0);
            if (cost < best_cost) { best_cost = cost; best = finish(c, a, p, tiles, ctas); }
        }
    }
    return best;
}

// Tiles of 256 rows on pairs of CTAs, in rounds of 74.  A fit to 151 measured launches (256 to 32768 rows, 320 to 1280 channels, W4 and
// W8, fp16 and per-head int8 rows; 6 and 5 % rms).  The per-head terms, below 0, are what the fit leaves between the two outputs, whose other
// parts are one number each, and no step's cost.
Choice choose_pair(const LinearArgs& a, int n_z, double& best_cost) {
    struct PairPace { int bn; double fixed, pair4, pair8, tile, q8; };
    constexpr PairPace PAIR_PACES[2] = {{160, 3.70, 0.628, 0.541, 1.25, -0.73}, {128, 3.16, 0.559, 0.504, 0.87, -0.22}};
    const Problem p = problem_of(a);
    Choice best{};
    best_cost = 1e30;
    for (const PairPace& m : PAIR_PACES) {
        Choice c{};
        if (!tile_carries(a, p, m.bn) || !(m.bn == 160 ? pair_rings<160>(a, p, c) : pair_rings<128>(a, p, c))) continue;
        const long long rows2 = (p.row_tiles + 1) / 2, tiles = rows2 * (a.n_out / m.bn) * (long long)n_z;
        if (tiles > (1 << 29)) continue;
        const long long per = (tiles + SMS / 2 - 1) / (SMS / 2), pairs = (tiles + per - 1) / per;
        const double cost = m.fixed + (double)per * ((p.n_kb + 1) / 2 * (a.bits == 4 ? m.pair4 : m.pair8) + m.tile) + (a.epi == EPI_Q8_HEAD ? m.q8 : 0);
        if (cost >= best_cost) continue;
        best_cost = cost;
        best = finish(c, a, p, tiles, 2 * pairs);
        best.lay.n_rows = (int)rows2;
        best.lay.mul_rows = multiplier(best.lay.n_rows, tiles);
    }
    return best;
}

// Pairs or one CTA per tile: the cheaper one, with three corrections.  Where a CTA would walk several tiles the model of one CTA per tile is 10 to
// 40 % short (in one problem's launches pairs were always faster there, by 2 to 45 %).  But requests of up to 128 rows leave half of every 256-row
// tile empty, and of 160 measured layers of such requests none is faster on pairs (18 requests x 34 rows, 1280 channels, heads of 64: 52.4 us, 43.4
// so).  In launches of one wave of 128 or 160 columns fp16 rows take 1.4 to 3.2 us more than the model says.  Of 248 single launches (16 to 32768
// rows) all but two get the kernel that is faster, or within 1.5 % of it, and of 224 layers of requests all within 2.6 %.  The two are of the
// third correction: scale groups that a cluster would share stay shared (heads of 160 channels, 600 to 1150 rows), for sums of all groups in a
// row lose bits that two halves keep.  1100 x 1280 x 1280, W4: scales' root mean square error 5.3e-8, on pairs 6.3e-8 (12.9 and 10.8 us); x 2560
// 5.8e-8 and 7.9e-8 (18.0 and 19.6 us).
Choice choose_anew(const LinearArgs& a, int n_z) {
    double cost, pair_cost;
    const Choice single = choose_single(a, n_z, cost), pair = choose_pair(a, n_z, pair_cost);
    if (single.lay.nsplit > 1 && single.lay.n_groups > 1) return single;
    const double limit = single.lay.persistent ? (a.rows <= BM ? 1.1 : 1.4) * cost : cost + (single.bn >= 128 ? 2.0 : 0.0);
    if (!pair.bn || (single.bn && pair_cost >= limit)) return single;
    return pair;
}

// The last few problems of the calling thread: a program runs the same layers again and again.
Choice choose(const LinearArgs& a, int n_z) {
    struct Key { long long rows; int n_out, k_in, bits, group, heads, epi, n_ctx, n_z, flags, max_trigger; };
    struct Known { Key key; Choice choice; };
    constexpr int N = 16;
    thread_local Known known[N] = {};
    thread_local int next = 0;
    const Key k = {a.rows, a.n_out, a.k_in, a.bits, a.group, a.heads, a.epi, a.n_ctx, n_z, 4 | (a.xq ? 1 : 0) | (a.reqs ? 2 : 0), a.max_trigger};
    for (const Known& e : known)
        if (memcmp(&e.key, &k, sizeof(k)) == 0) return e.choice;
    Known& e = known[next];
    next = (next + 1) % N;
    e.key = k;
    return e.choice = choose_anew(a, n_z);
}

// Shapes the tensor-core kernel takes at all (before looking for a layout).
bool takes_shape(const LinearArgs& a) {
    if (a.xq) {       // int8 activations: rows of 16-byte granularity, a scale group = one 128-element K block
        if (a.k_in % 16) return false;
        if (a.group != 0 && a.group != 2 * BK && a.group < a.k_in) return false;
    } else {
        if (a.k_in % BK) return false;
        if (a.group != 0 && a.group % BK) return false;
    }
    return a.rows >= 1 && a.rows <= (1LL << 31) - 1;
}

}  // namespace

bool sm100_linear_supported(const LinearArgs& a) {
    if (!takes_shape(a)) return false;
    if ((a.xq ? reinterpret_cast<uintptr_t>(a.xq) : reinterpret_cast<uintptr_t>(a.x)) & 15u) return false;
    if (a.epi != EPI_KV && (reinterpret_cast<uintptr_t>(a.y) & 15u)) return false;   // the output leaves in pieces of 16 bytes
    return choose(a, 1).bn != 0 && encode_tiled_fn() != nullptr;
}

// The launch plan of a dequant-GEMM as the launcher takes it (no GPU needed): tile width, ring depth in k-blocks, CTAs that share a tile's K
// loop, and the byte ranges of shared memory that the rings, the epilogue's staging area in them and the fixed sections occupy.  out: {bn,
// nstage, split, ring_bytes, staging_bytes, off_raw (the first fixed section), off_bias, off_bars, total, limit}.  bn = 0: the tensor-core
// kernels do not take it (pairs_only: it does not run on pairs of CTAs).
void linear_plan_of(const LinearArgs& a, int n_z, bool pairs_only, int out[10]) {
    for (int i = 0; i < 10; ++i) out[i] = 0;
    out[9] = SMEM_LIMIT;
    if (!takes_shape(a)) return;
    const Choice c = choose_anew(a, n_z);
    if (c.bn == 0 || (pairs_only && !c.pair)) return;
    const Plan& P = c.lay.plan;
    out[0] = c.bn; out[1] = 2 * (c.lay.nsa < c.lay.nsb ? c.lay.nsa : c.lay.nsb); out[2] = c.lay.nsplit; out[3] = P.ring_bytes; out[4] = c.staged;
    out[5] = P.off_scales; out[6] = P.off_bias; out[7] = P.off_bars; out[8] = P.total;
}

cudaError_t launch_linear_sm100(const LinearArgs& a, int n_z, cudaStream_t stream) {
    if (a.rows == 0 || n_z == 0) return cudaSuccess;
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return cudaErrorNotSupported;
    const Choice c = choose(a, n_z);
    CUtensorMap tmap;
    const bool i8 = a.xq != nullptr;
    const cuuint64_t esz = i8 ? 1 : 2;
    const cuuint64_t dims[3] = {(cuuint64_t)a.k_in, (cuuint64_t)a.rows, (cuuint64_t)n_z};
    const cuuint64_t strides[2] = {(cuuint64_t)a.k_in * esz, (cuuint64_t)a.k_in * esz * (cuuint64_t)a.rows};
    const cuuint32_t box[3] = {(cuuint32_t)(i8 ? 2 * BK : BK), c.lay.kv.x_bytes / 128, 1};       // 128 bytes of K either way; elements beyond k_in read as zero
    const cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(&tmap, i8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3,
                     i8 ? (void*)const_cast<int8_t*>(a.xq) : (void*)const_cast<__half*>(a.x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    if (c.pair) {
        // the output: boxes of 32 rows, 32 columns of fp16 (64-byte swizzle) or a tile's width of int8 codes (128 columns: swizzled)
        CUtensorMap tmap_y;
        const bool q8 = a.epi == EPI_Q8_HEAD;
        const cuuint64_t osz = q8 ? 1 : 2;
        const cuuint64_t ydims[3] = {(cuuint64_t)a.n_out, (cuuint64_t)a.rows, (cuuint64_t)n_z};
        const cuuint64_t ystrides[2] = {(cuuint64_t)a.n_out * osz, (cuuint64_t)a.n_out * osz * (cuuint64_t)a.rows};
        const cuuint32_t ybox[3] = {(cuuint32_t)(q8 ? c.bn : 32), 32, 1};
        r = enc(&tmap_y, q8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, a.y, ydims, ystrides, ybox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                !q8 ? CU_TENSOR_MAP_SWIZZLE_64B : c.bn == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
        return c.bn == 160 ? launch_pair<160>(tmap, a, c.lay, tmap_y, c.grid, c.total, stream) : launch_pair<128>(tmap, a, c.lay, tmap_y, c.grid, c.total, stream);
    }
    switch (c.bn) {
        case 64: return launch_tile<64>(tmap, a, c.lay, c.grid, c.total, stream);
        case 80: return launch_tile<80>(tmap, a, c.lay, c.grid, c.total, stream);
        case 128: return launch_tile<128>(tmap, a, c.lay, c.grid, c.total, stream);
        case 160: return launch_tile<160>(tmap, a, c.lay, c.grid, c.total, stream);
    }
    return cudaErrorNotSupported;
}

}  // namespace taq
