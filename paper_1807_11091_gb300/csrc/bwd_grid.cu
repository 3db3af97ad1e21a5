// bwd_grid.cu -- backward of a packed pruned stride-1 CONV layer for masked
// retraining (Sec. 4) on the padded pixel grid of grid.cuh: no im2col, no
// col2im, no atomics.
//
//   k_grid_front   in one launch: dZ = dY * [y > 0] of the kept filters as a grid
//                  copy (each element read once for dW, dx and db) with db's
//                  partial sums; x as a grid copy; the input gradient's weights
//                  (taps flipped, kept filters as channels) and output map; dW
//                  zeroed
//   k_grid_wgrad   dW: for a tap of shift s, dW[f][c] = sum over grid pixels q
//                  of x[c][q + s] * dZ[f][D0 + q].  Channels are the MMA's M
//                  side, filters its N side, pixels its K side: both operands
//                  are the copies themselves, read MN-major (core matrices of 8
//                  channels x 8 pixels); dZ is zero off the output, so the
//                  padded pixels add nothing.
//   k_grid_conv    dx: the slab GEMM over dZ (conv_grid.cu), every element
//                  written once
//   k_grid_wreduce the slices of the pixel ranges, in order, into dW's kept
//                  entries, and db's partial sums
//
// A layer of at most 64 channels fills half of the M side or less: its slab is
// then staged up to 16 / chunks times, each copy a pixel further on, and one
// MMA covers that many kernel columns.
// The tensor core truncates as it accumulates, so fp32 registers take over early: dW
// after kGwSegTiles tiles of 128 pixels (16 MMA steps), dx after dx_seg() steps; an
// item's sums leave the registers once, for its slice.  Errors against 64 bits (2-norm)
// of dW, beside the chunked path's: AlexNet conv2 1.4e-7 (2.2), conv3 1.1e-7 (1.9), a
// ResNet-50 3x3 layer 1.2e-7 (2.3), 64 channels at 224x224 and batch 8 1.5e-7 (2.3);
// with sums of 32 steps conv3's stand at 1.5e-7, of 48 at 2.1e-7.
//
// AlexNet conv2 at batch 128 (two groups of 64 kept filters x 48 channels, 5x5): 841
// us as six im2col / GEMM / col2im chunks, 161 us here; conv3 164 -> 52, a ResNet-50
// 3x3 layer (64 of 128 channels and filters kept) at batch 64 277 -> 42.2.
// One cold launch each (front, weight gradient, input gradient, reduction): conv2 35, 58,
// 74, 8 us, conv3 14, 21, 27, 10, the ResNet layer 14, 17, 21, 11.  Both gradients run at
// the issue rate of their MMAs (48 to 57 cycles a 128 x 64 x 16, set by the operands'
// shared-memory reads) between their first loads and their last stores; the front pass
// is 16 loads of 2 and 4 bytes an octet.
#include <string.h>

#include <algorithm>

#include "grid.cuh"

namespace sadmm {
namespace {

constexpr int kGwThreads = 10 * 32;
constexpr int kGwMaxStages = 6;
constexpr int kGwSegTiles = 2;       // 128-pixel tiles summed in TMEM: 8 MMA steps each
static_assert(kGwSegTiles % 2 == 0, "a segment ends with a stage of one or two tiles");
constexpr int kGwMaxTiles = 64;      // tiles of an item, summed in registers
constexpr int kDxStage = 27;         // most MMA steps of an input gradient's stage, where the kernel has no more taps
constexpr long long kGwCtas = 152;   // work items come in multiples of about this many (fixed: it sizes the workspace)
constexpr int kGwSmemLimit = 232448;
constexpr int kGwCols = 256;         // columns of an accumulator; TMEM holds two
constexpr int kGwChunks = kGwCols / kEpiCols / 2;  // 16-column chunks of an accumulator that a warp holds

// MMA steps of the input gradient summed in TMEM.  The chunked path sums a pixel's
// kept filters there, 16 a step, and adds the taps up in fp32: up to 256 filters a
// group 12 steps are held here, beyond that, where those sums are long themselves, 27.
// Errors against 64 bits, in 1e-8 (chunked path; here; with 27 steps): AlexNet conv3
// 7.0; 6.4; 9.4, conv2 8.2; 8.7; 12, a ResNet-50 3x3 layer 7.3; 11; 16, 7x7, 9x9 and
// 11x11 taps over 64 filters 13, 16, 19; 12, 14, 15; 19, 24, 21, 256 filters 3x3 16; 13;
// 17, 512 filters 30; 16 (27 steps).  A sum more to read takes about 750 cycles of an
// epilogue beside the MMAs: conv3's backward was 52.5 us, not 49.1, conv2's 162, not 149,
// the ResNet layer's 42.7, not 41.7 (with loads one by one: 52.0, 161 and 42.2 now).
int dx_seg(int filters) { return filters <= 256 ? 12 : 27; }

struct WgradShape {
    int nch;          // 8-channel chunks of x per conv group
    int blk, mblks;   // chunks per M block, blocks
    int rep, kwg;     // kernel columns per MMA, groups of them (macro taps) per kernel row
    int kws;          // a row's macro taps as items take them: kwg, or to a multiple of tpg where no item spans rows
    int rows;         // M rows in use: rep * blk * 8
    int nst, nft;     // filters per N tile, tiles
    int tpg, tgs;     // macro taps per item, items per kernel frame
    int types;        // items per pixel range
    int tiles, tps, Z;  // 128-pixel tiles, tiles per range, ranges
    int span;         // slots that an item's taps reach beyond its pixels, at most
    long long slice;  // floats of a pixel range's slice
    long long cycles;  // estimated time
};

// How the stages lie in shared memory for items of `nr` filters: slabs of one
// 128-pixel tile, or of two where that leaves two stages.  A bulk copy takes about
// 66 cycles whatever its size up to 4 KB at least, and a slab is a copy per chunk
// (with one tile: conv2's backward 172 us, not 162, conv3's 60, not 52.5).
struct GwStage {
    int tiles, spa, a_bytes, stride, count;  // tiles and slots a chunk, bytes of the slab and of a stage, stages
};
__host__ __device__ inline GwStage gw_stage(const WgradShape& w, int nr)
{
    GwStage st;
    for (st.tiles = 2;; st.tiles = 1) {
        st.spa = st.tiles * 128 + w.span;
        st.a_bytes = (w.rep * w.blk * st.spa * 16 + 127) / 128 * 128;
        st.stride = st.a_bytes + nr * 256 * st.tiles;
        // (the MMA reads 16 chunks whatever the rows in use: room past the last stage)
        st.count = (kGwSmemLimit - 1024 - 512 - (16 - w.rep * w.blk) * st.spa * 16) / st.stride;
        if (st.count > kGwMaxStages) st.count = kGwMaxStages;
        if (st.count >= 2 || st.tiles == 1) return st;
    }
}

// The most slots that the taps of an item span beyond its pixels.
int wgrad_span(const Grid& gr, const WgradShape& w)
{
    if (w.kws % w.tpg == 0) return (std::min(w.tpg, w.kwg) - 1) * w.rep;  // (no item spans rows)
    const int macro = gr.KH * w.kws;
    int span = 0;
    for (int t0 = 0; t0 < macro; t0 += w.tpg) {
        const int t1 = std::min(macro, t0 + w.tpg) - 1, r0 = t0 / w.kws, r1 = t1 / w.kws;
        const int first = r0 * gr.Wb + t0 % w.kws * w.rep, last = r1 * gr.Wb + t1 % w.kws * w.rep;
        int lo = std::min(first, last), hi = std::max(first, last);
        if (r1 > r0) {
            lo = std::min(lo, (r0 + 1) * gr.Wb);
            hi = std::max(hi, (r1 - 1) * gr.Wb + (w.kws - 1) * w.rep);
        }
        span = std::max(span, hi - lo);
    }
    return span;
}

// `nck` channels and at most `n_pad`, likely `likely`, filters per group.
bool wgrad_shape(const Grid& gr, int nck, int n_pad, int likely, int groups, WgradShape* out)
{
    WgradShape w;
    if (nck < 1) return false;
    w.nch = (nck + 7) / 8;
    w.rep = 1;
    if (w.nch <= 8) {
        w.rep = std::min(16 / w.nch, gr.KW);
        w.mblks = 1;
    } else {
        w.mblks = (w.nch + 15) / 16;
    }
    w.blk = (w.nch + w.mblks - 1) / w.mblks;
    w.kwg = (gr.KW + w.rep - 1) / w.rep;
    w.rows = w.rep * w.blk * 8;
    w.tiles = (gr.L + 127) / 128;
    const int macro = gr.KH * w.kwg;
    // The filter tiles (whole, about 128, 96, 64 and 48), the taps of an item (as many
    // as fill an accumulator with the likely filters, or fewer) and the pixel ranges of
    // least estimated time.  More columns an item mean fewer slab loads, more ranges
    // more slices to write and to add up.
    const int nft0 = (n_pad + kGwCols - 1) / kGwCols;
    long long best = -1;
    int seen = 0;
    for (const int aim : {kGwCols, 128, 96, 64, 48}) {
        w.nft = std::max(nft0, (n_pad + aim - 1) / aim);
        if (w.nft == seen) continue;
        seen = w.nft;
        w.nst = (int)round_up((n_pad + w.nft - 1) / w.nft, 16);
        const int nl = w.nft == 1 ? std::min(w.nst, (int)round_up(likely, 16)) : w.nst;
        const int tmax = std::min(std::min(kGwCols / nl, macro), 32), tg0 = (macro + tmax - 1) / tmax;
        for (int tgs = tg0, by_row = 0; tgs <= std::min(macro, tg0 + 3); tgs += by_row, by_row ^= 1) {
            w.tpg = (macro + tgs - 1) / tgs;
            if ((macro + w.tpg - 1) / w.tpg != tgs) continue;
            // also with items that span no rows, whose slabs are shorter (AlexNet conv3 in
            // pairs of taps fits stages of two tiles so)
            w.kws = by_row ? (int)round_up(w.kwg, w.tpg) : w.kwg;
            if (by_row && (w.kws == w.kwg || w.tpg > w.kwg)) continue;
            w.tgs = (gr.KH * w.kws + w.tpg - 1) / w.tpg;
            w.span = wgrad_span(gr, w);
            if (w.span + 256 >= (1 << 14) || gw_stage(w, w.nst).count < 2) continue;
            const GwStage sg = gw_stage(w, nl);
            const long long types = (long long)groups * w.nft * w.mblks * gr.KT * w.tgs;
            // Cycles of a tile: its MMAs (as in conv_grid.cu) or its share of the slab
            // copies, and 280 a stage for its waits and commits; of an item its tiles,
            // then its slice's stores (16 bytes a cycle, beside the next item's MMAs);
            // and the reduction's reads (16 bytes a cycle and SM).
            const long long cols = (long long)w.tpg * nl;
            const long long tile = std::max(w.tpg * 8ll * (std::max(32 + nl / 4, nl / 2) + 9),
                                            66ll * (w.rep * w.blk + nl / 8) / sg.tiles) + 280 / sg.tiles;
            const long long st = w.rows * cols / 4;
            for (int waves = 1; waves <= 4; ++waves) {
                // (ranges of at least four tiles, two stages: shorter ones start up and end longer
                // than they run: 26 drawn layers of up to 64 tiles took 3 % more with one, 1 % with two)
                const long long z = std::min<long long>((w.tiles + 3) / 4, std::max<long long>(std::max<long long>(1, kGwCtas * waves / types),
                                                                                               (w.tiles + kGwMaxTiles - 1) / kGwMaxTiles));
                w.tps = (int)((w.tiles + z - 1) / z);
                w.Z = (w.tiles + w.tps - 1) / w.tps;
                if (types * w.Z >= (1ll << 30)) continue;
                w.types = (int)types;
                w.slice = types * w.rows * w.tpg * w.nst;
                const long long item = w.tps * tile, rounds = (types * w.Z + kGwCtas - 1) / kGwCtas;
                const long long cost = rounds * std::max(item, st) + st + types * w.Z * w.rows * cols * 4 / (kGwCtas * 16);
                if (best < 0 || cost < best) {
                    best = w.cycles = cost;
                    *out = w;
                }
            }
        }
    }
    return best >= 0;
}

struct GwArgs {
    Grid gr;
    WgradShape w;
    const __nv_bfloat16* xs;
    const __nv_bfloat16* dz;
    long long xs_gstride, dz_gstride;
    const int* counts;
    const int* colidx;  // kept columns, ascending (NULL: every column of the kept channels)
    int nck, n_cols, taps;
    float* slices;
    int groups, units;
    FastDiv types_div;
    int* status;
};

// One work item: pixel range z and (group, filter tile, channel block, kernel
// frame, tap group).
struct GwItem {
    int z, type, g, ft, mb, kt, t0, nt, nr, base, span;
    int tp;  // taps that fill an accumulator: more take another pass over the pixels
};
SADMM_DEV GwItem gw_item(const GwArgs& a, int u)
{
    GwItem it;
    it.z = (int)fdiv((uint32_t)u, a.types_div);
    it.type = u - it.z * a.w.types;
    int r = it.type;
    const int tg = r % a.w.tgs;
    r /= a.w.tgs;
    it.kt = r % a.gr.KT;
    r /= a.gr.KT;
    it.mb = r % a.w.mblks;
    r /= a.w.mblks;
    it.ft = r % a.w.nft;
    it.g = r / a.w.nft;
    it.t0 = tg * a.w.tpg;
    it.nt = min(a.w.tpg, a.gr.KH * a.w.kws - it.t0);
    if (a.w.kws % a.w.tpg == 0) it.nt = min(it.nt, a.w.kwg - it.t0 % a.w.kws);
    const int cnt = min(a.w.nst, __ldg(a.counts + 2 * it.g) - it.ft * a.w.nst);
    it.nr = cnt > 0 ? (cnt + 15) & ~15 : 0;
    int lo = 1 << 30, hi = 0;
    for (int t = it.t0; t < it.t0 + it.nt; ++t) {
        const int s = (t / a.w.kws) * a.gr.Wb + (t % a.w.kws) * a.w.rep;
        lo = min(lo, s);
        hi = max(hi, s);
    }
    it.base = lo;
    it.span = hi - lo;
    it.tp = min(it.nt, it.nr > 0 ? kGwCols / it.nr : 1);
    return it;
}

// Bit j: the item's macro tap j holds a kept GEMM column of accumulator row `row`.
SADMM_DEV uint32_t gw_keep(const GwArgs& a, const GwItem& it, int row)
{
    const int per = a.w.blk * 8;
    const int rp = row / per, c = it.mb * per + row - rp * per;
    if (row >= a.w.rows || c >= a.nck) return 0;
    uint32_t keep = 0;
    for (int j = 0; j < it.nt; ++j) {
        const int t = it.t0 + j, kh = t / a.w.kws, kw = (t - kh * a.w.kws) * a.w.rep + rp;
        if (kw >= a.gr.KW) continue;
        bool ok = true;
        if (a.colidx) {
            const int want = c * a.taps + (it.kt * a.gr.KH + kh) * a.gr.KW + kw;
            int lo = 0, hi = a.n_cols;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (__ldg(a.colidx + mid) < want) lo = mid + 1;
                else hi = mid;
            }
            ok = lo < a.n_cols && __ldg(a.colidx + lo) == want;
        }
        if (ok) keep |= 1u << j;
    }
    return keep;
}

__global__ void __launch_bounds__(kGwThreads, 1) k_grid_wgrad(const __grid_constant__ GwArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem);  // the first 512 bytes
    uint8_t* stage0 = smem + 512;
    uint64_t* full = bars;
    uint64_t* empty = bars + kGwMaxStages;
    uint64_t* acc_full = bars + 2 * kGwMaxStages;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* drain = acc_empty + 2;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGwMaxStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 8); }
        mbar_init(drain, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_holder, 2u * kGwCols);
        tmem_relinquish();
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();  // after every thread's wait: k_grid_front has completed when a dependent starts
    const uint32_t tmem_base = *tmem_holder;
    // The stages hold what the groups' counts need, known on the device alone.
    int most = 0;
    for (int g = 0; g < a.groups; ++g) most = max(most, __ldg(a.counts + 2 * g));
    // (a reduction over the warp: the compiler then knows what follows from it as uniform)
    most = __reduce_max_sync(0xffffffffu, min(a.w.nst, (most + 15) & ~15));
    const GwStage sg = gw_stage(a.w, most);
    if (warp == 0) {
        int s = 0;
        uint32_t ph = 0, last = 0, issued = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < a.units; u += gridDim.x) {
            const GwItem it = gw_item(a, u);
            if (it.nr == 0) continue;
            const int nb = min(a.w.blk, a.w.nch - it.mb * a.w.blk);  // chunks of this block
            const int na = nb * a.w.rep, nd = it.nr / 8;
            const __nv_bfloat16* xg = a.xs + (size_t)it.g * a.xs_gstride;
            const __nv_bfloat16* dg = a.dz + (size_t)it.g * a.dz_gstride;
            const int b = it.z * a.w.tps, e = min(a.w.tiles, b + a.w.tps);
            for (int t0 = 0; ok && t0 < it.nt; t0 += it.tp) {  // a pass over the pixels for the taps t0 ..
                for (int t = b; t < e; t += sg.tiles) {
                    if (!mbar_wait_warp(&empty[s], ph ^ 1u, abort_flag, a.status)) { ok = false; break; }
                    const int n = min(sg.tiles, e - t);
                    const uint32_t abytes = (uint32_t)(n * 128 + it.span) * 16u, dbytes = (uint32_t)n * 2048u;
                    if (lane == 0) mbar_arrive_expect_tx(&full[s], (uint32_t)na * abytes + (uint32_t)nd * dbytes);
                    __syncwarp();
                    const uint32_t sa = smem_u32(stage0 + (size_t)s * sg.stride);
                    for (int k = lane; k < na + nd; k += 32) {
                        if (k < na) {
                            const int rp = k / nb, c = k - rp * nb;
                            bulk_load(sa + (uint32_t)((rp * a.w.blk + c) * sg.spa * 16),
                                      xg + ((size_t)(it.mb * a.w.blk + c) * a.gr.slots +
                                            (size_t)(t * 128 + it.kt * a.gr.HWb + it.base + rp)) * 8,
                                      abytes, &full[s]);
                        } else {
                            const int c = k - na;
                            bulk_load(sa + (uint32_t)(sg.a_bytes + c * sg.tiles * 2048),
                                      dg + ((size_t)(it.ft * (a.w.nst / 8) + c) * a.gr.slots +
                                            (size_t)(a.gr.D0 + t * 128)) * 8,
                                      dbytes, &full[s]);
                        }
                    }
                    last = (last & ~(1u << s)) | (ph << s);
                    issued |= 1u << s;
                    if (++s == sg.count) { s = 0; ph ^= 1u; }
                }
            }
        }
        for (int q = 0; q < sg.count; ++q) {
            if (!(issued & (1u << q))) continue;
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(&full[q], (last >> q) & 1u) && globaltimer() - t0 < kWaitLimitNs) {}
        }
        __syncwarp();
    } else if (warp == 1) {
        // The whole warp runs the loop; one elected lane issues.
        int s = 0, ab = 0;
        uint32_t ph = 0, acc_ph = 0;
        bool ok = true;
        const uint64_t ad0 = sdesc_kmajor_none(smem_u32(stage0), 128u, (uint32_t)sg.spa * 16u);
        const uint64_t bd0 = sdesc_kmajor_none(smem_u32(stage0) + (uint32_t)sg.a_bytes, 128u, (uint32_t)sg.tiles * 2048u);
        const uint64_t ahi = ad0 & 0xffffffff00000000ull, bhi = bd0 & 0xffffffff00000000ull;
        for (int u = blockIdx.x; ok && u < a.units; u += gridDim.x) {
            GwItem it = gw_item(a, u);
            // (uniform, as above)
            it.nr = __reduce_max_sync(0xffffffffu, it.nr);
            it.tp = __reduce_max_sync(0xffffffffu, it.tp);
            if (it.nr == 0) continue;
            const uint32_t idesc = idesc_bf16_f32(128, it.nr) | (1u << 15) | (1u << 16);  // A and B MN-major
            const int b = it.z * a.w.tps, e = min(a.w.tiles, b + a.w.tps);
            for (int t0 = it.t0; ok && t0 < it.t0 + it.nt; t0 += it.tp) {
                const int np = min(it.tp, it.t0 + it.nt - t0);
                const uint32_t kq0 = (uint32_t)(t0 % a.w.kws);
                const uint32_t to0 = (uint32_t)(t0 / a.w.kws * a.gr.Wb) + kq0 * (uint32_t)a.w.rep - (uint32_t)it.base;
                int in_seg = 0;
                uint32_t d0 = 0;
                for (int t = b; t < e; t += sg.tiles) {
                    if (in_seg == 0) {
                        if (!mbar_wait_warp(&acc_empty[ab], acc_ph ^ 1u, abort_flag, a.status)) { ok = false; break; }
                        d0 = tmem_base + (uint32_t)(ab * kGwCols);
                    }
                    if (!mbar_wait_warp(&full[s], ph, abort_flag, a.status)) { ok = false; break; }
                    tc_fence_after();
                    const int n = min(sg.tiles, e - t);
                    const uint32_t so = (uint32_t)(s * sg.stride) >> 4;
                    uint32_t to = to0, kq = kq0;  // the tap's shift in the slab, its place in the kernel row
                    for (int j = 0; j < np; ++j) {
                        uint32_t alo = (uint32_t)ad0 + so + to, blo = (uint32_t)bd0 + so;
                        const uint32_t d = d0 + (uint32_t)(j * it.nr);
                        uint32_t acc = in_seg > 0 ? 1u : 0u;
                        for (int q = 0; q < n; ++q) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk)  // 16 grid pixels each
                                mma_bf16_ss_elect(d, ahi | (alo + kk * 16u), bhi | (blo + kk * 16u), idesc, kk > 0 ? 1u : acc);
                            acc = 1u;
                            alo += 128u;
                            blo += 128u;
                        }
                        to += (uint32_t)a.w.rep;
                        if (++kq == (uint32_t)a.w.kws) {
                            kq = 0;
                            to += (uint32_t)(a.gr.Wb - a.w.kws * a.w.rep);
                        }
                    }
                    mma_commit_elect(&empty[s]);
                    if (++s == sg.count) { s = 0; ph ^= 1u; }
                    in_seg += n;
                    if (in_seg >= kGwSegTiles || t + n >= e) {
                        mma_commit_elect(&acc_full[ab]);
                        if (++ab == 2) { ab = 0; acc_ph ^= 1u; }
                        in_seg = 0;
                    }
                }
            }
        }
        mma_commit_elect(drain);
        if (lane == 0) {
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < kWaitLimitNs) {}
        }
        __syncwarp();
    } else {
        // epilogue: the item's segments added up in registers, then written to its
        // slice; lane = channel row, the two warps of a TMEM lane quadrant take its
        // 16-column chunks in turn
        const int q4 = warp & 3, h = (warp - 2) >> 2;
        const int row = q4 * 32 + lane;
        int ab = 0;
        uint32_t acc_ph = 0;
        bool alive = true;
        for (int u = blockIdx.x; alive && u < a.units; u += gridDim.x) {
            const GwItem it = gw_item(a, u);
            if (it.nr == 0) continue;
            // the item's taps whose column of this lane's channel is kept: only
            // those are written (found while the MMAs run)
            const uint32_t keep = gw_keep(a, it, row);
            const int per = it.nr / kEpiCols;
            const int b = it.z * a.w.tps, e = min(a.w.tiles, b + a.w.tps);
            float* dst = a.slices + (size_t)it.z * a.w.slice +
                         ((size_t)it.type * a.w.rows + row) * (size_t)(a.w.tpg * a.w.nst);
            for (int p0 = 0; alive && p0 < it.nt; p0 += it.tp) {
                const int n = min(it.tp, it.nt - p0) * per;
                float v[kGwChunks][kEpiCols];
#pragma unroll
                for (int c = 0; c < kGwChunks; ++c)
#pragma unroll
                    for (int i = 0; i < kEpiCols; ++i) v[c][i] = 0.0f;
                for (int t = b; t < e; t += kGwSegTiles) {
                    // warp-uniform outcome: the TMEM loads below are .sync.aligned
                    if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[ab], acc_ph, abort_flag, a.status))) {
                        alive = false;
                        break;
                    }
                    tc_fence_after();
                    if (q4 * 32 < a.w.rows) {
                        const uint32_t taddr = tmem_base + (uint32_t)(ab * kGwCols) + ((uint32_t)(q4 * 32) << 16);
#pragma unroll
                        for (int c = 0; c < kGwChunks; ++c) {
                            const int k = 2 * c + h;
                            if (k < n) {
                                uint32_t r[kEpiCols];
                                tmem_ld_32x32b_x16(taddr + (uint32_t)(k * kEpiCols), r);
                                tmem_ld_wait();
#pragma unroll
                                for (int i = 0; i < kEpiCols; ++i) v[c][i] += __uint_as_float(r[i]);
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[ab]);
                    if (++ab == 2) { ab = 0; acc_ph ^= 1u; }
                }
                if (!alive) break;
#pragma unroll
                for (int c = 0; c < kGwChunks; ++c) {
                    const int k = 2 * c + h, j = k / per;
                    if (k < n && ((keep >> (p0 + j)) & 1u) &&
                        dbg_in(dst + (p0 + j) * a.w.nst + (k - j * per) * kEpiCols + kEpiCols - 1 - a.slices,
                               a.w.Z * a.w.slice, a.status)) {
                        float4* d4 = reinterpret_cast<float4*>(dst + (p0 + j) * a.w.nst + (k - j * per) * kEpiCols);
#pragma unroll
                        for (int i = 0; i < kEpiCols / 4; ++i)
                            d4[i] = make_float4(v[c][4 * i], v[c][4 * i + 1], v[c][4 * i + 2], v[c][4 * i + 3]);
                    }
                }
                __syncwarp();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 2u * kGwCols);
    }
}

struct DbArgs {
    const float* part;  // NULL: no bias gradient
    const int* rowmap;
    const int* zeromap;
    const int* counts;
    int nparts, groups, n_pad, Fg;
    int more;  // 1: added to db, which an earlier pass over other images wrote
    float* db;
    int F;
    int* status;
};

// db, by blocks b, b + nb, ... of 256 threads: a warp per packed row adds its
// partial sums (fixed order); zeros for the pruned filters.
SADMM_DEV void db_blocks(const DbArgs& a, int b, int nb)
{
    const int lane = threadIdx.x & 31;
    for (int r = b * 8 + (threadIdx.x >> 5); r < a.groups * a.n_pad; r += nb * 8) {
        const int f = __ldg(a.rowmap + r);
        if (f < 0) continue;
        float s = 0.0f;
        for (int k = lane; k < a.nparts; k += 32) s += __ldg(a.part + (size_t)r * a.nparts + k);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0 && dbg_in(f, a.F, a.status)) a.db[f] = a.more ? a.db[f] + s : s;
    }
    for (int z = b * 256 + threadIdx.x; !a.more && z < a.groups * a.Fg; z += nb * 256) {
        const int g = z / a.Fg;
        if (z - g * a.Fg >= __ldg(a.counts + 2 * g + 1)) continue;
        const int f = __ldg(a.zeromap + z);
        if (dbg_in(f, a.F, a.status)) a.db[f] = 0.0f;
    }
}

__global__ void __launch_bounds__(256) k_grid_db(const DbArgs a)
{
    pdl_wait();  // after the kernel before it in the stream
    pdl_trigger();
    db_blocks(a, blockIdx.x, gridDim.x);
}

struct WrArgs {
    Grid gr;
    WgradShape w;
    const float* slices;
    const int* rowmap;
    const int* colidx;
    const int* counts;
    const __nv_bfloat16* xs;
    const __nv_bfloat16* dz;
    long long xs_gstride, dz_gstride;
    float* dW;
    int n_pad, n_cols, taps, chan_kind;
    int more;  // 1: added to dW, which an earlier pass over other images wrote
    long long K, dw_total;
    int* status;
};

// Where the slices of packed row i, K column col (packed column j) of group g lie, in
// the first range.
SADMM_DEV size_t wr_slice(const WrArgs& a, int g, int i, int j, int col)
{
    const int c = a.chan_kind ? j / a.taps : col / a.taps, tap = col % a.taps;
    const int kw = tap % a.gr.KW, kh = (tap / a.gr.KW) % a.gr.KH, kt = tap / (a.gr.KW * a.gr.KH);
    const int mb = (c >> 3) / a.w.blk, mt = kh * a.w.kws + kw / a.w.rep, ft = i / a.w.nst;
    const int m = (((kw % a.w.rep) * a.w.blk + ((c >> 3) - mb * a.w.blk)) << 3) + (c & 7);
    const int type = (((g * a.w.nft + ft) * a.w.mblks + mb) * a.gr.KT + kt) * a.w.tgs + mt / a.w.tpg;
    return ((size_t)type * a.w.rows + m) * (size_t)(a.w.tpg * a.w.nst) + (mt % a.w.tpg) * a.w.nst + (i - ft * a.w.nst);
}

// One entry of the weight gradient whose sum came out NaN, by a warp: a range's slice is
// NaN where a padded pixel's zero met an infinity or a NaN of x, which is no term of the
// sum, so such a range is added up again over its output pixels alone, until one of its
// terms is NaN itself.  Every lane returns the sum.
__device__ __noinline__ float wgrad_exact(const WrArgs& a, int g, int i, int j, int col)
{
    const int lane = threadIdx.x & 31;
    const int c = a.chan_kind ? j / a.taps : col / a.taps, tap = col % a.taps;
    const int kw = tap % a.gr.KW, kh = (tap / a.gr.KW) % a.gr.KH, kt = tap / (a.gr.KW * a.gr.KH);
    const int shift = kt * a.gr.HWb + kh * a.gr.Wb + kw;
    const __nv_bfloat16* xc = a.xs + (size_t)g * a.xs_gstride + (size_t)(c >> 3) * a.gr.slots * 8 + (c & 7);
    const __nv_bfloat16* dc = a.dz + (size_t)g * a.dz_gstride + (size_t)(i >> 3) * a.gr.slots * 8 + (i & 7);
    const float* src = a.slices + wr_slice(a, g, i, j, col);
    float acc = 0.0f;  // of the lane's ranges and pixels
    for (int z0 = 0; z0 < a.w.Z; z0 += 32) {
        const float v = z0 + lane < a.w.Z ? __ldcg(src + (size_t)(z0 + lane) * a.w.slice) : 0.0f;
        uint32_t bad = __ballot_sync(0xffffffffu, v != v);
        if (v == v) acc += v;
        for (; bad; bad &= bad - 1) {
            const int z = z0 + __ffs(bad) - 1;
            const int end = min(a.w.tiles, (z + 1) * a.w.tps) * 128;
            float sum = 0.0f;
            for (int q0 = z * a.w.tps * 128; q0 < end; q0 += 128) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int q = q0 + 32 * k + lane;
                    int n, t, h, w;
                    grid_decode(a.gr, q, n, t, h, w);
                    if (n < a.gr.N && t < a.gr.OT && h < a.gr.OH && w < a.gr.OW)
                        sum += __bfloat162float(dc[(size_t)(q + a.gr.D0) * 8]) * __bfloat162float(xc[(size_t)(q + shift) * 8]);
                }
                if (__any_sync(0xffffffffu, sum != sum)) return __uint_as_float(0x7fffffffu);
            }
            acc += sum;
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// dW[f_i][col_j] = sum over the pixel ranges of their slices: LANES threads per two
// columns of four filters take every LANES-th range, then their sums are added in order
// (deterministic).  Block (bx, by, g): 64 / LANES packed columns, packed rows
// by*32 .. +31; the slices are read along the filters, 16 bytes a load.
// Bound by latency: what counts is loads in flight (8 of 16 bytes a thread, four ranges)
// and what is done before the wait.  A thread has work for all of them when the lanes
// follow the ranges: with 32 lanes whatever their number, 512 filters x 512 channels 3x3
// over 8 images of 7x7, one range, stood at 217 us of the backward's 256.
constexpr int kWrCols = 2;

template <int LANES>
__global__ void __launch_bounds__(256) k_grid_wreduce(const __grid_constant__ WrArgs a, const DbArgs d)
{
    __shared__ float s_v[64][33];  // [part of the ranges][column][filter]
    __shared__ int s_f[32];        // the rows' filters
    if ((int)blockIdx.z == d.groups) {  // the last layer of blocks: the bias gradient
        pdl_wait();
        pdl_trigger();
        db_blocks(d, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
        return;
    }
    // The plan's tables: k_grid_front read them too and has completed.
    constexpr int ncol = 32 * kWrCols / LANES;
    const int g = blockIdx.z, cnt = __ldg(a.counts + 2 * g);
    const int i0 = blockIdx.y * 32, j0 = blockIdx.x * ncol;
    if (i0 >= cnt) {  // still waits: with no kept filter at all these are the launch's only blocks
        pdl_wait();
        return;
    }
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    const int rl = ty & (LANES - 1), jt = ty / LANES * kWrCols;  // range lane, first column in the block
    const int iq = i0 + tx * 4;  // (a filter tile is a multiple of 16)
    const float* src[kWrCols];
#pragma unroll
    for (int e = 0; e < kWrCols; ++e) {
        const int j = j0 + jt + e;
        const int col = j < a.n_cols ? __ldg(a.colidx + j) : -1;
        src[e] = a.slices;  // (nothing reads what this adds up)
        if (col < 0 || iq >= cnt) continue;
        src[e] = a.slices + wr_slice(a, g, iq, j, col);
    }
    // the column of the entries this thread writes (ncol divides the block), their filters
    const int oe = threadIdx.x & (ncol - 1);
    const int ocol = j0 + oe < a.n_cols ? __ldg(a.colidx + j0 + oe) : -1;
    if (threadIdx.x < 32) s_f[threadIdx.x] = i0 + (int)threadIdx.x < cnt ? __ldg(a.rowmap + g * a.n_pad + i0 + threadIdx.x) : -1;
    pdl_wait();  // after the kernel before it in the stream, and the one before that (see launch_grid_bwd)
    pdl_trigger();
    float v[kWrCols][4];
#pragma unroll
    for (int e = 0; e < kWrCols; ++e)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[e][q] = 0.0f;
#pragma unroll 1
    for (int z = rl; z < a.w.Z; z += 4 * LANES) {
        float4 t[4][kWrCols];  // every load first
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const bool in = z + r * LANES < a.w.Z;
            const size_t at = (size_t)(z + r * LANES) * a.w.slice;
#pragma unroll
            for (int e = 0; e < kWrCols; ++e) {
                t[r][e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (in && dbg_in(src[e] + at + 3 - a.slices, a.w.Z * a.w.slice, a.status))
                    t[r][e] = __ldcs(reinterpret_cast<const float4*>(src[e] + at));
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int e = 0; e < kWrCols; ++e) {
                v[e][0] += t[r][e].x;
                v[e][1] += t[r][e].y;
                v[e][2] += t[r][e].z;
                v[e][3] += t[r][e].w;
            }
    }
    // the range lanes of a warp (four values of ty), then the warps in order
    constexpr int parts = LANES > 4 ? LANES / 4 : 1;
#pragma unroll
    for (int e = 0; e < kWrCols; ++e)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float p = __shfl_xor_sync(0xffffffffu, v[e][q], 8);
            if (LANES > 1) v[e][q] += p;
            const float p2 = __shfl_xor_sync(0xffffffffu, v[e][q], 16);
            if (LANES > 2) v[e][q] += p2;
            if ((rl & 3) == 0) s_v[(rl >> 2) * ncol + jt + e][tx * 4 + q] = v[e][q];
        }
    __syncthreads();
    for (int i = threadIdx.x / ncol; i < 32; i += 256 / ncol) {  // (a warp's lanes alike)
        const int of = ocol >= 0 ? s_f[i] : -1;
        float acc = 0.0f;
        if (of >= 0)
            for (int z = 0; z < parts; ++z) acc += s_v[z * ncol + oe][i];
        for (uint32_t bad = __ballot_sync(0xffffffffu, acc != acc); bad; bad &= bad - 1) {
            const int l = __ffs(bad) - 1;
            const float e = wgrad_exact(a, g, __shfl_sync(0xffffffffu, i0 + i, l), __shfl_sync(0xffffffffu, j0 + oe, l),
                                        __shfl_sync(0xffffffffu, ocol, l));
            if ((int)(threadIdx.x & 31) == l) acc = e;
        }
        if (of < 0) continue;
        if (!dbg_in((long long)of * a.K + ocol, a.dw_total, a.status)) continue;
        float* dst = a.dW + (long long)of * a.K + ocol;
        *dst = a.more ? *dst + acc : acc;
    }
}

struct DzArgs {
    Grid gr;
    const __nv_bfloat16* dy;
    const void* y;
    const int* rowmap;
    const int* counts;
    int n_pad, F, plane, chunks, cb;
    __nv_bfloat16* dz;  // NULL: the bias gradient alone
    float* part;        // [groups*n_pad][bx], or NULL
    int bx, by;         // blocks
    int slots;          // slots of a block
    long long y_total, dz_total;  // elements of dY, octets of the copy
    int* status;
};

// Grid copy of dZ and the bias gradient's partial sums.  Block (bx, by), 256 threads: slots
// bx*slots .. of chunk by % chunks (8 kept filters) of conv group by / chunks.
// Four slots a thread where that leaves kDzBlocks blocks, else two: the block's
// bias sums cost as much as a slot (AlexNet conv2's backward 164.5 -> 160.2 us; one
// slot a thread instead of two 170.7 -> 177.4).
constexpr int kDzBlocks = 1024;

// One pixel's dZ of a chunk's filters (nf of them, 8 when FULL): every load
// first, then the products, the running bias sums and the packed octet.
template <bool RELU, typename Y, bool FULL>
SADMM_DEV void dz_octet(const unsigned short* dp, const Y* yp, const YCheck& in, const int (&off)[8], int nf, float (&sum)[8],
                        uint32_t (&o)[4])
{
    uint32_t dyv[8];
    Y yv[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        dyv[e] = (FULL || e < nf) && y_ok(in, off[e]) ? (uint32_t)__ldg(dp + off[e]) : 0u;
        if (RELU) yv[e] = (FULL || e < nf) && y_ok(in, off[e]) ? __ldg(yp + off[e]) : Y(0);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        float v = __uint_as_float(dyv[e] << 16);
        if (RELU) {
            const float yf = sizeof(Y) == 2 ? __uint_as_float((uint32_t)yv[e] << 16) : (float)yv[e];
            v *= yf > 0.0f ? 1.0f : 0.0f;
        }
        sum[e] += v;
        // v is a bf16 value (or a NaN, whose upper half is one)
        const uint32_t u = __float_as_uint(v);
        o[e >> 1] = (e & 1) ? __byte_perm(o[e >> 1], u, 0x7610) : u >> 16;
    }
}

template <bool RELU, typename Y>
SADMM_DEV void dz_block(const DzArgs& a, int bx, int by, int* s_off, float (*s_part)[8])
{
    const int g = by / a.chunks, ck = by - g * a.chunks;
    const int cnt = __ldg(a.counts + 2 * g);
    if (ck * 8 >= (cnt + a.cb - 1) / a.cb * a.cb && ck * 8 >= cnt + 15) return;  // past every reader's last filter
    const int nf = min(8, cnt - ck * 8);  // kept filters of this chunk (they come first)
    if (threadIdx.x < 8 && (int)threadIdx.x < nf)
        s_off[threadIdx.x] = __ldg(a.rowmap + g * a.n_pad + ck * 8 + threadIdx.x) * a.plane;
    __syncthreads();
    int off[8];
    float sum[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        off[e] = e < nf ? s_off[e] : 0;
        sum[e] = 0.0f;
    }
#pragma unroll 1
    for (int k = 0; k < a.slots; k += 256) {
        const int s = bx * a.slots + k + threadIdx.x;
        if (s >= a.gr.slots) break;
        int n = 0, t = 0, h = 0, w = 0;
        const int q = s - a.gr.D0;
        if (q >= 0) grid_decode(a.gr, q, n, t, h, w);
        uint32_t o[4] = {0u, 0u, 0u, 0u};
        if (q >= 0 && n < a.gr.N && t < a.gr.OT && h < a.gr.OH && w < a.gr.OW) {
            // every load first (32-bit offsets from the image's pixel), then the products
            const long long base = (long long)n * a.F * a.plane + (t * a.gr.OH + h) * a.gr.OW + w;
            const unsigned short* dp = reinterpret_cast<const unsigned short*>(a.dy) + base;
            const Y* yp = static_cast<const Y*>(a.y) + base;
            const YCheck in{base, a.y_total, a.status};
            if (nf == 8) dz_octet<RELU, Y, true>(dp, yp, in, off, 8, sum, o);
            else dz_octet<RELU, Y, false>(dp, yp, in, off, nf, sum, o);
        }
        const size_t at = ((size_t)g * a.chunks + ck) * a.gr.slots + s;
        if (a.dz && dbg_in((long long)at, a.dz_total, a.status))
            reinterpret_cast<uint4*>(a.dz)[at] = make_uint4(o[0], o[1], o[2], o[3]);
    }
    if (!a.part) return;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        for (int o = 16; o > 0; o >>= 1) sum[e] += __shfl_down_sync(0xffffffffu, sum[e], o);
        if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5][e] = sum[e];
    }
    __syncthreads();
    const int i = ck * 8 + threadIdx.x;
    if (threadIdx.x < 8 && i < a.n_pad) {
        float r = 0.0f;
        for (int w = 0; w < 8; ++w) r += s_part[w][threadIdx.x];
        a.part[(size_t)(g * a.n_pad + i) * a.bx + bx] = r;
    }
}

struct PrepArgs {
    const __nv_bfloat16* wp;
    const int* colidx;
    const int* counts;
    int n_pad, k_pad, n_cols, taps, Cg, groups, nck, chan_kind;
    int rows, ncpad, bn, cb, ksteps;  // rows 0: no input gradient
    __nv_bfloat16* wd;
    int* colmap;
    int* zmap;
    int* counts2;
    float* zero;  // dW (or NULL)
    long long zero_n;
    int zblocks;  // blocks that zero it
};

// Block b of 256 threads, of rows*kPrepSplit + zblocks: below rows*kPrepSplit, a
// share of the K columns of one output column (input channel) of the input
// gradient's weights; the others zero dW.
constexpr int kPrepSplit = 2;

SADMM_DEV void prep_block(const PrepArgs& a, int b, int* s_j)
{
    if (b >= a.rows * kPrepSplit) {
        const long long nb = (long long)a.zblocks * 256;
        for (long long i = (long long)(b - a.rows * kPrepSplit) * 256 + threadIdx.x; i < a.zero_n; i += nb) a.zero[i] = 0.0f;
        return;
    }
    const int row = b / kPrepSplit, share = b - row * kPrepSplit;
    const int g = row / a.ncpad, jc = row - g * a.ncpad;
    const int cnt = __ldg(a.counts + 2 * g);
    int c = jc < a.nck ? jc : -1;
    if (c >= 0 && a.chan_kind) {
        const int col = __ldg(a.colidx + jc * a.taps);
        c = col >= 0 ? col / a.taps : -1;
    }
    if (threadIdx.x == 0 && share == 0) a.colmap[row] = c >= 0 ? g * a.Cg + c : -1;
    for (int t = threadIdx.x; t < a.taps; t += 256) {
        int j = -1;
        if (c >= 0) {
            const int want = c * a.taps + t;
            int lo = 0, hi = a.n_cols;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (__ldg(a.colidx + mid) < want) lo = mid + 1;
                else hi = mid;
            }
            if (lo < a.n_cols && __ldg(a.colidx + lo) == want) j = lo;
        }
        s_j[a.taps - 1 - t] = j;
    }
    __syncthreads();
    // [step][K half][bn][8] of this column's tile: a thread fills the 8 filters
    // of one half of a step
    const int nt = jc / a.bn, h8 = a.cb / 8;
    uint4* wd = reinterpret_cast<uint4*>(a.wd) + ((size_t)(row / a.bn) * a.ksteps * 2) * a.bn + (jc - nt * a.bn);
    const unsigned short* wp = reinterpret_cast<const unsigned short*>(a.wp) + (size_t)g * a.n_pad * a.k_pad;
    const int kuse = min(a.ksteps, (cnt + a.cb - 1) / a.cb * a.taps * (a.cb / 16)) * 2;  // what an item may load
    for (int k = share * 256 + threadIdx.x; k < kuse; k += kPrepSplit * 256) {
        int t = k / h8;
        const int c8 = k - t * h8;
        const int blk = t / a.taps;
        t -= blk * a.taps;  // kt * KH*KW + tap
        const int i = blk * a.cb + c8 * 8, j = s_j[t];
        uint32_t v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            v[e] = 0;
            if (i + e < cnt) {
                v[e] = j >= 0 ? __ldg(wp + (size_t)(i + e) * a.k_pad + j) : 0x8000u;
                if (j >= 0 && v[e] == 0x8000u) v[e] = 0;
            }
        }
        wd[(size_t)k * a.bn] = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
    }
    if (jc == 0 && share == 0) {
        // the group's output columns and the pruned channels' planes
        const bool none = a.chan_kind && (a.n_cols == 0 || __ldg(a.colidx) < 0);
        const int ncols = none ? 0 : a.nck;
        if (threadIdx.x == 0) {
            a.counts2[2 * g] = ncols;
            a.counts2[2 * g + 1] = a.Cg - ncols;
        }
        if (a.chan_kind)
            for (int ch = threadIdx.x; ch < a.Cg; ch += 256) {
                int lo = 0, hi = ncols;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (__ldg(a.colidx + mid * a.taps) / a.taps < ch) lo = mid + 1;
                    else hi = mid;
                }
                if (!(lo < ncols && __ldg(a.colidx + lo * a.taps) / a.taps == ch)) a.zmap[g * a.Cg + ch - lo] = g * a.Cg + ch;
            }
    }
}

// The copies and the input gradient's weights in one launch: blocks of dZ, then
// of x, then of the weights and dW's zeros.
struct FrontArgs {
    DzArgs dz;
    GridX x;
    PrepArgs prep;
    int ndz, nx, np;  // blocks of each
};

template <bool RELU, typename Y>
__global__ void __launch_bounds__(256) k_grid_front(const __grid_constant__ FrontArgs a)
{
    pdl_wait();  // after the kernel before it in the stream
    pdl_trigger();
    __shared__ int s_i[256];
    __shared__ float s_part[8][8];
    // The input gradient's weights first: a block of them is a chain of dependent
    // loads (its search of the columns), hidden beside the copies and not behind them
    // (AlexNet conv3's backward 51.0 -> 49.5 us, the ResNet-50 3x3 layer's 47.7 -> 45.4).
    int b = blockIdx.x;
    if (b < a.np) {
        prep_block(a.prep, b, s_i);
        return;
    }
    b -= a.np;
    if (b < a.ndz)
        dz_block<RELU, Y>(a.dz, b % a.dz.bx, b / a.dz.bx, s_i, s_part);
    else
        grid_x_block(a.x, (b - a.ndz) % a.x.bx, (b - a.ndz) / a.x.bx, s_i);
}

struct GridBwd {
    int images;   // of a pass
    Grid gr;
    GridConvShape cs;
    WgradShape ws;
    int nck;      // channels of x per group that hold a kept column
    int dchunks;  // 8-filter chunks of dZ per group
    int dzslots;  // slots of a block of the dZ copy
    int nparts;   // its blocks along the slots
    size_t off_xs, off_dz, off_wd, off_maps, off_slices, off_part, total;
};

// One pass over the images of g.
bool grid_bwd_pass(const sadmm_plan* plan, const Geometry& g, GridBwd* out)
{
    GridBwd b;
    b.images = (int)g.n;
    if (plan->n_cols < 1 || plan->n_filt < 1 || g.taps > 256) return false;
    if (!grid_of(g, &b.gr)) return false;
    b.nck = plan->colkind == SADMM_COL_CHANNEL ? plan->n_colgroups : (int)g.cg;
    const int per = (int)((plan->n_filt + g.groups - 1) / g.groups);
    if (!grid_conv_shape(b.gr, plan->n_pad, b.nck, b.nck, (int)g.groups, (int)kGwCtas, kDxStage, dx_seg(per), true,
                         &b.cs)) return false;
    if (!wgrad_shape(b.gr, b.nck, plan->n_pad, per, (int)g.groups, &b.ws)) return false;
    b.dchunks = std::max(b.cs.k16 * 2, b.ws.nft * b.ws.nst / 8);
    b.dzslots = b.gr.slots / 1024 * g.groups * b.dchunks >= kDzBlocks ? 1024 : 512;
    b.nparts = (b.gr.slots + b.dzslots - 1) / b.dzslots;
    if ((long long)b.nparts * g.groups * b.dchunks + (b.gr.slots / 256 + 1) * g.groups * ((b.ws.nch + 1) / 2) +
            2 * g.groups * b.cs.npad + 256 >= (1ll << 31) ||
        g.groups * ((b.ws.nch + 1) / 2) > 65535)
        return false;
    size_t off = 0;
    auto take = [&off](long long bytes) {
        const size_t at = off;
        off += (size_t)round_up(bytes, 1024);
        return at;
    };
    b.off_xs = take(g.groups * b.ws.nch * (long long)b.gr.slots * 16);
    b.off_dz = take(g.groups * b.dchunks * (long long)b.gr.slots * 16);
    b.off_wd = take(g.groups * b.cs.npad * (long long)b.cs.ksteps * 32);
    b.off_maps = take((g.groups * b.cs.npad + g.c + 2 * g.groups) * 4);
    b.off_slices = take(b.ws.Z * b.ws.slice * 4);
    b.off_part = take(g.groups * plan->n_pad * (long long)b.nparts * 4);
    b.total = off;
    *out = b;
    return true;
}

// The layer in as few passes over equal shares of its images as keep the workspace
// within `cap` bytes; false when one image does not.
bool grid_bwd_shape(const sadmm_plan* plan, const Geometry& g, size_t cap, GridBwd* out)
{
    Geometry p = g;
    for (long long passes = 1;;) {
        p.n = (g.n + passes - 1) / passes;
        p.m = p.n * p.plane;
        const bool fits = grid_bwd_pass(plan, p, out);
        if (fits && out->total <= cap) return true;
        if (p.n == 1) return false;
        // the workspace is about proportional to the images; at least one image fewer
        const long long next = fits ? (long long)((double)passes * out->total / cap) : 2 * passes;
        passes = std::min(g.n, std::max(next, (g.n + p.n - 2) / (p.n - 1)));
    }
}

}  // namespace

// The estimate, fitted with the chunked path's (bwd.cu): launches, the two contractions'
// cycles at 1.95 GHz, and the copies; 0.8 to 1.15 of what 96 layers measured that take
// more than a third of the chunked path's time, less of the others.
size_t grid_bwd_bytes(const sadmm_plan* plan, const Geometry& g, size_t cap, long long* ns)
{
    GridBwd b;
    if (!grid_bwd_shape(plan, g, cap, &b)) return 0;
    const long long copies = 16ll * g.groups * b.gr.slots * (b.ws.nch + b.dchunks);
    *ns = (g.n + b.images - 1) / b.images * (16000 + (b.ws.cycles + b.cs.cycles * 5 / 4) * 100 / 195 + copies / 2000);
    return b.total;
}

// The images of g, a pass's or the last fewer, in b's workspace; `more`: dW and db add
// to what the passes before left.
static sadmm_status launch_pass(const sadmm_plan* plan, const Geometry& g, const GridBwd& b, const void* x, const void* dy,
                                const void* y, int ydt, int relu, float* dW, float* db, float* dx, void* ws, bool more,
                                cudaStream_t s)
{
    const char* base = static_cast<const char*>(plan->dev);
    char* w = static_cast<char*>(ws);
    const int* rowmap = reinterpret_cast<const int*>(base + plan->off_rowmap);
    const int* zeromap = reinterpret_cast<const int*>(base + plan->off_zeromap);
    const int* counts = reinterpret_cast<const int*>(base + plan->off_counts);
    const int* colidx = reinterpret_cast<const int*>(base + plan->off_colidx);
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(w + b.off_xs);
    __nv_bfloat16* dz = reinterpret_cast<__nv_bfloat16*>(w + b.off_dz);
    __nv_bfloat16* wd = reinterpret_cast<__nv_bfloat16*>(w + b.off_wd);
    int* colmap = reinterpret_cast<int*>(w + b.off_maps);
    int* zmap = colmap + g.groups * b.cs.npad;
    int* counts2 = zmap + g.c;
    float* slices = reinterpret_cast<float*>(w + b.off_slices);
    float* part = reinterpret_cast<float*>(w + b.off_part);
    const int chan_kind = plan->colkind == SADMM_COL_CHANNEL ? 1 : 0;
    const int* chans = chan_kind ? colidx : nullptr;
    const long long xs_g = (long long)b.ws.nch * b.gr.slots * 8, dz_g = (long long)b.dchunks * b.gr.slots * 8;

    FrontArgs fa;
    memset(&fa, 0, sizeof(fa));
    if (dW || dx) {
        PrepArgs& p = fa.prep;
        p.wp = reinterpret_cast<const __nv_bfloat16*>(base + plan->off_wp);
        p.colidx = colidx;
        p.counts = counts;
        p.n_pad = plan->n_pad;
        p.k_pad = plan->k_pad;
        p.n_cols = plan->n_cols;
        p.taps = (int)g.taps;
        p.Cg = (int)g.cg;
        p.groups = (int)g.groups;
        p.nck = b.nck;
        p.chan_kind = chan_kind;
        p.ncpad = b.cs.npad;
        p.rows = dx && !more ? (int)g.groups * b.cs.npad : 0;  // (they stay for the passes after the first)
        p.bn = b.cs.bn;
        p.cb = b.cs.cb;
        p.ksteps = b.cs.ksteps;
        p.wd = wd;
        p.colmap = colmap;
        p.zmap = zmap;
        p.counts2 = counts2;
        p.zero = dW;
        p.zero_n = dW && !more ? g.f * g.k : 0;
        p.zblocks = p.zero_n > 0 ? (int)std::min<long long>(256, (p.zero_n + 2047) / 2048) : 0;
        fa.np = p.rows * kPrepSplit + p.zblocks;
    }
    DzArgs& d = fa.dz;
    d.gr = b.gr;
    d.dy = static_cast<const __nv_bfloat16*>(dy);
    d.y = y;
    d.rowmap = rowmap;
    d.counts = counts;
    d.n_pad = plan->n_pad;
    d.F = (int)g.f;
    d.plane = (int)g.plane;
    d.chunks = b.dchunks;
    d.cb = b.cs.cb;
    d.dz = (dW || dx) ? dz : nullptr;
    d.part = db ? part : nullptr;
    d.bx = b.nparts;
    d.slots = b.dzslots;
    d.y_total = g.n * g.f * g.plane;
    d.dz_total = g.groups * b.dchunks * (long long)b.gr.slots;
    d.status = device_status_ptr();
    d.by = (int)(g.groups * b.dchunks);
    fa.ndz = d.bx * d.by;
    if (dW) {
        if (!grid_x_args(b.gr, g, x, chans, b.nck, b.ws.nch, xs, &fa.x)) return SADMM_EUNSUPPORTED;
        fa.nx = fa.x.bx * fa.x.by;
    }
    const dim3 fgrid((unsigned)(fa.ndz + fa.nx + fa.np));
    const cudaError_t fe =
        !relu ? launch_pdl(k_grid_front<false, float>, fgrid, dim3(256), 0, s, fa)
              : (ydt == SADMM_BF16 ? launch_pdl(k_grid_front<true, unsigned short>, fgrid, dim3(256), 0, s, fa)
                                   : launch_pdl(k_grid_front<true, float>, fgrid, dim3(256), 0, s, fa));
    if (fe != cudaSuccess) return SADMM_ECUDA;
    DbArgs dd;
    memset(&dd, 0, sizeof(dd));
    dd.part = part;
    dd.rowmap = rowmap;
    dd.zeromap = zeromap;
    dd.counts = counts;
    dd.nparts = b.nparts;
    dd.groups = (int)g.groups;
    dd.n_pad = plan->n_pad;
    dd.Fg = (int)g.fg;
    dd.db = db;
    dd.F = (int)g.f;
    dd.status = device_status_ptr();
    dd.more = more ? 1 : 0;
    if (db && !dW &&
        launch_pdl(k_grid_db, dim3((unsigned)((g.groups * plan->n_pad + 7) / 8)), dim3(256), 0, s, dd) != cudaSuccess)
        return SADMM_ECUDA;
    WrArgs r;
    if (dW) {
        GwArgs a;
        memset(&a, 0, sizeof(a));
        a.gr = b.gr;
        a.w = b.ws;
        a.xs = xs;
        a.dz = dz;
        a.xs_gstride = xs_g;
        a.dz_gstride = dz_g;
        a.counts = counts;
        a.colidx = plan->colkind == SADMM_COL_SHAPE ? colidx : nullptr;
        a.nck = b.nck;
        a.n_cols = plan->n_cols;
        a.taps = (int)g.taps;
        a.slices = slices;
        a.groups = (int)g.groups;
        a.units = b.ws.types * b.ws.Z;
        a.types_div = make_fastdiv((uint32_t)b.ws.types);
        a.status = device_status_ptr();
        static int configured_dev = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (configured_dev != dev) {
            if (cudaFuncSetAttribute(k_grid_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, kGwSmemLimit) != cudaSuccess)
                return SADMM_ECUDA;
            configured_dev = dev;
        }
        const int grid = std::min(a.units, device_sm_count());
        if (launch_pdl(k_grid_wgrad, dim3((unsigned)grid), dim3(kGwThreads), (size_t)kGwSmemLimit, s, a) != cudaSuccess)
            return SADMM_ECUDA;
        memset(&r, 0, sizeof(r));
        r.gr = b.gr;
        r.w = b.ws;
        r.slices = slices;
        r.rowmap = rowmap;
        r.colidx = colidx;
        r.counts = counts;
        r.xs = xs;
        r.dz = dz;
        r.xs_gstride = xs_g;
        r.dz_gstride = dz_g;
        r.dW = dW;
        r.n_pad = plan->n_pad;
        r.n_cols = plan->n_cols;
        r.taps = (int)g.taps;
        r.chan_kind = chan_kind;
        r.more = more ? 1 : 0;
        r.K = g.k;
        r.dw_total = g.f * g.k;
        r.status = device_status_ptr();
    }
    // The input gradient reads what k_grid_front wrote and nothing of k_grid_wgrad's.
    // Every CTA of k_grid_wgrad lets it start only after its own wait for
    // k_grid_front, so it does not wait first: its CTAs take the SMs as the weight
    // gradient's leave them (its two rounds of items end unevenly: AlexNet conv2 at
    // batch 128 189 -> 176 us, conv3 59.2 -> 55.1, a ResNet-50 3x3 layer at batch 64
    // 61.1 -> 58.4).  It waits for k_grid_wgrad at its end, for the reduction behind
    // it.  (The reduction between the two, beside the input gradient's start: 185, 55
    // and 58 us.)
    if (dx) {
        GridConvCall c;
        memset(&c, 0, sizeof(c));
        c.src = dz;
        c.chunks = b.dchunks;
        c.wd = wd;
        c.out = dx;
        c.colmap = colmap;
        c.cstride = b.cs.npad;
        c.zmap = zmap;
        c.zstride = (int)g.cg;
        c.counts = counts2;
        c.kcounts = counts;
        c.groups = (int)g.groups;
        c.planes = (int)g.c;
        c.VT = (int)g.t;
        c.VH = (int)g.h;
        c.VW = (int)g.w;
        c.out_total = g.n * g.c * g.t * g.h * g.w;
        c.src_dz = 1;
        c.late_wait = dW != nullptr;  // (k_grid_wgrad stands between)
        const sadmm_status st = launch_grid_conv(b.gr, b.cs, c, s);
        if (st != SADMM_OK) return st;
    }
    if (dW) {
        // As many range lanes as give each four ranges, or more while there are fewer
        // than two blocks an SM (idle lanes cost nothing then: with one range and lanes
        // for it alone, 2 images of 8x8 with 16 channels took 14.1 us, not 11.7).
        const long long rows = (plan->n_pad + 31) / 32 * g.groups;
        auto xblocks = [&](int lanes) { return (plan->n_cols * lanes + 32 * kWrCols - 1) / (32 * kWrCols); };
        int lanes = 1;
        while (lanes < 32 && (lanes * 4 < b.ws.Z || xblocks(lanes) * rows < 2 * kGwCtas)) lanes *= 2;
        const dim3 wgrid((unsigned)xblocks(lanes), (unsigned)((plan->n_pad + 31) / 32), (unsigned)g.groups + (db ? 1u : 0u));
        const auto kern = lanes == 1   ? k_grid_wreduce<1>
                          : lanes == 2 ? k_grid_wreduce<2>
                          : lanes == 4 ? k_grid_wreduce<4>
                          : lanes == 8 ? k_grid_wreduce<8>
                          : lanes == 16 ? k_grid_wreduce<16>
                                        : k_grid_wreduce<32>;
        if (launch_pdl(kern, wgrid, dim3(256), 0, s, r, dd) != cudaSuccess) return SADMM_ECUDA;
    }
    return cudaGetLastError() == cudaSuccess ? SADMM_OK : SADMM_ECUDA;
}

sadmm_status launch_grid_bwd(const sadmm_plan* plan, const Geometry& g, size_t cap, const void* x, const void* dy,
                             const void* y, int ydt, int relu, float* dW, float* db, float* dx, void* ws, cudaStream_t s)
{
    GridBwd b;
    if (!grid_bwd_shape(plan, g, cap, &b)) return SADMM_EINVAL;
    Geometry p = g;
    const long long xn = g.c * g.t * g.h * g.w, yn = g.f * g.plane;  // elements of an image
    for (long long n0 = 0; n0 < g.n; n0 += b.images) {
        p.n = std::min<long long>(b.images, g.n - n0);
        p.m = p.n * p.plane;
        if (p.n < b.images) {  // the last pass: fewer pixels, and ranges, in the same layout
            if (!grid_of(p, &b.gr)) return SADMM_EINVAL;
            b.ws.tiles = (b.gr.L + 127) / 128;
            b.ws.Z = (b.ws.tiles + b.ws.tps - 1) / b.ws.tps;
            b.nparts = (b.gr.slots + b.dzslots - 1) / b.dzslots;
        }
        const char* yp = static_cast<const char*>(y);
        const sadmm_status st =
            launch_pass(plan, p, b, static_cast<const __nv_bfloat16*>(x) + n0 * xn,
                        static_cast<const __nv_bfloat16*>(dy) + n0 * yn,
                        yp ? yp + n0 * yn * (ydt == SADMM_BF16 ? 2 : 4) : nullptr, ydt, relu, dW, db,
                        dx ? dx + n0 * xn : nullptr, ws, n0 > 0, s);
        if (st != SADMM_OK) return st;
    }
    return SADMM_OK;
}

}  // namespace sadmm
