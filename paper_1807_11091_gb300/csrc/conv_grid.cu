// conv_grid.cu -- stride-1 convolution as a slab GEMM on the tensor cores: the
// forward of a pruned layer (Sec. 3) and its input gradient (the forward with
// the taps flipped, over the kept filters; Sec. 4, masked retraining).
//
// GEMM row i of tile t is grid pixel 128t + i of the padded line (grid.cuh);
// every tap of a block of CB channels is the same shared-memory slab of
// 128*MT + maxshift slots, shifted: a K-major no-swizzle operand whose start
// moves by 16 bytes a slot.  So x is read about once per tile instead of once
// per tap, no element is gathered by a thread, and no thread touches the A
// operand: bulk copies bring the slabs, TMA the weights, one warp issues.
// Pruned columns cost tensor time (their weights are zero) but no traffic: at
// a quarter of the columns the 128 x 96 x 16 MMA of four times the steps is
// still shorter than gathering the kept ones 2 bytes at a time.
//
//   warp 0       slabs: CB/8 bulk copies per stage
//   warp 1       TMEM allocator, MMA issuer
//   warp 2       weights: resident, or a ring of a few MMA steps per slot
//   warps 3-10   epilogue: every segment (about `seg` MMA steps: whole stages, or
//                kernel rows of one) the accumulator is read from TMEM and added to
//                fp32 registers
//                (the tensor core truncates when it accumulates, about 1e-8 of
//                the result per step; short chains keep that below 5e-7), the
//                other TMEM buffers meanwhile taking the next stages; after the
//                last, bias, ReLU and coalesced stores (lane = pixel).
// A 0 * inf of a pruned weight would put a NaN where the kept sum has none:
// pruned entries are stored as -0.0 and an output that comes out NaN is summed
// again over the kept entries alone (grid_exact).
#include <string.h>

#include <algorithm>

#include "grid.cuh"

namespace sadmm {

namespace {

constexpr int kGcWarps = 11;
constexpr int kGcThreads = kGcWarps * 32;
constexpr int kGcEpiWarps = 8;
constexpr int kGcMaxA = 4, kGcMaxB = 8, kGcMaxBuf = 4;
constexpr int kGcTables = 2 * 256 * 4;
constexpr int kGcZcap = 1024;
constexpr int kGcBars = 512;
constexpr int kGcSmemLimit = 232448;

struct GcArgs {
    Grid gr;
    const __nv_bfloat16* src;
    const __nv_bfloat16* wd;
    void* out;
    const float* bias;
    const int* colmap;
    const int* zmap;
    const int* counts;
    const int* kcounts;
    int* status;
    long long out_total;
    long long gstride;  // source elements per group
    int late_wait;
    int src_dz;
    int zstride, groups, planes, plane, VT, VH, VW, VHW;
    int units, mtiles, ntiles;
    FastDiv mt_div, nt_div;
    int bn, ksteps;
    int cb, ncb, spt;   // channels per block, blocks (static), MMA steps per stage
    int h16, rsteps;    // 16-channel steps per tap, MMA steps per kernel row (a slot of the weight ring)
    int sp;             // slots of a slab
    // Accumulation segments: pps stages each or, where a stage is longer than a
    // segment (cut), pps pieces of psteps MMA steps of its kernel rows; ppst pieces
    // a stage (1 without cut).
    int cut, psteps, pps, ppst;
    int nbuf;  // accumulator buffers
    int cap_b, stages_a, a_bytes, a_stride;
    int cstride;
    int tmem_stride, tmem_cols;
    int relu;
};

// ---- outputs that come out NaN, summed again ----
// Their K columns lie in octets u: 8 channels of a tap, in the weights' order.
SADMM_DEV int gc_octets(const GcArgs& a, int kch)
{
    return (kch + a.cb - 1) / a.cb * a.gr.KT * a.gr.KH * a.gr.KW * (a.cb / 8);
}

// The kept terms (pruned entries are -0.0) of octet u of one output of grid pixel q:
// column `col` of the tile whose weights lie at wt, bnr rows apart.  Where the source is
// the output gradient, a tap that reads past the output's edge is no term; in the forward
// a padded pixel is one, as it is in the gathered path.
SADMM_DEV float gc_terms(const GcArgs& a, const uint4* wt, const uint4* src, int bnr, int col, int u, int q, int kch)
{
    const int per = a.cb / 8, t = u / per, taps = a.gr.KT * a.gr.KH * a.gr.KW;
    const int blk = t / taps, tap = t - blk * taps, kw = tap % a.gr.KW, r = tap / a.gr.KW;
    const int c = blk * a.cb + (u - t * per) * 8;
    const int slot = q + r / a.gr.KH * a.gr.HWb + r % a.gr.KH * a.gr.Wb + kw;
    if (c >= kch) return 0.0f;
    const uint4 w4 = __ldg(wt + (size_t)u * bnr + col), x4 = src[(size_t)(c >> 3) * a.gr.slots + slot];
    const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w}, x[4] = {x4.x, x4.y, x4.z, x4.w};
    float sum = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const uint32_t wb = (e & 1) ? w[e >> 1] & 0xffff0000u : w[e >> 1] << 16;
        const uint32_t xb = (e & 1) ? x[e >> 1] & 0xffff0000u : x[e >> 1] << 16;
        if (wb != 0x80000000u && c + e < kch) sum += __uint_as_float(wb) * __uint_as_float(xb);
    }
    if (sum != sum && a.src_dz) {
        int n = a.gr.N, t0 = 0, y0 = 0, x0 = 0;
        if (slot >= a.gr.D0) grid_decode(a.gr, slot - a.gr.D0, n, t0, y0, x0);
        if (n >= a.gr.N || t0 >= a.gr.OT || y0 >= a.gr.OH || x0 >= a.gr.OW) return 0.0f;
    }
    return sum;
}

// The first octets of grid pixel q, of four taps at most, whose source holds an infinity
// or a NaN (-1: no more): where a NaN of any of its outputs that is a kept term's shows
// first.  (One a tap: what is pruned is pruned for every filter.)
__device__ __noinline__ int4 grid_scan(const GcArgs& a, const uint4* src, int q, int kch)
{
    int4 f = make_int4(-1, -1, -1, -1);
    int u = 0;
    for (int c0 = 0; c0 < kch; c0 += a.cb)
        for (int kt = 0; kt < a.gr.KT; ++kt)
            for (int kh = 0; kh < a.gr.KH; ++kh)
                for (int kw = 0; kw < a.gr.KW; ++kw) {
                    const uint4* p = src + (size_t)(c0 >> 3) * a.gr.slots + (q + kt * a.gr.HWb + kh * a.gr.Wb + kw);
                    bool found = false;
                    for (int c8 = 0; c8 < a.cb / 8; ++c8, ++u, p += a.gr.slots) {
                        if (found) continue;
                        const uint4 x = *p;
                        bool bad = false;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t v = e == 0 ? x.x : e == 1 ? x.y : e == 2 ? x.z : x.w;
                            bad |= (v & 0x7f80u) == 0x7f80u || (v & 0x7f800000u) == 0x7f800000u;
                        }
                        if (!bad) continue;
                        found = true;
                        if (f.x < 0) f.x = u;
                        else if (f.y < 0) f.y = u;
                        else if (f.z < 0) f.z = u;
                        else {
                            f.w = u;
                            return f;
                        }
                    }
                }
    return f;
}

// Whether a kept term of the octets f is NaN: the output is then.
__device__ __noinline__ bool grid_nan_at(const GcArgs& a, const uint4* wt, const uint4* src, int bnr, int col, int q, int kch,
                                         int4 f)
{
    bool nan = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int u = k == 0 ? f.x : k == 1 ? f.y : k == 2 ? f.z : f.w;
        if (nan || u < 0) continue;
        const float t = gc_terms(a, wt, src, bnr, col, u, q, kch);
        nan = t != t;
    }
    return nan;
}

// The sum of one output over the kept K columns only, as the gathered path forms it, by a
// warp; every lane returns it.  NaN as soon as a term is.
__device__ __noinline__ float grid_exact(const GcArgs& a, const uint4* wt, const uint4* src, int bnr, int col, int q, int kch)
{
    const int units = gc_octets(a, kch), lane = threadIdx.x & 31;
    float acc = 0.0f;
    for (int u0 = 0; u0 < units; u0 += 64) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (u0 + 32 * k + lane < units) acc += gc_terms(a, wt, src, bnr, col, u0 + 32 * k + lane, q, kch);
        if (__any_sync(0xffffffffu, acc != acc)) return __uint_as_float(0x7fffffffu);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// Channel blocks a group's items contract over.
SADMM_DEV int gc_blocks(const GcArgs& a, int g)
{
    return a.kcounts ? min(a.ncb, (__ldg(a.kcounts + 2 * g) + a.cb - 1) / a.cb) : a.ncb;
}

// Work item u: pixel tile (fastest), column tile, group.
SADMM_DEV void gc_unit(const GcArgs& a, int u, int& g, int& nt, int& mt)
{
    const int t = (int)fdiv((uint32_t)u, a.mt_div);
    mt = u - t * a.mtiles;
    g = (int)fdiv((uint32_t)t, a.nt_div);
    nt = t - g * a.ntiles;
}

template <bool OUT_BF16>
SADMM_DEV void zero_at(float* yf, __nv_bfloat16* yh, const YCheck& yc, int off)
{
    if (!y_ok(yc, off)) return;
    if (OUT_BF16)
        yh[off] = __float2bfloat16_rn(0.0f);
    else
        __stcs(yf + off, 0.0f);
}

// Where an item's weights come from: shared memory for the whole group, a ring
// slot per stage, or one per kernel row where two stages of them do not fit.
enum { kResident, kStageSlots, kRowSlots };

// The barriers and operand bases of a CTA, for its issuing warp.
struct GcPipe {
    uint64_t *full_a, *empty_a, *full_b, *empty_b, *acc_full, *acc_empty, *b_full, *b_empty;
    volatile int* abort_flag;
    uint32_t sA, sB, tmem_base;
    int stages_b, bnr;
};

// The kernel rows gc_issue is instantiated for: KW taps of h16 16-channel steps, at
// most 14 MMAs.
inline bool unrolled_row(int kw, int h16)
{
    if (kw == 1 || kw == 3) return h16 <= 4;
    if (kw == 5 || kw == 7) return h16 <= 2;
    return h16 == 1 && (kw == 4 || kw == 6 || kw == 9 || kw == 11);
}

// The issuing warp's run over its work items.  The whole warp runs the loop,
// every branch on a parameter or a vote, and one elected lane issues.  KW taps
// of H steps of 16 channels make a kernel row, unrolled: an MMA then issues in
// the 48 cycles that a 128 x 64 x 16 takes (71 with the offsets read from a
// table in the parameters, 103 with the row chosen by a switch inside the loop,
// 120 and more with bounds the compiler cannot prove uniform).  KW = 0: any
// other row, one MMA at a time.
template <int KW, int H, int MT, bool CUT>
SADMM_DEV void gc_issue(const GcArgs& a, const GcPipe& p, const int mode)
{
    const bool resident = mode == kResident;
    int s = 0, sb = 0, ab = 0;
    uint32_t ph = 0, phb = 0, acc_ph = 0, bf_ph = 0;
    int cur = -1;
    bool ok = true;
    const uint64_t ad0 = sdesc_kmajor_none(p.sA, (uint32_t)a.sp * 16u, 128u);
    const uint64_t bd0 = sdesc_kmajor_none(p.sB, (uint32_t)p.bnr * 16u, 128u);
    const uint64_t ahi = ad0 & 0xffffffff00000000ull, bhi = bd0 & 0xffffffff00000000ull;
    const uint32_t alo0 = (uint32_t)ad0, blo0 = (uint32_t)bd0;
    const uint32_t bs16 = (uint32_t)p.bnr * 2u;   // one step of the weights, in 16-byte units
    const uint32_t half = 2u * (uint32_t)a.sp;   // 16 channels of a slab
    for (int u = blockIdx.x; ok && u < a.units; u += gridDim.x) {
        int g, nt, mt;
        gc_unit(a, u, g, nt, mt);
        const int cnt = min(a.bn, __ldg(a.counts + 2 * g) - nt * a.bn);
        const int nst = gc_blocks(a, g) * a.gr.KT;
        if (uniform(cnt <= 0 || nst == 0)) continue;
        const uint32_t idesc = idesc_bf16_f32(128, (cnt + 15) & ~15);
        if (resident && g != cur) {
            if (cur >= 0) mma_commit_elect(p.b_empty);  // the old weights are free once these MMAs finish
            if (!mbar_wait_warp(p.b_full, bf_ph, p.abort_flag, a.status)) break;
            bf_ph ^= 1u;
            cur = g;
        }
        uint32_t d = 0, blo = blo0;
        int in_seg = 0;  // stages (CUT: pieces) of the segment so far
        for (int st = 0; st < a.ncb * a.gr.KT; ++st) {
            if (uniform(st >= nst)) break;
            const bool last = uniform(st + 1 == nst);
            if (!CUT && in_seg == 0) {
                if (!mbar_wait_warp(&p.acc_empty[ab], acc_ph ^ 1u, p.abort_flag, a.status)) { ok = false; break; }
                d = p.tmem_base + (uint32_t)(ab * MT * a.tmem_stride);
            }
            if (!mbar_wait_warp(&p.full_a[s], ph, p.abort_flag, a.status)) { ok = false; break; }
            tc_fence_after();
            uint32_t ar = alo0 + ((uint32_t)(s * a.a_stride) >> 4);
            for (int kh = 0; kh < a.gr.KH; ++kh) {
                if (mode == kRowSlots || (mode == kStageSlots && kh == 0)) {
                    if (!mbar_wait_warp(&p.full_b[sb], phb, p.abort_flag, a.status)) { ok = false; break; }
                    tc_fence_after();
                    blo = blo0 + (uint32_t)(sb * (mode == kRowSlots ? a.rsteps : a.spt)) * bs16;
                }
                // CUT: a segment ends at a piece of the kernel row (the row itself when it is unrolled)
                for (int i0 = 0; i0 < (CUT && KW == 0 ? a.rsteps : 1); i0 += (CUT && KW == 0 ? a.psteps : 1)) {
                    if (CUT && in_seg == 0) {
                        if (!mbar_wait_warp(&p.acc_empty[ab], acc_ph ^ 1u, p.abort_flag, a.status)) { ok = false; break; }
                        tc_fence_after();
                        d = p.tmem_base + (uint32_t)(ab * MT * a.tmem_stride);
                    }
                    const uint32_t acc = (in_seg > 0 || (!CUT && kh > 0)) ? 1u : 0u;
                    if (KW > 0) {
#pragma unroll
                        for (int kw = 0; kw < KW; ++kw)
#pragma unroll
                            for (int j = 0; j < H; ++j) {
                                const uint32_t al = ar + kw + j * half, bl = blo + (kw * H + j) * bs16;
                                const uint32_t ac = (kw || j) ? 1u : acc;
                                mma_bf16_ss_elect(d, ahi | al, bhi | bl, idesc, ac);
                                if (MT == 2) mma_bf16_ss_elect(d + (uint32_t)a.tmem_stride, ahi | (al + 128u), bhi | bl, idesc, ac);
                            }
                    } else {
                        const int end = CUT ? min(i0 + a.psteps, a.rsteps) : a.rsteps;
                        for (int i = i0; i < end; ++i) {
                            const int kw = i / a.h16;
                            const uint32_t al = ar + kw + (i - kw * a.h16) * half, bl = blo + i * bs16;
                            const uint32_t ac = i > i0 ? 1u : acc;
                            mma_bf16_ss_elect(d, ahi | al, bhi | bl, idesc, ac);
                            if (MT == 2) mma_bf16_ss_elect(d + (uint32_t)a.tmem_stride, ahi | (al + 128u), bhi | bl, idesc, ac);
                        }
                    }
                    if (CUT && (++in_seg == a.pps || (last && kh + 1 == a.gr.KH && (KW > 0 || i0 + a.psteps >= a.rsteps)))) {
                        mma_commit_elect(&p.acc_full[ab]);
                        if (++ab == a.nbuf) { ab = 0; acc_ph ^= 1u; }
                        in_seg = 0;
                    }
                }
                if (CUT && !ok) break;
                ar += (uint32_t)a.gr.Wb;
                blo += (uint32_t)a.rsteps * bs16;
                if (mode == kRowSlots) {
                    mma_commit_elect(&p.empty_b[sb]);
                    if (++sb == p.stages_b) { sb = 0; phb ^= 1u; }
                }
            }
            if (!ok) break;
            if (mode == kStageSlots) {
                mma_commit_elect(&p.empty_b[sb]);
                if (++sb == p.stages_b) { sb = 0; phb ^= 1u; }
            }
            mma_commit_elect(&p.empty_a[s]);
            if (++s == a.stages_a) { s = 0; ph ^= 1u; }
            if (!CUT && (++in_seg == a.pps || last)) {
                mma_commit_elect(&p.acc_full[ab]);
                if (++ab == a.nbuf) { ab = 0; acc_ph ^= 1u; }
                in_seg = 0;
            }
        }
    }
}

// What the epilogue warps share.
struct GcEpi {
    uint64_t* acc_full;  // then acc_empty
    volatile int* abort_flag;
    int* t_off;          // [256], then t_bias [256], z_off [kGcZcap]
    uint32_t tmem_base;
    int bnr;
};

// The epilogue warps' run over the work items; a warp holds NCH chunks of 16 columns.
// With four, a segment's loads leave TMEM together: one by one each takes about 125
// cycles (AlexNet conv2's backward 162.5 -> 160.7 us, conv3's 53.0 -> 52.0, a 1x1 layer's
// of 256 channels and 64 filters at 56x56 164 -> 154).  Eight leave no registers for that (two in flight spilled 80 bytes and AlexNet
// conv2's forward took 60 us instead of 52), and both forms in the forward's kernel cost
// it 1 %, so the input gradient, whose segments are the short ones, has its own.
template <bool OUT_BF16, int MT, int NCH>
SADMM_DEV void gc_epilogue(const GcArgs& a, const GcEpi& ep)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int* t_off = ep.t_off;
    float* t_bias = reinterpret_cast<float*>(t_off + 256);
    int* z_off = t_off + 512;
    // Two warps per TMEM lane quadrant: with one pixel tile they take its
    // 16-column chunks in turn, with two a tile each.
    const int q4 = warp & 3;
    const int h = (warp - 3) >> 2;
    const int et = threadIdx.x - 3 * 32;
    int ab = 0, key = -1;
    uint32_t acc_ph = 0;
    bool alive = true;
    for (int u = blockIdx.x; u < a.units; u += gridDim.x) {
        int g, nt, mt;
        gc_unit(a, u, g, nt, mt);
        const int cnt = min(a.bn, __ldg(a.counts + 2 * g) - nt * a.bn);
        const int zc = nt == 0 ? __ldg(a.counts + 2 * g + 1) : 0;
        if (g * a.ntiles + nt != key) {
            key = g * a.ntiles + nt;
            asm volatile("bar.sync 1, %0;" ::"n"(kGcEpiWarps * 32) : "memory");  // the old tables are read
            for (int i = et; i < cnt; i += kGcEpiWarps * 32) {
                const int p = __ldg(a.colmap + g * a.cstride + nt * a.bn + i);
                t_off[i] = p >= 0 ? p * a.plane : 0;
                t_bias[i] = (p >= 0 && a.bias) ? __ldg(a.bias + p) : 0.0f;
            }
            for (int z = et; z < min(zc, kGcZcap); z += kGcEpiWarps * 32)
                z_off[z] = __ldg(a.zmap + g * a.zstride + z) * a.plane;
            asm volatile("bar.sync 1, %0;" ::"n"(kGcEpiWarps * 32) : "memory");
        }
        const int q = mt * (MT * 128) + (MT == 2 ? h * 128 : 0) + q4 * 32 + lane;
        int n, t, hh, w;
        grid_decode(a.gr, q, n, t, hh, w);
        const bool valid = q < a.gr.L && t < a.VT && hh < a.VH && w < a.VW;
        const long long pix =
            valid ? (long long)n * a.planes * a.plane + (long long)t * a.VHW + (long long)hh * a.VW + w : 0;
        float* yf = reinterpret_cast<float*>(a.out) + pix;
        __nv_bfloat16* yh = reinterpret_cast<__nv_bfloat16*>(a.out) + pix;
        const YCheck yc{pix, a.out_total, a.status};
        // zero planes, while the item's MMAs run: 16 at a time, the table read
        // four offsets to a load
        if (alive && valid) {
            const int zt = min(zc, kGcZcap) & ~15;
            for (int z = MT == 2 ? 0 : 16 * h; z < zt; z += MT == 2 ? 16 : 32) {
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    const int4 o = *reinterpret_cast<const int4*>(z_off + z + j);
                    zero_at<OUT_BF16>(yf, yh, yc, o.x);
                    zero_at<OUT_BF16>(yf, yh, yc, o.y);
                    zero_at<OUT_BF16>(yf, yh, yc, o.z);
                    zero_at<OUT_BF16>(yf, yh, yc, o.w);
                }
            }
            for (int z = zt + (MT == 2 ? 0 : h); z < zc; z += MT == 2 ? 1 : 2)
                zero_at<OUT_BF16>(yf, yh, yc, z < kGcZcap ? z_off[z] : __ldg(a.zmap + g * a.zstride + z) * a.plane);
        }
        if (cnt <= 0) continue;
        const int nch = (cnt + kEpiCols - 1) / kEpiCols;
        const int nst = gc_blocks(a, g) * a.gr.KT;
        float v[NCH][kEpiCols];
#pragma unroll
        for (int k = 0; k < NCH; ++k)
#pragma unroll
            for (int j = 0; j < kEpiCols; ++j) v[k][j] = 0.0f;
        const int pieces = nst * a.ppst;
        for (int pc = 0; alive && pc < pieces; pc += a.pps) {
            // warp-uniform outcome: the TMEM loads below are .sync.aligned
            if (!__all_sync(0xffffffffu, mbar_wait(&ep.acc_full[ab], acc_ph, ep.abort_flag, a.status))) {
                alive = false;
                break;
            }
            tc_fence_after();
            const uint32_t taddr = ep.tmem_base + (uint32_t)((ab * MT + (MT == 2 ? h : 0)) * a.tmem_stride) +
                                   ((uint32_t)(q4 * 32) << 16);
            if (NCH <= 4) {
                uint32_t r[NCH][kEpiCols];
#pragma unroll
                for (int k = 0; k < NCH; ++k) {
                    const int c = MT == 2 ? k : 2 * k + h;
                    if (c < nch) tmem_ld_32x32b_x16(taddr + (uint32_t)(c * kEpiCols), r[k]);
                }
                tmem_ld_wait();
                tc_fence_before();  // the buffer is free before the additions
                __syncwarp();
                if (lane == 0) mbar_arrive(&ep.acc_full[kGcMaxBuf + ab]);
#pragma unroll
                for (int k = 0; k < NCH; ++k) {
                    if ((MT == 2 ? k : 2 * k + h) < nch) {
#pragma unroll
                        for (int j = 0; j < kEpiCols; ++j) v[k][j] += __uint_as_float(r[k][j]);
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < NCH; ++k) {
                    const int c = MT == 2 ? k : 2 * k + h;
                    if (c < nch) {
                        uint32_t r[kEpiCols];
                        tmem_ld_32x32b_x16(taddr + (uint32_t)(c * kEpiCols), r);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < kEpiCols; ++j) v[k][j] += __uint_as_float(r[j]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ep.acc_full[kGcMaxBuf + ab]);
            }
            if (++ab == a.nbuf) { ab = 0; acc_ph ^= 1u; }
        }
        uint32_t nan = 0;         // chunks with NaN columns
        uint32_t nan_cols[NCH];     // theirs, 16 bits a chunk (in local memory: read by a runtime index)
#pragma unroll
        for (int k = 0; k < NCH; ++k) {
            const int c = MT == 2 ? k : 2 * k + h;
            if (alive && valid && c < nch) {
                bool bad = false;
#pragma unroll
                for (int j = 0; j < kEpiCols; ++j) bad |= v[k][j] != v[k][j];
                if (bad) {
                    uint32_t m = 0;
#pragma unroll
                    for (int j = 0; j < kEpiCols; ++j) m |= (v[k][j] != v[k][j] ? 1u : 0u) << j;
                    nan |= 1u << k;
                    nan_cols[k] = m;
                }
                store_cols<OUT_BF16>(v[k], c * kEpiCols, cnt, t_off, t_bias, a.relu, yf, yh, yc);
            }
        }
        // NaN columns: what a lane finds to be a kept term's stands, the others are
        // summed again by the warp
        if (__any_sync(0xffffffffu, nan != 0)) {
            const int kch = a.kcounts ? __ldg(a.kcounts + 2 * g) : a.ncb * a.cb;
            const uint4* wt = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(a.wd) +
                                                             (size_t)(g * a.ntiles + nt) * a.ksteps * a.bn * 32);
            const uint4* src = reinterpret_cast<const uint4*>(a.src + (size_t)g * a.gstride);
            int4 first = make_int4(-1, -1, -1, -1);
            if (nan) first = grid_scan(a, src, q, kch);
#pragma unroll 1
            for (int k = 0; k < NCH; ++k) {
                const int c0 = (MT == 2 ? k : 2 * k + h) * kEpiCols;
                uint32_t left = 0;
                for (uint32_t bits = (nan >> k) & 1u ? nan_cols[k] : 0u; bits; bits &= bits - 1) {
                    const int i = c0 + __ffs(bits) - 1;
                    if (i < cnt && !grid_nan_at(a, wt, src, ep.bnr, i, q, kch, first)) left |= bits & (0u - bits);
                }
                __syncwarp();
                for (uint32_t lanes = __ballot_sync(0xffffffffu, left != 0); lanes; lanes &= lanes - 1) {
                    const int l = __ffs(lanes) - 1;
                    const int ql = __shfl_sync(0xffffffffu, q, l);
                    for (uint32_t bits = __shfl_sync(0xffffffffu, left, l); bits; bits &= bits - 1) {
                        const int i = c0 + __ffs(bits) - 1;
                        float e = grid_exact(a, wt, src, ep.bnr, i, ql, kch) + t_bias[i];
                        if (lane != l || !y_ok(yc, t_off[i])) continue;
                        if (a.relu) e = fmaxf(e, 0.0f);
                        if (OUT_BF16)
                            yh[t_off[i]] = __float2bfloat16_rn(e);
                        else
                            yf[t_off[i]] = e;
                    }
                    __syncwarp();
                }
            }
        }
        __syncwarp();
    }
}

// DX: the input gradient, whose sums may be cut.
template <bool OUT_BF16, int MT, bool DX>
__global__ void __launch_bounds__(kGcThreads, 1)
    k_grid_conv(const __grid_constant__ GcArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sB = smem;
    uint8_t* sA = sB + a.cap_b;
    int* t_off = reinterpret_cast<int*>(sA + (size_t)a.stages_a * a.a_stride);
    float* t_bias = reinterpret_cast<float*>(t_off + 256);
    int* z_off = reinterpret_cast<int*>(t_bias + 256);
    uint64_t* bars = reinterpret_cast<uint64_t*>(z_off + kGcZcap);
    uint64_t* full_a = bars;
    uint64_t* empty_a = full_a + kGcMaxA;
    uint64_t* full_b = empty_a + kGcMaxA;
    uint64_t* empty_b = full_b + kGcMaxB;
    uint64_t* acc_full = empty_b + kGcMaxB;
    uint64_t* acc_empty = acc_full + kGcMaxBuf;
    uint64_t* b_full = acc_empty + kGcMaxBuf;
    uint64_t* b_empty = b_full + 1;
    uint64_t* drain = b_empty + 1;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGcMaxA; ++s) { mbar_init(&full_a[s], 1); mbar_init(&empty_a[s], 1); }
        for (int s = 0; s < kGcMaxB; ++s) { mbar_init(&full_b[s], 1); mbar_init(&empty_b[s], 1); }
        for (int b = 0; b < kGcMaxBuf; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], kGcEpiWarps); }
        mbar_init(b_full, 1);
        mbar_init(b_empty, 1);
        mbar_init(drain, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_holder, (uint32_t)a.tmem_cols);
        tmem_relinquish();
    }
    // Nothing above reads global memory: it overlaps the previous kernel's tail.
    if (!a.late_wait) pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();  // (every CTA has its TMEM: a dependent's allocation cannot come first)
    const uint32_t tmem_base = *tmem_holder;
    // The weights of a group stay in shared memory when there is one column
    // tile and every group's (as many steps as its channels need) fit.
    const int bnr = grid_rows(a.counts, a.groups, a.ntiles, a.bn);
    const uint32_t bstep = (uint32_t)bnr * 32u;               // one step of the weights
    const size_t btile = (size_t)a.ksteps * a.bn * 32;        // room of a tile's weights
    int most = 0;
    for (int g = 0; g < a.groups; ++g) most = max(most, gc_blocks(a, g) * a.gr.KT * a.spt);
    const bool resident = a.ntiles == 1 && uniform(most * (int)bstep <= a.cap_b);
    const bool stage_slots = uniform(2 * a.spt * (int)bstep <= a.cap_b);
    const int slot = stage_slots ? a.spt : a.rsteps;  // MMA steps of a ring slot
    const int stages_b = min(a.cap_b / (int)(bstep * slot), kGcMaxB);

    if (warp == 0) {
        // --------------------------------------------------- slab producer
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        uint32_t last = 0, issued = 0;  // bit s: parity of the last copy into stage s; whether there was one
        for (int u = blockIdx.x; ok && u < a.units; u += gridDim.x) {
            int g, nt, mt;
            gc_unit(a, u, g, nt, mt);
            if (__ldg(a.counts + 2 * g) <= nt * a.bn) continue;
            const int nblk = gc_blocks(a, g);
            const __nv_bfloat16* src = a.src + (size_t)g * a.gstride + (size_t)mt * (MT * 128) * 8;
            for (int c = 0; ok && c < nblk; ++c) {
                for (int kt = 0; kt < a.gr.KT; ++kt) {
                    if (!mbar_wait_warp(&empty_a[s], ph ^ 1u, abort_flag, a.status)) { ok = false; break; }
                    if (lane == 0) mbar_arrive_expect_tx(&full_a[s], (uint32_t)a.a_bytes);
                    __syncwarp();
                    if (lane < a.cb / 8)
                        bulk_load(smem_u32(sA + (size_t)s * a.a_stride) + (uint32_t)(lane * a.sp * 16),
                                  src + ((size_t)(c * (a.cb / 8) + lane) * a.gr.slots + (size_t)kt * a.gr.HWb) * 8,
                                  (uint32_t)a.sp * 16u, &full_a[s]);
                    last = (last & ~(1u << s)) | (ph << s);
                    issued |= 1u << s;
                    if (++s == a.stages_a) { s = 0; ph ^= 1u; }
                }
            }
        }
        // every copy issued has landed before the CTA retires
        for (int q = 0; q < a.stages_a; ++q) {
            if (!(issued & (1u << q))) continue;
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(&full_a[q], (last >> q) & 1u) && globaltimer() - t0 < kWaitLimitNs) {}
        }
        __syncwarp();
    } else if (warp == 2) {
        // ------------------------------------------------- weight producer
        if (lane == 0 && resident) {
            int cur = -1, loads = 0;
            uint32_t e_ph = 0;
            for (int u = blockIdx.x; u < a.units; u += gridDim.x) {
                int g, nt, mt;
                gc_unit(a, u, g, nt, mt);
                const int nst = gc_blocks(a, g) * a.gr.KT;
                if (__ldg(a.counts + 2 * g) <= 0 || nst == 0 || g == cur) continue;
                if (loads > 0) {
                    if (!mbar_wait(b_empty, e_ph, abort_flag, a.status)) break;
                    e_ph ^= 1u;
                }
                const uint32_t sbytes = bstep * (uint32_t)a.spt;
                mbar_arrive_expect_tx(b_full, sbytes * (uint32_t)nst);
                const char* w = reinterpret_cast<const char*>(a.wd) + (size_t)g * btile;
                for (int i = 0; i < nst; ++i)
                    bulk_load(smem_u32(sB) + (uint32_t)i * sbytes, w + (size_t)i * sbytes, sbytes, b_full);
                cur = g;
                ++loads;
            }
            if (loads > 0) {
                const unsigned long long t0 = globaltimer();
                while (!mbar_try_wait(b_full, (uint32_t)((loads - 1) & 1)) && globaltimer() - t0 < kWaitLimitNs) {}
            }
        } else if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            uint32_t last = 0, issued = 0;
            const uint32_t rbytes = bstep * (uint32_t)slot;
            for (int u = blockIdx.x; ok && u < a.units; u += gridDim.x) {
                int g, nt, mt;
                gc_unit(a, u, g, nt, mt);
                if (__ldg(a.counts + 2 * g) <= nt * a.bn) continue;
                const int nb = gc_blocks(a, g) * a.gr.KT * (stage_slots ? 1 : a.gr.KH);
                const char* w = reinterpret_cast<const char*>(a.wd) + (size_t)(g * a.ntiles + nt) * btile;
                for (int i = 0; i < nb; ++i) {
                    if (!mbar_wait(&empty_b[s], ph ^ 1u, abort_flag, a.status)) { ok = false; break; }
                    mbar_arrive_expect_tx(&full_b[s], rbytes);
                    bulk_load(smem_u32(sB) + (uint32_t)s * rbytes, w + (size_t)i * rbytes, rbytes, &full_b[s]);
                    last = (last & ~(1u << s)) | (ph << s);
                    issued |= 1u << s;
                    if (++s == stages_b) { s = 0; ph ^= 1u; }
                }
            }
            for (int q = 0; q < stages_b; ++q) {
                if (!(issued & (1u << q))) continue;
                const unsigned long long t0 = globaltimer();
                while (!mbar_try_wait(&full_b[q], (last >> q) & 1u) && globaltimer() - t0 < kWaitLimitNs) {}
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------- MMA issuer
        const GcPipe p{full_a, empty_a, full_b, empty_b, acc_full, acc_empty, b_full, b_empty, abort_flag,
                       smem_u32(sA), smem_u32(sB), tmem_base, stages_b, bnr};
        const int row = a.gr.KW * 8 + a.h16;
        const int mode = resident ? kResident : stage_slots ? kStageSlots : kRowSlots;
        // (a loop for each, so that the choice is not in them)
#define SADMM_MODES(KW, H, CUT)                                               \
    if (mode == kResident) gc_issue<KW, H, MT, CUT>(a, p, kResident);         \
    else if (mode == kStageSlots) gc_issue<KW, H, MT, CUT>(a, p, kStageSlots); \
    else gc_issue<KW, H, MT, CUT>(a, p, kRowSlots);
#define SADMM_ISSUE(KW, H) if (DX && a.cut) { SADMM_MODES(KW, H, true) } else { SADMM_MODES(KW, H, false) }
#define SADMM_ROW(KW, H) if (row == KW * 8 + H) { SADMM_ISSUE(KW, H) } else
        SADMM_ROW(1, 1) SADMM_ROW(1, 2) SADMM_ROW(1, 3) SADMM_ROW(1, 4)
        SADMM_ROW(3, 1) SADMM_ROW(3, 2) SADMM_ROW(3, 3) SADMM_ROW(3, 4)
        SADMM_ROW(5, 1) SADMM_ROW(5, 2) SADMM_ROW(7, 1) SADMM_ROW(7, 2)
        SADMM_ROW(4, 1) SADMM_ROW(6, 1) SADMM_ROW(9, 1) SADMM_ROW(11, 1)
        { SADMM_ISSUE(0, 0) }
#undef SADMM_ROW
#undef SADMM_ISSUE
#undef SADMM_MODES
        // Every MMA issued has completed before TMEM is freed.
        mma_commit_elect(drain);
        if (lane == 0) {
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(drain, 0) && globaltimer() - t0 < kWaitLimitNs) {}
        }
        __syncwarp();
    } else {
        // --------------------------------------------------------- epilogue
        const GcEpi ep{acc_full, abort_flag, t_off, tmem_base, bnr};
        if (DX && (a.bn / kEpiCols * MT + 1) / 2 <= 4)  // a warp's chunks
            gc_epilogue<OUT_BF16, MT, 4>(a, ep);
        else
            gc_epilogue<OUT_BF16, MT, 8>(a, ep);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)a.tmem_cols);
    }
    // TMEM is free: what this waits for may still need it.
    if (a.late_wait) pdl_wait();
}

__global__ void __launch_bounds__(256) k_grid_x(const GridX a)
{
    pdl_wait();  // after the kernel before it in the stream
    __shared__ int s_off[16];
    grid_x_block(a, blockIdx.x, blockIdx.y, s_off);
}

template <bool OUT_BF16, int MT, bool DX>
cudaError_t launch_gc(const GcArgs& a, int grid, size_t smem, cudaStream_t s)
{
    auto kern = k_grid_conv<OUT_BF16, MT, DX>;
    static int configured_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGcSmemLimit);
        if (e != cudaSuccess) return e;
        configured_dev = dev;
    }
    return launch_pdl(kern, dim3((unsigned)grid), dim3(kGcThreads), smem, s, a);
}

}  // namespace

bool grid_conv_shape(const Grid& gr, int chans, int cols, int likely, int groups, int sms, int stage, int seg, bool cut,
                     GridConvShape* out)
{
    if (chans < 1 || cols < 1) return false;
    GridConvShape r;
    r.seg = seg;
    r.cut = cut;
    const int taps = gr.KH * gr.KW;
    r.k16 = (chans + 15) / 16;
    const long long ksteps = (long long)r.k16 * gr.KT * taps;
    if (ksteps > (1 << 16)) return false;
    r.ksteps = (int)ksteps;
    const long long fixed = 1024 + kGcTables + kGcZcap * 4 + kGcBars;
    const int n16 = (int)round_up(cols, 16);
    if ((long long)(256 + (gr.KH - 1) * gr.Wb + gr.KW) >= (1 << 14)) return false;  // operand stride field
    const long long span = (gr.KH - 1) * gr.Wb + gr.KW - 1;
    // A block: as many 16s of channels as divide them, keep a stage to `stage`
    // MMA steps and its slab to 24 KB.
    // Where sums are cut, a kernel row that is unrolled (its issue is the slower
    // otherwise) and of which whole rows fill a segment best: the rest of one is a
    // segment more to read (AlexNet conv3: 12 steps of 2 rows, not 9 of 1).
    int m = 1;
    for (int k = 2, filled = 0; k <= 4; ++k) {
        if (r.k16 % k != 0 || taps * k > stage || (128 + span) * 32 * k > 24576) continue;
        if (cut) {
            if (unrolled_row(gr.KW, 1) && !unrolled_row(gr.KW, k)) continue;
            if (filled == 0) filled = std::max(gr.KW, seg / gr.KW * gr.KW);
            const int f = std::max(1, seg / (gr.KW * k)) * gr.KW * k;
            if (taps * k > seg && f < filled) continue;
            filled = std::max(filled, f);
        }
        m = k;
    }
    r.cb = 16 * m;
    const int rsteps = gr.KW * m;
    // The tiling of least estimated time: rounds of items over the SMs, each
    // item the longest of its MMAs (M = 128: the operands' shared-memory reads,
    // 32 + N/4 cycles, or N/2 at the tensor rate, and 9 more as issued; about
    // 400 a stage for its waits and commits), its stores (25 cycles per column
    // and tile: 512 bytes at 20 a cycle) and its streamed weights (32 bytes per
    // step and column at about 40 a cycle).
    long long best = -1;
    for (int mt = 1; mt <= 2; ++mt) {
        const long long stride = round_up((mt * 128 + span) * 16 * (m * 2), 128);
        const int nt0 = (n16 + 256 / mt - 1) / (256 / mt);
        for (int nt = nt0; nt <= nt0 + 3; ++nt) {
            const int bn = (int)round_up((n16 + nt - 1) / nt, 16);
            if (nt > nt0 && bn < 48) break;
            // three slabs and three slots of weights, two of each where that is too much
            long long room = kGcSmemLimit - fixed - 3 * stride;
            if (room < std::min(ksteps, 3ll * rsteps) * bn * 32) room = kGcSmemLimit - fixed - 2 * stride;
            if (room < std::min(ksteps, 2ll * rsteps) * bn * 32) continue;
            const long long cap = std::min(room / 128 * 128, ksteps * bn * 32);
            const int lb = nt == 1 ? std::min(bn, (int)round_up(likely, 16)) : bn;  // rows a tile is likely to have
            const bool res = nt == 1 && cap >= ksteps * lb * 32;
            const long long units = (gr.L + mt * 128 - 1) / (mt * 128) * nt * groups;
            const long long mma = ksteps * mt * (std::max(32 + lb / 4, lb / 2) + 9) + r.k16 / m * gr.KT * 400;
            const long long st = 25ll * mt * lb;
            // (an item's stores overlap the next one's MMAs about by half)
            const long long item = std::max(std::max(mma, st) + std::min(mma, st) / 2, res ? 0 : ksteps * lb * 32 / 40);
            const long long cost = (units + sms - 1) / sms * item + std::min(mma, st) / 2;
            if (best < 0 || cost < best) {
                best = cost;
                r.mt = mt;
                r.bn = bn;
                r.ntiles = nt;
                r.cap_b = (int)cap;
                const long long left = kGcSmemLimit - fixed - cap;
                r.stages_a = (int)std::min<long long>(kGcMaxA, left / stride);
                r.smem = (size_t)(fixed + cap + r.stages_a * stride);
            }
        }
    }
    if (best < 0) return false;
    r.cycles = best;
    r.npad = r.bn * r.ntiles;
    *out = r;
    return true;
}

sadmm_status launch_grid_conv(const Grid& gr, const GridConvShape& sh, const GridConvCall& c, cudaStream_t s)
{
    GcArgs a;
    memset(&a, 0, sizeof(a));
    a.gr = gr;
    a.src = c.src;
    a.wd = c.wd;
    a.out = c.out;
    a.bias = c.bias;
    a.colmap = c.colmap;
    a.cstride = c.cstride;
    a.zmap = c.zmap;
    a.zstride = c.zstride;
    a.counts = c.counts;
    a.kcounts = c.kcounts;
    a.status = device_status_ptr();
    a.out_total = c.out_total;
    a.late_wait = c.late_wait ? 1 : 0;
    a.src_dz = c.src_dz ? 1 : 0;
    a.gstride = (long long)c.chunks * gr.slots * 8;
    a.groups = c.groups;
    a.planes = c.planes;
    a.VT = c.VT;
    a.VH = c.VH;
    a.VW = c.VW;
    a.VHW = c.VH * c.VW;
    a.plane = c.VT * c.VH * c.VW;
    a.bn = sh.bn;
    a.ksteps = sh.ksteps;
    a.ntiles = sh.ntiles;
    a.mtiles = (gr.L + sh.mt * 128 - 1) / (sh.mt * 128);
    const long long units = (long long)a.mtiles * sh.ntiles * c.groups;
    if (units >= (1ll << 31) - (1ll << 20)) return SADMM_EUNSUPPORTED;
    a.units = (int)units;
    a.mt_div = make_fastdiv((uint32_t)a.mtiles);
    a.nt_div = make_fastdiv((uint32_t)a.ntiles);
    a.cb = sh.cb;
    a.ncb = sh.k16 * 16 / sh.cb;
    a.sp = sh.mt * 128 + (gr.KH - 1) * gr.Wb + gr.KW - 1;
    a.h16 = sh.cb / 16;
    a.rsteps = gr.KW * a.h16;
    a.spt = gr.KH * a.rsteps;
    a.cut = sh.cut && c.src_dz && a.spt > sh.seg ? 1 : 0;
    a.psteps = unrolled_row(gr.KW, a.h16) ? a.rsteps : std::min(a.rsteps, sh.seg);
    a.pps = std::max(1, sh.seg / (a.cut ? a.psteps : a.spt));
    a.ppst = a.cut ? gr.KH * ((a.rsteps + a.psteps - 1) / a.psteps) : 1;
    a.cap_b = sh.cap_b;
    a.stages_a = sh.stages_a;
    a.a_bytes = a.sp * 16 * (sh.cb / 8);
    a.a_stride = (int)round_up(a.a_bytes, 128);
    a.tmem_stride = (int)round_up(sh.bn, 32);
    a.nbuf = std::min(kGcMaxBuf, 512 / (sh.mt * a.tmem_stride));
    int cols = 32;
    while (cols < a.nbuf * sh.mt * a.tmem_stride) cols <<= 1;
    a.tmem_cols = cols;
    a.relu = c.relu ? 1 : 0;
    long long grid = c.ctas > 0 ? c.ctas : device_sm_count();
    if (grid > units) grid = units;
    cudaError_t e;
    if (c.src_dz)  // (its output is fp32)
        e = sh.mt == 2 ? launch_gc<false, 2, true>(a, (int)grid, sh.smem, s) : launch_gc<false, 1, true>(a, (int)grid, sh.smem, s);
    else if (sh.mt == 2)
        e = c.out_bf16 ? launch_gc<true, 2, false>(a, (int)grid, sh.smem, s) : launch_gc<false, 2, false>(a, (int)grid, sh.smem, s);
    else
        e = c.out_bf16 ? launch_gc<true, 1, false>(a, (int)grid, sh.smem, s) : launch_gc<false, 1, false>(a, (int)grid, sh.smem, s);
    return e == cudaSuccess ? SADMM_OK : SADMM_ECUDA;
}

bool grid_x_args(const Grid& gr, const Geometry& g, const void* x, const int* colidx, int nck, int chunks,
                 __nv_bfloat16* xs, GridX* a)
{
    a->gr = gr;
    a->x = static_cast<const __nv_bfloat16*>(x);
    a->colidx = colidx;
    a->xs = xs;
    a->C = (int)g.c;
    a->Cg = (int)g.cg;
    a->nck = nck;
    a->chunks = chunks;
    a->taps = (int)g.taps;
    a->x_total = g.n * g.c * g.t * g.h * g.w;
    a->xs_total = g.groups * chunks * (long long)gr.slots;
    a->status = device_status_ptr();
    a->bx = (gr.slots + 255) / 256;
    a->by = (int)(g.groups * ((chunks + 1) / 2));
    return a->by <= 65535;
}

static sadmm_status launch_grid_x(const Grid& gr, const Geometry& g, const void* x, const int* colidx, int nck, int chunks,
                                  __nv_bfloat16* xs, cudaStream_t s)
{
    GridX a;
    if (!grid_x_args(gr, g, x, colidx, nck, chunks, xs, &a)) return SADMM_EUNSUPPORTED;
    return launch_pdl(k_grid_x, dim3((unsigned)a.bx, (unsigned)a.by), dim3(256), 0, s, a) == cudaSuccess ? SADMM_OK
                                                                                                         : SADMM_ECUDA;
}

// The rule for the forward compares estimated times on a whole GB300, whatever
// the plan's cap: of 80 layers measured both ways (AlexNet conv2-5, ResNet-50,
// C3D and sweep layers, 1x1 to 5x5, densities 0.05 to 1, batch 8 to 128; each
// graph-replayed) it takes the slower one by more than 5 % on two, by at most
// 20 %.  Dense-in-taps work pays where the gathered kernel's rate is the gather's
// (up to 128 filters a group) or columns are mostly kept: AlexNet conv2 at half
// density 77 -> 50 us, all columns of conv3 63 -> 37, 64-channel 5x5 51 -> 23;
// conv3 at a quarter stays gathered (22 against 29 us), the 512-filter layer at
// half too (125 against 185).
constexpr long long kRuleSms = 152;

// MMA steps summed in TMEM, whole stages of one kernel frame: AlexNet conv2's error
// against 64 bits is 2.1e-7 (the gathered kernel's 3.3e-7); with 27 it would be
// 1.3e-7 and 55.8 us become 61.2.  A longer frame is one segment: 9x9 taps over 32
// channels, 81 steps, stand at 7.2e-7 where the gathered kernel's sums of all 162
// stand at 1.6e-6.
constexpr int kFwdSeg = 54;

// Channels of x per conv group that hold a kept column.
static int fwd_channels(const sadmm_plan* plan, const Geometry& g)
{
    return plan->colkind == SADMM_COL_CHANNEL ? plan->n_colgroups : (int)g.cg;
}

int grid_fwd_ksteps(const sadmm_plan* plan, const Geometry& g)
{
    return (fwd_channels(plan, g) + 15) / 16 * (int)g.taps;
}

bool grid_fwd_plan(const Geometry& g, sadmm_plan* plan, size_t* gx, size_t* gw, size_t* gcol)
{
    Grid gr;
    GridConvShape sh;
    if (plan->n_cols < 1 || plan->n_filt < 1 || plan->splits > 1 || g.groups > 64 || !grid_of(g, &gr)) return false;
    if (g.taps == 1) return false;  // one tap reads contiguous rows: no slab to share
    const long long units = (g.m + 127) / 128 * g.groups * ((plan->n_tiles + 1) / 2);
    if (units < kRuleSms) return false;
    const int nck = fwd_channels(plan, g);
    const int per = (int)((plan->n_filt + g.groups - 1) / g.groups);
    if (!grid_conv_shape(gr, nck, plan->n_pad, per, (int)g.groups, plan->ctas, kFwdSeg, kFwdSeg, false, &sh)) return false;
    const int chunks = sh.k16 * 2;
    if (g.groups * sh.k16 > 65535) return false;
    plan->gx_cb = sh.cb;
    plan->gx_mt = sh.mt;
    plan->gx_bn = sh.bn;
    plan->gx_ntiles = sh.ntiles;
    plan->gx_stages = sh.stages_a;
    plan->gx_cap = sh.cap_b;
    plan->gx_smem = (int)sh.smem;
    // The estimates, in ns.  Grid: launches and drain, the copy at 4 TB/s of x
    // read and written, the slab GEMM's cycles at 1.95 GHz, and y at 60 TB/s
    // for what its stores add.  Gathered: start-up, the busiest CTA's 64-column
    // stages (the gather's rate up to 128 filters, the MMAs' above), and the
    // stores, which overlap less when one accumulator set fills TMEM.
    GridConvShape rule;
    if (!grid_conv_shape(gr, nck, plan->n_pad, per, (int)g.groups, kRuleSms, kFwdSeg, kFwdSeg, false, &rule)) return false;
    const long long xb = 2 * g.n * g.groups * (long long)nck * g.t * g.h * g.w + 2 * g.groups * 16ll * sh.k16 * gr.L;
    const long long yb = 4 * g.m * g.f;
    const long long grid_ns = 8000 + xb / 4000 + rule.cycles * 100 / 195 + yb / 60000;
    const long long nks = plan->k_pad / 64, rows = (long long)std::min(plan->n_tiles, 2) * plan->bn;
    const long long whole = (units + kRuleSms - 1) / kRuleSms * nks, even = (units * nks + kRuleSms - 1) / kRuleSms;
    const bool sk = 2 * std::min(plan->n_tiles, 2) * round_up(plan->bn, 32) <= 512 && plan->k_pad >= 4ll * plan->bn &&
                    even >= nks && (whole - even) * 8 >= whole;
    const long long stages = sk ? even : whole;
    const long long gather_ns = 7000 + stages * (rows <= 128 ? 680 : rows <= 256 ? 800 : 950) +
                                yb / (plan->n_tiles > 1 ? 20000 : 40000);
    if (grid_ns * 100 > gather_ns * 95) return false;
    *gx = (size_t)(g.groups * chunks * (long long)gr.slots * 16);
    *gw = (size_t)(g.groups * sh.npad * (long long)sh.ksteps * 32);
    *gcol = (size_t)sh.ksteps * 16 * 4;
    return true;
}

sadmm_status launch_grid_fwd(const sadmm_plan* plan, const Geometry& g, const void* x, const float* bias, int relu,
                             void* y, int ydt, cudaStream_t s)
{
    Grid gr;
    if (!grid_of(g, &gr)) return SADMM_EINVAL;
    const int nck = fwd_channels(plan, g);
    GridConvShape sh;
    memset(&sh, 0, sizeof(sh));
    sh.cb = plan->gx_cb;
    sh.seg = kFwdSeg;
    sh.k16 = (nck + 15) / 16;
    sh.ksteps = grid_fwd_ksteps(plan, g);
    sh.mt = plan->gx_mt;
    sh.bn = plan->gx_bn;
    sh.ntiles = plan->gx_ntiles;
    sh.npad = sh.bn * sh.ntiles;
    sh.cap_b = plan->gx_cap;
    sh.stages_a = plan->gx_stages;
    sh.smem = (size_t)plan->gx_smem;
    const char* base = static_cast<const char*>(plan->dev);
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(const_cast<char*>(base) + plan->off_gx);
    const int* colidx = reinterpret_cast<const int*>(base + plan->off_colidx);
    sadmm_status st = launch_grid_x(gr, g, x, plan->colkind == SADMM_COL_CHANNEL ? colidx : nullptr, nck, sh.k16 * 2, xs, s);
    if (st != SADMM_OK) return st;
    GridConvCall c;
    memset(&c, 0, sizeof(c));
    c.src = xs;
    c.chunks = sh.k16 * 2;
    c.wd = reinterpret_cast<const __nv_bfloat16*>(base + plan->off_gw);
    c.out = y;
    c.out_bf16 = ydt == SADMM_BF16;
    c.bias = bias;
    c.relu = relu;
    c.colmap = reinterpret_cast<const int*>(base + plan->off_rowmap);
    c.cstride = plan->n_pad;
    c.zmap = reinterpret_cast<const int*>(base + plan->off_zeromap);
    c.zstride = (int)g.fg;
    c.counts = reinterpret_cast<const int*>(base + plan->off_counts);
    c.groups = (int)g.groups;
    c.planes = (int)g.f;
    c.VT = (int)g.ot;
    c.VH = (int)g.oh;
    c.VW = (int)g.ow;
    c.out_total = g.n * g.f * g.plane;
    c.ctas = plan->ctas;
    return launch_grid_conv(gr, sh, c, s);
}

}  // namespace sadmm
