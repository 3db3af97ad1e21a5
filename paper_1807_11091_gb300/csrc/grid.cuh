// grid.cuh -- the zero-padded pixel grid shared by the stride-1 kernels that
// read shifted slabs (conv_grid.cu, bwd_grid.cu).
//
// A stride-1 layer's input and output gradient are rewritten as channel-octet
// copies src[group][chunk][slot][8 channels] (bf16).  Slots run over the whole
// batch in one line: image n, frame t, row h, column w of the input sit at slot
//   n*P + (t + pt)*HWb + (h + ph)*Wb + (w + pw),
// Wb = W + pw, Hb = H + ph, Tb = T + pt, HWb = Hb*Wb, P = Tb*HWb.  Only the
// leading zeros of each row, frame and image are stored: the trailing ones are
// the next row's leading ones (pads are at most K - 1).  Output pixel
// (n, ot, oh, ow) is grid pixel q = n*P + ot*HWb + oh*Wb + ow and its tap
// (kt, kh, kw) reads slot q + kt*HWb + kh*Wb + kw, whatever the pixel: every
// tap is one shift of the whole line.  The output gradient sits D0 slots later
// (the flipped kernel's leading pad), so the same line serves the input
// gradient (a conv with the flipped taps) and, read from slot D0 on, the
// weight gradient.
#pragma once

#include "common.cuh"
#include "conv_common.cuh"
#include "internal.h"

namespace sadmm {

struct Grid {
    int N, T, H, W, OT, OH, OW, KT, KH, KW, pt, ph, pw;
    int Wb, HWb, P;
    int L;         // grid pixels N*P
    int slots;     // slots of a chunk, every one written: L to 256, the largest shift and 16 more, to 8
    int D0;        // slot of output pixel 0 in the output gradient's copy
    int maxshift;  // the last tap's shift
    FastDiv p_div, hw_div, w_div;
};

// The grid of a layer; false when it has none (a stride above 1, or a pad of K or more).
inline bool grid_of(const Geometry& g, Grid* out)
{
    if (g.st != 1 || g.sh != 1 || g.sw != 1 || g.pt >= g.kt || g.ph >= g.kh || g.pw >= g.kw) return false;
    const long long wb = g.w + g.pw, hb = g.h + g.ph, tb = g.t + g.pt;
    const long long p = wb * hb * tb, L = g.n * p;
    const long long ms = (g.kt - 1) * hb * wb + (g.kh - 1) * wb + g.kw - 1;
    const long long slots = round_up(round_up(L, 256) + ms + 16, 8);
    if (slots >= (1ll << 30)) return false;
    Grid r;
    r.N = (int)g.n; r.T = (int)g.t; r.H = (int)g.h; r.W = (int)g.w;
    r.OT = (int)g.ot; r.OH = (int)g.oh; r.OW = (int)g.ow;
    r.KT = (int)g.kt; r.KH = (int)g.kh; r.KW = (int)g.kw;
    r.pt = (int)g.pt; r.ph = (int)g.ph; r.pw = (int)g.pw;
    r.Wb = (int)wb;
    r.HWb = (int)(hb * wb);
    r.P = (int)p;
    r.L = (int)L;
    r.slots = (int)slots;
    r.maxshift = (int)ms;
    r.D0 = (int)((g.kt - 1 - g.pt) * hb * wb + (g.kh - 1 - g.ph) * wb + (g.kw - 1 - g.pw));
    r.p_div = make_fastdiv((uint32_t)p);
    r.hw_div = make_fastdiv((uint32_t)(hb * wb));
    r.w_div = make_fastdiv((uint32_t)wb);
    *out = r;
    return true;
}

// ---- slab GEMM over a grid copy (conv_grid.cu) ----
// out[plane(col)][pixel] = bias + sum over the K columns of Wd[col][k] * src:
// K column k = ((cb*KT + kt)*KH*KW + kh*KW + kw)*CB + ci reads channel
// cb*CB + ci at shift kt*HWb + kh*Wb + kw.  Wd lies as the MMA reads it, a step
// of 16 K columns at a time: [group][column tile][step][K half][row][8].
struct GridConvShape {
    int cb;      // channels per block (multiple of 16)
    int seg;     // MMA steps summed in TMEM before the fp32 registers take over,
    bool cut;    // also where that ends inside a stage (else a stage is never cut)
    int k16;     // 16-channel groups of the source (padded channels / 16)
    int ksteps;  // MMA steps of 16 K columns
    int mt;      // 128-pixel tiles per work item (1 or 2)
    int bn, ntiles, npad;  // output columns per tile, tiles, and bn*ntiles
    int cap_b;     // bytes of weights shared memory holds: all of an item's stay there, or a ring streams
    int stages_a;
    size_t smem;
    long long cycles;  // its estimated time
};
// The tiling for `chans` source channels and at most `cols`, likely `likely`,
// output columns per group over `groups` groups, stages of at most `stage` MMA steps
// where the kernel allows and sums of `seg` in TMEM; false when it does not fit.
// The blocks of channels (the order of the sums) follow the layer alone, not its
// batch or the device.
bool grid_conv_shape(const Grid& gr, int chans, int cols, int likely, int groups, int sms, int stage, int seg, bool cut,
                     GridConvShape* out);

// Rows of a column tile in the weights' layout: the most columns any group has,
// to 16, when there is one tile (the groups' counts are known on the device
// alone), else bn.
SADMM_DEV int grid_rows(const int* counts, int groups, int ntiles, int bn)
{
    if (ntiles > 1) return bn;
    int m = 16;
    for (int g = 0; g < groups; ++g) m = max(m, (__ldg(counts + 2 * g) + 15) & ~15);
    return min(m, bn);
}

struct GridConvCall {
    const __nv_bfloat16* src;  // [groups][chunks][slots][8]
    int chunks;                // chunks per group (k16 * 2)
    const __nv_bfloat16* wd;   // [groups][ntiles][ksteps][2][rows][8], rows = grid_rows() (a tile's room: bn); -0.0 at pruned entries
    void* out;
    int out_bf16;
    const float* bias;     // per plane, or NULL
    int relu;
    const int* colmap;     // [groups][cstride] column -> plane of an image (-1: none)
    int cstride;
    const int* zmap;       // [groups][zstride] planes written as zeros
    int zstride;
    const int* counts;     // [groups][2] columns, zero planes
    const int* kcounts;    // channels per group at [2*g] (NULL: all)
    int groups, planes;    // planes per image of the output
    int VT, VH, VW;        // its extents
    long long out_total;
    int ctas;
    int src_dz;  // 1: src is the output gradient's copy, pixel 0 at slot D0
    // 1: the kernel before this one in the stream writes nothing it reads, and lets
    // it start only when the one that wrote its inputs has completed.  It then
    // waits for that kernel at its end, so that its completion still means both.
    int late_wait;
};
sadmm_status launch_grid_conv(const Grid& gr, const GridConvShape& sh, const GridConvCall& c, cudaStream_t s);

// x (bf16 NCTHW) -> grid copy of `nck` channels per group (kept channels
// colidx[ci*taps]/taps when colidx != NULL, else 0..nck-1), `chunks` chunks, by
// bx x by blocks of 256 threads.
struct GridX {
    Grid gr;
    const __nv_bfloat16* x;
    const int* colidx;
    __nv_bfloat16* xs;
    int C, Cg, nck, chunks, taps, bx, by;
    long long x_total, xs_total;  // elements of x, octets of the copy
    int* status;
};
// False when by passes the grid limit.
bool grid_x_args(const Grid& gr, const Geometry& g, const void* x, const int* colidx, int nck, int chunks,
                 __nv_bfloat16* xs, GridX* a);

// ---- grid forward (conv_grid.cu) ----
// Whether the plan's forward takes the grid; its tiling then, and the bytes of
// the regions it adds to the plan's buffer.
bool grid_fwd_plan(const Geometry& g, sadmm_plan* plan, size_t* gx, size_t* gw, size_t* gcol);
int grid_fwd_ksteps(const sadmm_plan* plan, const Geometry& g);
sadmm_status launch_grid_fwd(const sadmm_plan* plan, const Geometry& g, const void* x, const float* bias, int relu,
                             void* y, int ydt, cudaStream_t s);

// ---- grid backward (bwd_grid.cu) ----
// The workspace, at most cap bytes: a layer that needs more takes its images in several
// passes.  0: the layer has no grid, or one image of it needs more.  *ns: its estimated
// time.
size_t grid_bwd_bytes(const sadmm_plan* plan, const Geometry& g, size_t cap, long long* ns);
sadmm_status launch_grid_bwd(const sadmm_plan* plan, const Geometry& g, size_t cap, const void* x, const void* dy,
                             const void* y, int ydt, int relu, float* dW, float* db, float* dx, void* ws, cudaStream_t s);

// ------------------------------------------------------------- device side --

// Bulk copy of `bytes` (a multiple of 16) from 16-byte aligned global memory
// into shared memory, completion as transaction bytes on `bar`.
SADMM_DEV void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// A condition every lane of the converged warp agrees on, as a vote: control
// flow the compiler cannot prove warp-uniform keeps the issuing warp's
// descriptors out of the uniform registers, and an MMA then takes about 140
// cycles to issue instead of 50.
SADMM_DEV bool uniform(bool c) { return __all_sync(0xffffffffu, c); }

// Grid pixel q -> image and coordinates.
SADMM_DEV void grid_decode(const Grid& gr, int q, int& n, int& t, int& h, int& w)
{
    n = (int)fdiv((uint32_t)q, gr.p_div);
    int r = q - n * gr.P;
    t = (int)fdiv((uint32_t)r, gr.hw_div);
    r -= t * gr.HWb;
    h = (int)fdiv((uint32_t)r, gr.w_div);
    w = r - h * gr.Wb;
}

// Block (bx, by) of the grid copy of x, 256 threads: thread t takes slot
// 256*bx + t of two chunks of conv group by / pairs (16 loads in flight, each
// coalesced along the row); s_off: 16 ints of shared memory.
SADMM_DEV void grid_x_block(const GridX& a, int bx, int by, int* s_off)
{
    const int pairs = (a.chunks + 1) / 2;
    const int g = by / pairs, c0 = (by - g * pairs) * 2;
    const int thw = a.gr.T * a.gr.H * a.gr.W;
    if (threadIdx.x < 16) {  // channel plane offsets (-1: zero)
        const int ci = c0 * 8 + threadIdx.x;
        int ch = ci < a.nck ? ci : -1;
        if (ch >= 0 && a.colidx) {
            const int col = __ldg(a.colidx + ci * a.taps);
            ch = col >= 0 ? col / a.taps : -1;
        }
        s_off[threadIdx.x] = ch >= 0 ? (g * a.Cg + ch) * thw : -1;
    }
    __syncthreads();
    const int s = bx * 256 + threadIdx.x;
    if (s >= a.gr.slots) return;
    int n, t, h, w;
    grid_decode(a.gr, s, n, t, h, w);
    const bool valid = n < a.gr.N && t >= a.gr.pt && h >= a.gr.ph && w >= a.gr.pw;
    const long long base = (long long)n * a.C * thw + (long long)(t - a.gr.pt) * (a.gr.H * a.gr.W) +
                           (long long)(h - a.gr.ph) * a.gr.W + (w - a.gr.pw);
    const unsigned short* xi = reinterpret_cast<const unsigned short*>(a.x);
    uint32_t v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int off = s_off[e];
        v[e] = (valid && off >= 0 && dbg_in(base + off, a.x_total, a.status)) ? (uint32_t)__ldg(xi + base + off) : 0u;
    }
    const size_t at = ((size_t)g * a.chunks + c0) * a.gr.slots + s;
    uint4* dst = reinterpret_cast<uint4*>(a.xs) + at;
    if (!dbg_in((long long)at, a.xs_total, a.status)) return;
    dst[0] = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
    if (c0 + 1 < a.chunks && dbg_in((long long)at + a.gr.slots, a.xs_total, a.status))
        dst[a.gr.slots] =
            make_uint4(v[8] | (v[9] << 16), v[10] | (v[11] << 16), v[12] | (v[13] << 16), v[14] | (v[15] << 16));
}

}  // namespace sadmm
