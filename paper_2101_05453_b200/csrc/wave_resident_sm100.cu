// Wavefront kernel for stacks whose weights fit in shared memory: the same schedule as wave_sm100.cu - every layer works on a step
// of its own, every layer's rows are split into row groups - but a (layer, row group) is one thread-block CLUSTER, and nothing of
// its recurrence leaves the cluster's shared memory.
//
// Such a step is a few kilobytes of weights per warp and one to four exchanges; what it costs is the length of its dependency
// chain.  In wave_small_sm100.cu that chain was, for two 256-cell layers at 8 rows (7000 cycles a step): publish to L2 1170, poll 1030,
// copy the operand back 1150, tcgen05 products of two k-blocks with their commit 1330, accumulators through tensor memory and gate sums
// through shared memory to other warps 1160, elementwise work 1140.  Here:
//   - h, m and the layer norm's sums go from registers into the peers' shared memory (st.async, completion counted in bytes on an
//     mbarrier there): 1100 cycles per exchange with its block barriers, against 3400;
//   - a warp owns eight cells and computes their four gates for eight rows with mma.sync m16n8k32: 20 cycles of latency, and 8 cycles
//     per 512 bytes of weights on each scheduler - with so few columns that is faster than tcgen05 (42 to 50 cycles per 4 KB for the SM),
//     whose 128 x 32 tiles leave their columns empty;
//   - a lane's accumulators are all gates of one cell and two rows, so that rescale, nonlinearities, cell update and hidden state
//     follow in registers: no block barrier but the layer norm's and the projection's.
//
// The shared-memory image of weights is [eight cells][64 bytes of K][gate][cell][64]: a lane's 16 bytes of a gate row are its A
// fragments of two k-steps, and 16 bytes of an activation row its B fragments (which k a fragment slot stands for is free, as long as
// both operands agree).  Activation rows are an odd multiple of 64 bytes apart: no bank conflicts.
//
// Warp 0 fetches x_{t+1} .. x_{t+4} (from the caller or, by bulk copy, from what the layer below wrote to global memory), warp 1 writes
// h^t for the layer above or y; neither is on the chain.  Buffers of h alternate between two; a peer's h^t is complete only after
// every block has read h^{t-2}, so that writing it needs no permission.
//
// Every wait is bounded: see wv_wait_cluster_slow.
#include <algorithm>
#include <cstring>

#include "wave_resident.h"

namespace ql {

namespace {

constexpr int RS_MAX_WARPS = 16;               // computing warps
constexpr int RS_THREADS = 32 * (RS_MAX_WARPS + 2);
constexpr int RS_NX = 4;                       // x buffers
constexpr int RS_MAX_CLUSTER = 16;
constexpr int RS_MAX_NT = 4;                   // tiles of eight rows
static_assert(RS_MAX_CLUSTER <= WC_WORDS && WC_WORDS <= 32, "a word per block in a line of counters, a lane per word");

struct ResLayer {
    int I, C, O;
    uint32_t flags;
    int m_bits, zp_m, zp_h;
    int cpc, opc;                  // cells and outputs per block (multiples of 8)
    int ki, kh, kc;                // 64-byte chunks of the three products
    int px, ph, pm;                // bytes between rows of x, h, m in shared memory
    size_t img_stride;             // bytes of a block's weights
    const int8_t *img;
    const int32_t *bx, *bh, *bln, *bp;
    const int16_t *P, *L;
    int x_left[4], h_left[4];
    FastScale f_x[4], f_h[4], f_c[4], f_ln[4], f_m, f_proj;
    DivMagic div_c;
    uint32_t sigma_min;
    const int8_t *in_img;          // [T][B][px] the layer below's outputs; null: x
    int8_t *out_img;               // [T][B][px of the layer above]; null: y
    int out_pitch;
    const unsigned *cnt_in;        // [row group][WC_WORDS]: by block of the group, the steps that it has written to in_img / out_img
    unsigned *cnt_out;
    int below;                     // blocks that write in_img
    int8_t *h; int16_t *c;
    int dir, y_off;
    const uint8_t *tab;
    ActLineLayout tab_lay;
};

struct ResCall {
    int T, B, n_layers, cl, rg, nt;            // cluster size, row groups, tiles of rows
    int hw, xw, pw;                            // warps for gate sums and cells, for X, for projections
    int x_bulk, y_wide;                        // x rows in 16-byte pieces; y in 8-byte pieces
    const int8_t *x;
    int8_t *y;
    int y_stride;
    unsigned *abort_word, *ticket, *cnt;       // cnt: a line of WC_WORDS per (layer, row group)
    int *status, *status2;
    unsigned long long limit_ns;
    unsigned missing;
    ResLayer layer[WV_MAX_LAYERS];
};

struct RsCtl {
    uint64_t w_full, x_full[RS_NX], x_empty[RS_NX], xg_full[2], xg_free[2], h_full[2], h_read[2], m_full, s_full[2], l_sync, p_sync;
    int abort_flag, x_issued;
    alignas(16) uint4 sc[18];
};

struct RsLayout { size_t x, xg, h, m, sx, ln, st, part, stage, consts, tab, ctl, total; };

__host__ __device__ inline RsLayout rs_layout(const ResLayer &L, int cl, int nt, int hw, int pw, bool ln, bool peep)
{
    const bool proj = L.flags & F_PROJECTION;
    const size_t r8 = (size_t)nt * 8, G = (L.flags & F_CIFG) ? 3 : 4;
    RsLayout l;
    size_t p = (size_t)(L.cpc / 8) * (L.ki + L.kh) * G * 512 + (proj ? (size_t)(L.opc / 8) * L.kc * 512 : 0);
    l.x = p;      p += RS_NX * r8 * L.px;
    l.xg = p;     p += 2 * (size_t)(L.cpc / 8) * nt * 512;
    l.h = p;      p += 2 * r8 * L.ph;
    l.m = p;      p += proj ? r8 * L.pm : 0;
    l.sx = p;     p += ln && cl > 1 ? (size_t)cl * r8 * (peep ? 5 : 4) * 16 : 0;
    l.ln = p;     p += ln ? 4 * r8 * sizeof(WvLnRow) : 0;
    l.st = p;     p += ln ? 2 * (size_t)(peep ? 15 : 12) * r8 * 4 : 0;
    l.part = p;   p += proj ? (size_t)pw * 512 : 0;
    l.stage = p;  p += (size_t)(hw + pw) * 64;
    l.consts = p; p += wv_up((size_t)L.cpc * (3 * 16 + 2 * 8) + (size_t)L.opc * 4, 16);
    l.tab = p;    p += wv_up(L.tab_lay.bytes, 16);
    l.ctl = p;    p += wv_up(sizeof(RsCtl), 16);
    l.total = p;
    return l;
}

// ---- waits and mma.sync -------------------------------------------------------------------------------------
// without waiting
__device__ __forceinline__ bool rs_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(ok)
        : "r"(ptx::smem_u32(bar)), "r"(parity)
        : "memory");
    return __all_sync(0xffffffffu, ok != 0);
}
__device__ __forceinline__ bool rs_wait(const ResCall &k, uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    return wv_wait_cluster(bar, parity, k.abort_word, k.limit_ns, abort_flag);
}
// one arrival of a warp, for what its lanes wrote
__device__ __forceinline__ void rs_arrive(uint64_t *bar, int lane)
{
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(bar);
}
__device__ __forceinline__ void rs_mma(int32_t (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Gate products of eight cells and eight rows: acc[0] slots 0 and 1, acc[1] slots 2 and 3; of a slot the lane has cell lane / 4, rows
// 2 (lane mod 4) and the next.  w, b: this lane's 16 bytes of the first chunk.
template <int G>
struct RsFrag { uint4 b, s[G]; };
template <int G>
__device__ __forceinline__ RsFrag<G> rs_fetch(const uint8_t *w, const uint8_t *b)
{
    RsFrag<G> f;
    f.b = *reinterpret_cast<const uint4 *>(b);
#pragma unroll
    for (int e = 0; e < G; ++e) f.s[e] = *reinterpret_cast<const uint4 *>(w + e * 512);
    return f;
}
// (A chunk's operands are requested before the products of the one before it.)
template <int G>
__device__ __forceinline__ void rs_gates(int32_t (&acc)[2][4], const uint8_t *w, const uint8_t *b, int nk)
{
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[0][j] = acc[1][j] = 0;
    RsFrag<G> f = rs_fetch<G>(w, b);
#pragma unroll 2
    for (int c = 1; c <= nk; ++c) {
        RsFrag<G> n = f;
        if (c < nk) n = rs_fetch<G>(w + c * (G * 512), b + c * 64);
        const uint4 z = make_uint4(0, 0, 0, 0), &s3 = G == 4 ? f.s[G - 1] : z;
        rs_mma(acc[0], f.s[0].x, f.s[1].x, f.s[0].y, f.s[1].y, f.b.x, f.b.y);
        rs_mma(acc[1], f.s[2].x, s3.x, f.s[2].y, s3.y, f.b.x, f.b.y);
        rs_mma(acc[0], f.s[0].z, f.s[1].z, f.s[0].w, f.s[1].w, f.b.z, f.b.w);
        rs_mma(acc[1], f.s[2].z, s3.z, f.s[2].w, s3.w, f.b.z, f.b.w);
        f = n;
    }
}
__device__ __forceinline__ int32_t rs_acc(const int32_t (&acc)[2][4], int g, int j) { return acc[g >> 1][2 * (g & 1) + j]; }

// Sums over the eight cells of a warp's lanes of eight values each (index i): afterwards a lane holds the sum of i = lane / 4.
__device__ __forceinline__ int32_t rs_sum_cells(const int32_t (&a)[8], int lane)
{
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
    int32_t b[4], c[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) b[i] = (h4 ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, h4 ? a[i] : a[i + 4], 16);
#pragma unroll
    for (int i = 0; i < 2; ++i) c[i] = (h3 ? b[i + 2] : b[i]) + __shfl_xor_sync(0xffffffffu, h3 ? b[i] : b[i + 2], 8);
    return (h2 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h2 ? c[0] : c[1], 4);
}

// Bytes (cell lane / 4, rows 2 q and 2 q + 1) of an 8 x 8 tile to `at`, the place of this lane's row (lane mod 8) in a buffer of this
// block's, and of the other blocks [0, n) of the cluster: whole rows of eight bytes, through the warp's stage.  peer[j]: distance from
// this block's shared memory to that of block lane / 8 + 4 j.
__device__ __forceinline__ void rs_send_tile(uint8_t *stage, int32_t v0, int32_t v1, uint8_t *at, bool valid, uint32_t bar, const uint32_t (&peer)[4], int rank, int n,
                                             int lane)
{
    const int g = lane >> 2, q = lane & 3;
    __syncwarp();
    stage[q * 16 + g] = (uint8_t)v0;
    stage[q * 16 + 8 + g] = (uint8_t)v1;
    __syncwarp();
    const uint2 v = *reinterpret_cast<const uint2 *>(stage + (lane & 7) * 8);
    const uint32_t a = ptx::smem_u32(at);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int p = (lane >> 3) + 4 * j;
        if (4 * j >= n) break;                                 // warp-uniform
        if (p < n && p != rank && valid) wv_send8(a + peer[j], v, bar + peer[j]);
    }
    if (lane < 8 && valid) *reinterpret_cast<uint2 *>(at) = v;
}

// rescale of Section 3.2.4 with its constants in one 16-byte word of shared memory: {m2, add_hi, rshift, left shift before it}
__device__ __forceinline__ uint4 rs_scale(const FastScale &f, int left) { return make_uint4(f.m2, f.add_hi, (uint32_t)f.rshift, (uint32_t)left); }
__device__ __forceinline__ int32_t rs_rescale(int32_t v, const uint4 &f) { return fast_rescale(v, FastScale{f.x, f.y, (int32_t)f.z}); }
enum { RS_SC_X = 0, RS_SC_H = 4, RS_SC_C = 8, RS_SC_LN = 12, RS_SC_M = 16, RS_SC_P = 17, RS_SCALES = 18 };

// A kernel argument that is wanted in a register: without this it is read from the constant bank again at every use.
__device__ __forceinline__ int rs_keep(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}

struct RsSmem {
    const uint4 *sc;               // [RS_SCALES]
    int4 *bx, *bh, *bln;           // [cell] by slot
    uint2 *L, *P;                  // [cell] four int16
    int32_t *bp;
    uint32_t *st;                  // [2][12 or 15][rows] layer-norm sums of the block: (slot, {sum, low 20 bits, rest of the squares})
    WvLnRow *ln;                   // [4][rows]
    uint4 *sx;                     // [block][4 or 5 slots][rows] the peers' sums
};
__device__ __forceinline__ int32_t rs_s16(const uint2 &v, int g) { return (g & 1) ? wv_hi(g < 2 ? v.x : v.y) : wv_lo(g < 2 ? v.x : v.y); }
__device__ __forceinline__ int32_t rs_i4(const int4 &v, int g) { return g == 0 ? v.x : g == 1 ? v.y : g == 2 ? v.z : v.w; }

// hidden state from the output gate's argument and the new cell state (Section 3.2.7)
__device__ __forceinline__ int32_t rs_hidden(const uint4 &f_m, int zp_m, const ActLines &at, int32_t o, int32_t c)
{
    return sat8(rs_rescale(line_sigmoid(at, o) * line_tanh_cell(at, c), f_m) + zp_m);
}

template <int G, bool LN, bool PEEP, int U>
__global__ void __launch_bounds__(RS_THREADS, 1) k_wave_resident(const __grid_constant__ ResCall k)
{
    constexpr int SI = 0, SF = (G == 4) ? 1 : 0, SZ = SF + 1, SO = SF + 2;
    constexpr int NA = PEEP ? G - 1 : G;                       // slots of the first exchange of layer-norm sums
    extern __shared__ __align__(128) uint8_t rs_smem[];
    uint8_t *const smem = rs_smem;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cl = k.cl, T = k.T, NT = k.nt, hw = k.hw, xw = k.xw;
    const int cluster = (int)blockIdx.x / cl, rank = (int)blockIdx.x - cluster * cl;
    const int li = cluster / k.rg, gu = cluster - li * k.rg;
    const ResLayer &L = k.layer[li];
    const bool proj = (L.flags & F_PROJECTION) != 0;
    const int row0 = (int)((long long)gu * k.B / k.rg), rows = (int)((long long)(gu + 1) * k.B / k.rg) - row0;
    const int r8 = NT * 8, ntr = (rows + 7) >> 3;
    // own cells and outputs, in groups of eight
    const int u0 = rank * L.cpc, o_lo = proj ? rank * L.opc : u0;
    int cells = L.C - u0 < L.cpc ? L.C - u0 : L.cpc, outs = proj ? (L.O - o_lo < L.opc ? L.O - o_lo : L.opc) : cells;
    if (cells < 0) cells = 0;
    if (outs < 0) outs = 0;
    const int ncg = (cells + 7) >> 3, nog = (outs + 7) >> 3;
    const int ncb = (L.C + L.cpc - 1) / L.cpc, nob = proj ? (L.O + L.opc - 1) / L.opc : ncb;       // blocks with cells, with outputs
    const int uw = (hw / NT < ncg ? hw / NT : ncg) * ntr, xn = ncg * ntr < xw ? ncg * ntr : xw;    // warps with cells; that compute X
    // projection: tasks of 16 outputs, eight rows and a part of K
    const int tn = proj ? ((nog + 1) >> 1) * ntr : 0;
    int parts = tn > 0 && tn < k.pw ? k.pw / tn : 1;
    if (parts > L.kc) parts = L.kc;
    const int pw = tn * parts < k.pw ? tn * parts : k.pw, fw = proj ? (tn < k.pw ? tn : k.pw) : uw;    // warps with such tasks; that write h
    const uint32_t h_remote = cells > 0 ? (uint32_t)(rows * 8 * (((L.O + 7) >> 3) - nog)) : 0u;
    const uint32_t m_remote = proj && outs > 0 ? (uint32_t)(rows * 8 * (((L.C + 7) >> 3) - ncg)) : 0u;
    const uint32_t s_remote = LN && cells > 0 ? (uint32_t)(rows * 16 * (ncb - 1)) : 0u;           // per slot

    const RsLayout lay = rs_layout(L, cl, NT, hw, k.pw, LN, PEEP);
    RsCtl *ctl = reinterpret_cast<RsCtl *>(smem + lay.ctl);
    volatile int *abort_flag = &ctl->abort_flag;
    const size_t w_r = (size_t)(L.cpc >> 3) * L.ki * G * 512, w_p = w_r + (size_t)(L.cpc >> 3) * L.kh * G * 512;
    RsSmem s;
    s.bx = (int4 *)(smem + lay.consts);
    s.bh = s.bx + L.cpc;
    s.bln = s.bh + L.cpc;
    s.L = (uint2 *)(s.bln + L.cpc);
    s.P = s.L + L.cpc;
    s.bp = (int32_t *)(s.P + L.cpc);
    s.st = (uint32_t *)(smem + lay.st);
    s.ln = (WvLnRow *)(smem + lay.ln);
    s.sx = (uint4 *)(smem + lay.sx);
    s.sc = ctl->sc;
    constexpr int ST = PEEP ? 15 : 12;

    if (threadIdx.x == 0) {
        const uint32_t stuck = k.missing;                      // arrivals that never come (failure-path check)
        ptx::mbar_init(&ctl->w_full, 1);
        for (int i = 0; i < RS_NX; ++i) { ptx::mbar_init(&ctl->x_full[i], 1); ptx::mbar_init(&ctl->x_empty[i], xn > 0 ? xn : 1); }
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(&ctl->h_full[i], fw + (h_remote ? 1u : 0u) + stuck + (fw + h_remote + stuck == 0u ? 1u : 0u));
            ptx::mbar_init(&ctl->h_read[i], 1);
            ptx::mbar_init(&ctl->xg_full[i], xn > 0 ? xn : 1);
            ptx::mbar_init(&ctl->xg_free[i], uw > 0 ? uw : 1);
            ptx::mbar_init(&ctl->s_full[i], 1);
        }
        ptx::mbar_init(&ctl->m_full, uw + (m_remote ? 1u : 0u) + (uw + m_remote == 0u ? 1u : 0u));
        ptx::mbar_init(&ctl->l_sync, uw > 0 ? uw : 1);
        ptx::mbar_init(&ctl->p_sync, pw > 0 ? pw : 1);
        ctl->abort_flag = 0;
        ctl->x_issued = 0;
        ptx::fence_barrier_init();
        if (h_remote) for (int i = 0; i < 2; ++i) ptx::mbar_arrive_expect_tx(&ctl->h_full[i], h_remote);
        if (m_remote) ptx::mbar_arrive_expect_tx(&ctl->m_full, m_remote);
        if (s_remote) {
            ptx::mbar_arrive_expect_tx(&ctl->s_full[0], s_remote * NA);
            if (PEEP) ptx::mbar_arrive_expect_tx(&ctl->s_full[1], s_remote);
        }
        // weights and tables
        if (ncg + nog > 0) {
            const int8_t *img = L.img + (size_t)rank * L.img_stride;
            const size_t at[3] = {0, w_r, w_p};
            const uint32_t n[3] = {(uint32_t)(ncg * L.ki * G * 512), (uint32_t)(ncg * L.kh * G * 512), proj ? (uint32_t)(nog * L.kc * 512) : 0u};
            ptx::mbar_arrive_expect_tx(&ctl->w_full, n[0] + n[1] + n[2] + L.tab_lay.bytes);
            ptx::bulk_load_1d(smem + lay.tab, L.tab, L.tab_lay.bytes, &ctl->w_full);
            for (int i = 0; i < 3; ++i)
                for (uint32_t d = 0; d < n[i]; d += 32768u)
                    ptx::bulk_load_1d(smem + at[i] + d, img + at[i] + d, n[i] - d < 32768u ? n[i] - d : 32768u, &ctl->w_full);
        }
    }
    for (int i = threadIdx.x; i < 4 * L.cpc; i += blockDim.x) {
        const int ul = i >> 2, g = i & 3, n = (u0 + ul) * G + g;
        const bool in = g < G && ul < cells;
        ((int32_t *)s.bx)[i] = in ? L.bx[n] : 0;
        ((int32_t *)s.bh)[i] = in ? L.bh[n] : 0;
        ((int32_t *)s.bln)[i] = in && LN ? L.bln[n] : 0;
        ((int16_t *)s.L)[i] = in && LN ? L.L[n] : (int16_t)0;
        ((int16_t *)s.P)[i] = in && PEEP ? L.P[n] : (int16_t)0;
    }
    if (proj)
        for (int i = threadIdx.x; i < L.opc; i += blockDim.x) s.bp[i] = i < outs ? L.bp[o_lo + i] : 0;
    if (threadIdx.x < RS_SCALES) {
        const int i = threadIdx.x, e = i & 3;
        ctl->sc[i] = i < RS_SC_H ? rs_scale(L.f_x[e], L.x_left[e]) : i < RS_SC_C ? rs_scale(L.f_h[e], L.h_left[e]) : i < RS_SC_LN ? rs_scale(L.f_c[e], 0)
                   : i < RS_SC_M ? rs_scale(L.f_ln[e], 0) : rs_scale(i == RS_SC_M ? L.f_m : L.f_proj, 0);
    }
    if (LN) {
        for (int i = threadIdx.x; i < 2 * ST * r8; i += blockDim.x) s.st[i] = 0u;
        // (rows that the group does not have: a sigma of zero, whose quotients are zero)
        for (int i = threadIdx.x; i < 16 * r8; i += blockDim.x) ((uint32_t *)s.ln)[i] = 0u;
    }
    if (cells > 0)
        for (int i = threadIdx.x; i < rows * L.O; i += blockDim.x) {
            const int r = i / L.O;
            smem[lay.h + (size_t)r * L.ph + (i - r * L.O)] = (uint8_t)L.h[(size_t)row0 * L.O + i];
        }
    wv_cluster_sync();

    if (warp == 0) {
        // ---------------- x ----------------
        if (cells > 0)
            for (int t = 0; t < T; ++t) {
                const int slot = t % RS_NX;
                if (t >= RS_NX && !rs_wait(k, &ctl->x_empty[slot], (uint32_t)(t / RS_NX - 1) & 1u, abort_flag)) break;
                uint8_t *dst = smem + lay.x + (size_t)slot * r8 * L.px;
                if (L.in_img) {
                    if (!wv_wait_blocks(k, L.cnt_in + gu * WC_WORDS, L.below, (unsigned)(t + 1), abort_flag)) break;
                    if (lane == 0) {
                        wv_fence_async_global();
                        ptx::mbar_arrive_expect_tx(&ctl->x_full[slot], (uint32_t)(rows * L.px));
                        ptx::bulk_load_1d(dst, L.in_img + ((size_t)t * k.B + row0) * L.px, (uint32_t)(rows * L.px), &ctl->x_full[slot]);
                        ctl->x_issued = t + 1;
                    }
                    __syncwarp();
                    continue;
                }
                const int8_t *src = k.x + ((size_t)(L.dir ? T - 1 - t : t) * k.B + row0) * L.I;
                if (k.x_bulk) {
                    if (lane == 0) { ptx::mbar_arrive_expect_tx(&ctl->x_full[slot], (uint32_t)(rows * L.I)); ctl->x_issued = t + 1; }
                    __syncwarp();
                    if (lane < rows) ptx::bulk_load_1d(dst + (size_t)lane * L.px, src + (size_t)lane * L.I, (uint32_t)L.I, &ctl->x_full[slot]);
                    __syncwarp();
                    continue;
                }
                // rows of any length: words from aligned words (x itself is aligned; nothing is read past its end)
                const int wpr = (L.I + 3) >> 2;
                const int8_t *end = k.x + (size_t)T * k.B * L.I;
                for (int r = 0; r < rows; ++r) {
#pragma unroll 4
                    for (int j = lane; j < wpr; j += 32) {
                        const int8_t *a = src + (size_t)r * L.I + 4 * j;
                        const uint32_t sh = (uint32_t)((uintptr_t)a & 3u) * 8u;
                        const int8_t *al = a - (sh >> 3);
                        uint32_t v = 0;
                        if (al + 8 <= end) {
                            const uint32_t lo = *reinterpret_cast<const uint32_t *>(al), hi = *reinterpret_cast<const uint32_t *>(al + 4);
                            v = __funnelshift_r(lo, hi, sh);
                        } else {
                            for (int b = 0; b < 4; ++b)
                                if (a + b < end) v |= (uint32_t)(uint8_t)a[b] << (8 * b);
                        }
                        *reinterpret_cast<uint32_t *>(dst + (size_t)r * L.px + 4 * j) = v;
                    }
                }
                rs_arrive(&ctl->x_full[slot], lane);
            }
    } else if (warp == 1) {
        // ---------------- h^t for the layer above, or y; the final h ----------------
        const int items = rows * nog;
        const bool last = L.out_img == nullptr;
        int t = 0;
        while (outs > 0 && t < T) {
            bool ok = true;
            unsigned n = 0;
            // two steps per arrival where two are there: the release waits for the stores, about as long as a short step
            while (t < T && n < 2) {
                const uint32_t par = (uint32_t)(t >> 1) & 1u;
                if (n == 0) { if (!rs_wait(k, &ctl->h_full[(t + 1) & 1], par, abort_flag)) { ok = false; break; } }
                else if (!rs_test(&ctl->h_full[(t + 1) & 1], par)) break;
                const uint8_t *src = smem + lay.h + (size_t)((t + 1) & 1) * r8 * L.ph + o_lo;
                const int ty = L.dir ? T - 1 - t : t;
                for (int i = lane; i < items; i += 32) {
                    const int r = i / nog, j = (i - r * nog) * 8, b = row0 + r;
                    const uint2 v = *reinterpret_cast<const uint2 *>(src + (size_t)r * L.ph + j);
                    const int valid = outs - j < 8 ? outs - j : 8;
                    if (!last) {
                        *reinterpret_cast<uint2 *>(L.out_img + ((size_t)t * k.B + b) * L.out_pitch + o_lo + j) = v;
                    } else {
                        int8_t *y = k.y + ((size_t)ty * k.B + b) * k.y_stride + L.y_off + o_lo + j;
                        if (k.y_wide && valid == 8) *reinterpret_cast<uint2 *>(y) = v;
                        else for (int e = 0; e < valid; ++e) y[e] = (int8_t)((e < 4 ? v.x >> (8 * e) : v.y >> (8 * (e - 4))) & 255u);
                    }
                    if (t == T - 1)
                        for (int e = 0; e < valid; ++e) L.h[(size_t)b * L.O + o_lo + j + e] = (int8_t)((e < 4 ? v.x >> (8 * e) : v.y >> (8 * (e - 4))) & 255u);
                }
                rs_arrive(&ctl->h_read[(t + 1) & 1], lane);
                ++t; ++n;
            }
            if (!ok) break;
            if (!last) {
                wv_fence_async_global();
                __syncwarp();
                if (lane == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(L.cnt_out + gu * WC_WORDS + rank), "r"(n) : "memory");
            }
        }
    } else if (warp < 2 + hw) {
        // ---------------- gate sums, layer norm, cells: h^{t-1} and X to m (h without a projection) ----------------
        const int cw = warp - 2, g = lane >> 2, q = lane & 3, nt = cw % NT, cg0 = cw / NT, cstep = hw / NT;
        const bool has_units = cg0 < ncg && nt * 8 < rows;
        const int uidx = cg0 * ntr + nt;                       // number of this warp among those with cells
        const int ra = nt * 8 + 2 * q, r_sh = NT == 1 ? 3 : NT == 2 ? 4 : 5;       // this lane's rows, within the group
        const int kh = rs_keep(L.kh), ph = rs_keep(L.ph), zp_m = rs_keep(L.zp_m), m_bits = rs_keep(L.m_bits), pm = rs_keep(L.pm);
        // this lane's operand fragments and the place of its row in the buffers
        const uint8_t *const w_h = smem + w_r + (size_t)cg0 * kh * G * 512 + lane * 16;
        const int h_unit = rs_keep(cstep * kh * G * 512), h_step = rs_keep(r8 * ph), xg_step = rs_keep((L.cpc >> 3) * NT * 512);
        const int bh_at = (nt * 8 + g) * ph + q * 16, row_at = nt * 8 + (lane & 7);
        const uint8_t *const xg0 = smem + lay.xg + (size_t)(cg0 * NT + nt) * 512 + lane * 16;
        const bool row_ok = row_at < rows;
        uint32_t peer[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = (lane >> 3) + 4 * j;
            peer[j] = (uint32_t)rs_keep((int)(wv_peer(ptx::smem_u32(smem), p < cl ? p : 0) - ptx::smem_u32(smem)));
        }
        const ActLines at = make_act_lines(ptx::smem_u32(smem + lay.tab), L.tab_lay);
        uint8_t *stage = smem + lay.stage + (size_t)cw * 64;
        uint8_t *const hbuf = smem + lay.h, *const mbuf = smem + lay.m;
        uint32_t c[U];                                         // cell states: low half row ra, high half the next
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int ul = (cg0 + i * cstep) * 8 + g;
            int32_t v[2] = {0, 0};
            for (int j = 0; j < 2; ++j)
                if (has_units && ul < cells && ra + j < rows) v[j] = L.c[(size_t)(row0 + ra + j) * L.C + u0 + ul];
            c[i] = (uint32_t)(uint16_t)v[0] | ((uint32_t)(uint16_t)v[1] << 16);
        }
        bool run = has_units && rs_wait(k, &ctl->w_full, 0, abort_flag);
        uint32_t ln_par = 0;                                   // parity of the next block-wide meeting of the layer norm
        int done = 0;
        for (int t = 0; run && t < T; ++t) {
            const uint32_t par = (uint32_t)t & 1u, par2 = (uint32_t)(t >> 1) & 1u;
            uint4 xg[U];
            if (!rs_wait(k, &ctl->xg_full[t & 1], par2, abort_flag)) break;
#pragma unroll
            for (int i = 0; i < U; ++i) xg[i] = *reinterpret_cast<const uint4 *>(xg0 + (t & 1) * xg_step + (cg0 + i * cstep < ncg ? i * cstep * NT * 512 : 0));
            rs_arrive(&ctl->xg_free[t & 1], lane);
            // h^t goes into buffer (t + 1) & 1, whose h^{t-2} has been written out
            if (!proj && t >= 2 && !rs_wait(k, &ctl->h_read[(t + 1) & 1], par2 ^ 1u, abort_flag)) break;
            if (t > 0) {
                if (!rs_wait(k, &ctl->h_full[t & 1], (uint32_t)((t - 1) >> 1) & 1u, abort_flag)) break;
                if (cw == 0 && lane == 0 && h_remote && t + 1 < T) ptx::mbar_arrive_expect_tx(&ctl->h_full[t & 1], h_remote);
            }
            const uint8_t *b = hbuf + bh_at + (t & 1) * h_step;
            const uint4 f_m = s.sc[RS_SC_M];
            uint32_t gw[U][4], xo[U];                          // gate sums
            int32_t sum[8], lo[8], hi[8];
            if (LN)
#pragma unroll
                for (int e = 0; e < 8; ++e) sum[e] = lo[e] = hi[e] = 0;
            int32_t mv[U][2];
            // nonlinearities, cell update and hidden state of unit i from its gate values
            auto cell = [&](int i, int cg, const int32_t (&a)[4][2], int32_t (&out)[2]) {
                int32_t cn[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int32_t f = line_sigmoid(at, a[SF][j]), z = line_tanh_gate(at, a[SZ][j]);
                    int32_t ig;
                    if (G == 4) ig = line_sigmoid(at, a[SI][j]);
                    else { ig = 32768 - f; if (ig > 32767) ig = 32767; }               // coupled input gate, Section 3.2.9
                    cn[j] = cell_update_fast(ig, z, f, j ? wv_hi(c[i]) : wv_lo(c[i]), m_bits);
                }
                c[i] = ptx::pack_sat_s16(cn[0], cn[1]);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    int32_t o = a[SO][j];
                    if (PEEP) o = sat16(o + sat16(rs_rescale(rs_s16(s.P[cg * 8 + g], SO) * cn[j], s.sc[RS_SC_C + SO])));     // Eq. 5
                    if (PEEP && LN) out[j] = o;                // waits for the row's statistics
                    else out[j] = rs_hidden(f_m, zp_m, at, o, cn[j]);
                }
            };
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int cg = cg0 + i * cstep;
                if (cg >= ncg) continue;
                int32_t acc[2][4], a[4][2];
                rs_gates<G>(acc, w_h + i * h_unit, b, kh);
                const int4 bh = s.bh[cg * 8 + g];
                const bool in = cg * 8 + g < cells;
                const uint32_t xw4[4] = {xg[i].x, xg[i].y, xg[i].z, xg[i].w};
                uint2 P = make_uint2(0, 0);
                if (PEEP) P = s.P[cg * 8 + g];
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    const uint4 f = s.sc[RS_SC_H + e];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        int32_t v = sat16(rs_rescale((rs_acc(acc, e, j) + rs_i4(bh, e)) << f.w, f));
                        v += j ? wv_hi(xw4[e]) : wv_lo(xw4[e]);
                        if (PEEP && e != SZ && e != SO) v += sat16(rs_rescale(rs_s16(P, e) * (j ? wv_hi(c[i]) : wv_lo(c[i])), s.sc[RS_SC_C + e]));
                        if (!(PEEP && e == SO)) v = sat16(v);                  // (output gate with a peephole: X + H, within 17 bits)
                        a[e][j] = v;
                        if (LN && !(PEEP && e == SO)) {
                            const int32_t w = in ? v : 0;
                            sum[2 * e + j] += w;
                            lo[2 * e + j] += (int32_t)((uint32_t)(w * w) & 0xfffffu);
                            hi[2 * e + j] += (int32_t)((uint32_t)(w * w) >> 20);
                        }
                    }
                }
                if (!LN) cell(i, cg, a, mv[i]);
                else {
#pragma unroll
                    for (int e = 0; e < G; ++e)
                        if (!(PEEP && e == SO)) gw[i][e] = ptx::pack_sat_s16(a[e][0], a[e][1]);
                    if (PEEP) { gw[i][SO] = (uint32_t)a[SO][0]; xo[i] = (uint32_t)a[SO][1]; }
                }
            }
            if (LN) {
                // sums of this warp's cells -> of the block -> of the cluster -> constants of each (slot, row)
                auto add = [&](uint32_t *st, int slot, int row, int32_t s1, int32_t s2, int32_t s3) {
                    atomicAdd(st + (slot * 3 + 0) * r8 + row, (uint32_t)s1);
                    atomicAdd(st + (slot * 3 + 1) * r8 + row, (uint32_t)s2);
                    atomicAdd(st + (slot * 3 + 2) * r8 + row, (uint32_t)s3);
                };
                // slots [e0, e0 + ne): block's sums in st at slot z0; peers' sums in sx
                auto exchange = [&](uint32_t *st, uint32_t *st_next, int z0, int e0, int ne, uint4 *sx, int sx_slots, uint64_t *bar) -> bool {
                    rs_arrive(&ctl->l_sync, lane);
                    if (!rs_wait(k, &ctl->l_sync, ln_par, abort_flag)) return false;
                    ln_par ^= 1u;
                    const int nc = ne * r8;                    // (slot, row) of a lane: rows are a power of two apart
                    if (ncb > 1)
                        for (int p = uidx; p < ncb; p += uw)
                            for (int w = lane; w < nc && p != rank; w += 32) {
                                const int e = w >> r_sh, r = w & (r8 - 1);
                                if (r >= rows) continue;
                                const uint32_t *v = st + (z0 + e) * 3 * r8 + r;
                                uint4 *dst = sx + ((size_t)rank * sx_slots + e) * r8 + r;
                                wv_send16(wv_peer(ptx::smem_u32(dst), p), make_uint4(v[0], v[r8], v[2 * r8], 0u), wv_peer(ptx::smem_u32(bar), p));
                            }
                    for (int i0 = uidx * 32; i0 < nc; i0 += uw * 32) {
                        if (ncb > 1 && !rs_wait(k, bar, par, abort_flag)) return false;
                        if (i0 == 0 && lane == 0 && ncb > 1 && t + 1 < T) ptx::mbar_arrive_expect_tx(bar, s_remote * (uint32_t)ne);
                        const int w = i0 + lane;
                        const int e = w >> r_sh, r = w & (r8 - 1);
                        if (w >= nc || r >= rows) continue;
                        const uint32_t *v = st + (z0 + e) * 3 * r8 + r;
                        int32_t s1 = (int32_t)v[0];
                        uint32_t s2 = v[r8], s3 = v[2 * r8];
                        uint32_t *nx = st_next + (z0 + e) * 3 * r8 + r;
                        nx[0] = nx[r8] = nx[2 * r8] = 0u;
#pragma unroll 4
                        for (int p = 0; p < ncb; ++p)
                            if (p != rank) {
                                const uint4 o = sx[((size_t)p * sx_slots + e) * r8 + r];
                                s1 += (int32_t)o.x; s2 += o.y; s3 += o.z;
                            }
                        s.ln[(e0 + e) * r8 + r] = wv_make_ln(s1, ((int64_t)s3 << 20) + s2, L.div_c, L.sigma_min);
                    }
                    rs_arrive(&ctl->l_sync, lane);
                    if (!rs_wait(k, &ctl->l_sync, ln_par, abort_flag)) return false;
                    ln_par ^= 1u;
                    return true;
                };
                uint32_t *st = s.st + (t & 1) * ST * r8, *st_next = s.st + ((t + 1) & 1) * ST * r8;
                {
                    const int32_t s1 = rs_sum_cells(sum, lane), s2 = rs_sum_cells(lo, lane), s3 = rs_sum_cells(hi, lane);
                    if ((g >> 1) < NA) add(st, g >> 1, nt * 8 + 2 * q + (g & 1), s1, s2, s3);
                }
                if (!exchange(st, st_next, 0, 0, NA, s.sx, 4, &ctl->s_full[0])) break;
                int32_t so[8], qlo[8], qhi[8];
                if (PEEP)
#pragma unroll
                    for (int e = 0; e < 8; ++e) so[e] = qlo[e] = qhi[e] = 0;
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const int cg = cg0 + i * cstep;
                    if (cg >= ncg) continue;
                    const int4 bln = s.bln[cg * 8 + g];
                    const uint2 Lw = s.L[cg * 8 + g];
                    int32_t a[4][2];
                    uint32_t slow = 0;
#pragma unroll
                    for (int e = 0; e < G; ++e)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            if (PEEP && e == SO) continue;
                            const WvLnRow r = s.ln[e * r8 + ra + j];
                            slow |= r.sigma;
                            a[e][j] = wv_ln_fast(j ? wv_hi(gw[i][e]) : wv_lo(gw[i][e]), r.m_hi, r.m_lo, r.mean, rs_s16(Lw, e), rs_i4(bln, e));
                        }
                    if (slow & WV_LN_SLOW) {
                        // (rows whose sigma is too small for 32-bit products)
#pragma unroll
                        for (int e = 0; e < G; ++e)
#pragma unroll
                            for (int j = 0; j < 2; ++j)
                                if (!(PEEP && e == SO))
                                    a[e][j] = wv_ln_slow(j ? wv_hi(gw[i][e]) : wv_lo(gw[i][e]), s.ln[e * r8 + ra + j], rs_s16(Lw, e), rs_i4(bln, e));
                    }
#pragma unroll
                    for (int e = 0; e < G; ++e) {
                        const uint4 f = s.sc[RS_SC_LN + e];
#pragma unroll
                        for (int j = 0; j < 2; ++j) a[e][j] = PEEP && e == SO ? (int32_t)(j ? xo[i] : gw[i][SO]) : sat16(rs_rescale(a[e][j], f));
                    }
                    cell(i, cg, a, mv[i]);
                    if (PEEP) {
                        const bool in = cg * 8 + g < cells;
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const int32_t w = in ? mv[i][j] : 0;
                            so[j] += w;
                            qlo[j] += (int32_t)((uint32_t)(w * w) & 0xfffffu);
                            qhi[j] += (int32_t)((uint32_t)(w * w) >> 20);
                        }
                    }
                }
                if (PEEP) {
                    const int32_t s1 = rs_sum_cells(so, lane), s2 = rs_sum_cells(qlo, lane), s3 = rs_sum_cells(qhi, lane);
                    if (g < 2) add(st, 4, nt * 8 + 2 * q + g, s1, s2, s3);
                    if (!exchange(st, st_next, 4, SO, 1, s.sx + (size_t)cl * 4 * r8, 1, &ctl->s_full[1])) break;
                    const WvLnRow r[2] = {s.ln[SO * r8 + ra], s.ln[SO * r8 + ra + 1]};
                    const uint4 f = s.sc[RS_SC_LN + SO];
#pragma unroll
                    for (int i = 0; i < U; ++i) {
                        const int cg = cg0 + i * cstep;
                        if (cg >= ncg) continue;
                        const int32_t b2 = rs_i4(s.bln[cg * 8 + g], SO), Lw = rs_s16(s.L[cg * 8 + g], SO);
                        int32_t v[2];
#pragma unroll
                        for (int j = 0; j < 2; ++j) v[j] = wv_ln_fast(mv[i][j], r[j].m_hi, r[j].m_lo, r[j].mean, Lw, b2);
                        if ((r[0].sigma | r[1].sigma) & WV_LN_SLOW)
                            for (int j = 0; j < 2; ++j) v[j] = wv_ln_slow(mv[i][j], s.ln[SO * r8 + ra + j], Lw, b2);
#pragma unroll
                        for (int j = 0; j < 2; ++j) mv[i][j] = rs_hidden(f_m, zp_m, at, sat16(rs_rescale(v[j], f)), j ? wv_hi(c[i]) : wv_lo(c[i]));
                    }
                }
            }
            // m, or h without a projection, to the blocks that read it
            uint8_t *dst = proj ? mbuf + row_at * pm : hbuf + ((t + 1) & 1) * h_step + row_at * ph;
            uint64_t *bar = proj ? &ctl->m_full : &ctl->h_full[(t + 1) & 1];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int cg = cg0 + i * cstep;
                if (cg < ncg) rs_send_tile(stage, mv[i][0], mv[i][1], dst + u0 + cg * 8, row_ok, ptx::smem_u32(bar), peer, rank, proj ? nob : ncb, lane);
            }
            rs_arrive(bar, lane);
            done = t + 1;
        }
        // nothing that peers send may be under way when the block ends; a block that did not get this far leaves the state as the caller had it
        if (done == T && rs_wait(k, &ctl->h_full[T & 1], (uint32_t)((T - 1) >> 1) & 1u, abort_flag))
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int ul = (cg0 + i * cstep) * 8 + g;
                for (int j = 0; j < 2; ++j)
                    if (ul < cells && ra + j < rows) L.c[(size_t)(row0 + ra + j) * L.C + u0 + ul] = (int16_t)(j ? wv_hi(c[i]) : wv_lo(c[i]));
            }
    } else if (warp < 2 + hw + xw) {
        // ---------------- X = rescaled W x_t, a step or two ahead ----------------
        const int xi = warp - 2 - hw, g = lane >> 2, q = lane & 3;
        const int ki = rs_keep(L.ki), px = rs_keep(L.px), xg_step = rs_keep((L.cpc >> 3) * NT * 512), x_step = rs_keep(r8 * L.px);
        bool run = xi < xn && rs_wait(k, &ctl->w_full, 0, abort_flag);
        for (int t = 0; run && t < T; ++t) {
            const int slot = t & (RS_NX - 1);
            if (!rs_wait(k, &ctl->x_full[slot], (uint32_t)((unsigned)t / RS_NX) & 1u, abort_flag)) break;
            if (t >= 2 && !rs_wait(k, &ctl->xg_free[t & 1], ((uint32_t)(t >> 1) & 1u) ^ 1u, abort_flag)) break;
            for (int cg = ntr == 1 ? xi : xi / ntr, nt = ntr == 1 ? 0 : xi % ntr; cg < ncg;) {
                int32_t acc[2][4];
                rs_gates<G>(acc, smem + (size_t)cg * ki * G * 512 + lane * 16, smem + lay.x + slot * x_step + (nt * 8 + g) * px + q * 16, ki);
                const int4 bx = s.bx[cg * 8 + g];
                uint32_t o[4] = {0, 0, 0, 0};
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    const uint4 f = s.sc[RS_SC_X + e];
                    o[e] = ptx::pack_sat_s16(rs_rescale((rs_acc(acc, e, 0) + rs_i4(bx, e)) << f.w, f), rs_rescale((rs_acc(acc, e, 1) + rs_i4(bx, e)) << f.w, f));
                }
                *reinterpret_cast<uint4 *>(smem + lay.xg + (t & 1) * xg_step + (size_t)(cg * NT + nt) * 512 + lane * 16) = make_uint4(o[0], o[1], o[2], o[3]);
                for (nt += xw; nt >= ntr; nt -= ntr) ++cg;
            }
            rs_arrive(&ctl->x_empty[slot], lane);
            if (lane == 0) ptx::mbar_arrive(&ctl->xg_full[t & 1]);
        }
    } else {
        // ---------------- projection: m to h ----------------
        const int pi = warp - 2 - hw - xw, g = lane >> 2, q = lane & 3;
        const int kc = rs_keep(L.kc), ph = rs_keep(L.ph), pm = rs_keep(L.pm), zp_h = rs_keep(L.zp_h), h_step = rs_keep(r8 * ph);
        uint32_t peer[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = (lane >> 3) + 4 * j;
            peer[j] = (uint32_t)rs_keep((int)(wv_peer(ptx::smem_u32(smem), p < cl ? p : 0) - ptx::smem_u32(smem)));
        }
        uint8_t *stage = smem + lay.stage + (size_t)(hw + pi) * 64;
        uint8_t *const hbuf = smem + lay.h, *const mbuf = smem + lay.m;
        const int task0 = tn > 0 ? pi % tn : 0, part = tn > 0 ? pi / tn : 0;       // (more tasks than warps: one part, task pi, pi + pw, ...)
        const int c0 = part * kc / parts, c1 = (part + 1) * kc / parts;
        bool run = proj && pi < pw && rs_wait(k, &ctl->w_full, 0, abort_flag);
        for (int t = 0; run && t < T; ++t) {
            const uint32_t par = (uint32_t)t & 1u, par2 = (uint32_t)(t >> 1) & 1u;
            if (part == 0 && t >= 2 && !rs_wait(k, &ctl->h_read[(t + 1) & 1], par2 ^ 1u, abort_flag)) break;
            if (!rs_wait(k, &ctl->m_full, par, abort_flag)) break;
            if (pi == 0 && lane == 0 && m_remote && t + 1 < T) ptx::mbar_arrive_expect_tx(&ctl->m_full, m_remote);
            const uint32_t bar = ptx::smem_u32(&ctl->h_full[(t + 1) & 1]);
            for (int task = task0; task < tn; task += k.pw) {
                const int tile = ntr == 1 ? task : task / ntr, rt = task - tile * ntr;
                const bool two = tile * 2 + 1 < nog;
                const uint8_t *w = smem + w_p + (tile * 2 * kc + c0) * 512 + lane * 16;
                const uint8_t *b = mbuf + (rt * 8 + g) * pm + q * 16 + c0 * 64;
                int32_t acc[2][4];
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[0][j] = acc[1][j] = 0;
                const int second = two ? kc * 512 : 0;         // (one group of eight outputs: its products twice)
#pragma unroll 4
                for (int ch = c0; ch < c1; ++ch, w += 512, b += 64) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(b), s0 = *reinterpret_cast<const uint4 *>(w);
                    const uint4 s1 = *reinterpret_cast<const uint4 *>(w + second);
                    rs_mma(acc[0], s0.x, s1.x, s0.y, s1.y, v.x, v.y);
                    rs_mma(acc[1], s0.z, s1.z, s0.w, s1.w, v.z, v.w);
                }
                int4 d = make_int4(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1], acc[0][2] + acc[1][2], acc[0][3] + acc[1][3]);
                if (parts > 1) {
                    int4 *pp = reinterpret_cast<int4 *>(smem + lay.part);
                    if (part > 0) pp[pi * 32 + lane] = d;
                    rs_arrive(&ctl->p_sync, lane);
                    if (part > 0) break;
                    if (!rs_wait(k, &ctl->p_sync, par, abort_flag)) { run = false; break; }
#pragma unroll 4
                    for (int e = 1; e < parts; ++e) {
                        const int4 o = pp[(e * tn + task) * 32 + lane];
                        d.x += o.x; d.y += o.y; d.z += o.z; d.w += o.w;
                    }
                }
                const int32_t v[4] = {d.x, d.y, d.z, d.w};
                const uint4 f = s.sc[RS_SC_P];
                uint8_t *dst = hbuf + ((t + 1) & 1) * h_step + (rt * 8 + (lane & 7)) * ph + o_lo + tile * 16;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (e == 1 && !two) break;
                    const int32_t bias = s.bp[(tile * 2 + e) * 8 + g];
                    rs_send_tile(stage, sat8(rs_rescale(v[2 * e] + bias, f) + zp_h), sat8(rs_rescale(v[2 * e + 1] + bias, f) + zp_h), dst + 8 * e,
                                 rt * 8 + (lane & 7) < rows, bar, peer, rank, ncb, lane);
                }
            }
            if (run && part == 0) rs_arrive(&ctl->h_full[(t + 1) & 1], lane);
        }
    }

    // ---------------- the end ----------------
    ptx::cta_sync();
    const bool aborted = *abort_flag != 0;
    if (aborted && warp == 0) {
        // copies under way end
        if (ncg + nog > 0) wv_drain(&ctl->w_full, 0);
        for (int i = 0; i < RS_NX; ++i) {
            const int n = (ctl->x_issued + RS_NX - 1 - i) / RS_NX;
            if (n > 0) wv_drain(&ctl->x_full[i], (uint32_t)(n - 1) & 1u);
        }
    }
    wv_cluster_sync();
    if (warp == 0) {
        if (aborted && lane == 0) {
            // what peers sent before they came here arrives within microseconds; this block does not end before
            atomicExch(k.abort_word, 1u);
            const unsigned long long t0 = wv_timer();
            while (wv_timer() - t0 < 50000ull) {}
        }
        // the last block reports, and leaves the counters as the next call wants them
        bool end = false;
        if (lane == 0) {
            __threadfence();
            end = atomicAdd(k.ticket, 1u) == gridDim.x - 1u;
            if (end) {
                __threadfence();
                *k.status = atomicExch(k.abort_word, 0u) ? 2 : 0;
                if (k.status2) *k.status2 = 0;
                *k.ticket = 0u;
            }
        }
        if (__any_sync(0xffffffffu, end))
            for (int i = lane; i < k.n_layers * k.rg * WC_WORDS; i += 32) k.cnt[i] = 0u;
    }
}

// A weight matrix into the blocks' images: [rank][eight rows' group][64 bytes of K][gate][row][64], rank images `stride` bytes apart.
__global__ void k_resident_tile(const int8_t *src, int8_t *dst, int G, int rows, int K, int n, int per, int nk, size_t stride)
{
    const int groups = per >> 3;
    const size_t total = (size_t)n * groups * nk * G * 32;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int piece = (int)(i & 3), r = (int)(i >> 2) & 7;
        size_t q = i >> 5;
        const int g = (int)(q % G); q /= G;
        const int ch = (int)(q % nk); q /= nk;
        const int cg = (int)(q % groups), rank = (int)(q / groups);
        const int row = (rank * per + cg * 8 + r) * G + g, k0 = ch * 64 + piece * 16;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (row < rows && k0 < K) v = wv_load16(src + (size_t)row * K + k0, K - k0);
        *reinterpret_cast<uint4 *>(dst + (size_t)rank * stride + ((((size_t)cg * nk + ch) * G + g) * 8 + r) * 64 + piece * 16) = v;
    }
}

template <int G, int U>
const void *rs_kernel_of(bool ln, bool peep)
{
    if (ln) return peep ? (const void *)k_wave_resident<G, true, true, U> : (const void *)k_wave_resident<G, true, false, U>;
    return peep ? (const void *)k_wave_resident<G, false, true, U> : (const void *)k_wave_resident<G, false, false, U>;
}
const void *rs_kernel(int G, bool ln, bool peep, int u)
{
    if (G == 4) return u == 1 ? rs_kernel_of<4, 1>(ln, peep) : u == 2 ? rs_kernel_of<4, 2>(ln, peep) : rs_kernel_of<4, 4>(ln, peep);
    return u == 1 ? rs_kernel_of<3, 1>(ln, peep) : u == 2 ? rs_kernel_of<3, 2>(ln, peep) : rs_kernel_of<3, 4>(ln, peep);
}

int rs_up(int v, int m) { return (v + m - 1) / m * m; }
int rs_pitch(int n) { return (rs_up(n, 64) / 64 | 1) * 64; }

// A stack shared out over clusters of one size.
struct ResShape {
    int cl = 0, clusters = 0;      // blocks per cluster, clusters that can be on the device together
    bool used = false;
    std::vector<ResLayer> layer;
};
struct ResPlan { int shape = -1, rg = 0, nt = 0, u = 0, hw = 0, xw = 0, pw = 0; size_t smem = 0; };

}  // namespace

struct ResidentStack {
    int max_T = 0, max_B = 0, G = 4, y_stride = 0;
    bool ln = false, peep = false, x_bulk = false, y_wide = false;
    std::vector<WaveLayer> base;
    std::vector<ResShape> shape;
    std::vector<ResPlan> by_rows;  // [B]
    unsigned *words = nullptr;     // abort word, ticket, counters: zero between calls
    size_t n_words = 0;
};

namespace {

// Clusters of cl blocks of this stack's kernel that fit on the device at once (a block per SM).
int rs_max_clusters(const ResidentStack *s, int cl, int max_smem)
{
    const void *f = rs_kernel(s->G, s->ln, s->peep, 1);
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(cl); c.blockDim = dim3(RS_THREADS); c.dynamicSmemBytes = (size_t)max_smem;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = (unsigned)cl; a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
    c.attrs = a; c.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, f, &c) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n;
}

// Shares of one layer's blocks.
void rs_share_layer(ResLayer &L, int cl)
{
    const bool proj = L.flags & F_PROJECTION;
    const int G = (L.flags & F_CIFG) ? 3 : 4;
    L.cpc = rs_up((L.C + cl - 1) / cl, 8);
    L.opc = proj ? rs_up((L.O + cl - 1) / cl, 8) : L.cpc;
    L.img_stride = (size_t)(L.cpc / 8) * (L.ki + L.kh) * G * 512 + (proj ? (size_t)(L.opc / 8) * L.kc * 512 : 0);
}

// The plan of calls of B rows under a shape, and an estimate of a step in us; false: does not fit.
// The estimate: least squares over 1900 calls of 64 steps, all cluster sizes, of 160 random stacks (one to eight layers of 32 to 900 cells with all
// variants, 1 to 256 rows), 9 % standard error.  What a warp does for its groups of eight cells one after the other costs more than an
// exchange saves, and with two or more groups per warp the layer norm's registers spill on top: many blocks of one group per warp are nearly
// always ahead (us per call of 64 steps in clusters of 1, 2, 4 and 8: two 208-cell layers with layer norm and projection, 4 rows 882, 353, 229 and
// 211; three 104-cell CIFG layers, 11 rows 187, 107, 83 and 76).  Over 130 other stacks the shape chosen was 2 % slower in the mean than the best
// one, 19 % at most, and no call was slower than on the kernels that take it otherwise (0.46 of their time in the mean, 0.96 at most; calls of 1, 4
// and 128 steps 1.01 to 5.5, 1.14 to 3.8 and 1.08 to 7.7 times as fast), so that a call that fits always comes here.
bool rs_try_plan(const ResidentStack *s, const ResShape &sh, int B, int max_smem, ResPlan &p, double &us)
{
    const int n = (int)sh.layer.size();
    int rg = std::min(B, sh.clusters / n);
    if (rg < 1) return false;
    const int rows = (B + rg - 1) / rg;
    rg = (B + rows - 1) / rows;
    p.rg = rg;
    p.nt = rows <= 8 ? 1 : rows <= 16 ? 2 : 4;
    if (rows > 8 * RS_MAX_NT) return false;
    int units = 0;
    bool proj = false;
    for (const ResLayer &L : sh.layer) {
        units = std::max(units, L.cpc / 8 * p.nt);
        proj = proj || (L.flags & F_PROJECTION);
    }
    p.hw = std::min(units, 8);
    const int u = (units + p.hw - 1) / p.hw;
    if (u > 4) return false;
    p.u = u == 3 ? 4 : u;
    p.xw = std::min(units, proj ? 4 : 8);
    p.pw = proj ? 4 : 0;
    p.smem = 0;
    us = 0;
    const int ntr = (rows + 7) / 8;
    const double ln = s->ln, ln_peep = s->ln && s->peep;
    for (const ResLayer &L : sh.layer) {
        p.smem = std::max(p.smem, rs_layout(L, sh.cl, p.nt, p.hw, p.pw, s->ln, s->peep).total);
        const double tiles = L.cpc / 8 * ntr, many = L.cpc < L.C;              // tiles of eight cells and rows; several blocks
        double e = 0.46 + 0.07 * L.kh * u + 0.088 * s->G * u + 0.07 * tiles + 0.0015 * tiles * L.ki * (s->G + 1) + many * 0.0001 * rows * L.O;
        if (p.u == 2) e += 0.06 + 0.99 * ln;
        if (p.u == 4) e += u * (0.13 + 0.83 * ln);
        e += ln * (1.16 + 0.144 * u + many * (0.0012 * rows * s->G + 0.058 * sh.cl)) + ln_peep * (1.16 + 0.07 * u + many * 0.33);
        if (L.flags & F_PROJECTION) {
            const int tasks = ((L.opc / 8 + 1) / 2) * ntr;
            e += 0.33 + 0.025 * L.kc * std::max(1.0, tasks / 4.0) + 0.067 * L.kc / std::max(1, p.pw / tasks);
        }
        us = std::max(us, e);
    }
    return p.smem <= (size_t)max_smem;
}

}  // namespace

ResidentStack *resident_plan(const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, int max_T, int max_B, int max_smem, int y_stride)
{
    const int n = (int)lp.size();
    size_t widest = 0;
    for (const LayerParams *p : lp)
        widest = std::max(widest, (size_t)p->N * (p->I + p->O) + ((p->flags & F_PROJECTION) ? (size_t)p->O * p->C : 0));
    if (widest > (size_t)RS_MAX_CLUSTER * max_smem) return nullptr;
    ResidentStack *s = new ResidentStack();
    s->max_T = max_T; s->max_B = max_B; s->G = lp[0]->G; s->y_stride = y_stride;
    s->ln = lp[0]->flags & F_LAYERNORM;
    s->peep = lp[0]->flags & F_PEEPHOLE;
    s->base = base;
    s->x_bulk = lp[0]->I % 16 == 0;
    s->y_wide = y_stride % 8 == 0;
    for (const WaveLayer &L : base)
        if (L.last && L.y_off % 8) s->y_wide = false;
    std::vector<ResLayer> layers;
    for (int l = 0; l < n; ++l) {
        const WaveLayer &W = base[l];
        ResLayer L;
        memset(&L, 0, sizeof(L));
        L.I = W.I; L.C = W.C; L.O = W.O; L.flags = W.flags; L.m_bits = W.m_bits; L.zp_m = W.zp_m; L.zp_h = W.zp_h;
        if (lp[l]->G == 3) L.flags |= F_CIFG;
        L.ki = (W.I + 63) / 64; L.kh = (W.O + 63) / 64; L.kc = (W.C + 63) / 64;
        L.px = rs_pitch(W.I); L.ph = rs_pitch(W.O); L.pm = rs_pitch(W.C);
        L.bx = W.bx; L.bh = W.bh; L.bln = W.bln; L.bp = W.bp; L.P = W.P; L.L = W.L;
        for (int g = 0; g < 4; ++g) {
            L.x_left[g] = W.x_left[g]; L.h_left[g] = W.h_left[g];
            L.f_x[g] = W.f_x[g]; L.f_h[g] = W.f_h[g]; L.f_c[g] = W.f_c[g]; L.f_ln[g] = W.f_ln[g];
        }
        L.f_m = W.f_m; L.f_proj = W.f_proj; L.div_c = W.div_c; L.sigma_min = W.sigma_min;
        L.dir = W.dir; L.y_off = W.y_off; L.tab_lay = W.tab_lay;
        layers.push_back(L);
    }
    // (setting an attribute loads a kernel, some milliseconds the first time in a process: the forms of several groups of cells per warp only
    // where a call takes them)
    bool loaded[5] = {};
    auto load = [&](int u) {
        if (loaded[u]) return true;
        const void *f = rs_kernel(s->G, s->ln, s->peep, u);
        loaded[u] = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem) == cudaSuccess &&
                    cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (!loaded[u]) cudaGetLastError();
        return loaded[u];
    };
    for (int cl = (int)std::max<size_t>(1, widest / max_smem); cl <= RS_MAX_CLUSTER; ++cl) {
        ResShape sh;
        sh.cl = cl;
        sh.layer = layers;
        bool fits = true;
        for (ResLayer &L : sh.layer) {
            rs_share_layer(L, cl);
            fits = fits && rs_layout(L, cl, 1, 1, 1, s->ln, s->peep).total <= (size_t)max_smem;
        }
        if (!fits) continue;
        if (!load(1)) break;
        sh.clusters = rs_max_clusters(s, cl, max_smem);
        if (sh.clusters < n) continue;
        s->shape.push_back(sh);
    }
    s->by_rows.resize((size_t)max_B + 1);
    size_t groups = 0;
    bool any = false;
    for (int B = max_B; B >= 1; --B) {
        // shapes that other calls of the handle take first: another one has to be 3 % ahead of them, for it has weight images of its own
        double line = 1e9;
        for (int fresh = 0; fresh < 2; ++fresh) {
            if (fresh && s->by_rows[B].shape >= 0) line *= 0.97;
            for (size_t i = 0; i < s->shape.size(); ++i) {
                ResPlan p;
                double us;
                if (s->shape[i].used == (fresh == 1) || !rs_try_plan(s, s->shape[i], B, max_smem, p, us) || us >= line || !load(p.u)) continue;
                line = us;
                p.shape = (int)i;
                s->by_rows[B] = p;
            }
        }
        if (s->by_rows[B].shape < 0) continue;
        any = true;
        s->shape[s->by_rows[B].shape].used = true;
        groups = std::max(groups, (size_t)s->by_rows[B].rg);
    }
    if (!any) { delete s; return nullptr; }
    s->n_words = 2 * WC_WORDS + (size_t)n * groups * WC_WORDS;
    return s;
}

void resident_destroy(ResidentStack *s) { delete s; }

int resident_place(ResidentStack *s, const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, WaveArena &keep, WaveArena &work, bool fill)
{
    const int n = (int)lp.size();
    keep.take(s->words, s->n_words * sizeof(unsigned));
    if (fill && cudaMemset(s->words, 0, s->n_words * sizeof(unsigned)) != cudaSuccess) return QLSTM_ERR_CUDA;
    std::vector<int8_t *> out(n, nullptr);
    for (int l = 0; l < n; ++l)
        if (!base[l].last) work.take(out[l], (size_t)s->max_T * s->max_B * rs_pitch(lp[l]->O));
    for (ResShape &sh : s->shape) {
        if (!sh.used) continue;
        for (int l = 0; l < n; ++l) {
            ResLayer &L = sh.layer[l];
            const LayerParams &p = *lp[l];
            int8_t *img;
            keep.take(img, (size_t)sh.cl * L.img_stride);
            L.img = img;
            L.tab = base[l].tab;
            L.out_img = out[l];
            L.out_pitch = rs_pitch(p.O);
            L.in_img = base[l].first ? nullptr : out[l - 1];
            if (!fill) continue;
            const size_t w_r = (size_t)(L.cpc / 8) * L.ki * p.G * 512, w_p = w_r + (size_t)(L.cpc / 8) * L.kh * p.G * 512;
            k_resident_tile<<<592, 256>>>(p.W, img, p.G, p.N, p.I, sh.cl, L.cpc, L.ki, L.img_stride);
            k_resident_tile<<<592, 256>>>(p.R, img + w_r, p.G, p.N, p.O, sh.cl, L.cpc, L.kh, L.img_stride);
            if (p.flags & F_PROJECTION) k_resident_tile<<<592, 256>>>(p.Wproj, img + w_p, 1, p.O, p.C, sh.cl, L.opc, L.kc, L.img_stride);
            if (cudaGetLastError() != cudaSuccess) return QLSTM_ERR_CUDA;
        }
    }
    return QLSTM_OK;
}

bool resident_supported(const ResidentStack *s, int T, int B)
{
    return s && T >= 1 && T <= s->max_T && B >= 1 && B <= s->max_B && s->by_rows[B].shape >= 0;
}

void resident_debug_plan(const ResidentStack *s, int T, int B, int *out4)
{
    const bool ok = resident_supported(s, T, B);
    const ResPlan p = ok ? s->by_rows[B] : ResPlan();
    out4[0] = ok ? s->shape[p.shape].cl : 0;
    out4[1] = p.rg; out4[2] = p.nt; out4[3] = p.u;
}

int launch_resident(const ResidentStack *s, const int8_t *x, int T, int B, int8_t *const (&h)[2], int16_t *const (&c)[2], int8_t *y, int *status,
                    int *status2, unsigned missing, unsigned long long limit_ns, bool refuse, cudaStream_t st)
{
    if (!resident_supported(s, T, B)) return QLSTM_ERR_DIM;
    const ResPlan &p = s->by_rows[B];
    const ResShape &sh = s->shape[p.shape];
    const int n = (int)sh.layer.size();
    ResCall k;
    k.T = T; k.B = B; k.n_layers = n; k.cl = sh.cl; k.rg = p.rg; k.nt = p.nt; k.hw = p.hw; k.xw = p.xw; k.pw = p.pw;
    k.x_bulk = s->x_bulk; k.y_wide = s->y_wide && ((uintptr_t)y & 7) == 0;
    k.x = x; k.y = y; k.y_stride = s->y_stride;
    k.abort_word = s->words; k.ticket = s->words + WC_WORDS; k.cnt = s->words + 2 * WC_WORDS;
    k.status = status; k.status2 = status2;
    k.limit_ns = limit_ns; k.missing = missing;
    for (int l = 0; l < n; ++l) {
        ResLayer &L = k.layer[l];
        L = sh.layer[l];
        L.cnt_out = k.cnt + (size_t)l * p.rg * WC_WORDS;
        if (L.in_img) {
            const ResLayer &D = sh.layer[l - 1];
            const int per = (D.flags & F_PROJECTION) ? D.opc : D.cpc;
            L.cnt_in = L.cnt_out - (size_t)p.rg * WC_WORDS;
            L.below = (D.O + per - 1) / per;
        }
        L.h = h[L.dir] + s->base[l].h_off * B;
        L.c = c[L.dir] + s->base[l].c_off * B;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n * p.rg * sh.cl)); cfg.blockDim = dim3((unsigned)(32 * (2 + p.hw + p.xw + p.pw))); cfg.dynamicSmemBytes = refuse ? WV_REFUSED_SMEM : p.smem; cfg.stream = st;
    cudaLaunchAttribute a[2];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = (unsigned)sh.cl; a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
    a[1].id = cudaLaunchAttributeCooperative;
    a[1].val.cooperative = 1;
    cfg.attrs = a; cfg.numAttrs = 2;
    void *args[] = {(void *)&k};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, rs_kernel(s->G, s->ln, s->peep, p.u), args);
    return e == cudaSuccess ? QLSTM_OK : wv_refused(e);
}

}  // namespace ql
