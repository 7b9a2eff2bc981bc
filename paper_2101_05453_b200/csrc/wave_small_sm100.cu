// Wavefront kernel for units of up to 32 batch rows.  The same schedule and the same exchanges as wave_sm100.cu (see the
// overview there), with the roles of the MMA operands swapped: the gate rows are the M side (128 tensor-memory lanes),
// the batch rows the N side (8 to 32 columns).  With so few rows a step is bound by the stream of weights and by its chain
// of exchanges, so the point of this form is that nothing else takes time:
//   - every lane holds a gate row, whatever the batch (with the batch as M, one row would use one lane of 128);
//   - a layer's input, its h and its m are a few kilobytes and arrive with one copy each;
//   - all accumulators of a step fit in tensor memory side by side, so X(t + 1) is accumulated as soon as the gate sums of
//     step t have been read, and is only rescaled together with H(t + 1).
// A gate tile holds up to 32 cells, gate slot g in the lanes 32 g .. 32 g + 31: a warp's lanes share a gate and its scales,
// and a row's layer-norm sums over a tile are warp-wide reductions.
//
// Two forms.  With CL a (layer, row group) is one thread-block cluster of up to 16 blocks, and what its own chain needs - layer-norm sums,
// m, h - goes from shared memory into the shared memory of the peers (16 or 8 bytes at a time, counted on an mbarrier there) instead of
// through L2 with a counter to poll and a copy back; only what the layer above reads is still written and published there, off the chain,
// each block in a word of its own (wv_wait_blocks).
// Without, groups may have any number of blocks.  A model fitted to measurements of both chooses (wave_cluster_plan).
#include <cstring>

#include "wave_common.cuh"

namespace ql {

namespace {

constexpr int WS_SLOTS = 8;
constexpr int WS_CHUNKS = 2;                   // gate chunks of a slot: a copy of 32 KB streams at 125 KB/us, one of 16 KB at 80, one
                                               // of 4 KB at 21 (about 0.2 us of the copying thread each)
constexpr int WS_MAX_TILES = 8;
constexpr int WS_ROWS = 32;

struct WsCtl {
    uint64_t w_full[WS_SLOTS], w_empty[WS_SLOTS];
    uint64_t op_full[3], op_empty[3];          // operands x, h, m
    uint64_t gate_full[WS_MAX_TILES], acc_empty, p_full, p_empty, tab_full, mma_done[2];
    uint64_t hx_full[2], mx_full, s_full[2];   // CL: what the cluster has sent to this block
    uint32_t tmem_base;
    int abort_flag, exit_at;
    int op_copies[3];              // copies of each operand that have been requested
    int end_slot;                  // where the weights' warp stopped in its ring
    uint32_t end_phase;
};

// [weight ring][x][h][m][control][constants][statistics][tables][gates][cell states][peers' sums][m and h on their way out]
struct WsLayout { size_t act[3], ctl, consts, st, ln, tab, gates, c, sx, stage_m, stage_h, total; };

__host__ __device__ inline WsLayout ws_layout(const WaveCall &k, int ns, int rows, bool peep)
{
    WsLayout l;
    l.act[0] = (size_t)ns * k.b_slot;
    l.act[1] = l.act[0] + (size_t)k.max_kb_i * k.ra * 128;
    l.act[2] = l.act[1] + (size_t)k.max_kb_h * k.ra * 128;
    if (k.cl) l.act[2] += (size_t)k.max_kb_h * k.ra * 128;     // (h in two buffers: peers may be a step ahead)
    l.ctl = l.act[2] + (size_t)k.max_kb_c * k.ra * 128;
    l.consts = l.ctl + wv_up(sizeof(WsCtl), 16);
    l.st = l.consts + wv_up((size_t)k.max_cpc * 4 * (3 * 4 + 2 * 2) + (size_t)k.max_opc * 4, 16);
    l.ln = l.st + 12 * WS_ROWS * 4;
    l.tab = l.ln + 4 * WS_ROWS * 16;
    l.gates = l.tab + wv_up((size_t)k.max_tab, 16);
    l.c = l.gates + wv_up((size_t)(peep ? 5 : 4) * rows * k.max_cpc * 2, 16);
    l.sx = l.c + wv_up((size_t)rows * k.max_cpc * 2, 16);
    l.stage_m = l.sx + (size_t)k.cl * k.cl_slots * k.ra * 16;
    l.stage_h = l.stage_m + (k.cl ? wv_up((size_t)rows * k.max_cpc, 16) : 0);
    l.total = l.stage_h + (k.cl ? wv_up((size_t)rows * k.max_opc, 16) : 0);
    // an MMA reads 128 rows of 128 bytes from where its k-block starts, whatever the tile holds
    if (l.total < l.act[0] + 128 * 128) l.total = l.act[0] + 128 * 128;
    l.total += 1024;                           // alignment of the ring
    return l;
}

struct WsSmem {
    int32_t *bx, *bh, *bln;        // [4][cpc]
    int16_t *L, *P;                // [4][cpc]
    int32_t *bp;                   // [opc]
    uint32_t *st;                  // [4][3][32] layer-norm sums: sum, low 20 bits and rest of the squares
    WvLnRow *ln;                   // [4][32]
    int16_t *g;                    // [slot][row][cpc] gate sums; slot 4: X of the output gate (peephole)
    int16_t *c;                    // [row][cpc]
    uint4 *sx, *sx2;               // CL: [block][4][ra] the cluster's sums of the first exchange, [block][ra] of the second
    uint8_t *stage_m, *stage_h;    // CL: [row][cpc], [row][opc]
    uint8_t *h_buf, *m_buf;        // CL: operands
};

struct WsRole {
    int li, rank;
    int u0, cells, o_lo, outs;
    int row0, rows, gu;
};

// Gate sums of eight rows from r0 of one tile, one lane per cell, for the gate `g` of this warp.
template <int G, bool LN, bool PEEP>
__device__ __forceinline__ void ws_gate_tile(const WaveCall &k, const WaveLayer &L, const WsSmem &s, const WsRole &r, uint32_t tx, uint32_t th,
                                             int tile, int g, int r0, int lane)
{
    constexpr int SF = (G == 4) ? 1 : 0, SZ = SF + 1, SO = SF + 2;
    const int cpc = L.cpc, ul = tile * L.ct + lane, rows = r.rows;
    const bool in = lane < L.ct && ul < r.cells;
    const int i0 = g * cpc + (in ? ul : 0);
    const int32_t bx = s.bx[i0], bh = s.bh[i0], P = PEEP ? (int32_t)s.P[i0] : 0;
    const FastScale fx = L.f_x[g], fh = L.f_h[g];
    const int xl = L.x_left[g], hl = L.h_left[g];
    const bool is_o = PEEP && g == SO;                         // warp-uniform
    uint32_t x[8], h[8];
    __syncwarp();
    ptx::tmem_ld_32x8(tx + (uint32_t)r0, x);
    ptx::tmem_ld_32x8(th + (uint32_t)r0, h);
    ptx::tmem_ld_wait();
    int32_t v[8];
    const int ne = rows - r0 < 8 ? rows - r0 : 8;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (e >= ne) break;
        const int32_t X = sat16(fast_rescale(((int32_t)x[e] + bx) << xl, fx));
        const int32_t H = sat16(fast_rescale(((int32_t)h[e] + bh) << hl, fh));
        v[e] = X + H;
        if (PEEP) {
            if (is_o) {
                if (in) s.g[(4 * rows + r0 + e) * cpc + ul] = (int16_t)X;
                v[e] = H;                                  // X + H + P c^t once c^t exists
            } else if (g != SZ) {
                const int32_t c_old = in ? s.c[(r0 + e) * cpc + ul] : 0;
                v[e] += sat16(fast_rescale(P * c_old, L.f_c[g]));
            }
        }
        v[e] = in ? sat16(v[e]) : 0;
        if (in) s.g[(g * rows + r0 + e) * cpc + ul] = (int16_t)v[e];
    }
    if (LN && !is_o) {
        uint32_t my_sum = 0, my_lo = 0, my_hi = 0;             // lane e keeps the sums of row r0 + e
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (e >= ne) break;
            const uint32_t sq = (uint32_t)(v[e] * v[e]);
            const uint32_t a = (uint32_t)__reduce_add_sync(0xffffffffu, v[e]);
            const uint32_t lo = __reduce_add_sync(0xffffffffu, sq & 0xfffffu), hi = __reduce_add_sync(0xffffffffu, sq >> 20);
            if (lane == e) { my_sum = a; my_lo = lo; my_hi = hi; }
        }
        if (lane < ne) {
            uint32_t *st = s.st + g * 3 * WS_ROWS + r0 + lane;
            atomicAdd(st, my_sum);
            atomicAdd(st + WS_ROWS, my_lo);
            atomicAdd(st + 2 * WS_ROWS, my_hi);
        }
    }
}

template <int G>
__device__ __forceinline__ void ws_push_stats(const WsSmem &s, long long *totals, int rows, unsigned mask, int tid)
{
    const int g = tid >> 5, row = tid & 31;
    if (g < G && row < rows && ((mask >> g) & 1u)) {
        uint32_t *st = s.st + g * 3 * WS_ROWS + row;
        const long long sum = (long long)(int32_t)st[0];
        const unsigned long long sq = ((unsigned long long)st[2 * WS_ROWS] << 20) + st[WS_ROWS];
        st[0] = st[WS_ROWS] = st[2 * WS_ROWS] = 0u;
        unsigned long long *dst = reinterpret_cast<unsigned long long *>(totals + (size_t)(row * 4 + g) * 2);
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst), "l"((unsigned long long)sum) : "memory");
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst + 1), "l"(sq) : "memory");
    }
}
template <int G>
__device__ __forceinline__ void ws_pull_stats(const WaveLayer &L, const WsSmem &s, const long long *totals, int rows, unsigned mask, int tid)
{
    const int g = tid >> 5, row = tid & 31;
    if (g < G && row < rows && ((mask >> g) & 1u)) {
        const longlong2 v = __ldcg(reinterpret_cast<const longlong2 *>(totals + (size_t)(row * 4 + g) * 2));
        s.ln[g * WS_ROWS + row] = wv_make_ln(v.x, v.y, L.div_c, L.sigma_min);
    }
}

// ---- exchanges within a cluster ----
// The block's sums of the gate slots in `mask` to every block; slots: of a block in sx, slot 0 of which is gate g0.
template <int G>
__device__ __forceinline__ void ws_send_stats(const WaveCall &k, const WsSmem &s, const WsRole &r, int n, uint4 *sx, int slots, int g0, unsigned mask, uint64_t *bar,
                                              int tid)
{
    const int g = (tid >> 5) & 3, row = tid & 31;
    if (g < G && row < r.rows && ((mask >> g) & 1u)) {
        const uint32_t *st = s.st + g * 3 * WS_ROWS + row;
        const uint4 v = make_uint4(st[0], st[WS_ROWS], st[2 * WS_ROWS], 0u);
        const uint32_t dst = ptx::smem_u32(sx + ((size_t)r.rank * slots + g - g0) * k.ra + row), b = ptx::smem_u32(bar);
        for (int p = tid >> 7; p < n; p += 4) wv_send16(wv_peer(dst, p), v, wv_peer(b, p));
    }
}
// The constants of those slots from what has come; false: leave.
template <int G>
__device__ __forceinline__ bool ws_merge_stats(const WaveCall &k, const WaveLayer &L, const WsSmem &s, const WsRole &r, const uint4 *sx, int slots, int g0,
                                               unsigned mask, uint64_t *bar, uint32_t par, WvPoint &pt, int tid)
{
    const int g = tid >> 5, row = tid & 31;
    const bool mine = g < G && ((mask >> g) & 1u);             // warp-uniform
    if (mine && wv_wait_cluster(bar, par, k.abort_word, k.limit_ns, pt.abort_flag)) {
        // (the first warp of them arms the barrier again; nobody sends to it before this block has sent m or h)
        if (row == 0 && (mask & ((1u << g) - 1u)) == 0u) ptx::mbar_arrive_expect_tx(bar, (uint32_t)(L.n * __popc(mask) * r.rows * 16));
        if (row < r.rows) {
            int32_t sum = 0;
            uint32_t lo = 0, hi = 0;
            const uint4 *src = sx + (size_t)(g - g0) * k.ra + row;
#pragma unroll 4
            for (int p = 0; p < L.n; ++p) {
                const uint4 o = src[(size_t)p * slots * k.ra];
                sum += (int32_t)o.x; lo += o.y; hi += o.z;
            }
            s.ln[g * WS_ROWS + row] = wv_make_ln(sum, ((int64_t)hi << 20) + lo, L.div_c, L.sigma_min);
        }
    }
    const bool stay = wv_point(pt, tid);
    // (every thread that sends them has read the block's sums)
    if (mine && row < r.rows) {
        uint32_t *st = s.st + g * 3 * WS_ROWS + row;
        st[0] = st[WS_ROWS] = st[2 * WS_ROWS] = 0u;
    }
    return stay;
}
// PIECE bytes at a time, rows of `n` values from column `col0` on into the image `buf` of the blocks [0, peers).
template <int PIECE>
__device__ __forceinline__ void ws_send_rows(const WaveCall &k, const uint8_t *stage, int pitch, int rows, int n, int col0, uint8_t *buf, uint64_t *bar, int peers,
                                             int tid)
{
    const int np = (n + PIECE - 1) / PIECE, tasks = rows * np;
    const uint32_t base = ptx::smem_u32(buf), b = ptx::smem_u32(bar);
    for (int i = tid & 127; i < tasks; i += 128) {
        const int row = i / np, j = (i - row * np) * PIECE;
        const uint32_t dst = base + wv_img_off(row, col0 + j, k.ra);
        if (PIECE == 16) {
            const uint4 v = *reinterpret_cast<const uint4 *>(stage + row * pitch + j);
            for (int p = tid >> 7; p < peers; p += 4) wv_send16(wv_peer(dst, p), v, wv_peer(b, p));
        } else {
            const uint2 v = *reinterpret_cast<const uint2 *>(stage + row * pitch + j);
            for (int p = tid >> 7; p < peers; p += 4) wv_send8(wv_peer(dst, p), v, wv_peer(b, p));
        }
    }
}
// Bytes of a piece of m.
__device__ __forceinline__ int ws_piece(const WaveLayer &L) { return (L.cpc & 15) == 0 ? 16 : 8; }
// h^t of this block is in global memory for the layer above (after a barrier of the epilogue threads; by a warp that is not the first to
// wait).  cnt: this block's word.
__device__ __forceinline__ void ws_signal(unsigned *cnt, int tid)
{
    if (tid == WV_EPI - 32) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
}

// layer norm of the gate slots in `mask` of one cell, in place
template <int G>
__device__ __forceinline__ void ws_ln_cell(const WaveLayer &L, const WsSmem &s, int row, int ul, unsigned mask, int32_t (&a)[4])
{
    int32_t v[4];
    uint32_t any = 0;
#pragma unroll
    for (int g = 0; g < G; ++g)
        if ((mask >> g) & 1u) {
            const WvLnRow r = s.ln[g * WS_ROWS + row];
            any |= r.sigma;
            v[g] = wv_ln_fast(a[g], r.m_hi, r.m_lo, r.mean, s.L[g * L.cpc + ul], s.bln[g * L.cpc + ul]);
        }
    if (any & WV_LN_SLOW) {
#pragma unroll
        for (int g = 0; g < G; ++g)
            if ((mask >> g) & 1u) v[g] = wv_ln_slow(a[g], s.ln[g * WS_ROWS + row], s.L[g * L.cpc + ul], s.bln[g * L.cpc + ul]);
    }
#pragma unroll
    for (int g = 0; g < G; ++g)
        if ((mask >> g) & 1u) a[g] = sat16(fast_rescale(v[g], L.f_ln[g]));
}

// m of one cell (h of a layer without a projection)
template <bool CL>
__device__ __forceinline__ void ws_store_m(const WaveCall &k, const WaveLayer &L, const WsSmem &s, int8_t *img_unit, int row, int ul, int u, int b, int t, int32_t m,
                                           bool last_layer)
{
    if (CL) s.stage_m[row * L.cpc + ul] = (uint8_t)m;
    if (!CL || (!(L.flags & F_PROJECTION) && !last_layer)) img_unit[wv_img_off(row, u, k.ra)] = (int8_t)m;
    if (L.flags & F_PROJECTION) return;
    if (last_layer) wv_y_row(k, L, t, b)[u] = (int8_t)m;
    if (t == k.T - 1) L.h[(size_t)b * L.O + u] = (int8_t)m;
}

// Everything between the gate sums and m, one cell per task, consecutive threads on consecutive cells of a row.
template <int G, bool LN, bool PEEP, bool CL>
__device__ __forceinline__ bool ws_elementwise(const WaveCall &k, const WaveLayer &L, const WsSmem &s, const WsRole &r, const ActLines &at, int t, bool last_layer,
                                               WvPoint &pt, WsCtl *ctl, int tid)
{
    constexpr int SI = 0, SF = (G == 4) ? 1 : 0, SZ = SF + 1, SO = SF + 2;
    constexpr unsigned ALL = (1u << G) - 1u;
    const int rows = r.rows, cells = r.cells, cpc = L.cpc, n_tasks = rows * cells;
    unsigned *cnt = L.cnt + (size_t)r.gu * WC_PER_UNIT * WC_WORDS;
    long long *tot = L.totals ? L.totals + ((size_t)(t & 1) * k.nu + r.gu) * k.ra * 8 : nullptr;
    if (LN && CL) {
        constexpr unsigned FIRST = PEEP ? ALL & ~(1u << SO) : ALL;
        ws_send_stats<G>(k, s, r, L.n, s.sx, 4, 0, FIRST, &ctl->s_full[0], tid);
        if (!ws_merge_stats<G>(k, L, s, r, s.sx, 4, 0, FIRST, &ctl->s_full[0], (uint32_t)t & 1u, pt, tid)) return false;
    } else if (LN) {
        ws_push_stats<G>(s, tot, rows, PEEP ? ALL & ~(1u << SO) : ALL, tid);
        if (!wv_publish(cnt + WC_STATS * WC_WORDS, false, pt, tid)) return false;
        if (!wv_meet(k, cnt + WC_STATS * WC_WORDS, (unsigned)(t + 1) * L.n, pt, tid)) return false;
        ws_pull_stats<G>(L, s, tot, rows, PEEP ? ALL & ~(1u << SO) : ALL, tid);
        // the other set of totals was read by everyone before this step's sums were complete: cleared for the next step
        long long *next = L.totals + ((size_t)((t + 1) & 1) * k.nu + r.gu) * k.ra * 8;
        for (int i = r.rank * WV_EPI + tid; i < rows * 8; i += L.n * WV_EPI) next[i] = 0;
        wv_epi_sync();
    }
    int8_t *img = (L.flags & F_PROJECTION) ? L.m_img + (size_t)r.gu * L.kb_c * k.ra * 128
                                           : L.out_img + ((size_t)(t + 1) * k.nu + r.gu) * L.kb_h * k.ra * 128;
    const bool fin = t == k.T - 1;
    const float inv_cells = 1.0f / (float)cells;               // (i + 1/2) / cells is 2^-9 or more away from an integer
#pragma unroll 1
    for (int i = tid; i < n_tasks; i += WV_EPI) {
        const int row = (int)(((float)i + 0.5f) * inv_cells), ul = i - row * cells, u = r.u0 + ul, b = r.row0 + row;
        int32_t a[4];
#pragma unroll
        for (int g = 0; g < G; ++g) a[g] = s.g[(g * rows + row) * cpc + ul];
        if (LN) ws_ln_cell<G>(L, s, row, ul, PEEP ? ALL & ~(1u << SO) : ALL, a);
        const int32_t f = line_sigmoid(at, a[SF]), z = line_tanh_gate(at, a[SZ]);
        int32_t ig;
        if (G == 4) ig = line_sigmoid(at, a[SI]);
        else { ig = 32768 - f; if (ig > 32767) ig = 32767; }               // coupled input gate, Section 3.2.9
        const int32_t c_new = cell_update_fast(ig, z, f, s.c[row * cpc + ul], L.m_bits);
        s.c[row * cpc + ul] = (int16_t)c_new;
        if (fin) L.c[(size_t)b * L.C + u] = (int16_t)c_new;
        int32_t ao = a[SO];
        if (PEEP) {
            ao = sat16((int32_t)s.g[(4 * rows + row) * cpc + ul] + a[SO] + sat16(fast_rescale((int32_t)s.P[SO * cpc + ul] * c_new, L.f_c[SO])));   // Eq. 5
            if (LN) {
                s.g[(SO * rows + row) * cpc + ul] = (int16_t)ao;           // waits for the row's statistics
                uint32_t *st = s.st + SO * 3 * WS_ROWS + row;
                const uint32_t sq = (uint32_t)(ao * ao);
                atomicAdd(st, (uint32_t)ao);
                atomicAdd(st + WS_ROWS, sq & 0xfffffu);
                atomicAdd(st + 2 * WS_ROWS, sq >> 20);
                continue;
            }
        }
        ws_store_m<CL>(k, L, s, img, row, ul, u, b, t, wv_hidden<true>(L, at, line_sigmoid(at, ao), c_new), last_layer);
    }
    if (LN && PEEP) {
        wv_epi_sync();
        if (CL) {
            ws_send_stats<G>(k, s, r, L.n, s.sx2, 1, SO, 1u << SO, &ctl->s_full[1], tid);
            if (!ws_merge_stats<G>(k, L, s, r, s.sx2, 1, SO, 1u << SO, &ctl->s_full[1], (uint32_t)t & 1u, pt, tid)) return false;
        } else {
            ws_push_stats<G>(s, tot, rows, 1u << SO, tid);
            if (!wv_publish(cnt + WC_STATS2 * WC_WORDS, false, pt, tid)) return false;
            if (!wv_meet(k, cnt + WC_STATS2 * WC_WORDS, (unsigned)(t + 1) * L.n, pt, tid)) return false;
            ws_pull_stats<G>(L, s, tot, rows, 1u << SO, tid);
            wv_epi_sync();
        }
#pragma unroll 1
        for (int i = tid; i < n_tasks; i += WV_EPI) {
            const int row = (int)(((float)i + 0.5f) * inv_cells), ul = i - row * cells;
            int32_t a[4] = {0, 0, 0, 0};
            a[SO] = s.g[(SO * rows + row) * cpc + ul];
            ws_ln_cell<G>(L, s, row, ul, 1u << SO, a);
            ws_store_m<CL>(k, L, s, img, row, ul, r.u0 + ul, r.row0 + row, t, wv_hidden<true>(L, at, line_sigmoid(at, a[SO]), s.c[row * cpc + ul]), last_layer);
        }
    }
    if (CL) {
        const bool proj = (L.flags & F_PROJECTION) != 0, publish = !proj && !last_layer;
        if (publish) wv_fence_async_global();
        if (!wv_point(pt, tid)) return false;
        if (proj || !fin) {
            uint8_t *buf = proj ? s.m_buf : s.h_buf + ((t + 1) & 1) * (k.max_kb_h * k.ra * 128);
            uint64_t *bar = proj ? &ctl->mx_full : &ctl->hx_full[(t + 1) & 1];
            const int peers = proj ? (L.O + L.opc - 1) / L.opc : L.n;
            if (ws_piece(L) == 16) ws_send_rows<16>(k, s.stage_m, cpc, rows, cells, r.u0, buf, bar, peers, tid);
            else ws_send_rows<8>(k, s.stage_m, cpc, rows, cells, r.u0, buf, bar, peers, tid);
        }
        if (publish) ws_signal(cnt + WC_H * WC_WORDS + r.rank, tid);
        return true;
    }
    return wv_publish(cnt + ((L.flags & F_PROJECTION) ? WC_M : WC_H) * WC_WORDS, true, pt, tid);
}

// One projection tile: a lane is an output, the four warps of a lane quarter share the rows.
template <bool CL>
__device__ __forceinline__ void ws_proj_tile(const WaveCall &k, const WaveLayer &L, const WsSmem &s, const WsRole &r, uint32_t tp, int o_first, int no,
                                             int quarter, int wq, int lane, int8_t *out_unit, int t, bool last_layer)
{
    const int j = quarter * 32 + lane, col = r.o_lo + o_first + j;
    const bool in = j < no;
    if (quarter * 32 >= no) return;                            // warp-uniform
    const int32_t bias = in ? s.bp[o_first + j] : 0;
    const bool fin = t == k.T - 1;
#pragma unroll 1
    for (int r0 = 8 * wq; r0 < r.rows; r0 += 32) {
        uint32_t a[8];
        __syncwarp();
        ptx::tmem_ld_32x8(tp + (uint32_t)r0, a);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int row = r0 + e, b = r.row0 + row;
            const int8_t h = (int8_t)sat8(fast_rescale((int32_t)a[e] + bias, L.f_proj) + L.zp_h);
            if (in && row < r.rows) {
                if (CL) s.stage_h[row * L.opc + o_first + j] = (uint8_t)h;
                if (!CL || !last_layer) out_unit[wv_img_off(row, col, k.ra)] = h;
                if (last_layer) wv_y_row(k, L, t, b)[col] = h;
                if (fin) L.h[(size_t)b * L.O + col] = h;
            }
        }
    }
}

// A block that leaves early: its copies and MMAs in flight end (whole warps; `warp` 0 to 3 are the service warps).  Out of line, so
// that the kernel's loops keep their shape (us per call of 100 steps, five 1024-cell CIFG layers, 4 rows: 660 without, 665 like this,
// 678 inline at the end of each role).
__device__ __noinline__ void ws_drain(WsCtl *ctl, int nb, int warp)
{
    if (warp == 0) {
        for (int op = 0; op < 3; ++op)
            if (ctl->op_copies[op]) wv_drain(&ctl->op_full[op], (uint32_t)(ctl->op_copies[op] - 1) & 1u);
        wv_drain(&ctl->tab_full, 0);
    } else if (warp == 1) {
        wv_drain_ring(ctl->w_full, nb, ctl->end_slot, ctl->end_phase);
    } else if (warp < WV_EPI_WARP0) {
        wv_drain_mmas(&ctl->mma_done[warp - 2]);
    }
}

template <int G, bool LN, bool PEEP, bool CL>
__global__ void __launch_bounds__(WV_THREADS, 1) k_wave_small_sm100(const __grid_constant__ WaveCall k)
{
    extern __shared__ uint8_t ws_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)ws_raw + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = blockIdx.x;
    WsRole r;
    r.li = -1;
    if (CL) {
        const int group = cta / k.cl;
        r.li = group / k.rg;
    } else {
        for (int l = 0; l < k.n_layers; ++l)
            if (cta >= k.layer[l].cta0 && cta < k.layer[l].cta0 + k.layer[l].n * k.rg) r.li = l;
        if (r.li < 0) return;
    }
    const WaveLayer &L = k.layer[r.li];
    const bool proj = (L.flags & F_PROJECTION) != 0, last_layer = L.last != 0;
    if (CL) {
        const int group = cta / k.cl;
        r.gu = group - r.li * k.rg;
        r.rank = cta - group * k.cl;
        if (r.rank >= L.n) {                                   // a block without cells
            wv_cluster_sync();
            wv_cluster_sync();
            return;
        }
    } else {
        r.gu = (cta - L.cta0) / L.n;
        r.rank = cta - L.cta0 - r.gu * L.n;
    }
    r.u0 = r.rank * L.cpc;
    r.cells = L.C - r.u0 < L.cpc ? L.C - r.u0 : L.cpc;
    r.o_lo = r.rank * L.opc;
    r.outs = proj ? (L.O - r.o_lo < L.opc ? L.O - r.o_lo : L.opc) : 0;
    if (r.outs < 0) r.outs = 0;
    r.row0 = (int)((long long)r.gu * k.B / k.nu);
    r.rows = (int)((long long)(r.gu + 1) * k.B / k.nu) - r.row0;
    if (!CL && r.rows == 0) return;                            // fewer rows than row groups: this group is idle

    const WsLayout lay = ws_layout(k, k.nb, (k.B + k.nu - 1) / k.nu, PEEP);
    WsCtl *ctl = reinterpret_cast<WsCtl *>(smem + lay.ctl);
    volatile int *abort_flag = &ctl->abort_flag;
    WsSmem s;
    {
        uint8_t *p = smem + lay.consts;
        const size_t q = (size_t)k.max_cpc * 4;
        s.bx = (int32_t *)p;  p += q * 4;
        s.bh = (int32_t *)p;  p += q * 4;
        s.bln = (int32_t *)p; p += q * 4;
        s.bp = (int32_t *)p;  p += (size_t)k.max_opc * 4;
        s.L = (int16_t *)p;   p += q * 2;
        s.P = (int16_t *)p;
        s.st = (uint32_t *)(smem + lay.st);
        s.ln = (WvLnRow *)(smem + lay.ln);
        s.g = (int16_t *)(smem + lay.gates);
        s.c = (int16_t *)(smem + lay.c);
        s.sx = (uint4 *)(smem + lay.sx);
        s.sx2 = s.sx + (size_t)k.cl * 4 * k.ra;
        s.stage_m = smem + lay.stage_m;
        s.stage_h = smem + lay.stage_h;
        s.h_buf = smem + lay.act[1];
        s.m_buf = smem + lay.act[2];
    }
    // CL: what a step brings
    const int piece = ws_piece(L);
    const uint32_t m_bytes = (uint32_t)(r.rows * ((L.C + piece - 1) & -piece)), h_bytes = proj ? (uint32_t)(r.rows * ((L.O + 7) & -8)) : m_bytes;
    if (threadIdx.x == 0) {
        for (int i = 0; i < WS_SLOTS; ++i) { ptx::mbar_init(&ctl->w_full[i], 1); ptx::mbar_init(&ctl->w_empty[i], 2); }
        for (int i = 0; i < 3; ++i) { ptx::mbar_init(&ctl->op_full[i], 1); ptx::mbar_init(&ctl->op_empty[i], 2); }
        for (int i = 0; i < WS_MAX_TILES; ++i) ptx::mbar_init(&ctl->gate_full[i], 1);
        ptx::mbar_init(&ctl->acc_empty, WV_EPI / 32);
        ptx::mbar_init(&ctl->p_full, 2);
        ptx::mbar_init(&ctl->p_empty, WV_EPI / 32);
        ptx::mbar_init(&ctl->tab_full, 1);
        for (int i = 0; i < 2; ++i) ptx::mbar_init(&ctl->mma_done[i], 1);
        if (CL) {
            // two arrivals: each of the issuing warps, when it has seen the phase before (k.missing: arrivals that never come)
            for (int i = 0; i < 2; ++i) ptx::mbar_init(&ctl->hx_full[i], 2 + k.missing);
            ptx::mbar_init(&ctl->mx_full, 2 + k.missing);
            for (int i = 0; i < 2; ++i) ptx::mbar_init(&ctl->s_full[i], 1 + k.missing);
        }
        ctl->abort_flag = 0;
        ctl->exit_at = 0x7fffffff;
        for (int i = 0; i < 3; ++i) ctl->op_copies[i] = 0;
        ptx::fence_barrier_init();
        if (CL) {
            for (int i = 0; i < 2; ++i) { ptx::mbar_arrive_expect_tx(&ctl->hx_full[i], h_bytes); ptx::mbar_arrive(&ctl->hx_full[i]); }
            ptx::mbar_arrive_expect_tx(&ctl->mx_full, m_bytes);
            ptx::mbar_arrive(&ctl->mx_full);
            ptx::mbar_arrive_expect_tx(&ctl->s_full[0], (uint32_t)(L.n * (PEEP ? G - 1 : G) * r.rows * 16));
            ptx::mbar_arrive_expect_tx(&ctl->s_full[1], (uint32_t)(L.n * r.rows * 16));
        }
        ptx::mbar_arrive_expect_tx(&ctl->tab_full, L.tab_lay.bytes);
        ptx::bulk_load_1d(smem + lay.tab, L.tab, L.tab_lay.bytes, &ctl->tab_full);
    }
    if (warp == 2) {
        ptx::tmem_alloc(&ctl->tmem_base, 512);
        ptx::tmem_relinquish();
    }
    for (int i = threadIdx.x; i < 4 * L.cpc; i += WV_THREADS) {
        const int g = i / L.cpc, u = r.u0 + i - g * L.cpc;
        const bool in = g < G && i - g * L.cpc < r.cells;
        const int n = u * G + g;
        s.bx[i] = in ? L.bx[n] : 0;
        s.bh[i] = in ? L.bh[n] : 0;
        s.bln[i] = in && LN ? L.bln[n] : 0;
        s.L[i] = in && LN ? L.L[n] : (int16_t)0;
        s.P[i] = in && PEEP ? L.P[n] : (int16_t)0;
    }
    for (int i = threadIdx.x; i < r.outs; i += WV_THREADS) s.bp[i] = L.bp[r.o_lo + i];
    for (int i = threadIdx.x; i < 12 * WS_ROWS; i += WV_THREADS) s.st[i] = 0u;
    for (int i = threadIdx.x; i < r.rows * r.cells; i += WV_THREADS) {
        const int row = i / r.cells, ul = i - row * r.cells;
        s.c[row * L.cpc + ul] = L.c[(size_t)(r.row0 + row) * L.C + r.u0 + ul];
    }
    ptx::tc_fence_before();
    ptx::cta_sync();
    ptx::tc_fence_after();
    if (CL) wv_cluster_sync();                                 // every block's barriers stand
    const uint32_t tmem_base = ctl->tmem_base;
    const int nt = (r.cells + L.ct - 1) / L.ct, ntp = proj ? (r.outs + L.opt - 1) / L.opt : 0, nr = k.ra, T = k.T;
    // accumulators: X tiles, H tiles, projection tiles
    const uint32_t col_h = (uint32_t)(nt * nr), col_p = (uint32_t)(2 * nt * nr);
    unsigned *cnt0 = L.cnt + (size_t)r.gu * WC_PER_UNIT * WC_WORDS;
    // the order of a step's products, which the service warps share: H(t), X(t + 1), P(t) - or P before X in calls too short to be
    // ahead of the layer below.  At the start H comes first: it does not wait for the layer below.
    auto walk = [&](auto f) -> bool {
        if (!f(1, 0) || !f(0, 0)) return false;
        for (int t = 0; t < T; ++t) {
            if (t > 0 && !f(1, t)) return false;
            if (k.early && t + 1 < T && !f(0, t + 1)) return false;
            if (ntp > 0 && !f(2, t)) return false;
            if (!k.early && t + 1 < T && !f(0, t + 1)) return false;
        }
        return true;
    };

    if (warp == 0) {
        // ---------------- operands: x, h, m of a unit, each one contiguous copy ----------------
        // (CL: the warp stays together, to look at a word per block of the layer below)
        if (CL || lane == 0) {
            walk([&](int op, int t) -> bool {
                if (CL && (op == 2 || (op == 1 && t > 0))) return true;        // (sent by the peers)
                const unsigned *cnt = nullptr;
                unsigned target = 0;
                const int8_t *src;
                uint32_t bytes = (uint32_t)nr * 128u;
                if (op == 0) {
                    bytes *= (uint32_t)L.kb_i;
                    src = L.in_img + ((size_t)(t + (L.below ? 1 : 0)) * k.nu + r.gu) * bytes;
                    if (L.below) {
                        cnt = k.layer[r.li - 1].cnt + ((size_t)r.gu * WC_PER_UNIT + WC_H) * WC_WORDS;
                        target = (unsigned)(t + 1) * (CL ? 1u : (unsigned)L.below);
                    }
                } else if (op == 1) {
                    bytes *= (uint32_t)L.kb_h;
                    src = L.out_img + ((size_t)t * k.nu + r.gu) * bytes;
                    if (t > 0) { cnt = cnt0 + WC_H * WC_WORDS; target = (unsigned)t * L.n; }
                } else {
                    bytes *= (uint32_t)L.kb_c;
                    src = L.m_img + (size_t)r.gu * bytes;
                    cnt = cnt0 + WC_M * WC_WORDS; target = (unsigned)(t + 1) * L.n;
                }
                if (CL) {
                    if (cnt && !wv_wait_blocks(k, cnt, L.below, target, abort_flag)) return false;
                    if (!wv_wait_warp(&ctl->op_empty[op], ((uint32_t)t & 1u) ^ 1u, abort_flag)) return false;
                } else {
                    if (cnt && !wv_wait_count(k, cnt, target, abort_flag)) return false;
                    if (!wv_wait(&ctl->op_empty[op], ((uint32_t)t & 1u) ^ 1u, abort_flag)) return false;
                }
                if (lane == 0) {
                    wv_fence_async_global();
                    ptx::mbar_arrive_expect_tx(&ctl->op_full[op], bytes);
                    ptx::bulk_load_1d(smem + lay.act[op], src, bytes, &ctl->op_full[op]);
                    ctl->op_copies[op] = t + 1;
                }
                if (CL) __syncwarp();
                return true;
            });
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- weights ----------------
        if (lane == 0) {
            int slot = 0; uint32_t phase = 0;
            // `total` bytes from src, a slot's worth (`most`) at a time
            auto put = [&](const int8_t *src, uint32_t total, uint32_t most) -> bool {
                for (uint32_t done = 0; done < total; done += most) {
                    const uint32_t bytes = total - done < most ? total - done : most;
                    if (!wv_wait(&ctl->w_empty[slot], phase ^ 1u, abort_flag)) return false;
                    ptx::mbar_arrive_expect_tx(&ctl->w_full[slot], bytes);
                    ptx::bulk_load_1d(smem + (size_t)slot * k.b_slot, src + done, bytes, &ctl->w_full[slot]);
                    if (++slot == k.nb) { slot = 0; phase ^= 1u; }
                }
                return true;
            };
            walk([&](int op, int) -> bool {
                if (op == 2) {
                    const uint32_t total = (uint32_t)(L.kb_c * L.opp * 128);
                    for (int j = 0; j < ntp; ++j)
                        if (!put(L.img_p + (size_t)(r.rank * L.ntp + j) * total, total, (uint32_t)(L.kpp * L.opp * 128))) return false;
                    return true;
                }
                const uint32_t total = (uint32_t)((((op == 0 ? L.kb_i : L.kb_h) + L.kpg - 1) / L.kpg) * G * 4096);
                for (int i = 0; i < nt; ++i)
                    if (!put((op == 0 ? L.img_w : L.img_r) + (size_t)(r.rank * L.nt + i) * total, total, WS_CHUNKS * G * 4096u)) return false;
                return true;
            });
            ctl->end_slot = slot; ctl->end_phase = phase;
        }
        __syncwarp();
    } else if (warp < WV_EPI_WARP0) {
        // ---------------- MMAs: weights x operand ----------------
        // Two warps take the tiles in turn: the waits and loop overhead around a slot (about 300 cycles) pass under the
        // other's MMAs.  Both watch every slot (a parity wait must not skip a round).  A gate tile's X and H have one issuer.
        const int me = warp - 2;
        int slot = 0; uint32_t phase = 0;
        const uint64_t w_desc0 = ptx::smem_desc_k_sw128(ptx::smem_u32(smem));
        const uint32_t idesc = ptx::idesc_i8(128, nr), b_step = (uint32_t)nr * 128u >> 4;
        // one tile of nkb k-blocks: kpc of them per chunk (kb_bytes apart), the chunks of a ring slot chunk_bytes apart
        auto tile = [&](bool mine, uint32_t d, size_t b_at, int nkb, int kpc, uint32_t kb_bytes, int n_chunks, uint32_t chunk_bytes) -> bool {
            const uint64_t b_desc0 = ptx::smem_desc_k_sw128(ptx::smem_u32(smem + b_at));
            for (int kb0 = 0; kb0 < nkb; kb0 += kpc * n_chunks) {
                if (!wv_wait_warp(&ctl->w_full[slot], phase, abort_flag)) return false;
                ptx::tc_fence_after();
                if (!mine) {
                    if (lane == 0) ptx::mbar_arrive(&ctl->w_empty[slot]);
                } else if (ptx::elect_one()) {
                    uint64_t ac = w_desc0 + (uint64_t)((uint32_t)slot * ((uint32_t)k.b_slot >> 4));
                    uint64_t bd = b_desc0 + (uint64_t)(b_step * (uint32_t)kb0);
                    int kb = kb0;
                    for (int c = 0; c < n_chunks; ++c, ac += chunk_bytes >> 4) {
                        uint64_t ad = ac;
                        for (int i = 0; i < kpc && kb < nkb; ++i, ++kb) {
                            wv_mma_kblock(d, ad, bd, idesc, kb == 0);
                            ad += kb_bytes >> 4;
                            bd += b_step;
                        }
                    }
                    ptx::mma_commit(&ctl->w_empty[slot]);
                }
                __syncwarp();
                if (++slot == k.nb) { slot = 0; phase ^= 1u; }
            }
            return true;
        };
        walk([&](int op, int t) -> bool {
            const uint32_t par = (uint32_t)t & 1u;
            // the gate accumulators of the step before have been read (X(t) waits for step t - 1 as well)
            if (op != 2 && t > 0 && !wv_wait_warp(&ctl->acc_empty, par ^ 1u, abort_flag)) return false;
            if (op == 2 && t > 0 && !wv_wait_warp(&ctl->p_empty, par ^ 1u, abort_flag)) return false;
            size_t b_at = lay.act[op];
            if (CL && (op == 2 || (op == 1 && t > 0))) {
                if (op == 1 && par) b_at += (size_t)k.max_kb_h * k.ra * 128;
                uint64_t *bar = op == 2 ? &ctl->mx_full : &ctl->hx_full[par];
                if (!wv_wait_cluster(bar, op == 2 ? par : (uint32_t)((t - 1) >> 1) & 1u, k.abort_word, k.limit_ns, abort_flag)) return false;
                if (lane == 0) {
                    if (me == 0) ptx::mbar_arrive_expect_tx(bar, op == 2 ? m_bytes : h_bytes);
                    else ptx::mbar_arrive(bar);
                }
                __syncwarp();
                ptx::fence_proxy_async();                      // (the peers' stores are ordinary ones, an MMA reads as copies do)
            } else if (!wv_wait_warp(&ctl->op_full[op], par, abort_flag)) return false;
            ptx::tc_fence_after();
            if (op == 2) {
                for (int j = 0; j < ntp; ++j)
                    if (!tile((j & 1) != me, tmem_base + col_p + (uint32_t)(j * nr), b_at, L.kb_c, L.kpp, (uint32_t)L.opp * 128u, 1, 0u)) return false;
                wv_commit(&ctl->p_full);
            } else {
                for (int i = 0; i < nt; ++i) {
                    if (!tile((i & 1) == me, tmem_base + (op ? col_h : 0u) + (uint32_t)(i * nr), b_at, op ? L.kb_h : L.kb_i, L.kpg, (uint32_t)L.ctp * 128u, WS_CHUNKS,
                              G * 4096u))
                        return false;
                    if (op == (t > 0 ? 1 : 0) && (i & 1) == me) wv_commit(&ctl->gate_full[i]);      // the step's last product
                }
            }
            if (!CL || op == 0) wv_commit(&ctl->op_empty[op]);
            return true;
        });
    } else if (warp >= WV_EPI_WARP0) {
        // ---------------- epilogues and elementwise work ----------------
        const int tid = threadIdx.x - 32 * WV_EPI_WARP0, quarter = warp & 3, wq = (warp - WV_EPI_WARP0) >> 2;
        const uint32_t tq = tmem_base + ((uint32_t)(quarter * 32) << 16);
        WvPoint pt{abort_flag, &ctl->exit_at, 0};
        const ActLines at = make_act_lines(ptx::smem_u32(smem + lay.tab), L.tab_lay);
        wv_wait(&ctl->tab_full, 0, abort_flag);
        bool stay = true;
        for (int t = 0; t < T && stay; ++t) {
            const uint32_t par = (uint32_t)t & 1u;
            // pieces of (tile, eight rows), dealt to the four warps of a lane quarter
            for (int i = 0, q = 0; i < nt && quarter < G; ++i) {
                bool seen = false, ok = true;
                for (int r0 = 0; r0 < r.rows && ok; r0 += 8, ++q) {
                    if ((q & 3) != wq) continue;
                    if (!seen) {
                        ok = __all_sync(0xffffffffu, wv_wait(&ctl->gate_full[i], par, abort_flag));
                        if (!ok) break;
                        ptx::tc_fence_after();
                        seen = true;
                    }
                    ws_gate_tile<G, LN, PEEP>(k, L, s, r, tq + (uint32_t)(i * nr), tq + col_h + (uint32_t)(i * nr), i, quarter, r0, lane);
                }
                if (!ok) break;                                // (on to the next meeting point)
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&ctl->acc_empty);
            wv_epi_sync();
            stay = ws_elementwise<G, LN, PEEP, CL>(k, L, s, r, at, t, last_layer, pt, ctl, tid);
            if (!stay || !proj) continue;
            if (ntp > 0 && __all_sync(0xffffffffu, wv_wait(&ctl->p_full, par, abort_flag))) {
                ptx::tc_fence_after();
                for (int j = 0; j < ntp; ++j) {
                    const int left = r.outs - j * L.opt;
                    ws_proj_tile<CL>(k, L, s, r, tq + col_p + (uint32_t)(j * nr), j * L.opt, left < L.opt ? left : L.opt, quarter, wq, lane,
                                 L.out_img + ((size_t)(t + 1) * k.nu + r.gu) * L.kb_h * k.ra * 128, t, last_layer);
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&ctl->p_empty);
            }
            if (CL) {
                if (!last_layer) wv_fence_async_global();
                stay = wv_point(pt, tid);
                if (!stay) continue;
                if (t + 1 < T)
                    ws_send_rows<8>(k, s.stage_h, L.opc, r.rows, r.outs, r.o_lo, s.h_buf + ((t + 1) & 1) * (k.max_kb_h * k.ra * 128), &ctl->hx_full[(t + 1) & 1], L.n,
                                    tid);
                if (!last_layer) ws_signal(cnt0 + WC_H * WC_WORDS + r.rank, tid);
                continue;
            }
            stay = wv_publish(cnt0 + WC_H * WC_WORDS, true, pt, tid);
        }
    }

    // ---------------- teardown ----------------
    ptx::cta_sync();
    const bool aborted = *abort_flag != 0;
    if (aborted) {
        // a wait ran out: copies and MMAs in flight end, then report
        ws_drain(ctl, k.nb, warp);
        if (threadIdx.x == 0) { atomicExch(k.abort_word, 1u); atomicExch(k.status, 2); }
    }
    ptx::cta_sync();
    if (CL) {
        wv_cluster_sync();                                     // no block ends while a peer may still store into it:
        if (aborted && threadIdx.x == 0) {
            // what peers sent before they came here arrives within microseconds (a block that has not given up has waited for all of it)
            const unsigned long long t0 = wv_timer();
            while (wv_timer() - t0 < 50000ull) {}
        }
    }
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, 512);
    }
}

// A weight matrix into the tiles its blocks stream.  Gate matrices (G > 0): [rank][tile][chunk of kps k-blocks][gate][k-block]
// [ctp cells][128 bytes]; W_proj (G = 0): [rank][tile][k-block][opp outputs][128 bytes]; 16-byte pieces swizzled by row mod 8.
__global__ void k_wave_small_tile_weights(const int8_t *src, int8_t *dst, int G, int rows, int K, int n, int per_rank, int nt, int per_tile, int padded,
                                          int nkb, int kps)
{
    const int gates = G > 0 ? G : 1, nch = (nkb + kps - 1) / kps, kbs = G > 0 ? nch * kps : nkb;
    const size_t total = (size_t)n * nt * kbs * gates * padded * 8;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int piece = (int)(i & 7);
        size_t q = i >> 3;
        const int c = (int)(q % padded); q /= padded;
        int kb, g = 0, tile, rank;
        if (G > 0) {
            const int kk = (int)(q % kps); q /= kps;
            g = (int)(q % G); q /= G;
            kb = (int)(q % nch) * kps + kk; q /= nch;
        } else {
            kb = (int)(q % nkb); q /= nkb;
        }
        tile = (int)(q % nt); rank = (int)(q / nt);
        const int u = tile * per_tile + c;                     // cell or output within the block
        int src_row = -1;
        if (c < per_tile && u < per_rank && (size_t)(rank * per_rank + u) * gates < (size_t)rows) src_row = (rank * per_rank + u) * gates + g;
        const int k0 = kb * 128 + piece * 16;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (src_row >= 0 && k0 < K) v = wv_load16(src + (size_t)src_row * K + k0, K - k0);
        *reinterpret_cast<uint4 *>(dst + (i >> 3) * 128 + ((piece ^ (c & 7)) << 4)) = v;
    }
}

}  // namespace

void wave_small_tile_weights(const int8_t *src, int8_t *dst, int G, int rows, int K, int n, int per_rank, int nt, int per_tile, int padded, int nkb, int kps)
{
    k_wave_small_tile_weights<<<2048, 256>>>(src, dst, G, rows, K, n, per_rank, nt, per_tile, padded, nkb, kps);
}

namespace {
template <bool CL>
const void *ws_kernel_of(int G, bool ln, bool peep)
{
    if (G == 4) {
        if (ln) return peep ? (const void *)k_wave_small_sm100<4, true, true, CL> : (const void *)k_wave_small_sm100<4, true, false, CL>;
        return peep ? (const void *)k_wave_small_sm100<4, false, true, CL> : (const void *)k_wave_small_sm100<4, false, false, CL>;
    }
    if (ln) return peep ? (const void *)k_wave_small_sm100<3, true, true, CL> : (const void *)k_wave_small_sm100<3, true, false, CL>;
    return peep ? (const void *)k_wave_small_sm100<3, false, true, CL> : (const void *)k_wave_small_sm100<3, false, false, CL>;
}
}  // namespace

const void *wave_small_kernel(int G, bool ln, bool peep, bool cluster)
{
    return cluster ? ws_kernel_of<true>(G, ln, peep) : ws_kernel_of<false>(G, ln, peep);
}

// shared memory of a launch with ns ring slots
size_t wave_small_smem(const WaveCall &k, int ns, bool peep) { return ws_layout(k, ns, (k.B + k.nu - 1) / k.nu, peep).total; }

}  // namespace ql
