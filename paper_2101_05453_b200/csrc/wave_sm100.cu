// Wavefront kernel: every layer and every time step of a stack in ONE cooperative launch, all matrix products on the
// tensor cores, batches up to 256 rows.
//
// A stack run layer after layer is a chain of T x L layer-steps, each of which crosses the whole machine three or four
// times (statistics, hidden state, output) and gives an SM only a few dozen cells to work on in between: at eight
// 2048-cell layers and 64 rows a layer-step took 20.6 us for 2 us of arithmetic.  Here the SMs are split into one group
// per layer (and, for shallow stacks, per range of batch rows), layer l + 1 works on a step while layer l works on a
// later one, and the exchanges involve the 18 or so blocks of a group.  The input term W x_t of Section 3.2.4 is part of
// the step, so no activation makes a round trip through memory beyond the layers' int8 outputs.
//
// A block owns a range of cells (all their gate rows) and a range of projection rows.  Its weights do not fit in shared
// memory (656 KB for an eighteenth of a 2048-cell layer): they lie in global memory in the order and in the
// shared-memory image in which the block's MMAs read them, and stream through a ring of contiguous bulk copies that runs
// ahead of the dependency chain.  The batch is the M side of the MMAs: a tensor-memory lane is a batch row.
//
//   X(t+1)  W x_{t+1}  -> rescale -> int16                                          needs the layer below at t + 1
//   H(t)    R h^{t-1}  -> + bias, rescale, + X(t) (+ peephole) -> gate sums, sums for the layer norm's statistics
//           [layer norm: the group adds its sums up in L2]
//   B(t)    layer norm, sigmoid / tanh, cell update, hidden state m (= h without a projection)
//   P(t)    W_proj m   -> h^t
//
// The rows are worked on in units of at most 128.  One unit: X(t+1) is computed while the block would otherwise wait for
// the statistics and for m.  Two units: each one's exchanges pass while the block works on the other.
//
// Warp roles: 0 copies activations, 1 copies weights, 2 issues MMAs, 4..19 epilogues and elementwise work.  All four
// walk the same table of operations, so that no role needs to tell another what comes next.
//
// Every wait is bounded; on expiry the block sets the abort word, all blocks see it at their next wait and leave, and the
// host reports QLSTM_ERR_TIMEOUT.
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <cmath>
#include <utility>
#include <vector>

#include "wave_resident.h"

namespace ql {

namespace {

constexpr int WV_A_SLOT = 128 * 128;                           // one k-block of 128 activation rows
constexpr int WV_MAX_SLOTS = 8;
constexpr int WV_MAX_OPS = 96;
constexpr int WV_ACC_COLS = 256;                               // columns of each of the two accumulators

enum { OP_X = 0, OP_H = 1, OP_P = 2, OP_S = 3, OP_B = 4, OP_F = 5 };
struct WaveOp { uint8_t kind, u, tile, pad; };

struct WaveCtl {
    uint64_t a_full[WV_MAX_SLOTS], a_empty[WV_MAX_SLOTS], b_full[WV_MAX_SLOTS], b_empty[WV_MAX_SLOTS];
    uint64_t t_full[2], t_empty[2], tab_full, mma_done;
    uint32_t tmem_base;
    int abort_flag;
    int end_slot[2];               // where the two copying warps stopped in their rings
    uint32_t end_phase[2];
    int exit_at;                   // meeting point of the epilogue threads at which they all leave
    int n_ops, n_pro;              // operations of a step; of the prologue (X of step 0)
    WaveOp ops[WV_MAX_OPS];
};

// What a block keeps in shared memory besides the rings.  Columns of a pair of cells: slot-major, [slot][cell of the pair].
struct WaveSmem {
    int32_t *bx, *bh, *bln;        // [ppc][8]
    int16_t *L, *P;                // [ppc][8]
    int32_t *bp;                   // [opc]
    uint32_t *st;                  // [4 slots][3][128] layer-norm sums of the block: sum, low 20 bits and rest of the squares
    WvLnRow *ln;                   // [4 slots][128]
    uint8_t *tab;
};

// Who a block is, and the buffers of its rows.
struct WaveRole {
    int li, rank, rgi;
    int pairs, u0;                 // own cell pairs, first cell
    int o_lo, outs;                // own projection outputs
    int row0[2], rows[2];          // units: first batch row, rows
    int gu[2];                     // unit numbers among all units
    uint4 *g[2];                   // gate buffers of the units: nbuf x [pairs][rows]
    uint32_t *c[2];                // cell states [pairs][rows]
    int n_rows_max;
};

// X and H epilogue of one tile for one thread = one batch row: pairs part, part + nparts, ... of the tile, two at a time.
// Per column:  X = sat16(rescale(acc + bx, eff_x));  H = sat16(rescale(acc + bh, eff_h)); gate = sat16(X + H [+ peephole])
// (the sums acc + b fit 32 bits: checked on the host).
template <int G, bool LN, bool PEEP, bool IS_H>
__device__ __forceinline__ void wv_gate_tile(const WaveLayer &L, const WaveSmem &s, uint32_t taddr, int pair0, int np, int part, int nparts,
                                             int row, int rows, bool valid, const uint4 *xbuf, uint4 *gbuf, const uint32_t *cbuf,
                                             uint64_t *full, uint32_t parity, volatile int *abort_flag)
{
    constexpr int SF = (G == 4) ? 1 : 0, SZ = SF + 1, SO = SF + 2;
    int32_t sum[4] = {0, 0, 0, 0};
    long long sq[4] = {0, 0, 0, 0};
    auto one = [&](const uint32_t (&r)[8], int p, const uint4 &x4) {
        const int pr = pair0 + p;
        const int32_t *bias = (IS_H ? s.bh : s.bx) + pr * 8;
        const int4 b0 = *reinterpret_cast<const int4 *>(bias), b1 = *reinterpret_cast<const int4 *>(bias + 4);
        const int32_t bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        const uint32_t xw[4] = {x4.x, x4.y, x4.z, x4.w};
        uint32_t w[4] = {0, 0, 0, 0};
        int32_t c_old[2] = {0, 0};
        uint32_t pw[4] = {0, 0, 0, 0};
        if (IS_H && PEEP) {
            const uint32_t cw = cbuf[pr * rows + row];
            c_old[0] = wv_lo(cw); c_old[1] = wv_hi(cw);
            const uint4 p4 = *reinterpret_cast<const uint4 *>(s.P + pr * 8);
            pw[0] = p4.x; pw[1] = p4.y; pw[2] = p4.z; pw[3] = p4.w;
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            int32_t v[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                int32_t acc = (int32_t)r[2 * g + k] + bb[2 * g + k];
                acc <<= IS_H ? L.h_left[g] : L.x_left[g];
                v[k] = fast_rescale(acc, IS_H ? L.f_h[g] : L.f_x[g]);
                if (IS_H && !(PEEP && g == SO)) {
                    v[k] = sat16(v[k]) + (k ? wv_hi(xw[g]) : wv_lo(xw[g]));
                    if (PEEP && g != SZ) {
                        const int32_t P = k ? wv_hi(pw[g]) : wv_lo(pw[g]);
                        v[k] += sat16(fast_rescale(P * c_old[k], L.f_c[g]));
                    }
                }
            }
            w[g] = ptx::pack_sat_s16(v[0], v[1]);          // (output gate with a peephole: H alone, the rest once c^t exists)
            if (IS_H && LN && !(PEEP && g == SO)) {
                const int32_t a = wv_lo(w[g]), b = wv_hi(w[g]);
                sum[g] = __dp2a_lo((int)w[g], 0x0101, sum[g]);
                sq[g] += (long long)a * a;
                sq[g] += (long long)b * b;
            }
        }
        gbuf[pr * rows + row] = make_uint4(w[0], w[1], w[2], w[3]);
    };
    // X(t) may lie in L2: the first trip's is requested before the accumulators are waited for, a later one's a trip ahead
    uint4 xa = make_uint4(0, 0, 0, 0), xb = xa;
    if (IS_H && valid) {
        const int p = G == 4 ? part : 2 * part, pb = G == 4 ? p + nparts : p + 1;
        if (p < np) xa = xbuf[(pair0 + p) * rows + row];
        if (pb < np) xb = xbuf[(pair0 + pb) * rows + row];
    }
    if (!__all_sync(0xffffffffu, wv_wait(full, parity, abort_flag))) return;
    ptx::tc_fence_after();
    // four gates: two pairs nparts apart, eight columns each; three gates: two adjacent pairs, twelve columns in pieces of
    // four (np is then even)
#pragma unroll 1
    for (int p = (G == 4 ? part : 2 * part); p < np; p += 2 * nparts) {
        const int pb = G == 4 ? p + nparts : p + 1;
        const bool two = G == 3 || pb < np;                // warp-uniform
        uint32_t acc[2][8];
        __syncwarp();
        if (G == 4) {
            ptx::tmem_ld_32x8(taddr + (uint32_t)(p * 8), acc[0]);
            if (two) ptx::tmem_ld_32x8(taddr + (uint32_t)(pb * 8), acc[1]);
        } else {
            uint32_t q[3][4];
#pragma unroll
            for (int i = 0; i < 3; ++i) ptx::tmem_ld_32x4(taddr + (uint32_t)(p * 6 + 4 * i), q[i]);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 12; ++i) acc[i / 6][i % 6] = q[i >> 2][i & 3];
            acc[0][6] = acc[0][7] = acc[1][6] = acc[1][7] = 0;
        }
        const uint4 x0 = xa, x1 = xb;
        if (IS_H && valid) {                               // the next trip's X
            const int pn = p + 2 * nparts, pbn = pb + 2 * nparts;
            if (pn < np) xa = xbuf[(pair0 + pn) * rows + row];
            if (pbn < np) xb = xbuf[(pair0 + pbn) * rows + row];
        }
        if (G == 4) ptx::tmem_ld_wait();
        if (valid) {
            one(acc[0], p, x0);
            if (two) one(acc[1], pb, x1);
        }
    }
    if (IS_H && LN && valid) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (PEEP && g == SO) continue;
            uint32_t *st = s.st + (g * 3) * 128 + row;
            atomicAdd(st, (uint32_t)sum[g]);
            atomicAdd(st + 128, (uint32_t)((unsigned long long)sq[g] & 0xfffffu));
            atomicAdd(st + 256, (uint32_t)((unsigned long long)sq[g] >> 20));
        }
    }
}

// Projection epilogue of one tile for one thread = one batch row, four outputs at a time.
__device__ __forceinline__ void wv_proj_tile(const WaveCall &k, const WaveLayer &L, const WaveSmem &s, const WaveRole &r, uint32_t taddr,
                                             int o_first, int no, int part, int nparts, int row, bool valid, int8_t *out_unit, int b, int t,
                                             bool last_layer)
{
    const int nq = (no + 3) >> 2;
#pragma unroll 1
    for (int q = part; q < nq; q += nparts) {
        uint32_t a[4];
        __syncwarp();
        ptx::tmem_ld_32x4(taddr + (uint32_t)(q * 4), a);
        ptx::tmem_ld_wait();
        const int col = r.o_lo + o_first + q * 4;
        if (!valid || col >= L.O) continue;
        const int4 b4 = *reinterpret_cast<const int4 *>(s.bp + o_first + q * 4);
        const int32_t bb[4] = {b4.x, b4.y, b4.z, b4.w};
        uint32_t w = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int32_t v = sat8(fast_rescale((int32_t)a[j] + bb[j], L.f_proj) + L.zp_h);
            w |= (uint32_t)(v & 0xff) << (8 * j);
        }
        *reinterpret_cast<uint32_t *>(out_unit + wv_img_off(row, col, k.ra)) = w;
        const bool fin = t == k.T - 1;
        if (last_layer || fin) {
            int8_t *dst[2] = {last_layer ? wv_y_row(k, L, t, b) + col : nullptr,
                              fin ? L.h + (size_t)b * L.O + col : nullptr};
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                if (!dst[d]) continue;
                if (((uintptr_t)dst[d] & 3) == 0 && col + 4 <= L.O) *reinterpret_cast<uint32_t *>(dst[d]) = w;
                else
                    for (int j = 0; j < 4; ++j)
                        if (col + j < L.O) dst[d][j] = (int8_t)(w >> (8 * j));
            }
        }
    }
}

// ---- elementwise phase -----------------------------------------------------------------------------------------------

// Layer-norm constants of a thread's row in registers: those that the fast form needs.
struct WvLnRegs { int32_t m_hi[4], m_lo[4], mean[4]; bool slow; };

template <int G>
__device__ __forceinline__ void wv_load_ln(const WaveSmem &s, int row, unsigned mask, WvLnRegs &r)
{
    uint32_t any = 0;
#pragma unroll
    for (int g = 0; g < G; ++g)
        if ((mask >> g) & 1u) {
            const WvLnRow v = s.ln[g * 128 + row];
            r.m_hi[g] = v.m_hi; r.m_lo[g] = v.m_lo; r.mean[g] = v.mean; any |= v.sigma;
        }
    r.slow = (any & WV_LN_SLOW) != 0u;
}

// The gate values of a pair after layer norm (slots in `mask`), in place.
template <int G>
__device__ __forceinline__ void wv_ln_pair(const WaveLayer &L, const WaveSmem &s, const WvLnRegs &r, int row, int pr, unsigned mask, int32_t (&a)[4][2])
{
    const uint4 lw = *reinterpret_cast<const uint4 *>(s.L + pr * 8);
    const uint32_t lws[4] = {lw.x, lw.y, lw.z, lw.w};
    const int4 b0 = *reinterpret_cast<const int4 *>(s.bln + pr * 8), b1 = *reinterpret_cast<const int4 *>(s.bln + pr * 8 + 4);
    const int32_t bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
    int32_t v[4][2];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if ((mask >> g) & 1u) v[g][k] = wv_ln_fast(a[g][k], r.m_hi[g], r.m_lo[g], r.mean[g], k ? wv_hi(lws[g]) : wv_lo(lws[g]), bb[2 * g + k]);
    if (r.slow) {
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if ((mask >> g) & 1u) v[g][k] = wv_ln_slow(a[g][k], s.ln[g * 128 + row], k ? wv_hi(lws[g]) : wv_lo(lws[g]), bb[2 * g + k]);
    }
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if ((mask >> g) & 1u) a[g][k] = sat16(fast_rescale(v[g][k], L.f_ln[g]));
}

// m of a pair of cells (h of a layer without a projection) to where the next product and the caller read it
__device__ __forceinline__ void wv_store_m(const WaveCall &k, const WaveLayer &L, int8_t *img_unit, int row, int u, int b, int t, int32_t m0, int32_t m1,
                                           bool last_layer)
{
    if (u >= L.C) return;
    const uint16_t w = (uint16_t)((m0 & 0xff) | ((m1 & 0xff) << 8));
    *reinterpret_cast<uint16_t *>(img_unit + wv_img_off(row, u, k.ra)) = w;
    if (L.flags & F_PROJECTION) return;
    const bool both = u + 1 < L.C, fin = t == k.T - 1;
    if (last_layer) {
        int8_t *y = wv_y_row(k, L, t, b) + u;
        if (both && ((uintptr_t)y & 1) == 0) *reinterpret_cast<uint16_t *>(y) = w;
        else { y[0] = (int8_t)m0; if (both) y[1] = (int8_t)m1; }
    }
    if (fin) {
        int8_t *h = L.h + (size_t)b * L.O + u;
        h[0] = (int8_t)m0;
        if (both) h[1] = (int8_t)m1;
    }
}

__device__ __forceinline__ void wv_store_c(const WaveCall &k, const WaveLayer &L, int u, int b, int32_t c0, int32_t c1)
{
    int16_t *c = L.c + (size_t)b * L.C + u;
    if (u < L.C) c[0] = (int16_t)c0;
    if (u + 1 < L.C) c[1] = (int16_t)c1;
}

// sums of a unit's rows (gate slots in `mask`) from shared memory into the group's totals; clears the block's own
template <int G>
__device__ __forceinline__ void wv_push_stats(const WaveSmem &s, long long *totals, int rows, unsigned mask, int tid)
{
    for (int i = tid; i < rows * G; i += WV_EPI) {
        const int g = i / rows, row = i - g * rows;
        if (!((mask >> g) & 1u)) continue;
        uint32_t *st = s.st + (g * 3) * 128 + row;
        const long long sum = (long long)(int32_t)st[0];
        const unsigned long long sq = ((unsigned long long)st[256] << 20) + st[128];
        st[0] = st[128] = st[256] = 0u;
        unsigned long long *dst = reinterpret_cast<unsigned long long *>(totals + (size_t)(row * 4 + g) * 2);
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst), "l"((unsigned long long)sum) : "memory");
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst + 1), "l"(sq) : "memory");
    }
}
// layer-norm constants of a unit's rows from the group's totals
template <int G>
__device__ __forceinline__ void wv_pull_stats(const WaveLayer &L, const WaveSmem &s, const long long *totals, int rows, unsigned mask, int tid)
{
    for (int i = tid; i < rows * G; i += WV_EPI) {
        const int g = i / rows, row = i - g * rows;
        if (!((mask >> g) & 1u)) continue;
        const longlong2 v = __ldcg(reinterpret_cast<const longlong2 *>(totals + (size_t)(row * 4 + g) * 2));
        s.ln[g * 128 + row] = wv_make_ln(v.x, v.y, L.div_c, L.sigma_min);
    }
}
// Everything between the gate sums and m for one unit.  Tasks are (pair, row) with the row fastest, so that the gate
// buffers are read as contiguous runs; a thread keeps one row, whose layer-norm constants stay in registers.
template <int G, bool LN, bool PEEP, bool TAB>
__device__ __forceinline__ bool wv_elementwise(const WaveCall &k, const WaveLayer &L, const WaveSmem &s, const WaveRole &r, const ActLines &at, int u,
                                               int t, bool last_layer, WvPoint &pt, int tid)
{
    constexpr int SI = 0, SF = (G == 4) ? 1 : 0, SZ = SF + 1, SO = SF + 2;
    constexpr unsigned ALL = (1u << G) - 1u;
    const int rows = r.rows[u], gu = r.gu[u];
    unsigned *cnt = L.cnt + (size_t)gu * WC_PER_UNIT * WC_WORDS;
    long long *tot = L.totals ? L.totals + ((size_t)(t & 1) * k.nu + gu) * k.ra * 8 : nullptr;
    if (LN) {
        if (!wv_meet(k, cnt + WC_STATS * WC_WORDS, (unsigned)(t + 1) * L.n, pt, tid)) return false;
        wv_pull_stats<G>(L, s, tot, rows, PEEP ? ALL & ~(1u << SO) : ALL, tid);
        // the other set of totals was read by everyone before this step's sums were complete: cleared for the next step,
        // each block a share
        long long *next = L.totals + ((size_t)((t + 1) & 1) * k.nu + gu) * k.ra * 8;
        for (int i = r.rank * WV_EPI + tid; i < rows * 8; i += L.n * WV_EPI) next[i] = 0;
        wv_epi_sync();
    }
    const int per = rows < WV_EPI ? WV_EPI / rows : 1;          // pairs in flight: threads beyond per * rows have no task
    const int row = tid % rows, p0 = tid / rows;
    const int b = r.row0[u] + row;
    uint4 *g_s = r.g[u];
    const uint4 *x_s = g_s + (size_t)(k.units == 1 ? 1 + (t & 1) : 1) * r.pairs * rows;    // peephole: X(t) is kept beside the sums
    uint32_t *c_s = r.c[u];
    int8_t *img = (L.flags & F_PROJECTION) ? L.m_img + (size_t)gu * L.kb_c * k.ra * 128
                                           : L.out_img + ((size_t)(t + 1) * k.nu + gu) * L.kb_h * k.ra * 128;
    const bool fin = t == k.T - 1;
    WvLnRegs lr = {};
    if (LN && p0 < per) wv_load_ln<G>(s, row, PEEP ? ALL & ~(1u << SO) : ALL, lr);
    if (p0 < per) {
        // the next pair's inputs are requested before the present one is worked on (the buffers may lie in L2)
        uint4 g_next = make_uint4(0, 0, 0, 0);
        uint32_t c_next = 0;
        if (p0 < r.pairs) { g_next = g_s[p0 * rows + row]; c_next = c_s[p0 * rows + row]; }
#pragma unroll 1
        for (int pr = p0; pr < r.pairs; pr += per) {
            const uint4 g4 = g_next;
            const uint32_t cw = c_next;
            if (pr + per < r.pairs) { g_next = g_s[(pr + per) * rows + row]; c_next = c_s[(pr + per) * rows + row]; }
            const uint32_t gw[4] = {g4.x, g4.y, g4.z, g4.w};
            int32_t a[4][2];
#pragma unroll
            for (int g = 0; g < G; ++g) { a[g][0] = wv_lo(gw[g]); a[g][1] = wv_hi(gw[g]); }
            if (LN) wv_ln_pair<G>(L, s, lr, row, pr, PEEP ? ALL & ~(1u << SO) : ALL, a);
            const int32_t c_old[2] = {wv_lo(cw), wv_hi(cw)};
            int32_t c_new[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int32_t f = wv_sigmoid<TAB>(at, a[SF][q]), z = wv_tanh<TAB>(at, a[SZ][q]);
                int32_t i;
                if (G == 4) i = wv_sigmoid<TAB>(at, a[SI][q]);
                else { i = 32768 - f; if (i > 32767) i = 32767; }          // coupled input gate, Section 3.2.9
                c_new[q] = cell_update_fast(i, z, f, c_old[q], L.m_bits);
            }
            c_s[pr * rows + row] = ((uint32_t)c_new[0] & 0xffffu) | ((uint32_t)c_new[1] << 16);
            const int uc = r.u0 + 2 * pr;
            if (fin) wv_store_c(k, L, uc, b, c_new[0], c_new[1]);
            int32_t ao[2] = {a[SO][0], a[SO][1]};
            if (PEEP) {
                const uint4 x4 = x_s[pr * rows + row];
                const uint32_t xo = G == 4 ? x4.w : x4.z;
                const int32_t X[2] = {wv_lo(xo), wv_hi(xo)};
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int32_t P = s.P[pr * 8 + 2 * SO + q];
                    ao[q] = sat16(X[q] + a[SO][q] + sat16(fast_rescale(P * c_new[q], L.f_c[SO])));     // Eq. 5: o sees c^t
                }
                if (LN) {
                    // waits for the row's statistics
                    const uint32_t w = ((uint32_t)ao[0] & 0xffffu) | ((uint32_t)ao[1] << 16);
                    reinterpret_cast<uint32_t *>(&g_s[pr * rows + row])[SO] = w;
                    uint32_t *st = s.st + (SO * 3) * 128 + row;
                    const unsigned long long sq = (unsigned long long)((long long)ao[0] * ao[0] + (long long)ao[1] * ao[1]);
                    atomicAdd(st, (uint32_t)(ao[0] + ao[1]));
                    atomicAdd(st + 128, (uint32_t)(sq & 0xfffffu));
                    atomicAdd(st + 256, (uint32_t)(sq >> 20));
                    continue;
                }
            }
            const int32_t m0 = wv_hidden<TAB>(L, at, wv_sigmoid<TAB>(at, ao[0]), c_new[0]);
            const int32_t m1 = wv_hidden<TAB>(L, at, wv_sigmoid<TAB>(at, ao[1]), c_new[1]);
            wv_store_m(k, L, img, row, uc, b, t, m0, m1, last_layer);
        }
    }
    if (LN && PEEP) {
        wv_epi_sync();
        wv_push_stats<G>(s, tot, rows, 1u << SO, tid);
        if (!wv_publish(cnt + WC_STATS2 * WC_WORDS, false, pt, tid)) return false;
        if (!wv_meet(k, cnt + WC_STATS2 * WC_WORDS, (unsigned)(t + 1) * L.n, pt, tid)) return false;
        wv_pull_stats<G>(L, s, tot, rows, 1u << SO, tid);
        wv_epi_sync();
        if (p0 < per) {
            wv_load_ln<G>(s, row, 1u << SO, lr);
#pragma unroll 1
            for (int pr = p0; pr < r.pairs; pr += per) {
                const uint32_t gw = reinterpret_cast<const uint32_t *>(&g_s[pr * rows + row])[SO];
                const uint32_t cw = c_s[pr * rows + row];
                int32_t a[4][2] = {};
                a[SO][0] = wv_lo(gw); a[SO][1] = wv_hi(gw);
                wv_ln_pair<G>(L, s, lr, row, pr, 1u << SO, a);
                const int32_t m0 = wv_hidden<TAB>(L, at, wv_sigmoid<TAB>(at, a[SO][0]), wv_lo(cw));
                const int32_t m1 = wv_hidden<TAB>(L, at, wv_sigmoid<TAB>(at, a[SO][1]), wv_hi(cw));
                wv_store_m(k, L, img, row, r.u0 + 2 * pr, b, t, m0, m1, last_layer);
            }
        }
    }
    return wv_publish(cnt + ((L.flags & F_PROJECTION) ? WC_M : WC_H) * WC_WORDS, true, pt, tid);
}

// ---- the table of operations -------------------------------------------------------------------------------------------

// first the prologue (X of step 0), then the operations of a step, in the order all roles follow
__device__ void wv_build_ops(const WaveCall &k, const WaveLayer &L, const WaveRole &r, WaveCtl *ctl)
{
    int n = 0;
    auto add = [&](int kind, int u, int tile) { ctl->ops[n].kind = (uint8_t)kind; ctl->ops[n].u = (uint8_t)u; ctl->ops[n].tile = (uint8_t)tile; ++n; };
    const bool proj = (L.flags & F_PROJECTION) != 0;
    const int nt = (r.pairs + L.ppt - 1) / L.ppt, ntp = proj ? (r.outs + L.opt - 1) / L.opt : 0;
    auto gates = [&](int kind, int u, int from, int to) { for (int i = from; i < to; ++i) add(kind, u, i); };
    auto project = [&](int u) {
        if (!proj) return;
        for (int i = 0; i < ntp; ++i) add(OP_P, u, i);
        add(OP_F, u, 0);
    };
    int nu = 0;
    while (nu < k.units && r.rows[nu] > 0) ++nu;
    for (int u = 0; u < nu; ++u) gates(OP_X, u, 0, nt);
    ctl->n_pro = n;
    if (nu == 1) {
        gates(OP_H, 0, 0, nt);
        add(OP_S, 0, 0);
        if (k.early) gates(OP_X, 0, 0, (nt + 1) / 2);
        add(OP_B, 0, 0);
        if (k.early) gates(OP_X, 0, (nt + 1) / 2, nt);
        project(0);
        if (!k.early) gates(OP_X, 0, 0, nt);
    } else if (nu == 2) {
        for (int u = 0; u < 2; ++u) { gates(OP_H, u, 0, nt); add(OP_S, u, 0); }
        for (int u = 0; u < 2; ++u) add(OP_B, u, 0);
        for (int u = 0; u < 2; ++u) { project(u); gates(OP_X, u, 0, nt); }
    }
    ctl->n_ops = n - ctl->n_pro;
}

// calls f(op, t) for every operation in order (X with the step it belongs to); stops when f returns false
template <class F>
__device__ __forceinline__ bool wv_walk(const WaveCtl *ctl, int T, F f)
{
    for (int i = 0; i < ctl->n_pro; ++i)
        if (!f(ctl->ops[i], 0)) return false;
    for (int t = 0; t < T; ++t)
        for (int i = 0; i < ctl->n_ops; ++i) {
            const WaveOp op = ctl->ops[ctl->n_pro + i];
            if (op.kind == OP_X && t + 1 == T) continue;
            if (!f(op, op.kind == OP_X ? t + 1 : t)) return false;
        }
    return true;
}

// shared memory of a block: [A slots][B slots][control][constants][statistics][tables][gate buffers, cell states]
struct WvLayout { size_t b_ring, ctl, consts, st, ln, tab, gates, total; };
__host__ __device__ inline WvLayout wv_layout(int na, int nb, int b_slot, int max_ppc, int max_opc, int max_tab, size_t gates_bytes)
{
    WvLayout l;
    l.b_ring = (size_t)na * WV_A_SLOT;
    l.ctl = l.b_ring + (size_t)nb * b_slot;
    l.consts = l.ctl + wv_up(sizeof(WaveCtl), 16);
    l.st = l.consts + (size_t)max_ppc * 8 * (3 * 4 + 2 * 2) + wv_up((size_t)max_opc * 4, 16);
    l.ln = l.st + 12 * 128 * 4;
    l.tab = l.ln + 4 * 128 * 16;
    l.gates = l.tab + wv_up((size_t)max_tab, 16);
    l.total = l.gates + gates_bytes + 1024;        // 1024: alignment of the rings
    return l;
}

// A block that leaves early: its copies and MMAs in flight end (whole warps; `warp` 0 to 3 are the service warps).  Out of line, so
// that the kernel's loops keep their shape.
__device__ __noinline__ void wv_drain_block(WaveCtl *ctl, int na, int nb, bool tab, int warp)
{
    if (warp == 0) wv_drain_ring(ctl->a_full, na, ctl->end_slot[0], ctl->end_phase[0]);
    else if (warp == 1) wv_drain_ring(ctl->b_full, nb, ctl->end_slot[1], ctl->end_phase[1]);
    else if (warp == 2) wv_drain_mmas(&ctl->mma_done);
    else if (warp == 3 && tab) wv_drain(&ctl->tab_full, 0);
}

template <int G, bool LN, bool PEEP, bool TAB>
__global__ void __launch_bounds__(WV_THREADS, 1) k_wave_sm100(const __grid_constant__ WaveCall k)
{
    extern __shared__ uint8_t wv_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)wv_raw + 1023) & ~(uintptr_t)1023);
    const WvLayout lay = wv_layout(k.na, k.nb, k.b_slot, k.max_ppc, k.max_opc, k.max_tab, 0);
    uint8_t *a_ring = smem, *b_ring = smem + lay.b_ring;
    WaveCtl *ctl = reinterpret_cast<WaveCtl *>(smem + lay.ctl);
    WaveSmem s;
    {
        uint8_t *p = smem + lay.consts;
        s.bx = (int32_t *)p;  p += (size_t)k.max_ppc * 32;
        s.bh = (int32_t *)p;  p += (size_t)k.max_ppc * 32;
        s.bln = (int32_t *)p; p += (size_t)k.max_ppc * 32;
        s.L = (int16_t *)p;   p += (size_t)k.max_ppc * 16;
        s.P = (int16_t *)p;   p += (size_t)k.max_ppc * 16;
        s.bp = (int32_t *)p;
        s.st = (uint32_t *)(smem + lay.st);
        s.ln = (WvLnRow *)(smem + lay.ln);
        s.tab = smem + lay.tab;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = blockIdx.x;
    volatile int *abort_flag = &ctl->abort_flag;

    WaveRole r;
    r.li = -1;
    for (int l = 0; l < k.n_layers; ++l)
        if (cta >= k.layer[l].cta0 && cta < k.layer[l].cta0 + k.layer[l].n * k.rg) r.li = l;
    if (r.li < 0) return;                                      // spare block: takes no part in any counter
    const WaveLayer &L = k.layer[r.li];
    const bool proj = (L.flags & F_PROJECTION) != 0, last_layer = L.last != 0;
    r.rgi = (cta - L.cta0) / L.n;
    r.rank = cta - L.cta0 - r.rgi * L.n;
    r.u0 = r.rank * L.ppc * 2;
    r.pairs = L.C > r.u0 ? (L.C - r.u0 + 1) / 2 : 0;
    if (r.pairs > L.ppc) r.pairs = L.ppc;
    if (G == 3) r.pairs = (r.pairs + 1) & ~1;
    r.o_lo = r.rank * L.opc;
    r.outs = proj ? (L.O - r.o_lo < L.opc ? L.O - r.o_lo : L.opc) : 0;
    if (r.outs < 0) r.outs = 0;
    r.n_rows_max = (k.B + k.nu - 1) / k.nu;
    for (int u = 0; u < 2; ++u) {
        r.gu[u] = u < k.units ? r.rgi * k.units + u : 0;
        r.row0[u] = (int)((long long)r.gu[u] * k.B / k.nu);
        r.rows[u] = u < k.units ? (int)((long long)(r.gu[u] + 1) * k.B / k.nu) - r.row0[u] : 0;
        const size_t per_unit = (size_t)k.nbuf * k.max_ppc * r.n_rows_max;
        if (k.gx_s) {
            r.g[u] = reinterpret_cast<uint4 *>(smem + lay.gates) + u * per_unit;
            r.c[u] = reinterpret_cast<uint32_t *>(smem + lay.gates + (size_t)k.units * per_unit * 16) + (size_t)u * k.max_ppc * r.n_rows_max;
        } else {
            r.g[u] = k.gbuf + ((size_t)cta * k.units + u) * per_unit;
            r.c[u] = k.cbuf + ((size_t)cta * k.units + u) * k.max_ppc * r.n_rows_max;
        }
    }
    if (r.rows[0] == 0) return;                                // fewer rows than row groups: this group is idle

    if (threadIdx.x == 0) {
        for (int i = 0; i < WV_MAX_SLOTS; ++i) {
            ptx::mbar_init(&ctl->a_full[i], 1); ptx::mbar_init(&ctl->a_empty[i], 1);
            ptx::mbar_init(&ctl->b_full[i], 1); ptx::mbar_init(&ctl->b_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) { ptx::mbar_init(&ctl->t_full[i], 1); ptx::mbar_init(&ctl->t_empty[i], WV_EPI / 32); }
        ptx::mbar_init(&ctl->tab_full, 1);
        ptx::mbar_init(&ctl->mma_done, 1);
        ctl->abort_flag = 0;
        ctl->exit_at = 0x7fffffff;
        ptx::fence_barrier_init();
        wv_build_ops(k, L, r, ctl);
        if (TAB) {
            ptx::mbar_arrive_expect_tx(&ctl->tab_full, L.tab_lay.bytes);
            ptx::bulk_load_1d(s.tab, L.tab, L.tab_lay.bytes, &ctl->tab_full);
        }
    }
    if (warp == 2) {
        ptx::tmem_alloc(&ctl->tmem_base, 512);
        ptx::tmem_relinquish();
    }
    // constants of the block's columns, slot-major within a pair of cells
    for (int i = threadIdx.x; i < r.pairs * 8; i += WV_THREADS) {
        const int pr = i >> 3, g = (i >> 1) & 3, u = r.u0 + 2 * pr + (i & 1);
        const bool in = g < G && u < L.C;
        const int n = u * G + g;
        s.bx[i] = in ? L.bx[n] : 0;
        s.bh[i] = in ? L.bh[n] : 0;
        s.bln[i] = in && LN ? L.bln[n] : 0;
        s.L[i] = in && LN ? L.L[n] : (int16_t)0;
        s.P[i] = in && PEEP ? L.P[n] : (int16_t)0;
    }
    for (int i = threadIdx.x; i < r.outs; i += WV_THREADS) s.bp[i] = L.bp[r.o_lo + i];
    for (int i = threadIdx.x; i < 12 * 128; i += WV_THREADS) s.st[i] = 0u;
    for (int u = 0; u < 2; ++u)
        for (int i = threadIdx.x; i < r.pairs * r.rows[u]; i += WV_THREADS) {
            const int pr = i / r.rows[u], b = r.row0[u] + i - pr * r.rows[u], c = r.u0 + 2 * pr;
            const int16_t *src = L.c + (size_t)b * L.C + c;
            const uint32_t lo = c < L.C ? (uint16_t)src[0] : 0u, hi = c + 1 < L.C ? (uint16_t)src[1] : 0u;
            r.c[u][i] = lo | (hi << 16);
        }
    ptx::tc_fence_before();
    ptx::cta_sync();
    ptx::tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    unsigned *cnt0 = L.cnt;
    auto gate_tile_pairs = [&](int tile) { const int left = r.pairs - tile * L.ppt; return left < L.ppt ? left : L.ppt; };

    if (warp == 0) {
        // ---------------- activations ----------------
        int slot = 0; uint32_t phase = 0;
        const uint32_t kb_bytes = (uint32_t)k.ra * 128u;
        const bool copier = lane < k.nrep;
        wv_walk(ctl, k.T, [&](const WaveOp &op, int t) -> bool {
            if (op.kind > OP_P) return true;
            const int gu = r.gu[op.u];
            const int8_t *src;
            const unsigned *cnt = nullptr;
            unsigned target = 0;
            int nkb;
            if (op.kind == OP_X) {
                nkb = L.kb_i;
                src = L.in_img + ((size_t)(t + (L.below ? 1 : 0)) * k.nu + gu) * nkb * kb_bytes;      // (slot 0 of a layer's outputs is h^-1)
                if (L.below) { cnt = k.layer[r.li - 1].cnt + ((size_t)gu * WC_PER_UNIT + WC_H) * WC_WORDS; target = (unsigned)(t + 1) * L.below; }
            } else if (op.kind == OP_H) {
                nkb = L.kb_h;
                src = L.out_img + ((size_t)t * k.nu + gu) * nkb * kb_bytes;
                if (t > 0) { cnt = cnt0 + ((size_t)gu * WC_PER_UNIT + WC_H) * WC_WORDS; target = (unsigned)t * L.n; }
            } else {
                nkb = L.kb_c;
                src = L.m_img + (size_t)gu * nkb * kb_bytes;
                cnt = cnt0 + ((size_t)gu * WC_PER_UNIT + WC_M) * WC_WORDS; target = (unsigned)(t + 1) * L.n;
            }
            if (cnt) {
                bool ok = true;
                if (lane == 0) ok = wv_wait_count(k, cnt, target, abort_flag);
                if (!__shfl_sync(0xffffffffu, (int)ok, 0)) return false;
                __syncwarp();
            }
            wv_fence_async_global();
            for (int kb = 0; kb < nkb; ++kb) {
                bool ok = true;
                if (lane == 0) {
                    ok = wv_wait(&ctl->a_empty[slot], phase ^ 1u, abort_flag);
                    if (ok) ptx::mbar_arrive_expect_tx(&ctl->a_full[slot], kb_bytes * (uint32_t)k.nrep);
                }
                if (!__shfl_sync(0xffffffffu, (int)ok, 0)) return false;
                if (copier)
                    ptx::bulk_load_1d(a_ring + (size_t)slot * WV_A_SLOT + (size_t)lane * (WV_A_SLOT / k.nrep), src + (size_t)kb * kb_bytes, kb_bytes,
                                      &ctl->a_full[slot]);
                if (++slot == k.na) { slot = 0; phase ^= 1u; }
            }
            return true;
        });
        if (lane == 0) { ctl->end_slot[0] = slot; ctl->end_phase[0] = phase; }
    } else if (warp == 1) {
        // ---------------- weights ----------------
        if (lane == 0) {
            const uint64_t policy = wv_weights_policy();
            int slot = 0; uint32_t phase = 0;
            wv_walk(ctl, k.T, [&](const WaveOp &op, int) -> bool {
                if (op.kind > OP_P) return true;
                const int8_t *src;
                uint32_t bytes;
                int nkb;
                if (op.kind == OP_P) {
                    nkb = L.kb_c; bytes = (uint32_t)L.npadp * 128u;
                    src = L.img_p + (size_t)(r.rank * L.ntp + op.tile) * nkb * bytes;
                } else {
                    nkb = op.kind == OP_X ? L.kb_i : L.kb_h; bytes = (uint32_t)L.npad * 128u;
                    src = (op.kind == OP_X ? L.img_w : L.img_r) + (size_t)(r.rank * L.nt + op.tile) * nkb * bytes;
                }
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!wv_wait(&ctl->b_empty[slot], phase ^ 1u, abort_flag)) return false;
                    ptx::mbar_arrive_expect_tx(&ctl->b_full[slot], bytes);
                    if (k.w_evict) wv_load_weights(b_ring + (size_t)slot * k.b_slot, src + (size_t)kb * bytes, bytes, &ctl->b_full[slot], policy);
                    else ptx::bulk_load_1d(b_ring + (size_t)slot * k.b_slot, src + (size_t)kb * bytes, bytes, &ctl->b_full[slot]);
                    if (++slot == k.nb) { slot = 0; phase ^= 1u; }
                }
                return true;
            });
            ctl->end_slot[1] = slot; ctl->end_phase[1] = phase;
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------- MMAs ----------------
        int sa = 0, sb = 0, job = 0;
        uint32_t pa = 0, pb = 0;
        const uint64_t a_desc0 = ptx::smem_desc_k_sw128(ptx::smem_u32(a_ring)), b_desc0 = ptx::smem_desc_k_sw128(ptx::smem_u32(b_ring));
        wv_walk(ctl, k.T, [&](const WaveOp &op, int) -> bool {
            if (op.kind > OP_P) return true;
            const int nkb = op.kind == OP_X ? L.kb_i : op.kind == OP_H ? L.kb_h : L.kb_c;
            const uint32_t idesc = ptx::idesc_i8(128, op.kind == OP_P ? L.npadp : L.npad);
            const uint32_t d = tmem_base + (uint32_t)(job & 1) * WV_ACC_COLS;
            if (!wv_wait_warp(&ctl->t_empty[job & 1], ((uint32_t)(job >> 1) & 1u) ^ 1u, abort_flag)) return false;
            ptx::tc_fence_after();
            for (int kb = 0; kb < nkb; ++kb) {
                const bool ok = wv_wait(&ctl->a_full[sa], pa, abort_flag) && wv_wait(&ctl->b_full[sb], pb, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) return false;
                ptx::tc_fence_after();
                if (ptx::elect_one()) {
                    wv_mma_kblock(d, a_desc0 + (uint64_t)(sa * (WV_A_SLOT >> 4)), b_desc0 + (uint64_t)(sb * (k.b_slot >> 4)), idesc, kb == 0);
                    ptx::mma_commit(&ctl->a_empty[sa]);
                    ptx::mma_commit(&ctl->b_empty[sb]);
                }
                __syncwarp();
                if (++sa == k.na) { sa = 0; pa ^= 1u; }
                if (++sb == k.nb) { sb = 0; pb ^= 1u; }
            }
            wv_commit(&ctl->t_full[job & 1]);
            ++job;
            return true;
        });
    } else if (warp >= WV_EPI_WARP0) {
        // ---------------- epilogues and elementwise work ----------------
        const int tid = threadIdx.x - 32 * WV_EPI_WARP0;
        const int quarter = warp & 3, qpr = 4 / k.nrep;        // quarters of the lanes that hold one copy of the rows
        const int row = (quarter % qpr) * 32 + lane, part = ((warp - WV_EPI_WARP0) >> 2) + 4 * (quarter / qpr), nparts = 4 * k.nrep;
        const ActLines at = make_act_lines(ptx::smem_u32(s.tab), L.tab_lay);
        WvPoint pt{abort_flag, &ctl->exit_at, 0};
        if (TAB) wv_wait(&ctl->tab_full, 0, abort_flag);
        int job = 0;
        wv_walk(ctl, k.T, [&](const WaveOp &op, int t) -> bool {
            const int u = op.u, rows = r.rows[u], gu = r.gu[u];
            if (op.kind <= OP_P) {
                // (after an abort the tile is skipped: on to the next meeting point)
                uint64_t *full = &ctl->t_full[job & 1];
                const uint32_t parity = (uint32_t)(job >> 1) & 1u;
                const uint32_t ta = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(job & 1) * WV_ACC_COLS;
                const bool valid = row < rows;
                uint4 *gb = r.g[u];
                uint4 *xb = gb + (size_t)(k.units == 1 ? 1 + (PEEP ? (t & 1) : 0) : (PEEP ? 1 : 0)) * r.pairs * rows;
                const int pair0 = op.tile * L.ppt;
                if (op.kind == OP_X) {
                    wv_gate_tile<G, LN, PEEP, false>(L, s, ta, pair0, gate_tile_pairs(op.tile), part, nparts, row, rows, valid, nullptr, xb, nullptr, full, parity,
                                                     abort_flag);
                } else if (op.kind == OP_H) {
                    wv_gate_tile<G, LN, PEEP, true>(L, s, ta, pair0, gate_tile_pairs(op.tile), part, nparts, row, rows, valid, xb, gb, r.c[u], full, parity,
                                                    abort_flag);
                } else if (__all_sync(0xffffffffu, wv_wait(full, parity, abort_flag))) {
                    ptx::tc_fence_after();
                    wv_proj_tile(k, L, s, r, ta, op.tile * L.opt, r.outs - op.tile * L.opt < L.opt ? r.outs - op.tile * L.opt : L.opt, part, nparts, row, valid,
                                 L.out_img + ((size_t)(t + 1) * k.nu + gu) * L.kb_h * k.ra * 128, r.row0[u] + row, t, last_layer);
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&ctl->t_empty[job & 1]);
                ++job;
                return true;
            }
            unsigned *cnt = cnt0 + (size_t)gu * WC_PER_UNIT * WC_WORDS;
            if (op.kind == OP_S) {
                wv_epi_sync();                                 // gate sums and their statistics are complete in this block
                if (!LN) return true;
                constexpr unsigned ALL = (1u << G) - 1u;
                wv_push_stats<G>(s, L.totals + ((size_t)(t & 1) * k.nu + gu) * k.ra * 8, rows, PEEP ? ALL & ~(1u << (G - 1)) : ALL, tid);
                return wv_publish(cnt + WC_STATS * WC_WORDS, false, pt, tid);
            }
            if (op.kind == OP_B) return wv_elementwise<G, LN, PEEP, TAB>(k, L, s, r, at, u, t, last_layer, pt, tid);
            return wv_publish(cnt + WC_H * WC_WORDS, true, pt, tid);        // OP_F: h^t of this block is written
        });
    }

    // ---------------- teardown ----------------
    ptx::cta_sync();
    if (*abort_flag) {
        // a wait ran out: copies and MMAs in flight end, then report
        wv_drain_block(ctl, k.na, k.nb, TAB, warp);
        if (threadIdx.x == 0) { atomicExch(k.abort_word, 1u); atomicExch(k.status, 2); }
    }
    ptx::cta_sync();
    if (warp == 2) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, 512);
    }
}

// ---- before the launch: operand images ---------------------------------------------------------------------------------

// The caller's x and h into activation images; counters, totals and status cleared.
__global__ void k_wave_prepare(const __grid_constant__ WaveCall k, const int8_t *x, unsigned *zero, size_t zero_words)
{
    const size_t step = (size_t)gridDim.x * blockDim.x, first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    auto put = [&](int8_t *img, int kbs, size_t block, int b, int chunk, const uint4 &v) {
        // unit of row b: units are floor(i B / nu) .. floor((i + 1) B / nu)
        int gu = (int)(((long long)(b + 1) * k.nu - 1) / k.B);
        const int row = b - (int)((long long)gu * k.B / k.nu);
        *reinterpret_cast<uint4 *>(img + (block * k.nu + gu) * kbs * k.ra * 128 + wv_img_off(row, chunk * 16, k.ra)) = v;
    };
    for (int l = 0; l < k.n_layers; ++l) {
        const WaveLayer &L = k.layer[l];
        if (!L.first) continue;
        const int per = (L.I + 15) >> 4;
        const size_t total = (size_t)k.T * k.B * per;
        for (size_t i = first; i < total; i += step) {
            const size_t rt = i / per, t = rt / k.B;
            const int chunk = (int)(i - rt * per), b = (int)(rt % k.B);
            put(L.in_img, L.kb_i, L.dir ? k.T - 1 - t : t, b, chunk, wv_load16(x + rt * L.I + chunk * 16, L.I - chunk * 16));
        }
    }
    for (int l = 0; l < k.n_layers; ++l) {
        const WaveLayer &L = k.layer[l];
        const int per = (L.O + 15) >> 4;
        for (size_t i = first; i < (size_t)k.B * per; i += step) {
            const int b = (int)(i / per), chunk = (int)(i - (size_t)b * per);
            put(L.out_img, L.kb_h, 0, b, chunk, wv_load16(L.h + (size_t)b * L.O + chunk * 16, L.O - chunk * 16));
        }
    }
    for (size_t i = first; i < zero_words; i += step) zero[i] = 0u;
    if (first == 0) {
        *k.status = 0;
        if (k.status2) *k.status2 = 0;
    }
}

// A weight matrix into the tiles its blocks stream: [rank][tile][k-block][column][128 bytes], swizzled.  Gate matrices
// (G > 0): column c of a tile is slot (c mod 2G) / 2, cell 2 (c / 2G) + c mod 2 of the tile.  W_proj (G = 0): plain rows.
__global__ void k_wave_tile_weights(const int8_t *src, int8_t *dst, int G, int rows, int K, int n, int per_rank, int nt, int per_tile, int npad, int nkb)
{
    const size_t total = (size_t)n * nt * nkb * npad * 8;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int chunk = (int)(i & 7);
        size_t q = i >> 3;
        const int c = (int)(q % npad); q /= npad;
        const int kb = (int)(q % nkb); q /= nkb;
        const int tile = (int)(q % nt), rank = (int)(q / nt);
        int src_row = -1;
        if (G > 0) {
            const int pr = tile * per_tile + c / (2 * G), in = c % (2 * G);
            const int u = 2 * (rank * per_rank + pr) + (in & 1);
            if (c / (2 * G) < per_tile && pr < per_rank && u * G < rows) src_row = u * G + (in >> 1);
        } else {
            const int o = tile * per_tile + c;
            if (c < per_tile && o < per_rank && rank * per_rank + o < rows) src_row = rank * per_rank + o;
        }
        const int k0 = kb * 128 + chunk * 16;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (src_row >= 0 && k0 < K) v = wv_load16(src + (size_t)src_row * K + k0, K - k0);
        *reinterpret_cast<uint4 *>(dst + (((size_t)(rank * nt + tile) * nkb + kb) * npad + c) * 128 + ((chunk ^ (c & 7)) << 4)) = v;
    }
}

int wv_round(int v, int m) { return (v + m - 1) / m * m; }

template <bool TAB>
const void *wave_kernel_of(int G, bool ln, bool peep)
{
    if (G == 4) {
        if (ln) return peep ? (const void *)k_wave_sm100<4, true, true, TAB> : (const void *)k_wave_sm100<4, true, false, TAB>;
        return peep ? (const void *)k_wave_sm100<4, false, true, TAB> : (const void *)k_wave_sm100<4, false, false, TAB>;
    }
    if (ln) return peep ? (const void *)k_wave_sm100<3, true, true, TAB> : (const void *)k_wave_sm100<3, true, false, TAB>;
    return peep ? (const void *)k_wave_sm100<3, false, true, TAB> : (const void *)k_wave_sm100<3, false, false, TAB>;
}

}  // namespace

constexpr int WV_MAX_ROWS = 256;

// One way of sharing a stack out over the SMs: mode 0 batch as the M side (this file), mode 1 gate rows as the M side, for up to
// 32 rows per row group (wave_small_sm100.cu).
struct WavePlan {
    int mode = 0, rg = 1, grid = 0;
    int cl = 0;                    // mode 1: blocks of a cluster that is a (layer, row group); 0: no clusters
    bool ok = true, used = false;
    int max_ppc = 0, max_cpc = 0, max_opc = 0, b_slot = 0;
    std::vector<WaveLayer> layer;
};

struct WaveStack {
    int n_layers = 0, max_T = 0, max_B = 0, max_smem = 0, sm_count = 0;
    int depth = 0;                 // layers of one stack (two of them: the directions of a bidirectional one)
    int y_stride = 0;
    int G = 4;
    bool ln = false, peep = false, tabs = false;
    bool proj = false;             // some layer has a projection
    bool ragged = false;           // some dimension is not a multiple of 16
    int max_C = 0;
    size_t weights = 0;            // bytes of all layers' weights
    size_t resident = 0;           // ... of the first layer's R and W_proj, which the per-layer kernel keeps in shared memory
    uint16_t fit_groups[WV_MAX_ROWS + 1];      // groups in which the few-row form could hold a call's rows, 0: none
    std::vector<WavePlan> plan;
    int8_t by_rows[2][WV_MAX_ROWS + 1];        // plan of a call by its rows, [0] without and [1] with memoised nonlinearities; -1: none
    int max_tab = 0, max_kb_i = 0, max_kb_h = 0, max_kb_c = 0;
    unsigned *zero = nullptr;      // abort word, counters, totals: cleared before every call
    uint4 *gbuf = nullptr;
    uint32_t *cbuf = nullptr;
    void *block[2] = {nullptr, nullptr};       // plans and tables; a call's activations, unless they lie in the caller's scratch
    ResidentStack *res = nullptr;  // wave_resident_sm100.cu; null: no call of this stack fits it
    int res_mode = 0;              // 1: never taken, 2: launches of clusters are refused
    unsigned dbg_missing = 0;
    unsigned long long dbg_limit_ns = 0;
};

void wave_destroy(WaveStack *s)
{
    if (!s) return;
    for (void *p : s->block) cudaFree(p);
    resident_destroy(s->res);
    delete s;
}

namespace {

constexpr int WV_SMALL_ROWS = 32;

// Rows a call of B rows is cut into: `rg` row groups times one or two units of at most 128 rows each.
void wave_units(int B, int rg, int &units, int &nu, int &ra)
{
    units = (B + rg - 1) / rg > 128 ? 2 : 1;
    nu = rg * units;
    ra = wv_round((B + nu - 1) / nu, 8);
}

// Whether wave_small_sm100.cu can take B rows in rg groups of blocks (shared memory and tensor memory of the widest layer).
bool wave_small_fits(const WaveStack *s, const std::vector<const LayerParams *> &lp, int rg, int B, int sm_count)
{
    const int per = sm_count / ((int)lp.size() * rg), rows = (B + rg - 1) / rg;
    if (per < 1 || rows > WV_SMALL_ROWS) return false;
    WaveCall k;
    memset(&k, 0, sizeof(k));
    k.B = B; k.nu = rg; k.ra = wv_round(rows, 8); k.b_slot = WS_SLOT_ROWS * 128; k.max_tab = s->max_tab;
    for (const LayerParams *p : lp) {
        const int cpc = (p->C + per - 1) / per, n = (p->C + cpc - 1) / cpc, nt = (cpc + 31) / 32;
        const bool proj = p->flags & F_PROJECTION;
        const int opc = proj ? (p->O + n - 1) / n : 0, ntp = (opc + 127) / 128;
        if (nt > 8 || (2 * nt + ntp) * k.ra > 512) return false;
        k.max_cpc = std::max(k.max_cpc, wv_round(cpc, 2));
        k.max_opc = std::max(k.max_opc, wv_round(opc, 4));
        k.max_kb_i = std::max(k.max_kb_i, (p->I + 127) / 128);
        k.max_kb_h = std::max(k.max_kb_h, (p->O + 127) / 128);
        if (proj) k.max_kb_c = std::max(k.max_kb_c, (p->C + 127) / 128);
    }
    return wave_small_smem(k, 2, s->peep) <= (size_t)s->max_smem;
}

// The fewest groups of at least 9 blocks in which the few-row kernel can hold the B rows of a call; 0: none.
int wave_fit_groups(const WaveStack *s, const std::vector<const LayerParams *> &lp, int B)
{
    for (int rg = 1;; rg *= 2) {
        if (wave_small_fits(s, lp, rg, B, s->sm_count)) return rg;
        if (2 * rg > B || s->sm_count / (2 * rg * (int)lp.size()) < 9) return 0;
    }
}

// How many groups the B rows of a call are split into.  (Deep stacks: the layers already share out the SMs.)
int wave_row_groups(const WaveStack *s, int mode, const std::vector<const LayerParams *> &lp, int B)
{
    const int n = (int)lp.size(), sm_count = s->sm_count;
    int rg = 1;
    if (mode == 0) {
        // more than 64 rows per group and at least 32 blocks left (two 1024-cell layers, 256 rows: 32 us per step as one group of two
        // units, 25 as two groups)
        while ((B + rg - 1) / rg > 64 && sm_count / (2 * rg * n) >= 32) rg *= 2;
        return rg;
    }
    // As many as it takes for the few-row kernel to hold a group's rows, down to 9 blocks: it is the faster one even then (us per
    // step against the many-row kernel as one group: five 1024-cell CIFG layers, 64 rows 12.0 as two groups against 14.1; four
    // 1024-cell layers, 100 rows 24 as four against 28; eight 2048-cell layers, 32 rows 37 as two against 41).
    // Every group streams all weights, though: above 128 MB per step (200 with layer norm, whose exchanges the few-row form has
    // cheaper) the many-row form, with its one group, is ahead of it (us per call, few-row, many-row and layer by layer: three 2048-cell
    // layers, 64 rows, 16 steps, four groups of 88 MB 951, 455 and 691; two 2048-cell layers, 33 rows, 218 MB 493, 352 and 417; below the
    // line four 1024-cell layers, 96 rows, 126 MB 4 % ahead).
    rg = wave_fit_groups(s, lp, B);
    if (rg == 0 || (rg > 1 && rg * s->weights > (size_t)(s->ln ? 200 : 128) * 1000000)) return 1;
    // Then, fewer blocks per group make every exchange cheaper (two 512-cell layers, 16 rows: 9.0 us per step with one group, 8.5
    // with four; one 2048-cell layer with layer norm and peephole, 32 rows: 26 and 17), but a block streams more weights per step:
    // below 16 blocks, or beyond 320 KB, the groups cost more than they save (the same layers with eight groups: 9.2 and 18; five
    // 1024-cell layers, 4 rows: 7.5 with one group, 10.3 with two), unless a block has little to do: up to 64 KB and 32 cells, groups go
    // down to 9 blocks (us per call of 100 steps, 16 blocks and 9: three 256-cell layers, 64 rows 493 and 446; two, 32 rows 404 and 385;
    // 107 cells per block, eight layers, 5 rows, 12 steps 180 and 191).
    size_t bytes = 0;
    for (const LayerParams *p : lp)
        bytes = std::max(bytes, (size_t)p->N * (p->I + p->O) + ((p->flags & F_PROJECTION) ? (size_t)p->O * p->C : 0));
    auto worth = [&](int per) { return per >= 16 ? bytes / per <= 320 * 1024 : per >= 9 && bytes / per <= 64 * 1024 && s->max_C <= 32 * per; };
    while (2 * rg <= B && worth(sm_count / (2 * rg * n))) rg *= 2;
    return rg;
}

// Shares of the blocks of one layer under `mode`, `per` blocks at most; false: the plan does not work.
bool wave_share_layer(int mode, const LayerParams &p, int per, bool cluster, WaveLayer &L)
{
    const bool proj = p.flags & F_PROJECTION;
    L.opc = 0; L.ntp = 0; L.opt = 4; L.npadp = 16; L.opp = 8; L.kpp = 1;
    // blocks without cells would only lengthen the exchanges: the projection keeps to the blocks that have some
    if (mode == 0) {
        const int pairs = (p.C + 1) / 2, grain = p.G == 3 ? 2 : 1, ppt_max = p.G == 4 ? 32 : 42;
        L.ppc = wv_round((pairs + per - 1) / per, grain);
        L.n = (pairs + L.ppc - 1) / L.ppc;
        L.nt = (L.ppc + ppt_max - 1) / ppt_max;
        L.ppt = wv_round((L.ppc + L.nt - 1) / L.nt, grain);
        L.npad = wv_round(L.ppt * 2 * p.G, 16);
        if (proj) {
            L.opc = wv_round((p.O + L.n - 1) / L.n, 4);
            L.ntp = (L.opc + 255) / 256;
            L.opt = wv_round((L.opc + L.ntp - 1) / L.ntp, 4);
            L.npadp = wv_round(L.opt, 16);
        }
        if (L.npad > WV_ACC_COLS || L.npadp > WV_ACC_COLS || 2 * (4 * L.nt + L.ntp + 4) > WV_MAX_OPS) return false;
    } else {
        L.cpc = (p.C + per - 1) / per;
        if (cluster) L.cpc = wv_round(L.cpc, 8);               // (m and h cross the cluster in pieces of at least 8 bytes)
        L.n = (p.C + L.cpc - 1) / L.cpc;
        L.nt = (L.cpc + 31) / 32;
        L.ct = (L.cpc + L.nt - 1) / L.nt;
        L.ctp = L.ct <= 8 ? 8 : L.ct <= 16 ? 16 : 32;                // (a chunk's gates are 32 rows apart and leave no gaps)
        L.kpg = 32 / L.ctp;
        if (proj) {
            L.opc = (p.O + L.n - 1) / L.n;
            if (cluster) L.opc = wv_round(L.opc, 8);
            L.ntp = (L.opc + 127) / 128;
            L.opt = (L.opc + L.ntp - 1) / L.ntp;
            L.opp = wv_round(L.opt, 8);
            L.kpp = WS_SLOT_ROWS / L.opp;
        }
        if (L.nt > 8 || (2 * L.nt + L.ntp) * 8 > 512) return false;
    }
    const size_t row_bytes = mode == 0 ? (size_t)L.n * L.nt * L.npad * 128 : (size_t)L.n * L.nt * p.G * L.ctp * 128;
    auto kbs = [&](int kb) { return (size_t)(mode == 0 ? kb : wv_round(kb, L.kpg)); };
    L.w_size[0] = row_bytes * kbs(L.kb_i);
    L.w_size[1] = row_bytes * kbs(L.kb_h);
    L.w_size[2] = proj ? (size_t)L.n * L.ntp * (mode == 0 ? L.npadp : L.opp) * 128 * L.kb_c : 0;
    return true;
}

// The plan of `mode` with rg row groups, made on first request; its number in s->plan.
int wave_plan(WaveStack *s, const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, int mode, int rg, int cl = 0)
{
    for (size_t i = 0; i < s->plan.size(); ++i)
        if (s->plan[i].mode == mode && s->plan[i].rg == rg && s->plan[i].cl == cl) return (int)i;
    WavePlan pl;
    pl.mode = mode; pl.rg = rg; pl.cl = cl;
    int prev_n = 0;
    for (size_t l = 0; l < lp.size() && pl.ok; ++l) {
        WaveLayer M = base[l];
        if (!wave_share_layer(mode, *lp[l], cl ? cl : s->sm_count / ((int)lp.size() * rg), cl > 0, M)) { pl.ok = false; break; }
        M.cta0 = pl.grid;
        pl.grid += (cl ? cl : M.n) * rg;
        M.below = M.first ? 0 : prev_n;
        prev_n = M.n;
        pl.max_ppc = std::max(pl.max_ppc, M.ppc);
        pl.max_cpc = std::max(pl.max_cpc, wv_round(M.cpc, 2));
        pl.max_opc = std::max(pl.max_opc, wv_round(M.opc, 4));
        pl.b_slot = mode == 1 ? WS_SLOT_ROWS * 128 : std::max(pl.b_slot, std::max(M.npad, (M.flags & F_PROJECTION) ? M.npadp : 0) * 128);
        pl.layer.push_back(M);
    }
    s->plan.push_back(pl);
    return (int)s->plan.size() - 1;
}

// The weight images of one layer of a plan.
int wave_fill_images(int mode, const LayerParams &p, const WaveLayer &L, int8_t *iw, int8_t *ir, int8_t *ip)
{
    const bool proj = p.flags & F_PROJECTION;
    if (mode == 0) {
        k_wave_tile_weights<<<2048, 256>>>(p.W, iw, p.G, p.N, p.I, L.n, L.ppc, L.nt, L.ppt, L.npad, L.kb_i);
        k_wave_tile_weights<<<2048, 256>>>(p.R, ir, p.G, p.N, p.O, L.n, L.ppc, L.nt, L.ppt, L.npad, L.kb_h);
        if (proj) k_wave_tile_weights<<<2048, 256>>>(p.Wproj, ip, 0, p.O, p.C, L.n, L.opc, L.ntp, L.opt, L.npadp, L.kb_c);
    } else {
        wave_small_tile_weights(p.W, iw, p.G, p.N, p.I, L.n, L.cpc, L.nt, L.ct, L.ctp, L.kb_i, L.kpg);
        wave_small_tile_weights(p.R, ir, p.G, p.N, p.O, L.n, L.cpc, L.nt, L.ct, L.ctp, L.kb_h, L.kpg);
        if (proj) wave_small_tile_weights(p.Wproj, ip, 0, p.O, p.C, L.n, L.opc, L.ntp, L.opt, L.opp, L.kb_c, L.kpp);
    }
    return cudaGetLastError() == cudaSuccess ? QLSTM_OK : QLSTM_ERR_CUDA;
}

// The description of a call of B rows under a plan; false if the plan cannot take it.
bool wave_describe(const WaveStack *s, const WavePlan &pl, int T, int B, bool tables, WaveCall &k, size_t &smem)
{
    if (!pl.ok) return false;
    memset(&k, 0, offsetof(WaveCall, layer));
    k.T = T; k.B = B; k.n_layers = s->n_layers; k.rg = pl.rg;
    wave_units(B, pl.rg, k.units, k.nu, k.ra);
    const int rows = (B + k.nu - 1) / k.nu;
    k.early = T >= 4 * s->depth;
    k.max_ppc = pl.max_ppc; k.max_cpc = pl.max_cpc; k.max_opc = pl.max_opc; k.b_slot = pl.b_slot;
    k.max_kb_i = s->max_kb_i; k.max_kb_h = s->max_kb_h; k.max_kb_c = s->max_kb_c;
    const size_t room = (size_t)s->max_smem;
    if (pl.mode == 1) {
        if (rows > WV_SMALL_ROWS || !tables || !s->tabs) return false;
        k.max_tab = s->max_tab;
        k.cl = pl.cl;
        k.cl_slots = s->ln ? (s->peep ? 5 : 4) : 0;
        for (const WaveLayer &L : pl.layer)
            if ((2 * L.nt + L.ntp) * k.ra > 512) return false;
        k.nb = 8;
        while (k.nb > 2 && wave_small_smem(k, k.nb, s->peep) > room) --k.nb;
        smem = wave_small_smem(k, k.nb, s->peep);
        return smem <= room;
    }
    k.nrep = rows <= 32 ? 4 : rows <= 64 ? 2 : 1;
    k.nbuf = k.units == 1 ? (s->peep ? 3 : 2) : (s->peep ? 2 : 1);
    const size_t gates = (size_t)k.units * pl.max_ppc * rows * (k.nbuf * 16 + 4);
    auto total = [&](int na, int nb, bool tab, bool in_smem) {
        return wv_layout(na, nb, pl.b_slot, pl.max_ppc, pl.max_opc, tab ? s->max_tab : 0, in_smem ? gates : 0).total;
    };
    if (total(2, 2, false, false) > room) return false;
    k.tab = tables && s->tabs && total(2, 2, true, false) <= room;
    k.gx_s = total(3, 3, k.tab, true) <= room;
    {
        // 100 MB of the 126: the rest goes to activations
        size_t used = k.gx_s ? 0 : gates * (size_t)pl.grid;
        for (const WaveLayer &L : pl.layer) used += L.w_size[0] + L.w_size[1] + L.w_size[2];
        k.w_evict = used > (size_t)100 << 20;
    }
    k.na = 2; k.nb = 2;
    while (k.na < 3 && total(k.na + 1, k.nb, k.tab, k.gx_s) <= room) ++k.na;
    // (two units keep their gate buffers in global memory and read them back through L1, which a third slot of weights would take
    // away: eight 2048-cell layers, 256 rows 110 us per step with three, 106 with two)
    while (k.nb < (k.units == 2 ? 2 : WV_MAX_SLOTS) && total(k.na, k.nb + 1, k.tab, k.gx_s) <= room) ++k.nb;
    while (k.units == 1 && k.na < WV_MAX_SLOTS && total(k.na + 1, k.nb, k.tab, k.gx_s) <= room) ++k.na;
    k.max_tab = k.tab ? s->max_tab : 0;
    smem = total(k.na, k.nb, k.tab, k.gx_s);
    return true;
}

// Clusters of cl blocks of the few-row kernel that fit on the device at once (a block per SM).  Asked only for sizes that some call would take
// (-1: not asked yet): the first question in a process loads the kernel, some milliseconds.
int wave_max_clusters(const WaveStack *s, int cl, int (&known)[17])
{
    if (known[cl] >= 0) return known[cl];
    const void *f = wave_small_kernel(s->G, s->ln, s->peep, true);
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(cl); c.blockDim = dim3(WV_THREADS); c.dynamicSmemBytes = (size_t)s->max_smem;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = (unsigned)cl; a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
    c.attrs = a; c.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, s->max_smem) != cudaSuccess ||
        cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, f, &c) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    return known[cl] = n;
}

// An estimate of a step of the few-row kernel in us: rg groups of `per` blocks, each a cluster or not.  Least squares over 2500 calls of 64
// steps, all cluster sizes and group counts that fit, of 300 random stacks (one to eight layers of 128 to 2048 cells with all variants, 1 to 100
// rows): 5 % standard error without clusters, 9 % with them.  A cluster's exchanges cost less, but its 16 blocks at most have the more weights
// to stream and the more cells to finish, and leave more of the SMs idle.
double wave_step_estimate(const WaveStack *s, const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, int rg, int per, bool cluster, int B)
{
    const double ln = s->ln, peep = s->peep, rows = (B + rg - 1) / rg, ra8 = wv_round((B + rg - 1) / rg, 8) / 8;
    double worst = 0;
    for (size_t l = 0; l < lp.size(); ++l) {
        WaveLayer L = base[l];
        if (!wave_share_layer(1, *lp[l], per, cluster, L)) return 1e9;
        const double proj = (L.flags & F_PROJECTION) ? 1 : 0, kb = 1.0 / 1024 / L.n;       // KB per block: all weights, those of the recurrent product
        const double stream = kb * (L.w_size[0] + L.w_size[1] + L.w_size[2]), rec = kb * L.w_size[1];
        const double ew = rows * L.cpc / 512, pieces = std::ceil(L.nt * ra8 / 4);          // cells, and pieces of gate tiles, per thread and warp
        const double proj_rows = proj * ra8 * std::max(1, L.ntp);
        const double e = cluster ? 1.2 + 0.0073 * stream + 0.0022 * rec + 0.78 * pieces + (0.67 + 0.73 * peep) * ew + 0.065 * rows * L.C / 1024 +
                                       ln * (0.72 + 0.053 * L.n + 0.094 * rows + 1.5 * peep) + proj * (1.7 + 0.03 * L.n) + 0.26 * proj_rows
                                 : 3.3 + 0.0028 * stream + 0.0056 * rec + (0.74 + 0.54 * peep) * ew + 0.059 * 8 * ra8 * L.C / 1024 +
                                       ln * (2.3 + 0.11 * pieces + 0.048 * rows + 2.3 * peep) + proj * 3.3 + 0.22 * proj_rows;
        worst = std::max(worst, e);
    }
    // the weights of all groups pass through L2 in every step
    return worst + (cluster ? 0.082 : 0.11) * std::max(0.0, 1e-6 * rg * s->weights - 60);
}

// Whether calls of B rows go to clusters, and to how many groups of clusters of which size.  `known`: see wave_max_clusters.  Where the
// estimates are close the form without clusters has it (us per call of 64 steps, without clusters and with the best ones: one 2048-cell layer with
// layer norm, peephole and projection, 32 rows 1116 and 1202; four 1120-cell layers with projection, 20 rows 700 and 756; three of 1000 cells with
// layer norm and projection, 37 rows 1011 and 898; one of 880 cells with projection, 15 rows 493 and 387; with the factor below none of 148
// other stacks was slower than without clusters, and the choice 1 % slower in the mean than the best of all, 14 % at most).
bool wave_cluster_plan(const WaveStack *s, const std::vector<const LayerParams *> &lp, const std::vector<WaveLayer> &base, int (&known)[17], int B, int rg_other,
                       int &rg, int &cl)
{
    const int n = (int)lp.size();
    double best = 0.93 * wave_step_estimate(s, lp, base, rg_other, s->sm_count / (n * rg_other), false, B);
    cl = 0;
    // sizes that other calls of the handle take first: another one has to be 3 % ahead of them, for it has weight images of its own
    for (int fresh = 0; fresh < 2; ++fresh) {
        double line = fresh && cl ? 0.97 * best : best;
        for (int size = 8; size <= 16; ++size) {
            bool taken = false;
            for (const WavePlan &pl : s->plan) taken = taken || (pl.used && pl.cl == size);
            if (taken == (fresh == 1)) continue;
            for (int groups = 1; groups <= B && groups * n * size <= s->sm_count; groups *= 2) {
                if ((B + groups - 1) / groups > WV_SMALL_ROWS) continue;
                const double e = wave_step_estimate(s, lp, base, groups, size, true, B);
                if (e >= line || groups * n > wave_max_clusters(s, size, known)) continue;
                best = line = e;
                rg = groups; cl = size;
            }
        }
    }
    return cl > 0;
}

// words of WaveStack::zero that a call of nu units of ra rows uses: abort word, counters, layer-norm totals
size_t wave_zero_words(const WaveStack *s, int nu, int ra)
{
    return WC_WORDS + (size_t)s->n_layers * nu * (WC_PER_UNIT * WC_WORDS + (s->ln ? 2 * ra * 8 * 2 : 0));
}

}  // namespace

// Plans the wavefront kernels for a handle - one stack of n_fwd layers, or two that read the same x, the second one backwards in
// time; *out stays null when the stack does not qualify (layers of different variants,
// a scale with a left shift where none is expected, sums that could leave int32) or device memory does not suffice.
int wave_create(const std::vector<const LayerParams *> &lp, int n_fwd, int max_T, int max_B, int sm_count, ActDomains &dom, void *scratch,
                size_t scratch_bytes, WaveStack **out)
{
    *out = nullptr;
    const int n = (int)lp.size();
    if (n < 1 || n > WV_MAX_LAYERS || sm_count / n < 2) return QLSTM_OK;
    for (const LayerParams *p : lp) {
        if (p->G != lp[0]->G || ((p->flags ^ lp[0]->flags) & (F_LAYERNORM | F_PEEPHOLE))) return QLSTM_OK;
        const bool proj = p->flags & F_PROJECTION, ln = p->flags & F_LAYERNORM, peep = p->flags & F_PEEPHOLE;
        const long long lim = 0x7fffffffll;
        for (int g = 0; g < p->G; ++g) {
            if ((ln && p->eff_ln[g].shift > 0) || (peep && p->eff_c[g].shift > 0)) return QLSTM_OK;
            const int xl = p->eff_x[g].shift > 0 ? p->eff_x[g].shift : 0, hl = p->eff_h[g].shift > 0 ? p->eff_h[g].shift : 0;
            if (xl > 15 || ((p->I * 16256ll + p->max_bx) << xl) > lim) return QLSTM_OK;
            if (hl > 15 || ((p->O * 16256ll + p->max_bh) << hl) > lim) return QLSTM_OK;
        }
        if (p->eff_m.shift > 0 || (proj && p->eff_proj.shift > 0)) return QLSTM_OK;
        if (proj && p->C * 16256ll + p->max_bp > lim) return QLSTM_OK;
    }
    WaveStack *s = new WaveStack();
    s->n_layers = n;
    s->depth = n_fwd;
    s->max_T = max_T;
    s->max_B = max_B < WV_MAX_ROWS ? max_B : WV_MAX_ROWS;
    s->sm_count = sm_count;
    s->G = lp[0]->G;
    s->ln = lp[0]->flags & F_LAYERNORM;
    s->peep = lp[0]->flags & F_PEEPHOLE;
    memset(s->by_rows, -1, sizeof(s->by_rows));
    for (const LayerParams *p : lp) {
        const size_t wp = (p->flags & F_PROJECTION) ? (size_t)p->O * p->C : 0;
        s->ragged = s->ragged || p->I % 16 || p->C % 16 || p->O % 16;
        s->proj = s->proj || wp;
        s->max_C = std::max(s->max_C, p->C);
        s->weights += (size_t)p->N * (p->I + p->O) + wp;
        if (p == lp[0]) s->resident = (size_t)p->N * p->O + wp;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&s->max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // no memory left for a path that a handle can go without is no failure of the handle
    auto fail = [&](int rc) {
        const bool mem = rc == QLSTM_ERR_NOMEM || cudaPeekAtLastError() == cudaErrorMemoryAllocation;
        if (mem) cudaGetLastError();
        wave_destroy(s);
        return mem ? QLSTM_OK : rc;
    };
    s->tabs = true;
    // one table per cell format
    std::vector<int> tab_of(n);
    std::vector<std::vector<uint8_t>> blobs;
    std::vector<ActLineLayout> tab_lays;
    for (int l = 0; l < n; ++l) {
        int same = 0;
        while (same < l && lp[same]->m_bits != lp[l]->m_bits) ++same;
        if (same == l) {
            tab_of[l] = (int)blobs.size();
            blobs.emplace_back();
            tab_lays.emplace_back();
            if (!act_lines_build(dom, lp[l]->m_bits, blobs.back(), &tab_lays.back())) return fail(QLSTM_ERR_CUDA);
            if (blobs.back().empty()) s->tabs = false;
            s->max_tab = std::max(s->max_tab, (int)tab_lays.back().bytes);
        }
        tab_of[l] = tab_of[same];
    }
    long long h_off = 0, c_off = 0;
    std::vector<WaveLayer> base;
    for (int l = 0; l < n; ++l) {
        const LayerParams &p = *lp[l];
        const bool proj = p.flags & F_PROJECTION;
        WaveLayer L;
        memset(&L, 0, sizeof(L));
        L.I = p.I; L.C = p.C; L.O = p.O; L.flags = p.flags; L.m_bits = p.m_bits; L.zp_m = p.zp_m; L.zp_h = p.zp_h;
        L.kb_i = (p.I + 127) / 128; L.kb_h = (p.O + 127) / 128; L.kb_c = (p.C + 127) / 128;
        s->max_kb_i = std::max(s->max_kb_i, L.kb_i);
        s->max_kb_h = std::max(s->max_kb_h, L.kb_h);
        if (proj) s->max_kb_c = std::max(s->max_kb_c, L.kb_c);
        L.bx = p.bx; L.bh = p.bh; L.bln = p.bln; L.bp = p.bp; L.P = p.P; L.L = p.L;
        for (int g = 0; g < p.G; ++g) {
            L.x_left[g] = p.eff_x[g].shift > 0 ? p.eff_x[g].shift : 0;
            L.h_left[g] = p.eff_h[g].shift > 0 ? p.eff_h[g].shift : 0;
            L.f_x[g] = make_fast_scale(p.eff_x[g]); L.f_h[g] = make_fast_scale(p.eff_h[g]);
            L.f_c[g] = make_fast_scale(p.eff_c[g]); L.f_ln[g] = make_fast_scale(p.eff_ln[g]);
        }
        L.f_m = make_fast_scale(p.eff_m); L.f_proj = make_fast_scale(p.eff_proj);
        L.div_c = make_div_magic((uint32_t)p.C);
        {
            // q' L + b stays inside an int32 for |q'| <= room, and |2^10 (2^10 q - mean)| <= 2^36
            const long long room = std::min(65535ll, (0x7fffffffll - p.max_bln) / (p.max_L > 0 ? p.max_L : 1)) - 1;
            L.sigma_min = room < 64 ? 0x7fffffffu : (uint32_t)((1ll << 36) / room + 1);
        }
        L.dir = l >= n_fwd ? 1 : 0;
        L.first = l == 0 || l == n_fwd;
        L.last = l == n_fwd - 1 || l == n - 1;
        if (L.first) h_off = c_off = 0;
        if (L.last) { L.y_off = s->y_stride; s->y_stride += p.O; }
        L.h_off = h_off; L.c_off = c_off;
        h_off += p.O; c_off += p.C;
        L.tab_lay = tab_lays[tab_of[l]];
        base.push_back(L);
    }
    // A plan for every number of rows that a call may have: the few-row form where it can hold them, else the many-row one.  Calls
    // of fewer rows than the handle was made for get the shares that a handle of their own would have (us per call of 100 steps, all
    // calls with the shares of the handle's rows and like this: five 1024-cell CIFG layers made for 64 rows, one row 968 and 641; two
    // 768-cell layers made for 256 rows, two rows 725 and 469, 64 rows 803 and 651).  The form that evaluates the nonlinearities by
    // definition is the many-row one; it has the plans that other calls need.
    WaveCall k;
    size_t smem, rows_alloc = 0, zero_words = 0, g_bytes = 0, c_bytes = 0;
    for (int B = 1; B <= s->max_B; ++B) s->fit_groups[B] = (uint16_t)wave_fit_groups(s, lp, B);
    int clusters[17];
    for (int &v : clusters) v = -1;
    for (int B = s->max_B; B >= 1 && s->tabs; --B) {
        int rg, cl;
        const int other = wave_row_groups(s, 1, lp, B);
        if (!wave_small_fits(s, lp, other, B, s->sm_count) || !wave_cluster_plan(s, lp, base, clusters, B, other, rg, cl)) continue;
        const int i = wave_plan(s, lp, base, 1, rg, cl);
        WavePlan &pl = s->plan[i];
        if (!wave_describe(s, pl, max_T, B, true, k, smem)) continue;
        pl.used = true;
        s->by_rows[1][B] = (int8_t)i;
        rows_alloc = std::max(rows_alloc, (size_t)k.nu * k.ra);
        zero_words = std::max(zero_words, wave_zero_words(s, k.nu, k.ra));
    }
    for (int tab = 1; tab >= 0; --tab)
        for (int B = 1; B <= s->max_B; ++B)
            for (int mode = tab; mode >= 0 && s->by_rows[tab][B] < 0; --mode) {
                const int rg = wave_row_groups(s, mode, lp, B);
                bool made = false;
                for (const WavePlan &pl : s->plan) made = made || (pl.mode == mode && pl.rg == rg && pl.used);
                if (tab == 0 && !made) continue;
                const int i = wave_plan(s, lp, base, mode, rg);
                WavePlan &pl = s->plan[i];
                if (!wave_describe(s, pl, max_T, B, tab, k, smem)) continue;
                pl.used = true;
                s->by_rows[tab][B] = (int8_t)i;
                rows_alloc = std::max(rows_alloc, (size_t)k.nu * k.ra);
                zero_words = std::max(zero_words, wave_zero_words(s, k.nu, k.ra));
                if (mode == 0 && !k.gx_s) {
                    // gate buffers and cell states in global memory, for batches whose buffers do not fit in shared memory
                    const size_t cells = (size_t)pl.grid * k.units * pl.max_ppc * ((B + k.nu - 1) / k.nu);
                    g_bytes = std::max(g_bytes, cells * k.nbuf * sizeof(uint4));
                    c_bytes = std::max(c_bytes, cells * sizeof(uint32_t));
                }
            }
    if (rows_alloc == 0) return fail(QLSTM_OK);
    // (only of the forms that some call takes: setting an attribute loads a kernel, some milliseconds the first time in a process)
    for (const WavePlan &pl : s->plan) {
        if (!pl.used) continue;
        if (pl.cl) continue;                                   // (set by wave_max_clusters)
        const void *f[2] = {wave_small_kernel(s->G, s->ln, s->peep, false), nullptr};
        if (pl.mode == 0) { f[0] = wave_kernel_of<true>(s->G, s->ln, s->peep); f[1] = wave_kernel_of<false>(s->G, s->ln, s->peep); }
        for (const void *kernel : f)
            if (kernel && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, s->max_smem) != cudaSuccess) return fail(QLSTM_ERR_CUDA);
    }
    if (s->tabs) s->res = resident_plan(lp, base, max_T, s->max_B, s->max_smem, s->y_stride);
    // everything in at most two allocations (a handle's creation is mostly allocations): counted first, then filled
    WaveArena keep, work, rwork;                               // (a call takes one path: their activations share memory)
    for (int pass = 0; pass < 2; ++pass) {
        keep.used = work.used = rwork.used = 0;
        std::vector<uint8_t *> tab(blobs.size());
        for (size_t i = 0; i < blobs.size(); ++i) {
            keep.take(tab[i], blobs[i].size());
            if (pass && !blobs[i].empty() && cudaMemcpy(tab[i], blobs[i].data(), blobs[i].size(), cudaMemcpyHostToDevice) != cudaSuccess)
                return fail(QLSTM_ERR_CUDA);
        }
        keep.take(s->zero, zero_words * sizeof(unsigned));
        work.take(s->gbuf, g_bytes);
        work.take(s->cbuf, c_bytes);
        int8_t *prev_img = nullptr;
        for (int l = 0; l < n; ++l) {
            WaveLayer &L = base[l];
            L.tab = tab[tab_of[l]];
            if (L.first) work.take(L.in_img, (size_t)max_T * rows_alloc * L.kb_i * 128);
            else L.in_img = prev_img;
            work.take(L.out_img, ((size_t)max_T + 1) * rows_alloc * L.kb_h * 128);
            if (L.flags & F_PROJECTION) work.take(L.m_img, rows_alloc * L.kb_c * 128);
            prev_img = L.out_img;
            for (WavePlan &pl : s->plan) {
                if (!pl.used) continue;
                WaveLayer &M = pl.layer[l];
                M.in_img = L.in_img; M.out_img = L.out_img; M.m_img = L.m_img; M.tab = L.tab;
                // (plans of one cluster size share their images: the blocks' shares are the same)
                const WavePlan *same = nullptr;
                for (const WavePlan *o = s->plan.data(); o < &pl && !same; ++o)
                    if (pl.cl && o->used && o->cl == pl.cl) same = o;
                if (same) {
                    const WaveLayer &S = same->layer[l];
                    M.img_w = S.img_w; M.img_r = S.img_r; M.img_p = S.img_p;
                    continue;
                }
                int8_t *img[3];
                for (int i = 0; i < 3; ++i) keep.take(img[i], M.w_size[i]);
                M.img_w = img[0]; M.img_r = img[1]; M.img_p = img[2];
                if (!pass) continue;
                const int rc = wave_fill_images(pl.mode, *lp[l], M, img[0], img[1], img[2]);
                if (rc != QLSTM_OK) return fail(rc);
            }
        }
        if (s->res) {
            const int rc = resident_place(s->res, lp, base, keep, rwork, pass);
            if (rc != QLSTM_OK) return fail(rc);
        }
        if (pass) break;
        const size_t activations = std::max(work.used, rwork.used);
        if (cudaMalloc(&s->block[0], keep.used) != cudaSuccess || (activations > scratch_bytes && cudaMalloc(&s->block[1], activations) != cudaSuccess)) {
            if (!s->res) return fail(QLSTM_ERR_NOMEM);
            // without the resident form, then
            cudaGetLastError();
            for (void *&b : s->block) { cudaFree(b); b = nullptr; }
            resident_destroy(s->res);
            s->res = nullptr;
            --pass;
            continue;
        }
        keep.base = (uint8_t *)s->block[0];
        work.base = rwork.base = activations > scratch_bytes ? (uint8_t *)s->block[1] : (uint8_t *)scratch;
    }
    if (cudaDeviceSynchronize() != cudaSuccess) return fail(QLSTM_ERR_CUDA);
    *out = s;
    return QLSTM_OK;
}

static const WavePlan *wave_plan_of(const WaveStack *s, int T, int B, bool tables)
{
    if (!s || B < 1 || B > s->max_B || T < 1 || T > s->max_T || s->by_rows[tables][B] < 0) return nullptr;
    return &s->plan[s->by_rows[tables][B]];
}

bool wave_supported(const WaveStack *s, int T, int B, bool tables) { return wave_plan_of(s, T, B, tables) != nullptr; }

// Calls of one or two rows that are over before a wavefront's fill and launch have paid for themselves, on the whole-stack kernel (us
// per call of that kernel over this one's): two or three steps of narrow stacks without layer norm or projection (one 256-cell layer 16
// and 19, two 21 and 23); with a projection, whose exchange of m costs more here, up to 16 steps (four 256-cell layers, 8 steps: 8 % ahead;
// with layer norm and at most two layers only up to three); one step of up to four rows or two of two rows of a narrow layer (128 cells
// 17 % and 16 %); two steps of stacks whose weights come from memory either way (eight 2048-cell layers without projection 205 and 260).
static bool wave_short_call(const WaveStack *s, int T, int B)
{
    if (T == 1 && B <= 2) return true;
    if (s->n_layers != s->depth || B > 4) return false;
    const int depth = s->depth, cells = depth * s->max_C;
    if (T == 2 && B <= 2 && s->weights > (size_t)200 * 1000000) return true;
    if (depth == 1 && !s->ln && ((T == 1 && s->max_C <= 512) || (T == 2 && B == 2 && s->max_C <= 1024))) return true;
    if (B > 1 || T < depth) return false;                          // (shorter than deep: its layers run one after the other)
    if (s->proj) return T <= (s->ln && depth <= 2 ? 3 : 16) && ((s->max_C <= 512 && cells <= 2048) || (cells <= 1024 && T <= 8));
    return !s->ln && T <= 3 && cells * (T - 1) <= 1024;
}

// Where the wavefront kernels are the faster path (measured, us per call, against the whole-stack kernel or layer after layer):
// one step of one or two rows stays with the whole-stack kernel (eight 2048-cell layers 137 against 151, one 512-cell layer 10
// against 15; two steps 266 against 186), and so do a few other short calls (above); calls of a few steps of many rows, in which a
// wavefront has little to overlap, run
// layer after layer (eight layers, 256 rows: one step 452 against 1057, four 1152 against 1404, sixteen 4050 against 2757; 64
// rows: one step 377 against 451, two 538 against 478; five layers, 256 rows: four steps 324 against 340, sixteen 926 against
// 628; two layers always).  A single layer with layer norm beyond 64 rows, with nothing to overlap, does so too (2048 cells, 128
// rows: 24.6 us per step against 28.2; 64 rows 20.9 against 17.7), and a single one without layer norm and peephole beyond 128 rows
// where the groups that hold them would stream more than 66 MB per step (100 with a projection) and the per-layer kernel keeps its
// weights in shared memory (16 steps, 192 rows: 2048 cells with projection 311 against 365, 1536 cells 222 against 243, 1536 with CIFG
// 218 against 231; under the lines, 1024 cells at 256 rows 191 against 168, 2048 cells with projection at 160 rows, 40 steps 679 against
// 620; 2048 cells without projection, 113 KB per SM, 256 rows 429 against 360).
bool wave_preferred(const WaveStack *s, int T, int B, bool tables)
{
    if (!wave_supported(s, T, B, tables)) return false;
    if (s->ragged) return true;
    if (wave_short_call(s, T, B)) return false;
    if (s->depth == 1 && s->ln && B > 64) return false;
    if (s->n_layers == 1 && !s->ln && !s->peep && B > 128 && s->fit_groups[B] * s->weights > (size_t)(s->proj ? 100 : 66) * 1000000 &&
        s->resident <= (size_t)s->sm_count * 96 * 1024)
        return false;
    return T * 256 > s->depth * (B - 32);
}

bool wave_resident_taken(const WaveStack *s, int T, int B, bool tables)
{
    return s && s->res_mode != 1 && tables && resident_supported(s->res, T, B);
}

int wave_resident_mode(WaveStack *s, int mode)
{
    if (s) s->res_mode = mode;
    return s && s->res ? 1 : 0;
}

int wave_resident_debug_plan(const WaveStack *s, int T, int B, int *out4)
{
    if (!out4) return QLSTM_ERR_ARG;
    if (s) resident_debug_plan(s->res, T, B, out4);
    else out4[0] = out4[1] = out4[2] = out4[3] = 0;
    return QLSTM_OK;
}

int launch_wave_resident(WaveStack *s, const int8_t *x, int T, int B, int8_t *const (&h)[2], int16_t *const (&c)[2], int8_t *y, int *status, int *status2,
                         cudaStream_t st)
{
    return launch_resident(s->res, x, T, B, h, c, y, status, status2, s->dbg_missing, s->dbg_limit_ns ? s->dbg_limit_ns : WV_WAIT_LIMIT_NS, s->res_mode == 2,
                           st);
}

int wave_debug_plan(const WaveStack *s, int T, int B, bool tables, int *out4)
{
    if (!out4) return QLSTM_ERR_ARG;
    const WavePlan *pl = wave_plan_of(s, T, B, tables);
    int units = 0, nu = 0, ra = 0;
    if (pl) wave_units(B, pl->rg, units, nu, ra);
    out4[0] = pl ? pl->mode : -1;
    out4[1] = pl ? pl->rg : 0;
    out4[2] = units;
    out4[3] = wave_preferred(s, T, B, tables) && !wave_resident_taken(s, T, B, tables) ? 1 : 0;
    return QLSTM_OK;
}

int wave_debug_cluster(const WaveStack *s, int T, int B)
{
    const WavePlan *pl = wave_plan_of(s, T, B, true);
    return pl ? pl->cl : 0;
}

void wave_debug_timeout(WaveStack *s, unsigned missing_arrivals, unsigned long long limit_ns)
{
    if (!s) return;
    s->dbg_missing = missing_arrivals;
    s->dbg_limit_ns = missing_arrivals ? limit_ns : 0;
}

int launch_wave(WaveStack *s, const int8_t *x, int T, int B, int8_t *const (&h)[2], int16_t *const (&c)[2], int8_t *y, int *status, int *status2,
                bool tables, cudaStream_t st, int *launches)
{
    if (launches) *launches = 0;
    WaveCall k;
    size_t smem = 0;
    const WavePlan *plan = wave_plan_of(s, T, B, tables);
    if (!plan || !wave_describe(s, *plan, T, B, tables, k, smem)) return QLSTM_ERR_DIM;
    const WavePlan &pl = *plan;
    k.y = y; k.y_stride = s->y_stride;
    k.gbuf = s->gbuf; k.cbuf = s->cbuf;
    k.abort_word = s->zero;
    k.status = status; k.status2 = status2;
    k.limit_ns = s->dbg_limit_ns ? s->dbg_limit_ns : WV_WAIT_LIMIT_NS;
    k.missing = s->dbg_missing;
    unsigned *cnt = s->zero + WC_WORDS;
    long long *totals = (long long *)(cnt + (size_t)s->n_layers * k.nu * WC_PER_UNIT * WC_WORDS);
    for (int l = 0; l < s->n_layers; ++l) {
        WaveLayer &L = k.layer[l];
        L = pl.layer[l];
        L.cnt = cnt + (size_t)l * k.nu * WC_PER_UNIT * WC_WORDS;
        L.totals = s->ln ? totals + (size_t)l * 2 * k.nu * k.ra * 8 : nullptr;
        L.h = h[L.dir] + L.h_off * B;
        L.c = c[L.dir] + L.c_off * B;
    }
    const size_t items = (size_t)T * B * ((pl.layer[0].I + 15) / 16);
    const int blocks = (int)std::min<size_t>(1184, (items + 255) / 256 + 32);
    k_wave_prepare<<<blocks, 256, 0, st>>>(k, x, s->zero, wave_zero_words(s, k.nu, k.ra));
    if (cudaGetLastError() != cudaSuccess) return QLSTM_ERR_CUDA;
    void *args[] = {(void *)&k};
    const void *f = pl.mode == 1 ? wave_small_kernel(s->G, s->ln, s->peep, pl.cl > 0)
                              : (k.tab ? wave_kernel_of<true>(s->G, s->ln, s->peep) : wave_kernel_of<false>(s->G, s->ln, s->peep));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.grid); cfg.blockDim = dim3(WV_THREADS); cfg.stream = st;
    cfg.dynamicSmemBytes = s->res_mode == 2 && pl.cl ? WV_REFUSED_SMEM : smem;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)pl.cl; attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = pl.cl ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, f, args);
    if (e != cudaSuccess) return wv_refused(e);
    if (launches) *launches = 2;
    return QLSTM_OK;
}

}  // namespace ql
