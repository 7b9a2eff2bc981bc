// What the wavefront kernels share: the description of a call, bounded waits, the exchanges between the blocks of a
// group, and the fixed-point pieces of a step.  wave_sm100.cu has the overview.
#pragma once

#include "../../include/qlstm.h"
#include "act_table.cuh"
#include "fast_kernels.h"
#include "sm100_ptx.cuh"
#include "wave_math.cuh"

namespace ql {

constexpr int WV_THREADS = 640;
constexpr int WV_EPI_WARP0 = 4;
constexpr int WV_EPI = WV_THREADS - 32 * WV_EPI_WARP0;         // 512 epilogue threads
constexpr int WV_MAX_LAYERS = 16;
constexpr int WS_SLOT_ROWS = 256;              // wave_small_sm100.cu: 128-byte rows of a weight slot
constexpr unsigned long long WV_WAIT_LIMIT_NS = 2000000000ull;

// counters of one (layer, unit), each on a line of its own
enum { WC_STATS = 0, WC_STATS2 = 1, WC_M = 2, WC_H = 3, WC_PER_UNIT = 4, WC_WORDS = 32 };

struct WaveLayer {
    int I, C, O;
    uint32_t flags;
    int m_bits, zp_m, zp_h;
    int cta0, n;                   // first block of row group 0, blocks per (layer, row group)
    int ppc;                       // cell pairs per block (wave_sm100.cu)
    int nt, ppt, npad;             // gate tiles: count, pairs per tile, MMA columns
    int opc, ntp, opt, npadp;      // outputs per block; projection tiles: count, outputs per tile, MMA columns
    int cpc, ct, ctp, kpg;         // wave_small_sm100.cu: cells per block; cells of a tile, rounded up; k-blocks per chunk
    int opp, kpp;                  // ... outputs of a projection tile rounded up to 8, k-blocks per ring slot
    int kb_i, kb_h, kb_c;          // 128-byte k-blocks of the three products
    size_t w_size[3];              // bytes of the three images
    const int8_t *img_w, *img_r, *img_p;       // weights in the order and image in which the blocks stream them
    const int32_t *bx, *bh, *bln, *bp;
    const int16_t *P, *L;
    int x_left[4], h_left[4];      // left shift before the rescale of the input / recurrent term (0 for scales below 1)
    FastScale f_x[4], f_h[4], f_c[4], f_ln[4], f_m, f_proj;      // by gate slot
    DivMagic div_c;
    uint32_t sigma_min;            // layer norm: from this sigma on every quotient is below 2^16 and q' L + b inside an int32
    int8_t *in_img;                // [T][units][kb_i][ra][128] input activations
    int8_t *out_img;               // [T + 1][units][kb_h][ra][128]: slot t + 1 holds h^t
    int8_t *m_img;                 // [units][kb_c][ra][128]
    long long *totals;             // [2][units][ra][4][2] layer-norm sums of the group
    unsigned *cnt;                 // [units][WC_PER_UNIT][WC_WORDS]
    int below;                     // blocks of the layer below, 0: none
    long long h_off, c_off;        // of this layer in its stack's state, in units of one batch row
    int8_t *h; int16_t *c;         // the caller's state of this layer (set per call)
    int first, last;               // of its stack
    int dir;                       // 1: the stack reads x from the last step backwards
    int y_off;                     // last layer: its columns within a row of y
    const uint8_t *tab;
    ActLineLayout tab_lay;
};

struct WaveCall {
    int T, B, n_layers, rg, units; // row groups; units of a row group
    int nu, ra;                    // units in all, rows of an activation image's k-block
    int nrep;                      // copies of a unit's rows in the 128 lanes
    int early;                     // one unit: X(t + 1) before B(t) and P(t)
    int tab;                       // memoised nonlinearities (resident in shared memory)
    int na, nb, b_slot;            // ring depths, bytes of a weight slot
    int max_cpc, max_kb_i, max_kb_h, max_kb_c;
    int gx_s;                      // gate buffers in shared memory
    int w_evict;                   // weights with an evict-first hint
    int nbuf;                      // gate buffers per unit: [gate sums | X ...]
    int max_ppc, max_opc, max_tab;
    int cl, cl_slots;              // wave_small_sm100.cu: blocks of a cluster (0: exchanges through global memory), its slots of layer-norm sums
    int8_t *y;
    int y_stride;                  // bytes of a row of y
    uint4 *gbuf;                   // [blocks][units][nbuf][max_ppc][max rows] gate buffers in global memory
    uint32_t *cbuf;                // [blocks][units][max_ppc][max rows] cell states
    unsigned *abort_word;
    int *status, *status2;         // status2: another word to clear, or null
    unsigned long long limit_ns;
    unsigned missing;
    WaveLayer layer[WV_MAX_LAYERS];
};

// the row of y that a last layer's step t and batch row b go to
__device__ __forceinline__ int8_t *wv_y_row(const WaveCall &k, const WaveLayer &L, int t, int b)
{
    return k.y + ((size_t)(L.dir ? k.T - 1 - t : t) * k.B + b) * k.y_stride + L.y_off;
}

// ---- waits ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ bool wv_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    // each attempt parks the thread for up to 20 us; 100 000 attempts bound the wait to about 2 s
    for (uint32_t i = 0; i < 100000u; ++i) {
        if (ptx::mbar_try_wait_parked(bar, parity, 20000u)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// The end of a copy or an MMA that has been issued, for a block that leaves early: none may be in flight then.  Bounded like the
// other waits.  (In the normal course all have been waited for.)
__device__ __forceinline__ void wv_drain(uint64_t *bar, uint32_t parity)
{
    for (uint32_t i = 0; i < 100000u; ++i)
        if (ptx::mbar_try_wait_parked(bar, parity, 20000u)) return;
}
// the copies of a ring whose next one would go to `slot` with parity `phase` (before a slot's first copy: passes at once)
__device__ __forceinline__ void wv_drain_ring(uint64_t *full, int n, int slot, uint32_t phase)
{
    for (int i = 0; i < n; ++i) wv_drain(&full[i], i < slot ? phase : phase ^ 1u);
}
__device__ __forceinline__ unsigned wv_ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long wv_timer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t)::"memory");
    return t;
}
__device__ __forceinline__ void wv_fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// one thread: until *cnt has reached target (bounded); false once an abort is seen
__device__ __forceinline__ bool wv_wait_count(const WaveCall &k, const unsigned *cnt, unsigned target, volatile int *abort_flag)
{
    target += k.missing;
    if (wv_ld_acquire(cnt) >= target) return *abort_flag == 0;
    const unsigned long long t0 = wv_timer();
    unsigned spins = 0;
    while (wv_ld_acquire(cnt) < target) {
        if ((++spins & 31u) == 0u) {
            if (*abort_flag) return false;
            if (wv_ld_acquire(k.abort_word) != 0u) { *abort_flag = 1; return false; }
            if (wv_timer() - t0 > k.limit_ns) { atomicExch(k.abort_word, 1u); *abort_flag = 1; return false; }
        }
    }
    return *abort_flag == 0;
}
// The same for a warp that stays together: one lane looks, all decide.  (A single thread that polls while its warp waits at the
// next barrier leaves the warp split, and everything after it then runs twice: 2 us per step.)
__device__ __forceinline__ void wv_wait_count_warp(const WaveCall &k, const unsigned *cnt, unsigned target, volatile int *abort_flag)
{
    const bool look = (threadIdx.x & 31) == 0;
    target += k.missing;
    const unsigned long long t0 = wv_timer();
    for (unsigned spins = 1;; ++spins) {
        unsigned v = 0;
        if (look) v = wv_ld_acquire(cnt);
        v = __shfl_sync(0xffffffffu, v, 0);
        if (v >= target) return;
        if ((spins & 31u) == 0u) {
            unsigned stop = 0;
            if (look) {
                if (*abort_flag) stop = 1;
                else if (wv_ld_acquire(k.abort_word) != 0u) { *abort_flag = 1; stop = 1; }
                else if (wv_timer() - t0 > k.limit_ns) { atomicExch(k.abort_word, 1u); *abort_flag = 1; stop = 1; }
            }
            if (__shfl_sync(0xffffffffu, stop, 0)) return;
        }
    }
}
// For a whole warp, a lane per block: until each of the n <= 32 blocks that write to a line of words has reached target.  For clusters, whose
// blocks exchange what their own recurrence needs through shared memory and do not wait for one another here: a sum over them would not say
// that all have.  Call: WaveCall or the like.
template <class Call>
__device__ __forceinline__ bool wv_wait_blocks(const Call &k, const unsigned *line, int n, unsigned target, volatile int *abort_flag)
{
    const int lane = threadIdx.x & 31;
    target += k.missing;
    const unsigned long long t0 = wv_timer();
    for (unsigned spins = 1;; ++spins) {
        const bool there = lane >= n || wv_ld_acquire(line + lane) >= target;
        if (__all_sync(0xffffffffu, there)) break;
        unsigned stop = 0;
        if (lane == 0 && (spins & 31u) == 0u) {
            if (*abort_flag) stop = 1;
            else if (wv_ld_acquire(k.abort_word) != 0u) { *abort_flag = 1; stop = 1; }
            else if (wv_timer() - t0 > k.limit_ns) { atomicExch(k.abort_word, 1u); *abort_flag = 1; stop = 1; }
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) return false;
    }
    __syncwarp();                              // (what the lanes acquired, to the lane that copies)
    return true;
}
__device__ __forceinline__ void wv_epi_sync() { asm volatile("barrier.sync 1, 512;" ::: "memory"); }

// all MMAs that this warp has issued, through a barrier of its own
__device__ __forceinline__ void wv_drain_mmas(uint64_t *bar)
{
    if (ptx::elect_one()) ptx::mma_commit(bar);
    __syncwarp();
    wv_drain(bar, 0);
}

// The same for a whole warp that stays together.
__device__ __forceinline__ bool wv_wait_warp(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    return __all_sync(0xffffffffu, wv_wait(bar, parity, abort_flag));
}

// The four MMAs of one k-block (128 bytes of K; both operands are zero-padded to that), by an elected lane of a warp that
// stays together.  The instruction wants its operands in uniform registers: in a rolled loop under a divergent branch an MMA
// took 200 cycles of issue, written like this 50 to 75 (N <= 128; the tensor core itself needs 50 at N <= 64 and 127 at N = 256).
__device__ __forceinline__ void wv_mma_kblock(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool fresh)
{
    ptx::mma_i8_ss(d, a, b, idesc, !fresh);
    ptx::mma_i8_ss(d, a + 2, b + 2, idesc, true);
    ptx::mma_i8_ss(d, a + 4, b + 4, idesc, true);
    ptx::mma_i8_ss(d, a + 6, b + 6, idesc, true);
}
__device__ __forceinline__ void wv_commit(uint64_t *bar)
{
    if (ptx::elect_one()) ptx::mma_commit(bar);
    __syncwarp();
}

// Where a stack's weights and the buffers between its phases together exceed L2 (WaveCall::w_evict), the weights pass through with
// an evict-first hint: of the two it is the buffers, read again within a step, that should stay (eight 2048-cell layers: 64 rows
// 46 -> 43 us per step, 256 rows 105 -> 100).  Weights that fit must not have it (five 1024-cell layers, 64 rows: 12.0 -> 16.3).
__device__ __forceinline__ uint64_t wv_weights_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void wv_load_weights(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t policy)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(ptx::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(ptx::smem_u32(bar)), "l"(policy)
                 : "memory");
}

// ---- thread-block clusters: stores into the shared memory of peers, counted in bytes on an mbarrier there ----------------------
__device__ __forceinline__ uint32_t wv_peer(uint32_t addr, int rank)
{
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
    return d;
}
__device__ __forceinline__ void wv_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void wv_send8(uint32_t dst, uint2 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void wv_send16(uint32_t dst, uint4 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool wv_try_cluster(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(ok)
        : "r"(ptx::smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// The rest of a wait (whole warp) whose first attempt has not seen its phase complete: until it does, another block has given up or
// the limit is over.
static __device__ __noinline__ bool wv_wait_cluster_slow(uint64_t *bar, uint32_t parity, unsigned *abort_word, unsigned long long limit_ns, volatile int *abort_flag)
{
    const unsigned long long t0 = wv_timer();
    for (unsigned n = 1;; ++n) {
        if (__all_sync(0xffffffffu, wv_try_cluster(bar, parity))) return true;
        unsigned stop = 0;
        if ((threadIdx.x & 31) == 0) {
            if (*abort_flag) stop = 1;
            else if ((n & 7u) == 0u) {
                if (wv_ld_acquire(abort_word) != 0u) { *abort_flag = 1; stop = 1; }
                else if (wv_timer() - t0 > limit_ns) { atomicExch(abort_word, 1u); *abort_flag = 1; stop = 1; }
            }
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) return false;
    }
}
// whole warp; what peers stored and counted on `bar` (wv_send8, wv_send16) has arrived; false once an abort is seen
__device__ __forceinline__ bool wv_wait_cluster(uint64_t *bar, uint32_t parity, unsigned *abort_word, unsigned long long limit_ns, volatile int *abort_flag)
{
    if (__all_sync(0xffffffffu, wv_try_cluster(bar, parity))) return true;
    return wv_wait_cluster_slow(bar, parity, abort_word, limit_ns, abort_flag);
}

// ---- fixed-point pieces ----------------------------------------------------------------------------------------------
__device__ __forceinline__ int32_t wv_lo(uint32_t w) { return (int32_t)(w << 16) >> 16; }
__device__ __forceinline__ int32_t wv_hi(uint32_t w) { return (int32_t)w >> 16; }

// byte offset of element (row, col) in a unit's activation image (see tile_off in recurrent_sm100.cu; k-blocks of ra rows)
__device__ __forceinline__ uint32_t wv_img_off(int row, int col, int ra)
{
    return (uint32_t)((col >> 7) * (ra * 128) + (row << 7) + (((((col >> 4) & 7) ^ (row & 7)) << 4) | (col & 15)));
}

// ---- layer norm and nonlinearities (wave_math.cuh) --------------------------------------------------------------------------------
// sat32(q' L + b) where q' and the sum are known to be in range
__device__ __forceinline__ int32_t wv_ln_fast(int32_t q, int32_t m_hi, int32_t m_lo, int32_t mean, int32_t Lw, int32_t b)
{
    return wv_ln_quotient(q, m_hi, m_lo, mean) * Lw + b;
}

// the same for any row, by division, out of line
static __device__ __noinline__ int32_t wv_ln_slow(int32_t q, WvLnRow row, int32_t Lw, int32_t b)
{
    const int32_t d = 1024 * q - row.mean;
    const uint32_t ad = (uint32_t)(d < 0 ? -d : d), sg = row.sigma & ~WV_LN_SLOW;
    const uint64_t quo = sg == 0u ? 0u : ((uint64_t)ad * 1024u + (sg >> 1)) / sg;
    const int64_t qp = d < 0 ? -(int64_t)quo : (int64_t)quo;
    return sat32_halves(qp * (int64_t)Lw + (int64_t)b);
}

template <bool TAB>
__device__ __forceinline__ int32_t wv_sigmoid(const ActLines &at, int32_t x)
{
    if constexpr (TAB) return line_sigmoid(at, x);
    else return sigmoid_q_fast(x, 3);
}
template <bool TAB>
__device__ __forceinline__ int32_t wv_tanh(const ActLines &at, int32_t x)
{
    if constexpr (TAB) return line_tanh_gate(at, x);
    else return tanh_q_fast(x, 3);
}
template <bool TAB>
__device__ __forceinline__ int32_t wv_hidden(const WaveLayer &L, const ActLines &at, int32_t o, int32_t c_new)
{
    int32_t tc;
    if constexpr (TAB) tc = line_tanh_cell(at, c_new);
    else tc = tanh_q_fast(c_new, L.m_bits);
    return sat8(fast_rescale(o * tc, L.f_m) + L.zp_m);                     // Section 3.2.7
}

// The epilogue threads meet at named barriers, so they have to agree on where to leave after an abort: one thread looks at
// the abort flag before the barrier of a meeting point and writes the point's number down; everybody leaves at the first
// point that is not before it.
struct WvPoint { volatile int *abort_flag, *exit_at; int n; };

__device__ __forceinline__ bool wv_point(WvPoint &pt, int tid)
{
    if (tid == 0 && *pt.abort_flag) { if (*pt.exit_at > pt.n) *pt.exit_at = pt.n; }
    wv_epi_sync();
    const bool stay = *pt.exit_at > pt.n;
    ++pt.n;
    return stay;
}
// all epilogue threads: publish their writes and add one arrival; false: leave
__device__ __forceinline__ bool wv_publish(unsigned *cnt, bool operands, WvPoint &pt, int tid)
{
    if (operands) wv_fence_async_global();
    const bool stay = wv_point(pt, tid);
    if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
    return stay;
}
// all epilogue threads: wait for the group; false: leave
__device__ __forceinline__ bool wv_meet(const WaveCall &k, const unsigned *cnt, unsigned target, WvPoint &pt, int tid)
{
    if (tid < 32) wv_wait_count_warp(k, cnt, target, pt.abort_flag);
    return wv_point(pt, tid);
}

__device__ __forceinline__ uint4 wv_load16(const int8_t *src, int valid)      // up to 16 bytes from any address, the rest zero
{
    if (valid >= 16 && ((uintptr_t)src & 15) == 0) return *reinterpret_cast<const uint4 *>(src);
    uint32_t w[4] = {0, 0, 0, 0};
    for (int j = 0; j < 16 && j < valid; ++j) w[j >> 2] |= (uint32_t)(uint8_t)src[j] << (8 * (j & 3));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// A launch that the runtime has refused: QLSTM_ERR_LAUNCH where a smaller or another one may still go through.
inline int wv_refused(cudaError_t e)
{
    cudaGetLastError();
    switch (e) {
        case cudaErrorCooperativeLaunchTooLarge:
        case cudaErrorLaunchOutOfResources:
        case cudaErrorInvalidClusterSize:
        case cudaErrorInvalidConfiguration:
        case cudaErrorInvalidValue:
        case cudaErrorNotSupported:
            return QLSTM_ERR_LAUNCH;
        default:
            return QLSTM_ERR_CUDA;
    }
}
constexpr size_t WV_REFUSED_SMEM = (size_t)1 << 20;            // more shared memory than a block can have (qlstm_debug_resident, mode 2)

__host__ __device__ inline size_t wv_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Memory handed out front to back; without a base it is only counted.  Pieces start 64 KB apart: packed at 256 bytes, what a step's
// exchanges touch lay closer together and took longer (us per call of 100 steps, median of eight handles: four 1024-cell layers with
// layer norm and projection, 16 rows 1345 and 1300; three of 1000 cells, 37 rows 1568 and 1545).
struct WaveArena {
    uint8_t *base = nullptr;
    size_t used = 0;
    template <class T>
    void take(T *&p, size_t bytes)
    {
        p = base ? (T *)(base + used) : nullptr;
        used += wv_up(bytes, 65536);
    }
};

// wave_small_sm100.cu
const void *wave_small_kernel(int G, bool ln, bool peep, bool cluster);
size_t wave_small_smem(const WaveCall &k, int ns, bool peep);
void wave_small_tile_weights(const int8_t *src, int8_t *dst, int G, int rows, int K, int n, int per_rank, int nt, int per_tile, int padded, int nkb, int kps);

}  // namespace ql
