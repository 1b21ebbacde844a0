// Conv contractions on sm_103a that take each part of their source image once:
// forward and dS by rows (tcgen05, bf16 operands, fp32 accumulation).
//
// A work item is a run of output rows of one image, NT tiles of output
// positions wide (ppt = 128 / Mp positions per 128-row MMA tile) and 64 channels
// deep: the forward of 64 -> 64 layers at stride 1 (one tile), dS of layers with
// 64 input channels (any number of output channels, strides 1 and 2). The item
// walks the source rows that its output rows read; the box of one source row
// (positions x grid steps x 64 channels, bf16, in shared memory) feeds every
// filter row and column that reads it, so up to k output rows are in flight,
// each in its own TMEM accumulator. The one-row-at-a-time kernels load a box per filter
// row and keep two in flight, 12 to 24 MMAs per load of about 1.4 us; here a
// box serves 36 to 72 MMAs. What bounds this kernel then: dS at 64 channels
// runs at 53 clocks per N = 64 MMA, of which reading the operands from shared
// memory takes 48 (64 -> 64 at 28 x 28, B = 256, M = 64: 1.35 -> 0.68 ms); the
// forward is bound by the scan's instructions (issue slots 68% busy, the tensor
// pipe 27%; the same layer: 2.38 -> 1.66 ms with the binning).
//
//   forward  the box holds the binned input and is generated on chip from 8
//            bytes per input spike (two nonzeros of Mp; generator warps erase
//            the last ones and write the new), so no binned input is written
//            to memory; the epilogue runs the scan/solve/select;
//   dS       the box holds dw^ rows, loaded by TMA; the epilogue takes the
//            input-time gradient.
//
// Per output element the products are added in the order of the
// one-row-at-a-time kernels: filter row, then (channel block, filter column)
// or (filter column, channel block) as those take them for the same shape, so
// both give the same w^.
//
// dW of 3x3 layers at stride 1 (k_conv_dw_cols) takes each column of the binned
// input once in the same spirit.
//
// Every mbarrier wait is bounded; an expired wait sets this unit's status
// word, the role stops, and the CTA still frees its TMEM.
#include "dstd_internal.cuh"
#include "dstd_tc_ptx.cuh"

#include <cuda.h>
#include <mutex>

namespace dstd {

__device__ unsigned int g_status_rows = 0;

cudaError_t conv_rows_status_read(unsigned int *out, int clear) {
    cudaError_t e = cudaMemcpyFromSymbol(out, g_status_rows, sizeof(unsigned int));
    if (e != cudaSuccess || !clear) return e;
    unsigned int z = 0;
    return cudaMemcpyToSymbol(g_status_rows, &z, sizeof(z));
}

namespace {

__device__ __forceinline__ void rows_set_status(unsigned int code) { atomicOr(&g_status_rows, code); }

constexpr int MAX_K = 7;       // filter rows and columns
constexpr int MAX_NSTA = 4;    // stages of source boxes
constexpr int MAX_NSTB = 8;    // stages of filter slices
constexpr int GEN_WARPS = 4;   // forward: generator warps
constexpr int MMA_WARPS = 4;   // issuing warps: output row n by warp n mod 4
constexpr int GEN_SLOTS = 5;   // (position, channel) slots of a generator thread per box, at most (7x7, 32 grid steps)
constexpr int ROWS_BN = 64;    // output channels of a tile
constexpr int EPI_LDF = 36;    // forward epilogue: floats per neuron row of 32 grid steps (read as float4)
constexpr int EPI_LDG = 33;    // dS epilogue: floats per grid-step row of 32 channels
constexpr int SILENT = -128;   // grid step of a record, and kept step of a slot, without a spike

struct RowsPlan {
    int n_items, n_xt, n_col, n_strip, R;  // items; position tiles, dS: column tiles (of 64 channels), strips of R output rows
    int gh, gw, sh, sw;                    // output and source grids
    int s, k, pad, ncb, cb_inner;          // forward: s = 1, ncb = 1
    int Mp, ppt;
    int nsta, nstb, npos;                  // stages; positions of a box
    int kwg;                               // filter columns per streamed stage (k or 1)
    int box_bytes, stage_bytes, res_bytes; // res_bytes > 0: all filter slices stay resident
    int nset;                              // epilogue warps / 4
    int xs_mul, xs_add;                    // first source position of tile xt: xt xs_mul + xs_add
    int off_b, off_epi, off_state, off_kept, off_bar, smem;  // shared-memory layout (from a 1 KB boundary), and its size
    int aoff[2][MAX_K];                    // offset (in 16 bytes) in the box of tile tau's first position under filter column kw, or -1
    int kfirst[2];                         // tile tau's first filter column
};

struct RowsArgs {
    const uint2 *rec;   // forward: the source's records (k_bin_rec), C_t channels
    const float *t_in;  // dS: the layer input's spike times, C_t channels
    int C_t;
    float *t_out;       // forward
    int *q_out;
    float *s_out, *vdot_out;
    const float *rowsum;
    float *penalty;
    float *g_t_in;      // dS
    LifConst c;
};

__host__ __device__ constexpr uint32_t idesc_kk(int N) {  // M = 128, both operands K-major bf16
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void rows_sts_u16(uint32_t addr, uint16_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}

// byte offset of element (row r, column c) of a K-major tile of 128-byte rows
// in the 128-byte swizzle
__device__ __forceinline__ uint32_t rows_sw128(int r, int c) {
    return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((((c >> 3) ^ (r & 7)) & 7) << 4) + (c & 7) * 2);
}

// One work item and the source rows it walks: forward upwards, dS downwards
// (the order in which an output row's filter rows come up).
template <bool FWD>
struct Item {
    int b, xt, ct, ya, yb, sr, sr_end;  // (ct: dS only) sr steps by +-1 up to and including sr_end
    __device__ __forceinline__ void decode(const RowsPlan &p, int it) {
        if (!FWD) {  // rows_pick takes one column tile; but dS without the index came out 2 to 3% slower
            ct = it % p.n_col;
            it /= p.n_col;
        }
        xt = it % p.n_xt;
        it /= p.n_xt;
        const int strip = it % p.n_strip;
        b = it / p.n_strip;
        ya = strip * p.R;
        yb = ya + p.R < p.gh ? ya + p.R : p.gh;
        if (FWD) {
            sr = ya - p.pad;
            if (sr < 0) sr = 0;
            sr_end = yb - 1 - p.pad + p.k - 1;
            if (sr_end > p.sh - 1) sr_end = p.sh - 1;
        } else {
            sr = (yb - 1 + p.pad) >> (p.s - 1);  // strides are 1 or 2
            if (sr > p.sh - 1) sr = p.sh - 1;
            const int lo = ya + p.pad - (p.k - 1);
            sr_end = lo <= 0 ? 0 : (lo + p.s - 1) >> (p.s - 1);
        }
    }
    __device__ __forceinline__ int rows() const { return yb - ya; }
    __device__ __forceinline__ bool done(int r) const { return FWD ? r > sr_end : r < sr_end; }
    // output row that source row r reaches through filter row kh, or -1
    __device__ __forceinline__ int out_row(const RowsPlan &p, int r, int kh) const {
        const int y = FWD ? r + p.pad - kh : r * p.s - p.pad + kh;
        return y >= ya && y < yb ? y : -1;
    }
    __device__ __forceinline__ int seq(int y) const { return FWD ? y - ya : yb - 1 - y; }
    // whether source row r is the first / the last that output row y reads
    __device__ __forceinline__ bool first_of(const RowsPlan &p, int r, int y) const {
        if (FWD) {
            const int f = y - p.pad;
            return r == (f < 0 ? 0 : f);
        }
        const int f = (y + p.pad) >> (p.s - 1);
        return r == (f > p.sh - 1 ? p.sh - 1 : f);
    }
    __device__ __forceinline__ bool last_of(const RowsPlan &p, int r, int y) const {
        if (FWD) {
            const int l = y - p.pad + p.k - 1;
            return r == (l > p.sh - 1 ? p.sh - 1 : l);
        }
        const int l = y + p.pad - (p.k - 1);
        return r == (l <= 0 ? 0 : (l + p.s - 1) >> (p.s - 1));
    }
};

// What the MMA warp does with source row r under filter row kh, in 8 bits:
// whether an output row of the item reads it, whether it starts or completes
// that row, its accumulator (bits 4-6) and the phase of the accumulator's
// empty barrier (bit 7). n0: output rows of the items before.
constexpr uint32_t ROW_ON = 1, ROW_FIRST = 2, ROW_LAST = 4;
template <int NA, bool FWD>
__device__ __forceinline__ uint32_t row_plan(const Item<FWD> &w, const RowsPlan &p, int r, int kh, uint32_t n0) {
    const int y = w.out_row(p, r, kh);
    if (y < 0) return 0;
    const uint32_t q = n0 + (uint32_t)w.seq(y);
    return ROW_ON | (w.first_of(p, r, y) ? ROW_FIRST : 0u) | (w.last_of(p, r, y) ? ROW_LAST : 0u) |
           ((q & (uint32_t)(NA - 1)) << 4) | ((((q / NA) & 1u) ^ 1u) << 7);
}

// four bins in the bare recurrence: rounding as the group took it in the pass
// over the bins (fused or not, see scan_walk)
__device__ __forceinline__ void walk_group(const LifConst &c, const float *x, bool fused, float &v, float &I) {
    float i0 = __fadd_rn(I, x[0]);
    v = walk_v(c, v, i0);
#pragma unroll
    for (int u = 1; u < 4; ++u) {
        i0 = fused ? fmaf(c.rI, i0, x[u]) : __fadd_rn(__fmul_rn(c.rI, i0), x[u]);
        v = walk_v(c, v, i0);
    }
    I = __fmul_rn(c.rI, i0);
}

// scan_walk over the 32 bins m0 .. m0+31 of one neuron, whose w^ values sit in
// row[0 .. 32) (shared memory, 16-byte aligned, zero past mend), starting from
// the state (v, I) at T_m0: the same results, in a loop that is not unrolled.
// On a spike, fills st (bin, state at its start, bracket end) and returns true;
// otherwise leaves (v, I) at the end of the block.
//
// A pass over the bins, four at a time, flags those that may hold the spike
// (v^ at v_th at the end, or an interior maximum, dv^/ds > 0 at the start and
// < 0 at the end, that may reach v_th); the flagged bins are then walked to
// from the state kept at the start of the first flagged eight and tested
// exactly, in order. Cheap bounds keep the flags rare:
//   - a group of four whose potential stays below v_th by max(v, 0) + Kmax4
//     (max(I, 0) + the positive inputs) in every lane takes the bare
//     recurrence;
//   - else flags are looked at only if max(v, 0) + Kmax max(I0, 0) over the
//     group's bins comes near v_th in a lane that is still looking. A lane
//     stops looking once v^ is clearly above v_th at the end of a group;
//   - e^{av s} dv^/ds falls along a bin, so v^ climbs from v at most at the
//     rate d0 and comes down to ve at most at the rate -dE e^{av dt}: if the
//     times that takes to v_th (less a margin far above the rounding) and
//     back exceed dt, the maximum stays below and the bin is not flagged.
// Beside the kernel's other roles the unrolled walk overran the instruction
// cache (64 -> 64 at 28 x 28, B = 256, M = 64: 3.2 ms against 2.2 ms); where it
// runs alone, in the dense scan, unrolled is the faster one (16384 wide, M =
// 128: 295 against 320 us).
__device__ __forceinline__ bool walk_rolled(unsigned lanes, const LifConst &c, const float *row, int m0, int mend,
                                            float &v, float &I, ScanState &st) {
    float cv = v, cI = I;             // state at the start of the current eight bins
    float kv = v, kI = I;             // and of the first flagged eight, kb
    int kb = -1;
    uint32_t mask = 0u, fused = 0u;   // flagged bins; groups that took the bare recurrence
    bool looking = true;
    const float vlow = c.vth * 0.99999f, vhigh = c.vth * 1.00001f;
#pragma unroll 1
    for (int g = 0; g < 32; g += 4) {
        if ((g & 7) == 0) {
            cv = v;
            cI = I;
        }
        float xs[4];
        const float4 x = *reinterpret_cast<const float4 *>(row + g);
        xs[0] = x.x; xs[1] = x.y; xs[2] = x.z; xs[3] = x.w;
        const float ipos = fmaxf(I, 0.0f) + fmaxf(xs[0], 0.0f) + fmaxf(xs[1], 0.0f) + fmaxf(xs[2], 0.0f) +
                           fmaxf(xs[3], 0.0f);
        const bool quiet = fmaf(ipos, c.Kmax4, fmaxf(v, 0.0f)) < vlow;
        if (__all_sync(lanes, quiet)) {
            walk_fused<4>(c, xs, v, I);
            fused |= 1u << (g >> 2);
        } else {
            float vs[5], I0[4], In[4];
            vs[0] = v;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                I0[u] = __fadd_rn(u == 0 ? I : In[u > 0 ? u - 1 : 0], xs[u]);
                vs[u + 1] = walk_v(c, vs[u], I0[u]);
                In[u] = __fmul_rn(c.rI, I0[u]);
            }
            v = vs[4];
            I = In[3];
            const float vm = fmaxf(fmaxf(fmaxf(vs[0], vs[1]), fmaxf(vs[2], vs[3])), 0.0f);
            const float Im = fmaxf(fmaxf(fmaxf(I0[0], I0[1]), fmaxf(I0[2], I0[3])), 0.0f);
            looking = looking & !(mask != 0u && vs[0] >= vhigh);
            const bool near = looking & !quiet & (fmaf(Im, c.Kmax, vm) >= vlow);
            if (__any_sync(lanes, near)) {
                uint32_t nib = 0u;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float d0 = fmaf(-c.av, vs[u], I0[u]), dE = fmaf(-c.av, vs[u + 1], In[u]);
                    const float below = fmaf(-4e-6f, c.vth + fabsf(vs[u]), c.vth);
                    const float fall = -dE * c.fall;
                    const bool apart = fmaf(below - vs[u], fall, (below - vs[u + 1]) * d0) > d0 * fall * c.dt;
                    const bool peak = (d0 > 0.0f) & (dE < 0.0f) & !apart &
                                      (fmaf(fmaxf(I0[u], 0.0f), c.Kmax, fmaxf(vs[u], 0.0f)) >= c.vth);
                    if ((vs[u + 1] >= c.vth) | peak) nib |= 1u << u;
                }
                if (near & (nib != 0u)) {
                    mask |= nib << g;
                    if (kb < 0) {
                        kb = g >> 3;
                        kv = cv;
                        kI = cI;
                    }
                }
            }
        }
    }
    if (mend < 32) mask &= (1u << mend) - 1u;
    while (mask) {
        const int m = __ffs(mask) - 1;
        mask &= mask - 1u;
        for (; kb < (m >> 3); ++kb) {  // a later eight: the state at its start
            walk_group(c, row + kb * 8, (fused >> (kb * 2)) & 1u, kv, kI);
            walk_group(c, row + kb * 8 + 4, (fused >> (kb * 2 + 1)) & 1u, kv, kI);
        }
        float vw = kv, Iw = kI;
        walk_to<false>(c, row + kb * 8, m & 7, vw, Iw);
        const float I0 = __fadd_rn(Iw, row[m]);
        const float ve = walk_v(c, vw, I0);
        float hi = -1.0f;
        if (ve >= c.vth)
            hi = c.dt;
        else if ((fmaf(-c.av, vw, I0) > 0.0f) & (fmaf(-c.av, ve, __fmul_rn(c.rI, I0)) < 0.0f) &
                 (fmaf(fmaxf(I0, 0.0f), c.Kmax, fmaxf(vw, 0.0f)) >= c.vth))
            hi = interior_test(c.av, c.aI, c.lam, c.lam_zero, c.rI, c.dt, c.vth, vw, I0, ve);
        if (hi >= 0.0f) {
            st.q = m0 + m;
            st.v0 = vw;
            st.I0 = I0;
            st.hi = hi;
            return true;
        }
    }
    return false;
}

// Warps (FWD): 0-3 generators, 4 filter TMA, 5-8 MMA issue, 9.. epilogue
// (4 nset); (dS): 0 source TMA, 1 filter TMA, 2-5 MMA issue, 6.. epilogue. An
// epilogue warp reads TMEM lane quarter (warp mod 4): grid steps of one
// position. Output row n is issued by MMA warp n mod 4: the tensor core queues
// hardly any MMAs, and between two runs of them a warp spends 500 to 900 clocks
// on waits, addresses and commits, which the other warps' MMAs now cover (one
// warp: 82 to 130 clocks per N = 64 MMA over the whole loop, of which the
// tensor core needs 48).
template <int NT, bool FWD>
struct Roles {
    static constexpr int W_B = FWD ? GEN_WARPS : 1;  // the filter warp
    static constexpr int W_MMA = W_B + 1;
    static constexpr int W_EPI = W_MMA + MMA_WARPS;
    static constexpr int SLOT_COLS = NT * ROWS_BN;
    static constexpr int NA = 512 / SLOT_COLS > 8 ? 8 : 512 / SLOT_COLS;  // accumulators (output rows)
    static constexpr int CH = SLOT_COLS / 32;                            // 32-channel chunks of an output row
    static __host__ __device__ constexpr int threads(int nset) { return (W_EPI + 4 * nset) * 32; }
};
constexpr int FWD_MAX_THREADS = (GEN_WARPS + 1 + MMA_WARPS + 16) * 32;
constexpr int DS_MAX_THREADS = (2 + MMA_WARPS + 8) * 32;

// SLOTS: (position, channel) slots of a generator thread per box (forward)
template <int NT, bool FWD, int SLOTS>
__global__ void __launch_bounds__(FWD ? FWD_MAX_THREADS : DS_MAX_THREADS, 1)
    k_conv_rows(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ RowsArgs a, const __grid_constant__ RowsPlan p) {
    using Ro = Roles<NT, FWD>;
    static_assert(!FWD || NT == 1, "the forward takes one position tile");
    constexpr int NA = Ro::NA, CH = Ro::CH;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int SLICE = ROWS_BN * 128;  // one filter slice: ROWS_BN channels x 64 of K
    uint8_t *bbuf = smem + p.off_b;  // resident filters, or the ring of slices
    float *epi = reinterpret_cast<float *>(smem + p.off_epi);
    float4 *state = reinterpret_cast<float4 *>(smem + p.off_state);
    int8_t *kept = reinterpret_cast<int8_t *>(smem + p.off_kept);
    uint64_t *full_a = reinterpret_cast<uint64_t *>(smem + p.off_bar);
    uint64_t *empty_a = full_a + MAX_NSTA;
    uint64_t *full_b = empty_a + MAX_NSTA;
    uint64_t *empty_b = full_b + MAX_NSTB;
    uint64_t *acc_full = empty_b + MAX_NSTB;
    uint64_t *acc_empty = acc_full + 8;
    uint64_t *res_full = acc_empty + 8;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(res_full + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Mp = p.Mp, k = p.k, ncb = p.ncb;  // forward: one channel block (as constants 3% slower)
    const bool cb_inner = p.cb_inner != 0;
    const int cbo_n = cb_inner ? 1 : ncb, cbi_n = cb_inner ? ncb : 1;  // boxes outside / inside the filter columns
    const int kc = ncb * 64;

    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_NSTA; ++s) {
            tc::mbar_init(&full_a[s], FWD ? GEN_WARPS : 1);
            tc::mbar_init(&empty_a[s], MMA_WARPS);
        }
        for (int s = 0; s < MAX_NSTB; ++s) {
            tc::mbar_init(&full_b[s], 1);
            tc::mbar_init(&empty_b[s], MMA_WARPS);
        }
        for (int s = 0; s < 8; ++s) {
            tc::mbar_init(&acc_full[s], 1);
            // forward: one arrival per chunk and lane quarter; dS: every warp of the groups that read the row
            tc::mbar_init(&acc_empty[s], FWD ? CH * 4 : (NT == 2 ? 8 : 4));
        }
        tc::mbar_init(res_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (FWD) {  // zero boxes and no kept steps: the generators then write only nonzeros
        for (int i = threadIdx.x; i < p.nsta * p.stage_bytes / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = threadIdx.x; i < p.off_bar - p.off_kept; i += blockDim.x) kept[i] = (int8_t)SILENT;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == Ro::W_MMA) tc::tmem_alloc(tmem_slot, NA * Ro::SLOT_COLS);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (FWD && warp < GEN_WARPS) {
        // Generators: thread (g, c) writes channel c of the box positions
        // g, g + 2, ...; its records are loaded one box ahead. (The weights are
        // computed once per input by k_bin_rec: computed here, twice or more
        // per input, they took a quarter of the kernel's issue slots and left
        // the generators 3600 clocks per box.)
        const int g0 = threadIdx.x >> 6, c = threadIdx.x & 63;
        Item<FWD> nx;
        int n_it = blockIdx.x, n_sr = 0;
        if (n_it < p.n_items) {
            nx.decode(p, n_it);
            n_sr = nx.sr;
        }
        uint2 tn[SLOTS];
        auto load_next = [&]() {
            const bool on = n_it < p.n_items && c < a.C_t;
            const int x0 = on ? nx.xt * p.xs_mul + p.xs_add : 0;
            const uint2 *src = on ? a.rec + (((long long)nx.b * p.sh + n_sr) * p.sw + x0) * a.C_t + c : nullptr;
#pragma unroll
            for (int u = 0; u < SLOTS; ++u) {
                const int i = g0 + 2 * u;
                tn[u] = make_uint2((uint32_t)SILENT, 0u);
                if (on && i < p.npos && x0 + i >= 0 && x0 + i < p.sw) tn[u] = __ldg(src + (long long)i * a.C_t);
            }
            if (n_it < p.n_items && nx.done(++n_sr)) {
                n_it += gridDim.x;
                if (n_it < p.n_items) {
                    nx.decode(p, n_it);
                    n_sr = nx.sr;
                }
            }
        };
        load_next();
        int sa = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < p.n_items && ok; it += gridDim.x) {
            Item<FWD> w;
            w.decode(p, it);
            for (int sr = w.sr; !w.done(sr); ++sr) {
                uint2 cur[SLOTS];
#pragma unroll
                for (int u = 0; u < SLOTS; ++u) cur[u] = tn[u];
                load_next();
                int got = 1;  // the stage's previous MMAs are done with it
                if (lane == 0) got = tc::mbar_wait_spin(&empty_a[sa], ph ^ 1u) ? 1 : 0;
                if (!__shfl_sync(0xffffffffu, got, 0)) {
                    if (lane == 0) rows_set_status(STATUS_TIMEOUT);
                    ok = false;
                    break;
                }
                const uint32_t box = tc::smem_u32(smem + sa * p.stage_bytes);
                int8_t *kp = kept + sa * p.npos * 64 + c;
#pragma unroll
                for (int u = 0; u < SLOTS; ++u) {
                    const int i = g0 + 2 * u;
                    if (i >= p.npos) break;
                    const int kk = (int)cur[u].x;
                    const uint32_t wq = cur[u].y;
                    const int row0 = i * Mp, old = kp[i * 64];
                    if (old != SILENT) {
                        if (old >= 0) rows_sts_u16(box + rows_sw128(row0 + old, c), 0);
                        if (old + 1 < a.c.M) rows_sts_u16(box + rows_sw128(row0 + old + 1, c), 0);
                    }
                    if (kk != SILENT) {
                        if (kk >= 0) rows_sts_u16(box + rows_sw128(row0 + kk, c), (uint16_t)(wq & 0xffffu));
                        if (kk + 1 < a.c.M) rows_sts_u16(box + rows_sw128(row0 + kk + 1, c), (uint16_t)(wq >> 16));
                    }
                    if (kk != old) kp[i * 64] = (int8_t)kk;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&full_a[sa]);
                if (++sa == p.nsta) {
                    sa = 0;
                    ph ^= 1u;
                }
            }
        }
    } else if (!FWD && warp == 0) {
        // source boxes by TMA (the whole warp steps the loop, one lane issues)
        const uint32_t lead = tc::elect_one();
        uint32_t n = 0;
        int sa = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < p.n_items && ok; it += gridDim.x) {
            Item<FWD> w;
            w.decode(p, it);
            for (int sr = w.sr; !w.done(sr) && ok; --sr) {
                for (int cbo = 0; cbo < cbo_n; ++cbo, ++n) {
                    if (!tc::mbar_wait_warp(&empty_a[sa], ph ^ 1u)) {
                        ok = false;
                        break;
                    }
                    tc::mbar_expect_tx_if(lead, &full_a[sa], (uint32_t)(cbi_n * p.box_bytes));
                    for (int cbi = 0; cbi < cbi_n; ++cbi)
                        tc::tma_load_5d_if(lead, tc::smem_u32(smem + sa * p.stage_bytes + cbi * p.box_bytes), &mapA,
                                           &full_a[sa], (cbo + cbi) * 64, 0, w.xt * p.xs_mul + p.xs_add, sr, w.b);
                    if (++sa == p.nsta) {
                        sa = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
        if (!ok && lead) rows_set_status(STATUS_TIMEOUT);
        const uint32_t tail = n < (uint32_t)p.nsta ? n : (uint32_t)p.nsta;
        for (uint32_t i = n - tail; i < n; ++i) tc::mbar_wait_spin(&full_a[i % p.nsta], (i / p.nsta) & 1u);
        __syncwarp();
    } else if (warp == Ro::W_B) {
        const uint32_t lead = tc::elect_one();
        if (p.res_bytes) {  // every slice, once
            const int n = k * k * ncb;
            tc::mbar_expect_tx_if(lead, res_full, (uint32_t)(n * SLICE));
            for (int q = 0; q < n; ++q) {
                const int tap = q / ncb, cb = q - tap * ncb;
                tc::tma_load_2d_if(lead, tc::smem_u32(bbuf + q * SLICE), &mapB, res_full, tap * kc + cb * 64, 0);
            }
            tc::mbar_wait_spin(res_full, 0);
        } else {  // groups of slices in the order the MMAs take them
            uint32_t n = 0;
            int sb = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < p.n_items && ok; it += gridDim.x) {
                Item<FWD> w;
                w.decode(p, it);
                for (int sr = w.sr; !w.done(sr) && ok; sr += FWD ? 1 : -1)
                    for (int cbo = 0; cbo < cbo_n && ok; ++cbo)
                        for (int kh = k - 1; kh >= 0 && ok; --kh) {
                            if (w.out_row(p, sr, kh) < 0) continue;
                            for (int kw0 = 0; kw0 < k; kw0 += p.kwg, ++n) {
                                if (!tc::mbar_wait_warp(&empty_b[sb], ph ^ 1u)) {
                                    ok = false;
                                    break;
                                }
                                tc::mbar_expect_tx_if(lead, &full_b[sb], (uint32_t)(p.kwg * cbi_n * SLICE));
                                uint32_t dst = tc::smem_u32(bbuf + sb * p.kwg * cbi_n * SLICE);
                                for (int kw = kw0; kw < kw0 + p.kwg; ++kw)
                                    for (int cbi = 0; cbi < cbi_n; ++cbi, dst += SLICE)
                                        tc::tma_load_2d_if(lead, dst, &mapB, &full_b[sb],
                                                           (kh * k + kw) * kc + (cbo + cbi) * 64, FWD ? 0 : w.ct * ROWS_BN);
                                if (++sb == p.nstb) {
                                    sb = 0;
                                    ph ^= 1u;
                                }
                            }
                        }
            }
            if (!ok && lead) rows_set_status(STATUS_TIMEOUT);
            const uint32_t tail = n < (uint32_t)p.nstb ? n : (uint32_t)p.nstb;
            for (uint32_t i = n - tail; i < n; ++i) tc::mbar_wait_spin(&full_b[i % p.nstb], (i / p.nstb) & 1u);
        }
        __syncwarp();
    } else if (warp >= Ro::W_MMA && warp < Ro::W_EPI) {
        const uint32_t mw = (uint32_t)(warp - Ro::W_MMA);
        constexpr uint32_t idesc = idesc_kk(ROWS_BN);
        const uint32_t lead = tc::elect_one();
        const bool res = p.res_bytes != 0;
        int sa = 0, sb = 0;
        uint32_t pa = 0, pb = 0;
        uint32_t n0 = 0;  // output rows of the items before
        // low descriptor words; slices of one channel block are ncb apart when resident
        const uint32_t res_lo = tc::sdesc_kk_lo(tc::smem_u32(bbuf));
        const uint32_t b_step = (uint32_t)((res && !cb_inner ? ncb : 1) * (SLICE >> 4));
        const bool three = k == 3 && p.kwg == 3 && cbi_n == 1;
        const uint32_t tmem_u = tc::uniform(tmem);
        bool ok = !res || tc::mbar_wait_warp(res_full, 0);
        for (int it = blockIdx.x; it < p.n_items && ok; it += gridDim.x) {
            Item<FWD> w;
            w.decode(p, it);
            const int nsteps = (FWD ? w.sr_end - w.sr : w.sr - w.sr_end) + 1;
            uint32_t plan_lo = 0, plan_hi = 0;
            for (int j = 0; j < nsteps && ok; ++j) {
                if ((j & 31) == 0) {  // lane l works out source row j + l: the issuing loop is left with few instructions
                    const int sr = FWD ? w.sr + j + lane : w.sr - j - lane;
                    plan_lo = plan_hi = 0;
                    for (int kh = 0; kh < k && j + lane < nsteps; ++kh) {
                        const uint32_t f = row_plan<NA>(w, p, sr, kh, n0);
                        if (kh < 4) plan_lo |= f << (8 * kh);
                        else plan_hi |= f << (8 * (kh - 4));
                    }
                }
                const uint32_t lo = tc::uniform(__shfl_sync(0xffffffffu, plan_lo, j & 31));
                const uint32_t hi = k > 4 ? tc::uniform(__shfl_sync(0xffffffffu, plan_hi, j & 31)) : 0u;
                for (int cbo = 0; cbo < cbo_n && ok; ++cbo) {
                    if (!tc::mbar_wait_warp(&full_a[sa], pa)) {
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after();
                    const uint32_t st =
                        tc::uniform(tc::sdesc_kk_lo(tc::smem_u32(smem)) + (uint32_t)(sa * (p.stage_bytes >> 4)));
                    for (int kh = k - 1; kh >= 0; --kh) {  // the row that completes first
                        const uint32_t f = ((kh < 4 ? lo : hi) >> (8 * (kh & 3))) & 0xffu;
                        if (!(f & ROW_ON)) continue;
                        const uint32_t slot = (f >> 4) & 7u;
                        const bool mine = (slot & (MMA_WARPS - 1)) == mw;  // NA is a multiple of MMA_WARPS
                        if (!mine && res) continue;
                        const uint32_t acc = tmem_u + slot * Ro::SLOT_COLS;
                        const bool fresh = cbo == 0 && (f & ROW_FIRST);
                        if (fresh && mine) {
                            if (!tc::mbar_wait_warp(&acc_empty[slot], f >> 7)) {
                                ok = false;
                                break;
                            }
                            tc::tc_fence_after();
                        }
                        for (int kw0 = 0; kw0 < k; kw0 += p.kwg) {
                            uint32_t blo;
                            if (res) {
                                blo = res_lo + (uint32_t)(((kh * k + kw0) * ncb + cbo) * (SLICE >> 4));
                            } else {
                                if (!tc::mbar_wait_warp(&full_b[sb], pb)) {
                                    ok = false;
                                    break;
                                }
                                tc::tc_fence_after();
                                blo = tc::uniform(res_lo + (uint32_t)(sb * p.kwg * cbi_n * (SLICE >> 4)));
                            }
                            // (every warp passes every stage of the ring, so that none is ever two phases off)
                            auto tap = [&](int kw, int cbi, uint32_t bo) {
#pragma unroll
                                for (int t = 0; t < NT; ++t) {
                                    const int o = p.aoff[t][kw];
                                    if (NT == 2 && o < 0) continue;
                                    const uint32_t alo = st + (uint32_t)(cbi * (p.box_bytes >> 4) + o);
                                    const uint32_t on = !(fresh && kw == p.kfirst[t] && cbi == 0);  // adds to the tile
                                    tc::mma_kk(acc + t * ROWS_BN, alo, bo, idesc, on);
#pragma unroll
                                    for (int kk = 1; kk < 4; ++kk)
                                        tc::mma_kk(acc + t * ROWS_BN, alo + 2 * kk, bo + 2 * kk, idesc, 1u);
                                }
                            };
                            if (lead && mine) {
                                if (three) {  // a 3-wide filter row, one channel block: 12 NT MMAs back to back
#pragma unroll
                                    for (int kw = 0; kw < 3; ++kw) tap(kw, 0, blo + kw * b_step);
                                } else {
                                    for (int kw = kw0; kw < kw0 + p.kwg; ++kw)
                                        for (int cbi = 0; cbi < cbi_n; ++cbi, blo += b_step) tap(kw, cbi, blo);
                                }
                            }
                            __syncwarp();
                            if (!res) {
                                if (mine) tc::mma_commit_if(lead, &empty_b[sb]);
                                else if (lead) tc::mbar_arrive(&empty_b[sb]);
                                if (++sb == p.nstb) {
                                    sb = 0;
                                    pb ^= 1u;
                                }
                            }
                        }
                        if (!ok) break;
                        if (mine && cbo == cbo_n - 1 && (f & ROW_LAST)) tc::mma_commit_if(lead, &acc_full[slot]);
                    }
                    if (!ok) break;
                    tc::mma_commit_if(lead, &empty_a[sa]);
                    if (++sa == p.nsta) {
                        sa = 0;
                        pa ^= 1u;
                    }
                }
            }
            n0 += (uint32_t)w.rows();
        }
        if (!ok && lead) rows_set_status(STATUS_TIMEOUT);
        __syncwarp();
    } else if (FWD) {
        // Scan in the epilogue. Chunk c (32 channels) of output row n belongs
        // to epilogue set (n CH + c) mod nset. A warp reads its lane quarter
        // (32 grid steps of one position) of the chunk, turns it into neuron
        // rows in its own buffer and walks them, one neuron per lane. With 64
        // grid steps the lower quarter's warp hands the states to the upper
        // one's and gets them back to solve for the spike times, which balances
        // the two (the upper quarter holds most crossings): shared memory,
        // double buffered both ways, one named barrier per pair and chunk,
        // which also ends both after an expired wait.
        const int ew = warp - Ro::W_EPI, set = ew >> 2, quarter = warp & 3;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const bool two = Mp == 64;
        const int pp = two ? quarter >> 1 : quarter;
        const bool upper = two && (quarter & 1);
        float *tb = epi + ew * 32 * EPI_LDF;
        const int pair = set * 2 + (quarter >> 1), bar_id = 1 + pair;
        float4 *stb = state + pair * 128;  // lower -> upper [2][32], upper -> lower [2][32]
        auto pair_any = [&](bool x) -> bool {
            uint32_t r;
            asm volatile(
                "{\n"
                ".reg .pred pi, po;\n"
                "setp.ne.u32 pi, %1, 0;\n"
                "barrier.cta.red.or.pred po, %2, 64, pi;\n"
                "selp.u32 %0, 1, 0, po;\n"
                "}\n"
                : "=r"(r)
                : "r"((uint32_t)x), "r"(bar_id)
                : "memory");
            return r != 0;
        };
        float pacc[4] = {0.f, 0.f, 0.f, 0.f};
        // one loop over this set's chunks, so that each part's code is there
        // once (the instruction cache is shared with the other roles); with 64
        // grid steps one more round, without a chunk, for the last spikes
        uint32_t n = 0, cnt = 0;               // output rows before this one; chunks done
        int it = blockIdx.x, r = 0, c = -1, nrow = 0;
        int last_pos = -1, last_ch = 0;        // the lower warp's previous chunk, whose spikes it solves
        bool ok = true, more = it < p.n_items;
        Item<FWD> w;
        if (more) {
            w.decode(p, it);
            nrow = w.rows();
        }
        while (more) {
            do {  // the next chunk of the set
                if (++c == CH) {
                    c = 0;
                    ++n;
                    if (++r == nrow) {
                        r = 0;
                        it += gridDim.x;
                        more = it < p.n_items;
                        if (more) {
                            w.decode(p, it);
                            nrow = w.rows();
                        }
                    }
                }
            } while (more && (int)((n * CH + c) % (uint32_t)p.nset) != set);
            if (!more && (!two || cnt == 0)) break;
            bool fail = false;
            const uint32_t slot = n & (NA - 1);
            if (more) {
                fail = __any_sync(0xffffffffu, !tc::mbar_wait_sleep(&acc_full[slot], (n / NA) & 1u));
                if (!fail) {
                    tc::tc_fence_after();
                    float v[32];
                    tc::tmem_ld32(tmem + lane_base + slot * Ro::SLOT_COLS + c * 32, v);
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&acc_empty[slot]);
#pragma unroll
                    for (int u = 0; u < 32; ++u) tb[u * EPI_LDF + lane] = v[u];
                }
                __syncwarp();
            }
            const int x = w.xt * p.ppt + pp;
            const bool on = more && x < p.gw && !fail;
            const int pos = (w.b * p.gh + w.ya + r) * p.gw + x, ch = c * 32 + lane;
            // the state the walk starts from (upper: the lower quarter's end), then the spike's bin or the end
            // state: (q, v0, I0, hi) or (-1, v, I, -)
            float4 h = make_float4(__int_as_float(-1), 0.f, 0.f, 0.f);
            if (upper) {
                if (pair_any(fail)) {
                    ok = false;
                    break;
                }
                h = stb[(cnt & 1u) * 32 + lane];
            }
            const bool walks = on && __float_as_int(h.x) < 0;
            const unsigned lanes = __ballot_sync(0xffffffffu, walks);
            if (walks) {
                ScanState st;
                scan_reset(st, a.c.M);
                const int m0 = upper ? 32 : 0, mend = two && !upper ? 32 : a.c.M - m0;
                if (walk_rolled(lanes, a.c, tb + lane * EPI_LDF, m0, mend, h.y, h.z, st))
                    h = make_float4(__int_as_float(st.q), st.v0, st.I0, st.hi);
            }
            int f_pos = on ? pos : -1, f_ch = ch;  // the neuron to solve now
            if (two) {
                stb[(upper ? 64 : 0) + (cnt & 1u) * 32 + lane] = h;
                if (!upper) {
                    if (pair_any(fail)) {
                        ok = false;
                        break;
                    }
                    h = stb[64 + ((cnt - 1u) & 1u) * 32 + lane];  // the upper warp is past the previous chunk
                    f_pos = last_pos;
                    f_ch = last_ch;
                    last_pos = on ? pos : -1;
                    last_ch = ch;
                }
                ++cnt;
            } else if (fail) {
                ok = false;
                break;
            }
            if (!upper && f_pos >= 0) {
                ScanState st;
                scan_reset(st, a.c.M);
                if (__float_as_int(h.x) >= 0) {
                    st.q = __float_as_int(h.x);
                    st.v0 = h.y;
                    st.I0 = h.z;
                    st.hi = h.w;
                }
                scan_finish(a.c, st);
                finish_neuron(a.c, st, f_pos, f_ch, ROWS_BN, a.rowsum, a.t_out, a.q_out, a.s_out, a.vdot_out, pacc);
            }
            __syncwarp();
        }
        if (!ok) rows_set_status(STATUS_TIMEOUT);
        if (a.penalty) {
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) {
                const float sum = warp_sum(pacc[k2]);
                if (lane == 0 && sum != 0.f) atomicAdd(&a.penalty[k2], sum);
            }
        }
    } else {
        // dS: with two tiles per row, group g takes tile g; with one, every
        // other row. A warp reads its lane quarter of all ROWS_BN columns; lane u of
        // a chunk then owns input channel u and picks its two grid steps.
        const int ew = warp - Ro::W_EPI, group = ew >> 2, quarter = warp & 3;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        float *tb = epi + ew * 32 * EPI_LDG;
        const int pp = (quarter * 32) / Mp, m_base = (quarter * 32) % Mp;
        constexpr int NCH = ROWS_BN / 32;
        uint32_t n = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < p.n_items && ok; it += gridDim.x) {
            Item<FWD> w;
            w.decode(p, it);
            const int nrow = w.rows();
            for (int r = 0; r < nrow; ++r, ++n) {
                if (NT == 1 && (int)(n & 1u) != group) continue;
                const uint32_t slot = n & (NA - 1);
                const int tau = NT == 2 ? group : 0;
                // stride 1: tiles side by side; stride s: one tile per class x mod s
                const int x = p.s == 1 ? (w.xt * NT + tau) * p.ppt + pp : tau + p.s * (w.xt * p.ppt + pp);
                const int y = w.yb - 1 - r;
                const long long pos = ((long long)w.b * p.gh + y) * p.gw + x;
                // the inputs this lane will own, loaded ahead of the row
                float ti[NCH];
#pragma unroll
                for (int h = 0; h < NCH; ++h) {
                    const int col = w.ct * ROWS_BN + h * 32 + lane;
                    ti[h] = x < p.gw && col < a.C_t ? __ldg(a.t_in + pos * a.C_t + col) : INFINITY;
                }
                if (__any_sync(0xffffffffu, !tc::mbar_wait_sleep(&acc_full[slot], (n / NA) & 1u))) {
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                const uint32_t acc = tmem + lane_base + slot * Ro::SLOT_COLS + tau * ROWS_BN;
#pragma unroll 1
                for (int h = 0; h < NCH; ++h) {
                    {
                        float v[32];
                        tc::tmem_ld32(acc + h * 32, v);
#pragma unroll
                        for (int u = 0; u < 32; ++u) tb[lane * EPI_LDG + u] = v[u];
                    }
                    if (h == NCH - 1) {
                        tc::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&acc_empty[slot]);
                    }
                    __syncwarp();
                    float t = ti[0];
#pragma unroll
                    for (int z = 1; z < NCH; ++z) t = h == z ? ti[z] : t;
                    if (isfinite(t)) {
                        const int kb = bin_index(a.c, t), k0 = kb - m_base;
                        if (k0 >= -1 && k0 < 32 && kb < a.c.M) {  // this quarter holds one of its grid steps
                            const BinW bw = bin_weights(a.c, t, true);
                            float g = 0.f;
                            if (k0 >= 0) g = fmaf(tb[k0 * EPI_LDG + lane], bw.dR, g);
                            if (k0 + 1 < 32 && kb + 1 < a.c.M) g = fmaf(tb[(k0 + 1) * EPI_LDG + lane], bw.dL, g);
                            if (g != 0.f) atomicAdd(a.g_t_in + pos * a.C_t + w.ct * ROWS_BN + h * 32 + lane, g);
                        }
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok) rows_set_status(STATUS_TIMEOUT);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == Ro::W_MMA) tc::tmem_dealloc(tmem, NA * Ro::SLOT_COLS);
}

// ---------------------------------------------------------------------------
// dW of 3x3 layers at stride 1, walking the output rows position by position:
//   dW[o, (kh, kw), c] = sum_{y, x, m} dw^[(y, x, m), o] S[(y + kh, x + kw, m), c]
// A K step is one output position (Mp grid steps). Its nine taps read three
// columns of S, two of which the step before has taken: a ring of columns in
// shared memory (the S boxes of the rows y - pad .. for one x, and the dw^ box
// of the position that the column completes) is filled once per position where
// a box per tap and position was loaded before: 32 KB instead of 88 KB per step
// (64 channels, Mp = 64), with three and more columns in flight instead of one
// step. With 64 output channels generator warps write the columns from 8 bytes
// per input spike, so that the backward writes no S; with 128 the MMAs of a
// column are too short for them (128 -> 128 at 14 x 14: 0.84 ms generated,
// 0.58 ms from S) and S comes by TMA.
// The filter rows of the layer's channel block form 128-row MMA blocks: the
// taps (0, kw) and (1, kw) together (their boxes lie side by side), tap
// (2, kw) alone (the other 64 rows of the block are not used); with 64 output
// channels per tile all six blocks share a CTA, with 128 the first three and
// the last three are tiles of their own (TMEM holds four accumulators of 128
// columns). Split over output rows; fp32 atomics into g_W. Warps: 0 TMA, 1-4
// MMA issue (block b by warp b mod 4), 5-12 epilogue, 13.. generators. Bound by
// the MMAs: the tensor pipe is 55% busy with N = 64, whose operand reads cap it
// at 67%, and 75% with N = 128. Measured, a box per tap before and by columns
// (B = 256, M = 64): 64 -> 64 at 28 x 28 1.29 -> 0.92 ms
// (and 0.27 ms of writing S -> 0.07 of records), 128 -> 128 at 14 x 14 0.79 -> 0.61.
// ---------------------------------------------------------------------------
constexpr int DWC_MAX_RING = 8;
constexpr int DWC_MMA_WARPS = 4;
template <int BN>
struct DwCols {
    static constexpr bool GEN = BN == 64;           // columns generated on chip, else S by TMA
    static constexpr int BOXES = BN == 64 ? 3 : 2;  // source boxes of a slot
    static constexpr int GW = GEN ? 2 * BOXES : 0;  // generator warps: two per box, a thread per channel
    static constexpr int THREADS = (1 + DWC_MMA_WARPS + 8 + GW) * 32;
    static constexpr int SLOT_BOXES = BOXES + BN / 64;
    static constexpr int EXTRA = 1024 + (2 * DWC_MAX_RING + 2) * 8 + 8 + DWC_MAX_RING * GW * 32;  // beside the ring
};

struct DwColsPlan {
    int H, W, Ho, Wo, pad, M, Mp, ncb, n_col;
    int rows, rows_per, n_tiles, ring;
    const uint2 *rec;     // [ni H W][C_t] records of the input
    int C_t;              // the layer's input channels (below 64: padded to 64)
    float *g_W;           // [C_out][9][C_t]
    const float *count;   // silent neurons per output channel, or null
    float qcoef;
};

template <int BN>
__global__ void __launch_bounds__(DwCols<BN>::THREADS, 1)
    k_conv_dw_cols(const __grid_constant__ CUtensorMap mapS0, const __grid_constant__ CUtensorMap mapS1,
                   const __grid_constant__ CUtensorMap mapD, const __grid_constant__ DwColsPlan p) {
    constexpr int NGRP = BN == 64 ? 1 : 2, NBOX = DwCols<BN>::BOXES, GW = DwCols<BN>::GW;
    constexpr bool GEN = DwCols<BN>::GEN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int box = p.Mp * 128;
    const int slot_bytes = DwCols<BN>::SLOT_BOXES * box;  // (the second group leaves one source box unused)
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + p.ring * slot_bytes);
    uint64_t *empty = full + DWC_MAX_RING;
    uint64_t *acc_full = empty + DWC_MAX_RING;
    uint64_t *acc_empty = acc_full + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 1);
    int8_t *kept = reinterpret_cast<int8_t *>(tmem_slot + 2);  // [ring][GW 32] grid steps in the boxes

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int per = p.ncb * NGRP * p.n_col;  // tiles of one range of rows

    if (threadIdx.x == 0) {
        for (int s = 0; s < DWC_MAX_RING; ++s) {
            tc::mbar_init(&full[s], 1 + GW);
            tc::mbar_init(&empty[s], DWC_MMA_WARPS);
        }
        tc::mbar_init(acc_full, DWC_MMA_WARPS);
        tc::mbar_init(acc_empty, 8);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (GEN) {  // zero boxes and no kept steps: the generators then write only nonzeros
        for (int i = threadIdx.x; i < p.ring * slot_bytes / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = threadIdx.x; i < p.ring * GW * 32; i += blockDim.x) kept[i] = (int8_t)SILENT;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tc::tmem_alloc(tmem_slot, 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // tile t: rows [r0, r1) of the (image, y) rows, channel block, group, column tile
    auto decode = [&](int t, int &r0, int &r1, int &cb, int &grp, int &ct) {
        const int sp = t / per;
        int q = t - sp * per;
        ct = q % p.n_col;
        q /= p.n_col;
        grp = q % NGRP;
        cb = q / NGRP;
        r0 = sp * p.rows_per;
        r1 = r0 + p.rows_per < p.rows ? r0 + p.rows_per : p.rows;
    };

    if (warp == 0) {
        const uint32_t lead = tc::elect_one();
        uint32_t n = 0;
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x) {
            int r0, r1, cb, grp, ct;
            decode(t, r0, r1, cb, grp, ct);
            const int nbox = GEN ? 0 : 2 - grp;  // source boxes of a column that come by TMA
            int b = r0 / p.Ho, y = r0 - b * p.Ho;
            for (int r = r0; r < r1 && ok; ++r) {
                for (int cx = 0; cx < p.Wo + 2; ++cx, ++n) {
                    if (!tc::mbar_wait_warp(&empty[s], ph ^ 1u)) {
                        ok = false;
                        break;
                    }
                    // columns 0 and 1 complete no position
                    tc::mbar_expect_tx_if(lead, &full[s], (uint32_t)((nbox + (cx >= 2 ? BN / 64 : 0)) * box));
                    const uint32_t st = tc::smem_u32(smem + s * slot_bytes);
                    if (!GEN)
                        tc::tma_load_5d_if(lead, st, grp == 0 ? &mapS0 : &mapS1, &full[s], cb * 64, 0, cx - p.pad,
                                           y - p.pad + 2 * grp, b);
                    if (cx >= 2)
#pragma unroll
                        for (int h = 0; h < BN / 64; ++h)
                            tc::tma_load_5d_if(lead, st + (uint32_t)((NBOX + h) * box), &mapD, &full[s],
                                               ct * BN + h * 64, 0, cx - 2, y, b);
                    if (++s == p.ring) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (++y == p.Ho) {
                    y = 0;
                    ++b;
                }
            }
        }
        if (!ok && lead) rows_set_status(STATUS_TIMEOUT);
        const uint32_t tail = n < (uint32_t)p.ring ? n : (uint32_t)p.ring;
        for (uint32_t i = n - tail; i < n; ++i) tc::mbar_wait_spin(&full[i % p.ring], (i / p.ring) & 1u);
        __syncwarp();
    } else if (warp <= DWC_MMA_WARPS) {
        const int mw = warp - 1;
        const uint32_t lead = tc::elect_one();
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                   ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);  // both MN-major
        // low descriptor words: the next 64 columns (of A or of N) one box on
        const uint32_t base = ((tc::smem_u32(smem) & 0x3FFFFu) >> 4) | ((uint32_t)(box >> 4) << 16);
        const uint32_t tmem_u = tc::uniform(tmem);
        const int nkk = p.Mp >> 4;
        uint32_t j = 0;
        int s = 0;  // slot of the current column
        uint32_t ph = 0;
        bool ok = true;
        auto back = [&](int q, int d) { return q - d < 0 ? q - d + p.ring : q - d; };
        for (int t = blockIdx.x; t < p.n_tiles && ok; t += gridDim.x, ++j) {
            int r0, r1, cb, grp, ct;
            decode(t, r0, r1, cb, grp, ct);
            constexpr int NBLK = NGRP == 1 ? 6 : 3;
            if (j >= 1) {
                if (!tc::mbar_wait_warp(acc_empty, (j - 1) & 1u)) {
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
            }
            uint32_t more = 0;
            for (int r = r0; r < r1 && ok; ++r) {
                for (int cx = 0; cx < p.Wo + 2; ++cx) {
                    if (!tc::mbar_wait_warp(&full[s], ph)) {
                        ok = false;
                        break;
                    }
                    if (cx >= 2) {
                        tc::tc_fence_after();
                        const uint32_t cols =
                            tc::uniform((uint32_t)(back(s, 2) | (back(s, 1) << 8) | (s << 16)));  // slots of kw = 0, 1, 2
                        if (lead) {
                            const uint32_t blo = base + ((cols >> 16) * (uint32_t)slot_bytes + (uint32_t)(NBOX * box)) / 16u;
                            for (int bk = mw; bk < NBLK; bk += DWC_MMA_WARPS) {
                                const int kw = bk < 3 ? bk : bk - 3, bx = bk < 3 ? 0 : 2;
                                const uint32_t alo =
                                    base + (((cols >> (8 * kw)) & 0xffu) * (uint32_t)slot_bytes + (uint32_t)(bx * box)) / 16u;
                                const uint32_t acc = tmem_u + (uint32_t)(bk * BN);
                                for (int kk = 0; kk < nkk; ++kk)
                                    tc::mma_kk(acc, alo + (uint32_t)(kk * 128), blo + (uint32_t)(kk * 128), idesc,
                                               kk > 0 ? 1u : more);
                            }
                        }
                        __syncwarp();
                        more = 1u;
                        tc::mma_commit_if(lead, &empty[back(s, 2)]);
                        if (cx == p.Wo + 1) {  // the row's last position
                            tc::mma_commit_if(lead, &empty[back(s, 1)]);
                            tc::mma_commit_if(lead, &empty[s]);
                        }
                    }
                    if (++s == p.ring) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (ok) tc::mma_commit_if(lead, acc_full);
        }
        if (!ok && lead) rows_set_status(STATUS_TIMEOUT);
        __syncwarp();
    } else if (GEN && warp > DWC_MMA_WARPS + 8) {
        // Generators: warps 2 h and 2 h + 1 write box h of every column, a
        // thread one channel; its record is loaded one column ahead.
        const int gi = threadIdx.x - (1 + DWC_MMA_WARPS + 8) * 32, h = gi >> 6, c = gi & 63;
        struct Col {
            int t, r, r1, cx, b, y, cb;
        };
        auto open = [&](Col &q) {
            int r0, grp, ct;
            decode(q.t, r0, q.r1, q.cb, grp, ct);
            q.r = r0;
            q.cx = 0;
            q.b = r0 / p.Ho;
            q.y = r0 - q.b * p.Ho;
        };
        auto step = [&](Col &q) {
            if (++q.cx < p.Wo + 2) return;
            q.cx = 0;
            if (++q.y == p.Ho) {
                q.y = 0;
                ++q.b;
            }
            if (++q.r == q.r1) {
                q.t += gridDim.x;
                if (q.t < p.n_tiles) open(q);
            }
        };
        auto load = [&](const Col &q) {
            const int y = q.y - p.pad + h, x = q.cx - p.pad, ch = q.cb * 64 + c;
            if (q.t >= p.n_tiles || y < 0 || y >= p.H || x < 0 || x >= p.W || ch >= p.C_t)
                return make_uint2((uint32_t)SILENT, 0u);
            return __ldg(p.rec + (((long long)q.b * p.H + y) * p.W + x) * p.C_t + ch);
        };
        Col q, nx;
        nx.t = blockIdx.x;
        if (nx.t < p.n_tiles) open(nx);
        q = nx;
        uint2 tn = load(nx);
        int s = 0;
        uint32_t ph = 0;
        for (; q.t < p.n_tiles; step(q)) {
            const uint2 cur = tn;
            step(nx);
            tn = load(nx);
            int got = 1;
            if (lane == 0) got = tc::mbar_wait_spin(&empty[s], ph ^ 1u) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, got, 0)) {
                if (lane == 0) rows_set_status(STATUS_TIMEOUT);
                break;
            }
            const uint32_t bx = tc::smem_u32(smem + s * slot_bytes + h * box);
            int8_t *kp = kept + s * GW * 32 + gi;
            const int kk = (int)cur.x, old = *kp;
            if (old != SILENT) {
                if (old >= 0) rows_sts_u16(bx + rows_sw128(old, c), 0);
                if (old + 1 < p.M) rows_sts_u16(bx + rows_sw128(old + 1, c), 0);
            }
            if (kk != SILENT) {
                if (kk >= 0) rows_sts_u16(bx + rows_sw128(kk, c), (uint16_t)(cur.y & 0xffffu));
                if (kk + 1 < p.M) rows_sts_u16(bx + rows_sw128(kk + 1, c), (uint16_t)(cur.y >> 16));
            }
            if (kk != old) *kp = (int8_t)kk;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&full[s]);
            if (++s == p.ring) {
                s = 0;
                ph ^= 1u;
            }
        }
        __syncwarp();
    } else {
        const int quarter = warp & 3, half = (warp - 1 - DWC_MMA_WARPS) >> 2;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const int r = quarter * 32 + lane;
        uint32_t j = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < p.n_tiles; t += gridDim.x, ++j) {
            int r0, r1, cb, grp, ct;
            decode(t, r0, r1, cb, grp, ct);
            if (__any_sync(0xffffffffu, !tc::mbar_wait_sleep(acc_full, j & 1u))) {
                ok = false;
                break;
            }
            tc::tc_fence_after();
            constexpr int NBLK = NGRP == 1 ? 6 : 3;
            for (int bk = 0; bk < NBLK; ++bk) {
                const bool pair = NGRP == 1 ? bk < 3 : grp == 0;
                const int kw = bk < 3 ? bk : bk - 3, kh = pair ? r >> 6 : 2;
                const int ch = cb * 64 + (r & 63);
                const bool on = (pair || r < 64) && ch < p.C_t;
                const long long k0 = (long long)(kh * 3 + kw) * p.C_t + ch;
                for (int cc = half; cc < BN / 32; cc += 2) {
                    float v[32];
                    tc::tmem_ld32(tmem + lane_base + bk * BN + cc * 32, v);
                    if (on) {
                        const int o0 = ct * BN + cc * 32;
#pragma unroll
                        for (int u = 0; u < 32; ++u) {
                            const float add = r0 == 0 && p.count ? p.qcoef * p.count[o0 + u] : 0.f;
                            atomicAdd(p.g_W + (long long)(o0 + u) * 9 * p.C_t + k0, v[u] + add);
                        }
                    }
                }
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(acc_empty);
        }
        if (!ok) rows_set_status(STATUS_TIMEOUT);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
typedef CUresult (*RowsEncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

RowsEncodeFn rows_encode() {
    static RowsEncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *q = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &q, 12000, cudaEnableDefault, &r) ==
                cudaSuccess &&
            r == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<RowsEncodeFn>(q);
    });
    return fn;
}

// activation [ni][h][w][Mp][C] bf16, boxes of (64, Mp, box_x, box_y, 1), zeros outside
bool rows_map_act(CUtensorMap *m, const void *ptr, int ni, int h, int w, int Mp, int C, int box_x, int box_y = 1) {
    RowsEncodeFn enc = rows_encode();
    if (!enc || box_x > 256) return false;
    cuuint64_t dims[5] = {(cuuint64_t)C, (cuuint64_t)Mp, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)ni};
    cuuint64_t strides[4] = {(cuuint64_t)C * 2, (cuuint64_t)Mp * C * 2, (cuuint64_t)w * Mp * C * 2,
                             (cuuint64_t)h * w * Mp * C * 2};
    cuuint32_t box[5] = {64, (cuuint32_t)Mp, (cuuint32_t)box_x, (cuuint32_t)box_y, 1};
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(ptr), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool rows_map_mat(CUtensorMap *m, const void *ptr, int rows, int cols, int box_rows) {
    RowsEncodeFn enc = rows_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int rows_num_sms() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
    }
    return n;
}

constexpr int ROWS_SMEM_MAX = 227 * 1024;
constexpr int BAR_BYTES = (2 * MAX_NSTA + 2 * MAX_NSTB + 16 + 1) * 8 + 8;  // barriers and the TMEM address

// lays the shared memory out for the plan's stages; false if it does not fit.
// Behind the source boxes: filters, epilogue rows (32 x 32 values a warp),
// forward: the lower quarters' states (64 grid steps) and the kept grid steps
// of the generator slots; the barriers last
bool rows_layout(bool fwd, RowsPlan &p) {
    constexpr int slice = ROWS_BN * 128;
    const int cbi = p.cb_inner ? p.ncb : 1;
    const long long b = p.res_bytes ? (long long)p.res_bytes : (long long)p.nstb * p.kwg * cbi * slice;
    const long long off_epi = (long long)p.nsta * p.stage_bytes + b;
    const int warps = 4 * p.nset;
    const long long off_state = off_epi + warps * 32 * (fwd ? EPI_LDF : EPI_LDG) * 4;
    const long long off_kept = off_state + (fwd && p.Mp == 64 ? p.nset * 2 * 4 * 32 * 16 : 0);
    const long long off_bar = off_kept + (fwd ? (p.nsta * cbi * p.npos * 64 + 127) / 128 * 128 : 0);
    const long long total = off_bar + BAR_BYTES + 1024;  // and the alignment of the start
    if (total > ROWS_SMEM_MAX) return false;
    p.off_b = p.nsta * p.stage_bytes;
    p.off_epi = (int)off_epi;
    p.off_state = (int)off_state;
    p.off_kept = (int)off_kept;
    p.off_bar = (int)off_bar;
    p.smem = (int)total;
    return true;
}

// rows per strip: the fewest (rounds of items on the SMs) x (rows + 1), the
// one for the item's first box and last epilogue
void rows_strips(RowsPlan &p, int ni) {
    const long long per = (long long)ni * p.n_xt * p.n_col;
    const int sms = rows_num_sms();
    long long best = -1;
    for (int n = 1; n <= p.gh; ++n) {
        const int R = (p.gh + n - 1) / n, ns = (p.gh + R - 1) / R;
        const long long cost = (per * ns + sms - 1) / sms * (R + 1);
        if (best < 0 || cost < best) {
            best = cost;
            p.R = R;
            p.n_strip = ns;
        }
    }
    p.n_items = (int)(per * p.n_strip);
}

// The plan of one launch, or false where the shape stays on the
// one-row-at-a-time kernels: strides above 2, filters wider than their
// padding allows (an output row without a source row), more output rows in
// flight than accumulators, or too little shared memory.
bool rows_plan(bool fwd, const ConvGeom &g, int ni, int C_out, int Mp, bool cb_inner, int NT, int nset, RowsPlan &p) {
    p = RowsPlan{};
    p.s = g.s;
    p.k = g.k;
    p.pad = g.p;
    p.Mp = Mp;
    p.ppt = 128 / Mp;
    p.gh = fwd ? g.Ho : g.H;
    p.gw = fwd ? g.Wo : g.W;
    p.sh = fwd ? g.H : g.Ho;
    p.sw = fwd ? g.W : g.Wo;
    p.ncb = fwd ? 1 : C_out / 64;
    p.cb_inner = cb_inner && p.ncb > 1;
    p.nset = nset;
    p.n_col = fwd ? 1 : g.C / ROWS_BN;
    if (g.s > 2 || g.k > MAX_K || g.k < g.s || g.p > g.k - 1) return false;
    for (int t = 0; t < 2; ++t)
        for (int kw = 0; kw < MAX_K; ++kw) p.aoff[t][kw] = -1;
    if (fwd) {
        p.n_xt = (p.gw + p.ppt - 1) / p.ppt;
        p.npos = p.ppt - 1 + p.k;
        for (int kw = 0; kw < p.k; ++kw) p.aoff[0][kw] = kw;
        p.xs_mul = p.ppt;
        p.xs_add = -p.pad;
    } else if (p.s == 1) {
        p.n_xt = (p.gw + NT * p.ppt - 1) / (NT * p.ppt);
        p.npos = NT * p.ppt + p.k - 1;
        for (int t = 0; t < NT; ++t)
            for (int kw = 0; kw < p.k; ++kw) p.aoff[t][kw] = t * p.ppt + p.k - 1 - kw;
        p.xs_mul = NT * p.ppt;
        p.xs_add = p.pad - (p.k - 1);
    } else {
        // class t = x mod 2: filter columns kw = t + pad (mod 2) read source
        // position (x - t) / 2 + (t + pad - kw) / 2
        if (NT != 2) return false;
        p.n_xt = ((p.gw + 1) / 2 + p.ppt - 1) / p.ppt;
        int lo = 1 << 20, hi = -(1 << 20);
        for (int t = 0; t < 2; ++t)
            for (int kw = (t + p.pad) % 2; kw < p.k; kw += 2) {
                const int d = (t + p.pad - kw) / 2;  // even numerator
                lo = d < lo ? d : lo;
                hi = d > hi ? d : hi;
            }
        for (int t = 0; t < 2; ++t)
            for (int kw = (t + p.pad) % 2; kw < p.k; kw += 2) p.aoff[t][kw] = (t + p.pad - kw) / 2 - lo;
        p.npos = p.ppt + hi - lo;
        p.xs_mul = p.ppt;
        p.xs_add = lo;
    }
    // output rows in flight at one source row, and one for the epilogue
    const int flight = p.k + 1;
    int NA = 512 / (NT * ROWS_BN);
    if (NA > 8) NA = 8;
    if (flight > NA) return false;
    // every output row reads at least one source row
    for (int y = 0; y < p.gh; ++y) {
        bool any = false;
        for (int kh = 0; kh < p.k && !any; ++kh) {
            int r;
            if (fwd) {
                r = y - p.pad + kh;
            } else {
                if ((y + p.pad - kh) < 0 || (y + p.pad - kh) % p.s != 0) continue;
                r = (y + p.pad - kh) / p.s;
            }
            any = r >= 0 && r < p.sh;
        }
        if (!any) return false;
    }
    for (int t = 0; t < 2; ++t) {
        p.kfirst[t] = -1;
        for (int kw = p.k - 1; kw >= 0; --kw)
            if (p.aoff[t][kw] >= 0) {
                p.aoff[t][kw] *= Mp * 8;
                p.kfirst[t] = kw;
            }
    }
    p.box_bytes = p.npos * Mp * 128;
    p.stage_bytes = p.box_bytes * (p.cb_inner ? p.ncb : 1);
    const long long res = (long long)p.k * p.k * p.ncb * ROWS_BN * 128;
    p.nsta = 2;
    p.nstb = 0;
    p.kwg = p.k;
    if (res < ROWS_SMEM_MAX) {
        p.res_bytes = (int)res;
        if (!rows_layout(fwd, p)) p.res_bytes = 0;
    }
    if (!p.res_bytes) {
        // as many stages of a whole filter row as fit, at least two; else of single filter columns
        for (int pass = 0; pass < 2; ++pass) {
            p.kwg = pass == 0 ? p.k : 1;
            for (p.nstb = MAX_NSTB; p.nstb >= 2 && !rows_layout(fwd, p);) --p.nstb;
            if (p.nstb >= 2) break;
        }
        if (p.nstb < 2) return false;
    }
    while (!fwd && p.nsta < MAX_NSTA) {
        RowsPlan m = p;
        ++m.nsta;
        if (!rows_layout(fwd, m)) break;
        p = m;
    }
    rows_strips(p, ni);
    return true;
}

template <int NT, bool FWD, int SLOTS>
cudaError_t rows_launch(const CUtensorMap &mA, const CUtensorMap &mB, const RowsArgs &a, const RowsPlan &p,
                        cudaStream_t st) {
    cudaError_t e = allow_smem<k_conv_rows<NT, FWD, SLOTS>>(p.smem);
    if (e != cudaSuccess) return e;
    const int grid = p.n_items < rows_num_sms() ? p.n_items : rows_num_sms();
    k_conv_rows<NT, FWD, SLOTS><<<grid, Roles<NT, FWD>::threads(p.nset), p.smem, st>>>(mA, mB, a, p);
    return cudaGetLastError();
}

// Expected time of dS by rows under plan p: launch, and per round of items on
// the SMs a source box (of one channel block), a pair of a source row and a
// filter row, its taps, an output row and the item. Fitted, as in
// conv_ds_tap_us, for each way the filters come (resident, a filter row or one
// filter column at a time) and each order of the products (2 to 8% rms).
double rows_ds_us(const RowsPlan &p, int NT) {
    struct Fit {
        double launch, box, pair, tap, row, item;
    };
    static const Fit fits[2][3][2] = {  // [NT - 1][resident, rows, columns][cb_inner]
        {{{13.3, 0.857, 0.0, 0.070, 0.0, 0.21}, {10.9, 0.349, 0.0, 0.0, 0.0, 0.0}},
         {{13.0, 0.806, 0.0, 0.123, 0.156, 0.163}, {13.0, 0.806, 0.0, 0.123, 0.156, 0.163}},
         {{8.7, 1.667, 0.0, 0.313, 0.0, 0.0}, {13.6, 0.0, 0.0, 0.239, 0.0, 0.55}}},
        {{{12.7, 0.254, 0.236, 0.0, 1.227, 0.12}, {12.1, 0.079, 0.0, 0.424, 0.0, 0.12}},
         {{13.1, 0.815, 0.0, 0.100, 0.14, 0.0}, {13.1, 0.815, 0.0, 0.100, 0.14, 0.0}},
         {{14.0, 0.265, 0.0, 0.156, 0.0, 0.09}, {14.0, 0.265, 0.0, 0.156, 0.0, 0.09}}}};
    const Fit &f = fits[NT - 1][p.res_bytes ? 0 : (p.kwg > 1 || p.k == 1) ? 1 : 2][p.cb_inner ? 1 : 0];
    long long src = 0, pairs = 0;  // over the strips of an image's columns
    for (int s = 0; s < p.n_strip; ++s) {
        const int ya = s * p.R, yb = ya + p.R < p.gh ? ya + p.R : p.gh;
        for (int r = 0; r < p.sh; ++r) {  // rows ya .. yb - 1 through filter rows of 0 .. k - 1
            const int lo = ya > r * p.s - p.pad ? ya : r * p.s - p.pad;
            const int hi = yb - 1 < r * p.s - p.pad + p.k - 1 ? yb - 1 : r * p.s - p.pad + p.k - 1;
            if (hi < lo) continue;
            ++src;
            pairs += hi - lo + 1;
        }
    }
    const double rounds = (double)((p.n_items + rows_num_sms() - 1) / rows_num_sms()), per = rounds / p.n_strip;
    return f.launch + per * p.ncb * (f.box * src + pairs * (f.pair + f.tap * p.k * (p.s == 1 ? NT : 1))) +
           per * f.row * p.gh + f.item * rounds;
}

struct Tile {
    int NT, nset;
};

// Where this kernel is the faster one, measured against the one-row-at-a-time
// kernels over 3 to 32 wide images:
//   forward  64 output channels of one channel block at stride 1, from about
//            300 output positions per SM on: with the filters resident or
//            streamed a filter row at a time, 2x2 to 4x4 filters 1.02 to 1.54
//            times faster (3x3 at 28 x 28, M = 64: 1.07 to 1.13, binning
//            included); 5x5 1.1 to 1.3 where the other kernel has no row boxes
//            (the position tile does not divide the image's width), 0.85 to 1
//            where it has; streamed a filter column at a time (4x4 and wider at
//            64 grid steps, 6x6 and wider) 0.5 to 0.87. Fewer positions 0.86 to
//            0.96. With 64 grid steps and little decay over the window (the
//            lesser rate times its length below 0.9) the scan is light and this
//            kernel only pays for 3x3 and wider where the other has no row boxes
//            (1.1 to 1.3; else 0.84 to 1.05). Not built: two channel blocks
//            (0.82), stride 2 (0.95 to 1.02), 128 and more output channels (0.6
//            to 0.9); 1x1 0.91;
//   dS       64 input channels, by the expected times: 64 -> 64 at 28 x 28 and 64
//            -> 128 at stride 2 1.6 and 2.0 times faster; slower where the tile
//            is twice as wide as the image (M = 32 at 4 wide, 0.4 to 0.8) and
//            where the filters stream past row boxes (64 -> 128 at 14 x 14, M = 64:
//            0.84 to 0.92; 64 -> 64, 7x7: 0.6 to 0.8). Over the fitted layers the
//            choice costs 0.4% against the better of the two; taken always, these
//            kernels lost up to 2.4 times.
bool rows_faster(bool fwd, const ConvGeom &g, int ni, int C_out, int Mp, bool cb_inner, float decay,
                 const RowsPlan &p, const Tile &t) {
    if (!fwd) return rows_ds_us(p, t.NT) < conv_ds_tap_us(g, ni, C_out, Mp);
    if (!p.res_bytes && !(p.kwg > 1 && (g.k < 5 || cb_inner))) return false;
    return Mp < 64 || decay >= 0.9f || (g.k > 2 && cb_inner);
}

// the plan of a shape that the kernel takes: the most epilogue warps, or the
// widest tile, that fits
bool rows_pick(bool fwd, const ConvGeom &g, int ni, int C_out, int Mp, bool cb_inner, RowsPlan &p, Tile &t) {
    if (fwd) {
        if (C_out != 64 || g.C != 64 || g.s != 1 || g.k == 1) return false;
        if ((long long)ni * g.Ho * g.Wo < 300ll * rows_num_sms()) return false;
        for (t = Tile{1, 4}; t.nset >= 2; --t.nset)
            if (rows_plan(true, g, ni, C_out, Mp, cb_inner, t.NT, t.nset, p)) return true;
    } else {
        if (g.C != 64 || (long long)ni * g.H * g.W < 20ll * rows_num_sms()) return false;
        for (t = Tile{2, 2}; t.NT >= 1; --t.NT)
            if (rows_plan(false, g, ni, C_out, Mp, cb_inner, t.NT, t.nset, p)) return true;
    }
    return false;
}

}  // namespace

bool conv_rows_fwd_faster(const ConvGeom &g, int ni, int C_out, int Mp, bool cb_inner, float decay) {
    RowsPlan p;
    Tile t;
    return rows_pick(true, g, ni, C_out, Mp, cb_inner, p, t) && rows_faster(true, g, ni, C_out, Mp, cb_inner, decay, p, t);
}

cudaError_t launch_conv_rows_fwd(const ConvGeom &g, int ni, int C_out, const LifConst &c, bool cb_inner,
                                 const uint2 *rec, int C_t, const __nv_bfloat16 *Wf, const float *rowsum,
                                 float *t_out, int *q, float *s, float *vdot, float *penalty, cudaStream_t st) {
    RowsPlan p;
    Tile t;
    if (!rows_pick(true, g, ni, C_out, c.Mp, cb_inner, p, t)) return cudaErrorInvalidConfiguration;
    RowsArgs a{};
    a.rec = rec;
    a.C_t = C_t;
    a.t_out = t_out;
    a.q_out = q;
    a.s_out = s;
    a.vdot_out = vdot;
    a.rowsum = rowsum;
    a.penalty = penalty;
    a.c = c;
    CUtensorMap mB;
    if (!rows_map_mat(&mB, Wf, C_out, g.k * g.k * g.C, ROWS_BN)) return cudaErrorInvalidValue;
    // the generator's code is laid out for its slots (2 or 3 for 3x3 filters, 3 or 4 for 5x5): unrolled for more than
    // it needs, it overran the instruction cache
    const int slots = (p.npos + 1) / 2;
    if (slots <= 2) return rows_launch<1, true, 2>(mB, mB, a, p, st);
    if (slots <= 3) return rows_launch<1, true, 3>(mB, mB, a, p, st);
    return rows_launch<1, true, GEN_SLOTS>(mB, mB, a, p, st);
}

bool conv_rows_ds_faster(const ConvGeom &g, int ni, int C_out, int Mp, bool cb_inner) {
    RowsPlan p;
    Tile t;
    return rows_pick(false, g, ni, C_out, Mp, cb_inner, p, t) && rows_faster(false, g, ni, C_out, Mp, cb_inner, 0.f, p, t);
}

cudaError_t launch_conv_rows_ds(const ConvGeom &g, int ni, int C_out, const LifConst &c, bool cb_inner,
                                const __nv_bfloat16 *dW_hat, const __nv_bfloat16 *Wt, const float *t_in, float *g_t_in, int C_t, cudaStream_t st) {
    RowsPlan p;
    Tile t;
    if (!rows_pick(false, g, ni, C_out, c.Mp, cb_inner, p, t)) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaMemsetAsync(g_t_in, 0, sizeof(float) * (size_t)ni * g.H * g.W * C_t, st);
    if (e != cudaSuccess) return e;
    RowsArgs a{};
    a.t_in = t_in;
    a.C_t = C_t;
    a.g_t_in = g_t_in;
    a.c = c;
    CUtensorMap mA, mB;
    if (!rows_map_act(&mA, dW_hat, ni, g.Ho, g.Wo, c.Mp, C_out, p.npos) ||
        !rows_map_mat(&mB, Wt, g.C, g.k * g.k * C_out, ROWS_BN))
        return cudaErrorInvalidValue;
    if (t.NT == 2) return rows_launch<2, false, 1>(mA, mB, a, p, st);
    return rows_launch<1, false, 1>(mA, mB, a, p, st);
}

bool conv_dw_cols_records(int C_out) { return C_out == 64; }

// The ranges of rows: the fewest rounds of tiles on the SMs x (rows + the cost
// of a tile's epilogue, about two rows of 28 positions), but at least as many
// as splits in k_conv_dw_tma where the chunk has that many rows, with 128
// columns half as many again: the tensor core cuts its sums off, so the error
// of a range grows with its length. With one round of tiles dW of 64 -> 64 at
// 28 x 28 was 24e-6 off and of 128 -> 128 at 14 x 14 8e-6, against 16e-6 and
// 2e-6 of that kernel.
static ConvDwColsSplit dw_cols_split(const ConvGeom &g, int ni, int C_out) {
    const int BN = C_out == 64 ? 64 : 128, ncb = g.C / 64, n_col = C_out / BN, rows = ni * g.Ho;
    const int per = ncb * (BN == 64 ? 1 : 2) * n_col, sms = rows_num_sms();
    const int G = BN == 64 ? 5 : 3, row_tiles = (9 * ncb + 1) / 2;
    int least = (BN == 64 ? 2 : 3) * sms / ((row_tiles + G - 1) / G * n_col);
    if (least > rows) least = rows;
    const double tail = 56.0 / g.Wo;
    double best = -1.0;
    ConvDwColsSplit sp{1, 0};
    for (int n = least < 1 ? 1 : least; n <= rows && (n <= least || n <= 4 * sms); ++n) {
        const int rp = (rows + n - 1) / n, ns = (rows + rp - 1) / rp;
        const double cost = (double)(((long long)per * ns + sms - 1) / sms) * (rp + tail);
        if (best < 0.0 || cost < best) {
            best = cost;
            sp = ConvDwColsSplit{rp, per * ns};
        }
    }
    return sp;
}

// Shapes: 3x3 at stride 1, 64 output channels, or a multiple of 128 with 64
// grid steps. (With 32 a K step of those is one position of 32, half of whose
// MMA block (2, kw) is not used: 0.68 to 0.99 of the speed of a box per tap.)
// Of those, where the kernel is expected to be the faster one. By columns it
// pays for two more columns per row and for atomics per range, so it loses on
// few positions and on narrow images, unless a single round of short rows does
// it. Measured, a box per tap / by columns (with 64 output channels S or the
// records included), us: 64 -> 64, M = 64: 12 images of 2 x 2 25 / 23, 250 of
// 2 x 2 26 / 35, one of 28 x 28 26 / 39, 20 of 14 x 14 46 / 47, 82 of 14 x 14
// 150 / 108, 82 of 28 x 28 520 / 349; M = 32: 165 of 11 x 11 116 / 107;
// 128 -> 64, M = 32: 40 of 10 x 10 49 / 63; 128 -> 128: 12 of 2 x 2 23 / 16, 250 of
// 2 x 2 35 / 51, 20 of 14 x 14 64 / 82, 163 of 14 x 14 480 / 414; 256 -> 256: 50 of
// 2 x 2 27 / 46, 82 of 14 x 14 841 / 756; 512 -> 512: 62 of 4 x 4 213 / 241. The
// times are fitted as in conv_dw_tma_us (3% rms): launch, a position of a row, a
// row's two more columns, a tile's epilogue; S at 5.7 TB/s, the records at 2.5, or
// 4.3 with no decay at all (no exponentials).
// Over the fitted shapes the choice costs 0.2% against the better of the two.
// Where both are expected within 2% it stays by columns.
bool conv_dw_cols_pick(const ConvGeom &g, int ni, int C_out, int Mp, int C_t, bool decay, ConvDwColsSplit &sp) {
    if (g.k != 3 || g.s != 1 || g.C % 64 != 0) return false;
    if (!(C_out == 64 && (Mp == 32 || Mp == 64)) && !(C_out % 128 == 0 && Mp == 64)) return false;
    sp = dw_cols_split(g, ni, C_out);
    struct Fit {
        double launch, pos, row, epi;
    };
    const Fit f = C_out != 64 ? Fit{8.2, 0.406, 0.285, 6.42}
                  : Mp == 64  ? Fit{9.0, 0.623, 0.473, 6.42}
                  : C_t < 64  ? Fit{8.5, 0.486, 0.560, 6.19}   // (its generators have less to write)
                              : Fit{9.0, 0.538, 0.641, 5.33};
    const double rounds = (double)((sp.n_tiles + rows_num_sms() - 1) / rows_num_sms());
    double cols = f.launch + rounds * (sp.rows_per * (g.Wo * f.pos + f.row) + f.epi);
    double taps = conv_dw_tma_us(g, ni, C_out, Mp);
    if (conv_dw_cols_records(C_out)) {
        const double in_mb = 1e-6 * ni * g.H * g.W;
        cols += 5.5 + in_mb * C_t * 12 * (decay ? 0.405 : 0.233);
        taps += 6.3 + in_mb * g.C * Mp * 2 * 0.177;
    }
    return 0.98 * cols < taps;
}

cudaError_t launch_conv_dw_cols(const ConvGeom &g, int ni, int C_out, const LifConst &c, const ConvDwColsSplit &sp,
                                const uint2 *rec, const __nv_bfloat16 *S, const __nv_bfloat16 *dW_hat,
                                const float *count, float qcoef, float *g_W, int C_t, cudaStream_t st) {
    DwColsPlan p{};
    p.H = g.H;
    p.W = g.W;
    p.M = c.M;
    p.rec = rec;
    p.Ho = g.Ho;
    p.Wo = g.Wo;
    p.pad = g.p;
    p.Mp = c.Mp;
    p.ncb = g.C / 64;
    const int BN = C_out == 64 ? 64 : 128, sms = rows_num_sms();
    p.n_col = C_out / BN;
    p.rows = ni * g.Ho;
    if (p.rows == 0) return cudaSuccess;
    p.C_t = C_t;
    p.g_W = g_W;
    p.count = count;
    p.qcoef = qcoef;
    p.rows_per = sp.rows_per;
    p.n_tiles = sp.n_tiles;
    const int slot = (BN == 64 ? DwCols<64>::SLOT_BOXES : DwCols<128>::SLOT_BOXES) * c.Mp * 128;
    const int extra = BN == 64 ? DwCols<64>::EXTRA : DwCols<128>::EXTRA;
    p.ring = (ROWS_SMEM_MAX - extra) / slot;
    if (p.ring > DWC_MAX_RING) p.ring = DWC_MAX_RING;
    if (p.ring < 4) return cudaErrorInvalidConfiguration;
    CUtensorMap mS0{}, mS1{}, mD;
    if (!rec && (!rows_map_act(&mS0, S, ni, g.H, g.W, c.Mp, g.C, 1, 2) ||
                 !rows_map_act(&mS1, S, ni, g.H, g.W, c.Mp, g.C, 1)))
        return cudaErrorInvalidValue;
    if (!rows_map_act(&mD, dW_hat, ni, g.Ho, g.Wo, c.Mp, C_out, 1)) return cudaErrorInvalidValue;
    const int smem = p.ring * slot + extra;
    const int grid = p.n_tiles < sms ? p.n_tiles : sms;
    if (BN == 64) {
        cudaError_t e = allow_smem<k_conv_dw_cols<64>>(smem);
        if (e != cudaSuccess) return e;
        k_conv_dw_cols<64><<<grid, DwCols<64>::THREADS, smem, st>>>(mS0, mS1, mD, p);
    } else {
        cudaError_t e = allow_smem<k_conv_dw_cols<128>>(smem);
        if (e != cudaSuccess) return e;
        k_conv_dw_cols<128><<<grid, DwCols<128>::THREADS, smem, st>>>(mS0, mS1, mD, p);
    }
    return cudaGetLastError();
}

}  // namespace dstd
