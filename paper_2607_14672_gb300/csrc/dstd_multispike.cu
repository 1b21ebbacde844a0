// Multi-spike regime (App. D, "Extension to multi-spike regime"): a neuron
// may fire up to F times; at each spike v is reset to 0 and I is kept
// (Eq. Vmem_multiSpikes). Every input spike is discretised on its own and
// the grid weights of an input's spikes are summed (s_jm = sum_f s_jm^f), so
// the contraction w^ = W s is unchanged; the scan continues after each spike
// from the state (0, I(t_k)), and the spikes are found one after another.
//
//   k_binning_ms_rows  forward operand [B*Mp, ld]: row (b, m), column j
//   k_binning_ms_cols  dW operand      [N, ld]:    row j, column (b, m)
//   k_scan_ms          one thread per neuron: the walk over the M intervals
//                      with the decayed (v, I) state; on a spike, the reset
//                      and a new test of the rest of the same interval
//   k_dwhat_ms         dC/dw^ through the chain of spikes (implicit function
//                      theorem per spike, adjoints from the last spike back)
//   k_gt_ms            the input-time gradient of every input spike from dS
#include "dstd_internal.cuh"

namespace dstd {

namespace {

inline unsigned ms_blocks(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int OP>
__device__ __forceinline__ void ms_store(void *hi, void *lo, long long o, float v) {
    if (OP == 3) {
        const __half h = __float2half_rn(v);
        static_cast<__half *>(hi)[o] = h;
        static_cast<__half *>(lo)[o] = __float2half_rn(v - __half2float(h));
    } else {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        static_cast<__nv_bfloat16 *>(hi)[o] = h;
        if (OP == 1) static_cast<__nv_bfloat16 *>(lo)[o] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
}

// two neighbouring elements, o even (rows of operands start on 16-byte boundaries)
template <int OP>
__device__ __forceinline__ void ms_store2(void *hi, void *lo, long long o, float v0, float v1) {
    if (OP == 3) {
        const __half2 h = __floats2half2_rn(v0, v1);
        *reinterpret_cast<__half2 *>(static_cast<__half *>(hi) + o) = h;
        *reinterpret_cast<__half2 *>(static_cast<__half *>(lo) + o) =
            __floats2half2_rn(v0 - __low2float(h), v1 - __high2float(h));
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
        *reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(hi) + o) = h;
        if (OP == 1)
            *reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(lo) + o) =
                __floats2bfloat162_rn(v0 - __low2float(h), v1 - __high2float(h));
    }
}

// the grid weights of one spike; no bin when it never comes
constexpr int MS_NO_BIN = -100;
struct MsSpike {
    int k;
    float wR, wL;
};
__device__ __forceinline__ MsSpike ms_spike(const LifConst &c, float x) {
    MsSpike s{MS_NO_BIN, 0.f, 0.f};
    if (isfinite(x)) {
        const BinW w = bin_weights(c, x, false);
        s = MsSpike{w.k, w.wR, w.wL};
    }
    return s;
}
// adds the spike's weight at bin m < M
__device__ __forceinline__ void ms_add(const MsSpike &s, int m, float &v) {
    if (m == s.k) v += s.wR;
    if (m == s.k + 1) v += s.wL;
}

}  // namespace

// A thread per sample b and two neighbouring inputs: 4-byte stores, and the
// spikes' weights in registers (indexed by a count they lay in local memory
// and were read back for every bin). Bound by the compares of every bin with
// every spike (800 inputs, B = 256, M = 32, 4 spikes: 43 -> 26 us).
template <int OP>
__global__ void __launch_bounds__(128) k_binning_ms_rows(const float *__restrict__ t, int B, int N, int F, LifConst c,
                                                         void *hi, void *lo, int ld) {
    const int b = blockIdx.y;
    const int j = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (j >= ld) return;  // ld is even
    MsSpike s[2][kMsMaxSpikes];
#pragma unroll
    for (int f = 0; f < kMsMaxSpikes; ++f) {
        if (f >= F) break;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            s[h][f] = ms_spike(c, j + h < N ? t[((long long)b * N + j + h) * F + f] : INFINITY);
    }
    for (int m = 0; m < c.Mp; ++m) {
        float v0 = 0.f, v1 = 0.f;
        if (m < c.M) {
#pragma unroll
            for (int f = 0; f < kMsMaxSpikes; ++f) {
                if (f >= F) break;
                ms_add(s[0][f], m, v0);
                ms_add(s[1][f], m, v1);
            }
        }
        ms_store2<OP>(hi, lo, ((long long)b * c.Mp + m) * ld + j, v0, v1);
    }
}

// Half a warp per (input j, sample b): lane f < F of the half discretises spike
// f, the half shares the results, and lane l writes bins 2 l, 2 l + 1, 2 l + 32,
// ... of the row segment (contiguous: column b*Mp + m), 4 bytes a store. Bound by
// its stores' instructions (800 inputs, B = 256, M = 32, 4 spikes: 65 -> 44 us, a warp per
// (input, sample) with 2-byte stores before).
constexpr int MS_COLS_ITER = 4;  // up to 128 bins
template <int OP>
__global__ void __launch_bounds__(256) k_binning_ms_cols(const float *__restrict__ t, int B, int N, int F, LifConst c,
                                                         void *hi, void *lo, int ld) {
    const int lane = threadIdx.x & 31, l = lane & 15, h = lane & 16;
    const int j = blockIdx.x;
    const int b = blockIdx.y * 16 + (threadIdx.x >> 4);
    const MsSpike own = ms_spike(c, b < B && l < F ? t[((long long)b * N + j) * F + l] : INFINITY);
    float v0[MS_COLS_ITER], v1[MS_COLS_ITER];  // bins 2 l + 32 i and the one after
#pragma unroll
    for (int i = 0; i < MS_COLS_ITER; ++i) v0[i] = v1[i] = 0.f;
    for (int f = 0; f < F; ++f) {  // in the spikes' order, as the rows add them
        const MsSpike s{__shfl_sync(0xffffffffu, own.k, h + f), __shfl_sync(0xffffffffu, own.wR, h + f),
                        __shfl_sync(0xffffffffu, own.wL, h + f)};
#pragma unroll
        for (int i = 0; i < MS_COLS_ITER; ++i) {
            const int m = 2 * l + 32 * i;
            if (m < c.M) ms_add(s, m, v0[i]);
            if (m + 1 < c.M) ms_add(s, m + 1, v1[i]);
        }
    }
    if (b >= B) return;
    const long long o = (long long)j * ld + (long long)b * c.Mp;
#pragma unroll
    for (int i = 0; i < MS_COLS_ITER; ++i) {
        const int m = 2 * l + 32 * i;
        if (m < c.Mp) ms_store2<OP>(hi, lo, o + m, v0[i], v1[i]);
    }
}

cudaError_t launch_binning_ms(const float *t, int B, int N, int F, const LifConst &c, OpKind op, bool transposed,
                              void *hi, void *lo, int ld, cudaStream_t st) {
    if (F < 1 || F > kMsMaxSpikes || c.Mp > 32 * MS_COLS_ITER || ld % 2) return cudaErrorInvalidValue;
#define DSTD_MS_BIN(OPV)                                                                                        \
    if (transposed)                                                                                             \
        k_binning_ms_cols<OPV><<<dim3((unsigned)N, (unsigned)((B + 15) / 16)), 256, 0, st>>>(t, B, N, F, c, hi, \
                                                                                           lo, ld);             \
    else                                                                                                        \
        k_binning_ms_rows<OPV><<<dim3((unsigned)((ld + 255) / 256), (unsigned)B), 128, 0, st>>>(t, B, N, F, c, \
                                                                                                hi, lo, ld);
    switch (op) {
        case OpKind::F32: return cudaErrorInvalidValue;
        case OpKind::BF16X3: DSTD_MS_BIN(1) break;
        case OpKind::BF16: DSTD_MS_BIN(2) break;
        default: DSTD_MS_BIN(3) break;
    }
#undef DSTD_MS_BIN
    return cudaGetLastError();
}

// One thread per neuron (b, i): w^ of bin m at what[b*sb + i*si + m]. On
// interval m the state (v, I0) at its start is tested exactly (the same
// test and root as the first-spike scan, with the interval's remaining
// length); on a spike at s the state becomes (0, I0 e^{-aI s}) and the rest
// of the interval, of length L - s, is tested again. Outputs per spike k
// (index (b*N + i)*F + k): t, the bin q, I at the spike and dv^/dt there;
// t = +inf, q = M after the last spike.
//
// The neurons of a warp come to their exact tests on different intervals, and a
// test is some hundred instructions: each lane walks on to its next interval
// that needs one, and the warp then runs them together, so it pays for the
// largest number of such intervals of a lane instead of for every interval that
// any lane tests (800 outputs, B = 256, M = 32, up to 4 spikes: 107 -> 44 us).
__global__ void __launch_bounds__(256) k_scan_ms(const float *__restrict__ what, long long sb, long long si, int B,
                                                 int N, LifConst c, int F, float *t_out, int *q_out, float *I_out,
                                                 float *vd_out, int vec4) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = idx < (long long)B * N;
    const int b = (int)(idx / N), i = (int)(idx % N);
    const float *w = what + b * sb + i * si;  // read by live lanes only
    float v = 0.f, I = 0.f;
    int nk = 0;
    const long long o = idx * F;
    float4 w4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int m = live ? 0 : c.M;; ++m) {
        float v0 = 0.f, I0 = 0.f;
        for (; m < c.M && nk < F; ++m) {
            if (vec4) {
                if ((m & 3) == 0) w4 = __ldg(reinterpret_cast<const float4 *>(w + m));
            }
            const float wm = vec4 ? ((m & 3) == 0 ? w4.x : (m & 3) == 1 ? w4.y : (m & 3) == 2 ? w4.z : w4.w) : w[m];
            v0 = v;
            I0 = I + wm;
            // a whole interval with no spike in it yet: the cheap tests of the
            // first-spike scan decide whether the exact test is needed
            const float ve = fmaf(c.KD, I0, c.rv * v0);
            const bool endp = ve >= c.vth;
            const bool peak = (fmaf(-c.av, v0, I0) > 0.0f) & (fmaf(-c.av, ve, c.rI * I0) < 0.0f) &
                              (fmaf(fmaxf(I0, 0.0f), c.Kmax, fmaxf(v0, 0.0f)) >= c.vth);
            if (endp | peak) break;
            v = ve;
            I = c.rI * I0;
        }
        const bool test = m < c.M && nk < F;
        if (!__any_sync(0xffffffffu, test)) break;
        if (!test) continue;
        float L = c.dt, start = c.T0 + (float)m * c.dt;
        // at most F spikes in all, so the inner loop ends
        while (nk < F) {
            const float rI = expf(-c.aI * L);
            const float ve = fmaf(expf(-c.av * L) * phi_f(c, L), I0, expf(-c.av * L) * v0);
            const float hi = interval_test(c.av, c.aI, c.lam, c.lam_zero, rI, L, c.vth, v0, I0, ve);
            if (hi < 0.0f) break;
            const float s = hi > 0.0f ? interval_root(c, v0, I0, hi) : 0.0f;
            const float Ik = I0 * expf(-c.aI * s);
            t_out[o + nk] = start + s;
            q_out[o + nk] = m;
            I_out[o + nk] = Ik;
            vd_out[o + nk] = fmaxf(fmaf(-c.av, c.vth, Ik), c.vdot_floor);
            ++nk;
            v0 = 0.f;
            I0 = Ik;
            start += s;
            L -= s;
            if (!(L > 1e-7f * c.dt)) break;  // the spike closed the interval
        }
        // the state at T_{m+1}
        const float e = expf(-c.av * L);
        v = fmaf(e * phi_f(c, L), I0, e * v0);
        I = I0 * expf(-c.aI * L);
    }
    if (!live) return;
    for (int k = nk; k < F; ++k) {
        t_out[o + k] = INFINITY;
        q_out[o + k] = c.M;
        I_out[o + k] = 0.f;
        vd_out[o + k] = 0.f;
    }
}

cudaError_t launch_scan_ms(const float *what, long long sb, long long si, int B, int N, const LifConst &c, int F,
                           float *t_out, int *q, float *I, float *vd, cudaStream_t st) {
    if (F < 1 || F > kMsMaxSpikes) return cudaErrorInvalidValue;
    // 16-byte loads when every row of bins starts on a 16-byte boundary
    const int vec4 = (sb % 4 == 0) && (si % 4 == 0) && (reinterpret_cast<uintptr_t>(what) % 16 == 0) && (c.Mp % 4 == 0);
    k_scan_ms<<<ms_blocks((long long)B * N, 256), 256, 0, st>>>(what, sb, si, B, N, c, F, t_out, q, I, vd, vec4);
    return cudaGetLastError();
}

// dC/dw^_im of one neuron from dC/dt_k of its spikes. With v'_k the saved
// dv^/dt at spike k:
//   spike 0:  dt_0/dw^_m = -K(t_0 - T_m)/v'_0, m <= q_0;
//   spike k:  dt_k/dw^_m = -e^{-aI (t_{k-1} - T_m)} K(t_k - t_{k-1}) / v'_k  for m <= q_{k-1},
//                        = -K(t_k - T_m) / v'_k                             for q_{k-1} < m <= q_k,
//             dt_k/dt_{k-1} = -I_{k-1} [(av - aI) K(s) - e^{-aI s}] / v'_k, s = t_k - t_{k-1}
// (the current kept through the reset decays at aI; dK/ds = -av K + e^{-aI s}).
// The adjoints a_k = dC/dt_k + a_{k+1} dt_{k+1}/dt_k run from the last
// spike back; dC/dw^_m = sum_k a_k dt_k/dw^_m.
//
// A bin m with q_{k-1} < m <= q_k takes one K (spike k) and one exponential per
// later spike. The lanes of a warp take the K together, then the exponentials:
// a loop over the spikes with either in it ran both for every spike of the lanes
// (800 outputs, B = 256, M = 32, up to 4 spikes, with 4-byte stores: 87 -> 62 us).
// The running sum of the later spikes' terms (one exponential per bin in all)
// takes 50 us, but differs by 1e-5 where a spike only just reaches the threshold
// and the terms cancel, so each term is taken as it stands above.
//
// A block takes 32 neurons of one sample: thread i < 32 runs neuron i's
// adjoints into shared memory, the block fills a [Mp][32] tile of dC/dw^
// (zero after a neuron's last spike), and writes it to both layouts with
// contiguous stores: the (i, (b, m)) rows (a warp per neuron, lanes over m)
// and, when b_hi is given, the ((b, m), i) rows (lanes over the 32 neurons).
constexpr int MS_DW_NEURONS = 32;
template <int OP>
__global__ void __launch_bounds__(256) k_dwhat_ms(const float *__restrict__ t_out, const int *__restrict__ qv,
                                                  const float *__restrict__ Iv, const float *__restrict__ vdv,
                                                  const float *__restrict__ g_up, int B, int N, int F, LifConst c,
                                                  void *a_hi, void *a_lo, int lda, void *b_hi, void *b_lo, int ldb) {
    extern __shared__ __align__(16) float dsm[];
    float *tile = dsm;                                        // [Mp][33]
    float *stk = tile + c.Mp * (MS_DW_NEURONS + 1);           // [32][F] spike times
    float *scf = stk + MS_DW_NEURONS * F;                     // [32][F] coefficients -a_k / v'_k
    float *sKk = scf + MS_DW_NEURONS * F;                     // [32][F] K(t_k - t_{k-1})
    int *sq = reinterpret_cast<int *>(sKk + MS_DW_NEURONS * F);  // [32][F] bins
    int *sn = sq + MS_DW_NEURONS * F;                         // [32] spike counts
    const int b = blockIdx.y;
    const int i0 = blockIdx.x * MS_DW_NEURONS;
    const int tid = threadIdx.x;
    if (tid < MS_DW_NEURONS) {
        const int i = i0 + tid;
        int n = 0;
        if (i < N) {
            const long long o = ((long long)b * N + i) * F;
            float tk[kMsMaxSpikes], Ik[kMsMaxSpikes], coef[kMsMaxSpikes];
            for (int k = 0; k < F; ++k) {
                if (qv[o + k] >= c.M) break;
                tk[k] = t_out[o + k];
                Ik[k] = Iv[o + k];
                coef[k] = g_up ? g_up[o + k] : 0.f;
                sq[tid * F + k] = qv[o + k];
                n = k + 1;
            }
            // adjoints, last spike first; coef_k = -a_k / v'_k
            for (int k = n - 1; k >= 0; --k) {
                coef[k] = -coef[k] / vdv[o + k];
                float K = 0.f;
                if (k > 0) {
                    const float s = tk[k] - tk[k - 1];
                    K = kernel_K(c, s);
                    const float dv_dprev = Ik[k - 1] * fmaf(c.av - c.aI, K, -expf(-c.aI * s));
                    coef[k - 1] += coef[k] * dv_dprev;  // a_{k-1} += a_k (-dv_dprev / v'_k)
                }
                stk[tid * F + k] = tk[k];
                scf[tid * F + k] = coef[k];
                sKk[tid * F + k] = K;
            }
        }
        sn[tid] = n;
    }
    __syncthreads();
    // the tile: thread (neuron il, bins m = row, row + 8, ...)
    for (int e = tid; e < c.Mp * MS_DW_NEURONS; e += blockDim.x) {
        const int il = e % MS_DW_NEURONS, m = e / MS_DW_NEURONS;
        const int n = sn[il];
        float val = 0.f;
        if (n > 0 && m <= sq[il * F + n - 1]) {
            int k = 0;
            while (m > sq[il * F + k]) ++k;  // the spike whose bins hold m (m <= the last spike's)
            const float Tm = c.T0 + (float)m * c.dt;
            val = scf[il * F + k] * kernel_K(c, stk[il * F + k] - Tm);
            for (++k; k < n; ++k)
                val = fmaf(scf[il * F + k], expf(-c.aI * (stk[il * F + k - 1] - Tm)) * sKk[il * F + k], val);
        }
        tile[m * (MS_DW_NEURONS + 1) + il] = val;
    }
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    // two neurons per warp, two bins per lane: 4-byte stores
    for (int p = warp; p < MS_DW_NEURONS / 2; p += blockDim.x / 32) {
        const int il = 2 * p + (lane >> 4), i = i0 + il;
        if (i >= N) continue;
        const long long oa = (long long)i * lda + (long long)b * c.Mp;
        for (int m = 2 * (lane & 15); m < c.Mp; m += 32)
            ms_store2<OP>(a_hi, a_lo, oa + m, tile[m * (MS_DW_NEURONS + 1) + il],
                          tile[(m + 1) * (MS_DW_NEURONS + 1) + il]);
    }
    if (b_hi) {
        const int i = i0 + lane;
        if (i < N)
            for (int m = warp; m < c.Mp; m += blockDim.x / 32)
                ms_store<OP>(b_hi, b_lo, ((long long)b * c.Mp + m) * ldb + i, tile[m * (MS_DW_NEURONS + 1) + lane]);
    }
}

cudaError_t launch_dwhat_ms(const float *t_out, const int *q, const float *I, const float *vd, const float *g_up,
                            int B, int N, int F, const LifConst &c, OpKind op, void *a_hi, void *a_lo, int lda,
                            void *b_hi, void *b_lo, int ldb, cudaStream_t st) {
    if (F < 1 || F > kMsMaxSpikes || op == OpKind::F32) return cudaErrorInvalidValue;
    const size_t smem = sizeof(float) * ((size_t)c.Mp * (MS_DW_NEURONS + 1) + 4 * MS_DW_NEURONS * F + MS_DW_NEURONS);
    const dim3 g((unsigned)((N + MS_DW_NEURONS - 1) / MS_DW_NEURONS), (unsigned)B);
    if (op == OpKind::BF16X3)
        k_dwhat_ms<1><<<g, 256, smem, st>>>(t_out, q, I, vd, g_up, B, N, F, c, a_hi, a_lo, lda, b_hi, b_lo, ldb);
    else
        k_dwhat_ms<2><<<g, 256, smem, st>>>(t_out, q, I, vd, g_up, B, N, F, c, a_hi, a_lo, lda, b_hi, b_lo, ldb);
    return cudaGetLastError();
}

// g_t of input spike f of input j in sample b: sum over its two bins of
// dS[j, (b, m)] ds_jm/dt (Tab. DSTD_kernels' derivative); 0 when silent.
__global__ void k_gt_ms(const float *__restrict__ D, long long ldd, const float *__restrict__ t_in, int B, int N,
                        int F, LifConst c, float *g_t_in) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)B * N * F) return;
    const long long bj = idx / F;
    const int b = (int)(bj / N), j = (int)(bj % N);
    const float x = t_in[idx];
    float g = 0.f;
    if (isfinite(x)) {
        const BinW w = bin_weights(c, x, true);
        const float *row = D + (long long)j * ldd + (long long)b * c.Mp;
        if (w.k >= 0 && w.k < c.M) g += row[w.k] * w.dR;
        if (w.k + 1 >= 0 && w.k + 1 < c.M) g += row[w.k + 1] * w.dL;
    }
    g_t_in[idx] = g;
}

cudaError_t launch_gt_ms(const float *D, long long ldd, const float *t_in, int B, int N, int F, const LifConst &c,
                         float *g_t_in, cudaStream_t st) {
    const long long n = (long long)B * N * F;
    k_gt_ms<<<ms_blocks(n, 256), 256, 0, st>>>(D, ldd, t_in, B, N, F, c, g_t_in);
    return cudaGetLastError();
}

}  // namespace dstd
